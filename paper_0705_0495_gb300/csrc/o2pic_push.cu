// o2pic_push.cu -- the fused per-step particle kernel of libo2pic.
//
// One launch advances every live superparticle of every discharge by one time
// step (paper Sec. II (i) and Sec. III):
//   four consecutive slots per thread: gather E at x^n (linear
//   interpolation from a shared-memory copy of the node field) -> leapfrog
//   v^{n+1/2}, x^{n+1} -> absorption at x < 0 or x >= L -> null-collision
//   test against nu_max (one Philox4x32-10 block serves the four slots) ->
//   linear charge assignment of x^{n+1} into per-block shared-memory sums
//   (warp aggregated, exact integers), flushed to the global accumulators with
//   one atomic per touched node -> candidates listed for k_collide.
// k_collide, one candidate per thread: a gas molecule from the Maxwellian at T,
// the channel walk over sum_j n_j sigma_j(E) u and the kinematics of the chosen
// reaction; a particle that dies leaves the global charge again; births are
// staged per 128-slot sub-tile and appended in parent order by k_births.
// k_dsmc: the sequential gas scheme's channels in its place.
//
// Particles are SoA with the position as (int32 cell, offset in [0,1)) and
// velocities in cells per step.  Slots are processed in tiles of 1024
// (256 threads x 4 consecutive slots, 16-byte vector loads) by a persistent
// grid: a block takes TILES_PER_TICKET tiles at a time from an atomic ticket,
// or one contiguous share when there are few tiles per block.  No block ever
// waits for another.
//
// What bounds it: instruction issue and latency in FP32 (5e7 superparticles,
// 4096 cells: 251 us against 177 us for its bytes), the FP64 units in FP64.
// A warp whose 128 slots are live and stay on the grid (nearly all) takes a
// path without masks and selects, with its floors from packed adds (FP32) or
// off the FP64 units where a slot stays in its cell: FP32 push 293 -> 251 us,
// FP64 1968 -> 1000 us, results bit for bit the same.  The FP64 sums in 32-bit
// words per cell took it to 733 us (4e4 superparticles: 17 -> 10.6 us), the
// field's steps from a table, floors and energy bins off the FP64 units and one
// block per SM to 578 us (835 with diagnostics, 1350 before; 9.2 us): about
// five FP64 instructions a particle, 340 us for its bytes.
#include <algorithm>
#include <cstdio>

#include "o2pic_launch.h"

namespace o2 {

// tiles ahead of the current one whose particle data a push block asks the
// L2 cache to fetch (a bulk prefetch issued by one thread; 0 = none)
#ifndef O2_PUSH_L2_AHEAD
#define O2_PUSH_L2_AHEAD 2
#endif
// Up to STATIC_TILES tiles per block of the grid, each block takes one
// contiguous share.  Tickets of 8 tiles left most blocks idle on a small
// discharge (4e4 superparticles: 6 blocks of 456 busy; FP32 push 21 -> 8 us,
// FP64 104 -> 30 us) and ran a middle one in two uneven waves (4e6: 34 ->
// 28 us).  Above the limit shares lose: electron tiles cost more than ion
// tiles, and no block can take over from a slower one (5e7: 400 time steps
// 163.8 ms with tickets, 170.3 ms with shares; FP64 54.4 against 83.3 ms per
// 40).  Between 16 and 64 tiles per block both took the same time.
#ifndef O2_STATIC_TILES
#define O2_STATIC_TILES 16
#endif
constexpr int STATIC_TILES = O2_STATIC_TILES;


template <typename Real> struct AccT;
template <> struct AccT<float> { using T = unsigned long long; };
template <> struct AccT<double> { using T = double; };

template <typename Real> struct GasTab;
template <> struct GasTab<float> {
    static constexpr int VEC = 4;
    static __device__ __forceinline__ const float *ptr(const WsPtrs &W) { return W.gtabf; }
    static __device__ __forceinline__ const float *bound(const WsPtrs &W) { return W.gpmf; }
    static __device__ __forceinline__ void load(const float *p, float v[4])
    {
        const float4 t = __ldg(reinterpret_cast<const float4 *>(p));
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    }
};
template <> struct GasTab<double> {
    static constexpr int VEC = 2;
    static __device__ __forceinline__ const double *ptr(const WsPtrs &W) { return W.gtab; }
    static __device__ __forceinline__ const double *bound(const WsPtrs &W) { return W.gpm; }
    static __device__ __forceinline__ void load(const double *p, double v[2])
    {
        const double2 t = __ldg(reinterpret_cast<const double2 *>(p));
        v[0] = t.x; v[1] = t.y;
    }
};

template <typename Real> struct Lut;
template <> struct Lut<float> {
    static __device__ __forceinline__ const float *E(const WsPtrs &W) { return W.lutEf; }
    static __device__ __forceinline__ const float *S(const WsPtrs &W) { return W.lutSf; }
};
template <> struct Lut<double> {
    static __device__ __forceinline__ const double *E(const WsPtrs &W) { return W.lutE; }
    static __device__ __forceinline__ const double *S(const WsPtrs &W) { return W.lutS; }
};

__device__ __forceinline__ void ld4(const int *p, int v[4])
{
    int4 t = *reinterpret_cast<const int4 *>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void st4(int *p, const int v[4])
{
    *reinterpret_cast<int4 *>(p) = make_int4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void ld4(const float *p, float v[4])
{
    float4 t = *reinterpret_cast<const float4 *>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void st4(float *p, const float v[4])
{
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void ld4(const double *p, double v[4])
{
    double2 a = reinterpret_cast<const double2 *>(p)[0];
    double2 b = reinterpret_cast<const double2 *>(p)[1];
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
__device__ __forceinline__ void st4(double *p, const double v[4])
{
    reinterpret_cast<double2 *>(p)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2 *>(p)[1] = make_double2(v[2], v[3]);
}

// a < b for values that are not negative: FP64 compares as integers (their
// bit patterns have the same order), off the few FP64 units
__device__ __forceinline__ bool less_pos(float a, float b) { return a < b; }
__device__ __forceinline__ bool less_pos(double a, double b)
{
    return __double_as_longlong(a) < __double_as_longlong(b);
}

// Interpolation of the gas-channel cross sections of one projectile at the
// centre-of-mass energy E [eV]: piecewise linear in E on the shared geometric
// grid, end values held outside it, zero below each channel's threshold.
template <typename Real>
struct XsPoint {
    int k;       // segment
    Real f;      // fraction inside the segment
    int region;  // 0 below the grid, 1 inside, 2 above
};

template <typename Real>
__device__ __forceinline__ XsPoint<Real> xs_locate(const SpeciesC &S, const Real *lutE, Real E)
{
    XsPoint<Real> p;
    const Real *nodes = lutE + S.grid_off;
    const int n = S.grid_n;
    if (!less_pos(pick<Real>(S.grid_lo, S.grid_lo_f), E)) {
        p.region = 0; p.k = 0; p.f = Real(0);
        return p;
    }
    if (!less_pos(E, pick<Real>(S.grid_hi, S.grid_hi_f))) {
        p.region = 2; p.k = n - 2; p.f = Real(1);
        return p;
    }
    // the logarithm only guesses the segment, so a fast FP32 one will do in
    // both precisions; the node comparison decides.  Both ends of the guess
    // are loaded at once.
    const float t = (__logf((float)E) - S.grid_lnlo_f) * S.grid_inv_f;
    int k = (int)t;
    k = k < 0 ? 0 : (k > n - 2 ? n - 2 : k);
    Real a = nodes[k], b = nodes[k + 1];
    while (k > 0 && less_pos(E, a)) {
        --k;
        b = a;
        a = nodes[k];
    }
    while (k < n - 2 && !less_pos(E, b)) {
        ++k;
        a = b;
        b = nodes[k + 1];
    }
    p.region = 1;
    p.k = k;
    p.f = (E - a) / (b - a);
    return p;
}

// centre-of-mass binary collision in normalised units: relative speed
// sqrt(u^2 - dloss) along n (Eq. 5 with dloss = 2 dE/mu (dt/dx)^2)
template <typename Real>
__device__ __forceinline__ void cm_scatter(Real mfrac, Real Mfrac, const Real v[3],
                                           const Real V[3], Real dloss, const Real n[3],
                                           Real vo[3], Real Vo[3])
{
    Real g0 = v[0] - V[0], g1 = v[1] - V[1], g2 = v[2] - V[2];
    Real u2 = g0 * g0 + g1 * g1 + g2 * g2 - dloss;
    Real up = u2 > Real(0) ? sqrt(u2) : Real(0);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        Real vcm = mfrac * v[q] + Mfrac * V[q];
        vo[q] = vcm + Mfrac * up * n[q];
        Vo[q] = vcm - mfrac * up * n[q];
    }
}

template <typename Real>
__device__ __forceinline__ void ee_elastic(Real a[3], Real b[3], const Real n[3])
{
    Real g0 = a[0] - b[0], g1 = a[1] - b[1], g2 = a[2] - b[2];
    Real u = sqrt(g0 * g0 + g1 * g1 + g2 * g2);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        Real c = Real(0.5) * (a[q] + b[q]);
        a[q] = c + Real(0.5) * u * n[q];
        b[q] = c - Real(0.5) * u * n[q];
    }
}

// charge of one particle added to (sign > 0) or removed from the global
// accumulator of its species (births, pair-pass kills)
__device__ __forceinline__ void deposit_global(unsigned long long *acc, int c, float off, int sign)
{
    unsigned w1 = __float2uint_rn(off * (float)(1 << FIX_BITS));
    unsigned w0 = (1u << FIX_BITS) - w1;
    unsigned long long a = w0, b = w1;
    if (sign < 0) { a = 0ull - a; b = 0ull - b; }
    atomicAdd(&acc[c], a);
    atomicAdd(&acc[c + 1], b);
}
__device__ __forceinline__ void deposit_global(double *acc, int c, double off, int sign)
{
    atomicAdd(&acc[c], sign * (1.0 - off));
    atomicAdd(&acc[c + 1], sign * off);
}

template <typename Real> __device__ __forceinline__ typename AccT<Real>::T *acc_global(const WsPtrs &W);
template <> __device__ __forceinline__ unsigned long long *acc_global<float>(const WsPtrs &W) { return W.acc_fix; }
template <> __device__ __forceinline__ double *acc_global<double>(const WsPtrs &W) { return W.acc_dbl; }

// Births of one candidate go straight to its sub-tile's records, in any
// order; the tag restores parent order when they are appended.  Their charge
// is deposited here, so that the next field does not wait for the append (which
// takes it back from a birth that finds no room).
template <typename Real>
struct BirthSink {
    BirthRec<Real> *rec;  // the sub-tile's birth_cap records
    int *n;               // the sub-tile's record count
    int *blk;             // births per product species of the sub-tile's birth-append block
    int *all;             // births of the step
    typename AccT<Real>::T *acc;  // the discharge's charge accumulators, first species
    int acc_ld;           // from one species' accumulators to the next
    Ctl *ctl;
    int cap;
};

template <typename Real>
__device__ __forceinline__ BirthSink<Real> birth_sink(const WsPtrs &W, const Disc &Dd, int par, int sub)
{
    return BirthSink<Real>{reinterpret_cast<BirthRec<Real> *>(W.births) + (size_t)sub * W.birth_cap, W.tile_cnt + sub,
                           birth_words(W, par) + (size_t)(sub / BIRTHS_TILES) * NSP, W.ctl->births + par,
                           acc_global<Real>(W) + Dd.gbase, W.total_nodes, W.ctl, W.birth_cap};
}

// ask the L2 cache to fetch [p, p + bytes) (16-byte aligned, a multiple of
// 16 bytes); no completion to wait for
__device__ __forceinline__ void l2_prefetch(const void *p, unsigned bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

template <typename Real>
__device__ __forceinline__ void stage_birth(const BirthSink<Real> &B, int tag, int sp, int c, Real off,
                                            const Real v[3])
{
    const int pos = atomicAdd(B.n, 1);
    if (pos >= B.cap) {
        set_status(B.ctl, ST_BIRTHBUF);
        return;
    }
    atomicAdd(B.blk + sp, 1);
    atomicAdd(B.all, 1);
    deposit_global(B.acc + (size_t)sp * B.acc_ld, c, off, 1);
    BirthRec<Real> &r = B.rec[pos];
    r.c = c;
    r.tag = (tag << 2) | sp;
    r.off = off;
    r.vx = v[0];
    r.vy = v[1];
    r.vz = v[2];
}

// Energy bin of an electron's lab energy K [eV] for the collision-frequency
// bound: with K = m 2^e, m in [1, 2), bin 4 (e + 6) + floor(4 (m - 1)) (the
// exponent and the top two mantissa bits), clamped to [0, nb - 1].  K is a
// sum of squares times a positive factor: for K >= 0 the exponent and the
// top two mantissa bits are the bits above the lower 21 (FP32), and +0 falls
// below bin 0.  (FP64: K <= 0 or NaN gives bin 0.)
__device__ __forceinline__ int energy_bin(float K, int nb)
{
    const int b = (int)(__float_as_uint(K) >> 21) - 4 * (127 + NUBIN_LOG2_E0);
    return min(max(b, 0), nb - 1);
}
__device__ __forceinline__ int energy_bin(double K, int nb)
{
    if (!(K > 0.0)) return 0;
    const unsigned long long u = (unsigned long long)__double_as_longlong(K);
    const int b = 4 * ((int)((u >> 52) & 0x7FFull) - 1023 - NUBIN_LOG2_E0) + (int)((u >> 50) & 3ull);
    return b < 0 ? 0 : (b > nb - 1 ? nb - 1 : b);
}

// One gas-target candidate (null-collision method).  Returns false if the
// particle died.  v is updated in place; products are staged.  The cell and
// offset are read from cP, offP (into c, off) only when the collision has
// products or kills the particle.
struct Outcome {
    bool alive;     // the particle survives
    bool viol;      // sum_j n_j sigma_j u exceeded the bound
    int reaction;   // reaction number, -1 for a null event
};

// Products of one gas event: species, product index (the tag's product
// bit) and velocity
template <typename Real>
struct GasProducts {
    int n;
    int sp[2], prod[2];
    Real v[2][3];
};

// Kinematics of gas channel ch for a particle of species s with velocity v
// that meets a gas molecule of velocity V at centre-of-mass energy E; nd is
// an isotropic direction, nd2 a second one used by (18).  Returns whether
// the particle lives on (with velocity vo) and its products.  One centre-of-
// mass scattering serves every channel that scatters: elastic (4), (5),
// isotropic (6) with no loss, (7)-(12) and (18) with the loss of Eq. 5; its
// result is unused by (15)-(17) and resonant (6).
template <typename Real>
__device__ __forceinline__ bool gas_event(const WsPtrs &W, const Disc &Dd, const SpeciesC &S, const GasChan &ch,
                                          const Real v[3], const Real V[3], Real E, const Real nd[3],
                                          const Real nd2[3], Real vo[3], GasProducts<Real> &pr)
{
    const int r = ch.reaction;
    const Real mf = pick<Real>(S.mfrac, S.mfrac_f), Mf = pick<Real>(S.Mfrac, S.Mfrac_f);
    const bool elastic = r <= 6;
    const bool dies = r >= 15 && r <= 17;
    Real Vo[3];
    cm_scatter<Real>(mf, Mf, v, V, elastic ? Real(0) : pick<Real>(ch.dloss, ch.dloss_f), nd, vo, Vo);
    const bool swap = r == 6 && !Dd.cx_iso;  // resonant exchange: the ion takes the gas velocity
#pragma unroll
    for (int q = 0; q < 3; ++q) vo[q] = swap ? V[q] : vo[q];
    pr.n = 0;
    if (r == 18) {
        // ionisation: the O2 splits into O2+ and a second electron with the
        // post-collision O2 velocity, then the two electrons collide
        // elastically (isotropic in their centre of mass)
        Real e2[3] = {Vo[0], Vo[1], Vo[2]};
        ee_elastic<Real>(vo, e2, nd2);
        pr.n = 2;
        pr.sp[0] = 0;
        pr.prod[0] = 0;
        pr.sp[1] = 2;
        pr.prod[1] = 1;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            pr.v[0][q] = e2[q];
            pr.v[1][q] = Vo[q];
        }
    }
    if (!dies) return true;
    // (15) attachment: O- with the CM velocity plus half the relative
    // energy above threshold shared back to back with O; (16) detachment:
    // electron with a tenth of the O- energy, isotropic; (17) associative
    // detachment: electron with the CM energy about the CM velocity
    Real w;
    if (r == 16) {
        w = sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]) * pick<Real>(Dd.f16, Dd.f16_f);
    } else {
        Real arg;
        if (r == 15) {
            const TableDesc &Tc = W.tables[ch.table];
            const Real Ea = E - pick<Real>(Tc.th, Tc.th_f);
            arg = (Ea > Real(0) ? Ea : Real(0)) * pick<Real>(Dd.f15, Dd.f15_f);
        } else {
            arg = E * pick<Real>(Dd.f17, Dd.f17_f);
        }
        w = sqrt(arg);
    }
    const Real A = r == 16 ? Real(0) : Real(1);
    pr.n = 1;
    pr.sp[0] = r == 15 ? 1 : 0;
    pr.prod[0] = 0;
#pragma unroll
    for (int q = 0; q < 3; ++q) pr.v[0][q] = A * (mf * v[q] + Mf * V[q]) + w * nd[q];
    return false;
}

template <typename Real>
__device__ __forceinline__ Outcome gas_collide(const WsPtrs &W, const Disc &Dd, int s, unsigned idx,
                                            unsigned long long step, Real numax_n, Real &vx, Real &vy,
                                            Real &vz, const int *cP, const Real *offP, int &c, Real &off,
                                            int tag, const BirthSink<Real> &B)
{
    const SpeciesC &S = Dd.sp[s];
    const Real *lutE = Lut<Real>::E(W);
    uint4 a = rng_block(Dd.seed, Dd.discharge, s, 1, 0, 0, step, idx);
    uint4 b = rng_block(Dd.seed, Dd.discharge, s, 1, 0, 1, step, idx);
    Real n0, n1, n2, n3;
    box_muller<Real>(a.x, a.y, n0, n1);
    box_muller<Real>(a.z, a.w, n2, n3);
    const Real vg = pick<Real>(S.vgas_n, S.vgas_n_f);
    Real V[3] = {vg * n0, vg * n1, vg * n2};
    Real v[3] = {vx, vy, vz};
    Real g0 = v[0] - V[0], g1 = v[1] - V[1], g2 = v[2] - V[2];
    Real u2 = g0 * g0 + g1 * g1 + g2 * g2;
    Real u = sqrt(u2);
    Real E = pick<Real>(S.Ek, S.Ek_f) * u2;
    Real target = unif<Real>(b.x) * numax_n;
    XsPoint<Real> pt = xs_locate<Real>(S, lutE, E);
    // node-major table of n_j dx sigma_j(E_k): the rows k and k+1 of every
    // channel come in a few 16-byte loads
    const Real *row = GasTab<Real>::ptr(W) + S.gtab_off;
    const int ld = S.gtab_ld;
    const Real *ra = row + (size_t)pt.k * ld;
    const Real *rb = ra + ld;
    Real cum = Real(0);
    int chosen = -1;
    // channel walk with selects only: the lanes of a warp stay together; the
    // next channels' rows are loaded before the present ones are walked
    constexpr int VEC = GasTab<Real>::VEC;
    Real xa[VEC], xb[VEC];
    GasTab<Real>::load(ra, xa);
    GasTab<Real>::load(rb, xb);
    for (int j0 = 0; j0 < S.nch; j0 += VEC) {
        Real a[VEC], b[VEC];
#pragma unroll
        for (int q = 0; q < VEC; ++q) {
            a[q] = xa[q];
            b[q] = xb[q];
        }
        if (j0 + VEC < ld) {
            GasTab<Real>::load(ra + j0 + VEC, xa);
            GasTab<Real>::load(rb + j0 + VEC, xb);
        }
#pragma unroll
        for (int q = 0; q < VEC; ++q) {
            const int j = j0 + q;
            if (j >= S.nch) break;  // uniform: one species per warp
            // below the grid f = 0 gives a exactly; above it, the last node
            Real v = pt.region == 2 ? b[q] : a[q] + pt.f * (b[q] - a[q]);
            v = less_pos(E, pick<Real>(S.thv[j], S.thv_f[j])) ? Real(0) : v;
            cum += v * u;
            chosen = (chosen < 0 && less_pos(target, cum)) ? j : chosen;
        }
    }
    const bool viol = cum > numax_n;
    if (chosen < 0) return Outcome{true, viol, -1};  // null event
    const GasChan &ch = S.ch[chosen];
    const int r = ch.reaction;
    Real nd[3], nd2[3] = {Real(0), Real(0), Real(1)};
    iso_dir<Real>(unif<Real>(b.y), unif<Real>(b.z), nd);
    if (r == 18) {
        uint4 e = rng_block(Dd.seed, Dd.discharge, s, 1, 0, 2, step, idx);
        iso_dir<Real>(unif<Real>(e.x), unif<Real>(e.y), nd2);
    }
    GasProducts<Real> pr;
    Real vo[3];
    const bool alive = gas_event<Real>(W, Dd, S, ch, v, V, E, nd, nd2, vo, pr);
    // the position is needed only by products and by a dying particle
    if (pr.n > 0 || !alive) {
        c = *cP;
        off = *offP;
    }
    for (int q = 0; q < pr.n; ++q) stage_birth<Real>(B, tag | pr.prod[q], pr.sp[q], c, off, pr.v[q]);
    if (alive) {
        vx = vo[0]; vy = vo[1]; vz = vo[2];
    }
    return Outcome{alive, viol, r};
}

template <typename Acc> __device__ __forceinline__ void acc_add(Acc *a, Acc v);
template <> __device__ __forceinline__ void acc_add(unsigned long long *a, unsigned long long v)
{
    atomicAdd(a, v);
}
template <> __device__ __forceinline__ void acc_add(double *a, double v) { atomicAdd(a, v); }

// Split 64-bit shared sums of the FP32 path: the 8 bytes hold two signed
// 32-bit sums, of the low SPLIT_BITS bits of each added weight (word 0) and
// of the rest (word 1); the value is word1 * 2^SPLIT_BITS + word0.  Adds are
// plain 32-bit atomics whose result is not needed (no carry), and both sums
// stay exact while a block adds at most FLUSH_TILES tiles of weights
// before it flushes (each particle's weight is at most 2^FIX_BITS, so word 1
// grows by at most 2^(FIX_BITS - SPLIT_BITS) per particle and word 0 by less
// than 2^SPLIT_BITS per add).
constexpr int SPLIT_BITS = 12;
constexpr int FLUSH_TILES = 256;
static_assert((long long)FLUSH_TILES * CHUNK * (1LL << (FIX_BITS - SPLIT_BITS)) < (1LL << 31),
              "split sums must stay within int32");
__device__ __forceinline__ void split_add(unsigned long long *node, unsigned v)
{
    unsigned *w = reinterpret_cast<unsigned *>(node);  // w[0] low part, w[1] high part
    atomicAdd(&w[0], v & ((1u << SPLIT_BITS) - 1u));
    atomicAdd(&w[1], v >> SPLIT_BITS);
}
__host__ __device__ __forceinline__ unsigned long long split_value(unsigned long long node)
{
    const long long lo = (int)(unsigned)(node & 0xFFFFFFFFull);
    const long long hi = (int)(unsigned)(node >> 32);
    return (unsigned long long)(hi * (1LL << SPLIT_BITS) + lo);
}

// The FP64 path's shared grid holds exact 64-bit integer sums of the
// weights in units of 2^-FIX_BITS_64 (a particle's two weights add up to
// exactly 2^FIX_BITS_64); they become doubles once per node and flush.  A
// block adds at most FLUSH_TILES tiles of weights before a flush, far
// below the 2^63 / 2^FIX_BITS_64 particles a node could hold.  (Shared-memory
// double atomics took nine tenths of the FP64 push.)
constexpr int FIX_BITS_64 = 40;
static_assert((long long)FLUSH_TILES * CHUNK < (1LL << (63 - FIX_BITS_64)),
              "FP64 shared sums must stay within int64");

// A node's integer sum as the global accumulators' type.
template <typename Real> __device__ __forceinline__ typename AccT<Real>::T sacc_value(unsigned long long node);
template <> __device__ __forceinline__ unsigned long long sacc_value<float>(unsigned long long node) { return node; }
template <> __device__ __forceinline__ double sacc_value<double>(unsigned long long node)
{
    return (double)(long long)node * (1.0 / (double)(1ull << FIX_BITS_64));
}

// A node's integer sum (units of 2^-FIX_BITS or 2^-FIX_BITS_64 of a
// particle) from the block's sums per cell: count_i - W_i + W_(i-1).
// FP32: sCnt[i], and the split words of sAcc[i].  FP64: sCnt[i], and W in
// three words of SPLIT64 bits, two of them the halves of sAcc[i] and the
// third sCnt[stride + i] (FLUSH_TILES tiles of particles stay below 2^32 in
// each).
constexpr int SPLIT64_0 = 14, SPLIT64_1 = 27;  // first bits of the second and third words
static_assert((long long)FLUSH_TILES * CHUNK <= (1LL << 18) && FIX_BITS_64 - SPLIT64_1 == 13, "words must fit 32 bits");
template <typename Real>
__device__ __forceinline__ unsigned long long sacc_cells(const unsigned long long *sAcc, const unsigned *sCnt, int stride,
                                                         int i);
template <>
__device__ __forceinline__ unsigned long long sacc_cells<float>(const unsigned long long *sAcc, const unsigned *sCnt, int,
                                                                int i)
{
    const unsigned long long lw = i > 0 ? split_value(sAcc[i - 1]) : 0ull;
    return ((unsigned long long)sCnt[i] << FIX_BITS) - split_value(sAcc[i]) + lw;
}
template <>
__device__ __forceinline__ unsigned long long sacc_cells<double>(const unsigned long long *sAcc, const unsigned *sCnt,
                                                                 int stride, int i)
{
    auto w = [&](int j) {
        const unsigned long long a = sAcc[j];
        return (a & 0xFFFFFFFFull) + ((a >> 32) << SPLIT64_0) + ((unsigned long long)sCnt[stride + j] << SPLIT64_1);
    };
    return ((unsigned long long)sCnt[i] << FIX_BITS_64) - w(i) + (i > 0 ? w(i - 1) : 0ull);
}

// Charge of the four slots of a thread into the block's shared sums.  The
// FP32 sums are kept per CELL: the particles that land in it (sCnt, one
// 32-bit add) and the sum of their upper CIC weights w1 = rn(offset
// 2^FIX_BITS) (sAcc, split words); node i is then
// count_i 2^FIX_BITS - W1_i + W1_(i-1), the same integer as the sum of the
// particles' two node weights, with three shared atomics per particle
// instead of four.  The lanes whose four slots sit in the first lane's cell
// (sorted, slow particles: most of a warp, even when a few have left) sum
// their weights over the warp and one lane adds them
// (4 * 32 * 2^FIX_BITS < 2^32); every other lane adds its own (its four
// summed first when they share a cell).  No lane matching: it runs on a
// narrow pipe.  DEP_LANES (lanes worth a warp sum) between 1 and 12 gave the
// same time.
#ifndef O2_DEP_LANES
#define O2_DEP_LANES 4
#endif
constexpr int DEP_LANES = O2_DEP_LANES;
__device__ __forceinline__ void deposit4(unsigned long long *sAcc, unsigned *sCnt, int, const int dep[4],
                                         const float off[4])
{
    unsigned w1[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) w1[k] = dep[k] >= 0 ? __float2uint_rn(off[k] * (float)(1 << FIX_BITS)) : 0u;
    const bool same = dep[0] >= 0 && dep[1] == dep[0] && dep[2] == dep[0] && dep[3] == dep[0];
    const unsigned a = w1[0] + w1[1] + w1[2] + w1[3];
    const int c0 = __shfl_sync(0xffffffffu, dep[0], 0);
    const bool in = same && dep[0] == c0;
    const unsigned m = __ballot_sync(0xffffffffu, in);
    if (__popc(m) >= DEP_LANES) {
        const unsigned sa = __reduce_add_sync(0xffffffffu, in ? a : 0u);
        if ((threadIdx.x & 31) == 0) {
            atomicAdd(&sCnt[c0], 4u * (unsigned)__popc(m));
            split_add(&sAcc[c0], sa);
        }
        if (in) return;
    }
    if (same) {
        atomicAdd(&sCnt[dep[0]], 4u);
        split_add(&sAcc[dep[0]], a);
        return;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        // an empty slot adds nothing to cell 0
        const int ck = dep[k] >= 0 ? dep[k] : 0;
        atomicAdd(&sCnt[ck], dep[k] >= 0 ? 1u : 0u);
        split_add(&sAcc[ck], w1[k]);
    }
}

// The same for the FP64 sums: four 32-bit shared atomics where two 64-bit
// ones per particle (compare-and-swap loops here) contended for the few cells
// of a sorted warp.
__device__ __forceinline__ void split_add64(unsigned long long *sAcc, unsigned *sCnt, int stride, int c,
                                            unsigned long long v, unsigned n)
{
    unsigned *w = reinterpret_cast<unsigned *>(&sAcc[c]);
    atomicAdd(&sCnt[c], n);
    atomicAdd(&w[0], (unsigned)v & ((1u << SPLIT64_0) - 1u));
    atomicAdd(&w[1], (unsigned)(v >> SPLIT64_0) & ((1u << (SPLIT64_1 - SPLIT64_0)) - 1u));
    atomicAdd(&sCnt[stride + c], (unsigned)(v >> SPLIT64_1));
}
// rn(off 2^FIX_BITS_64) from one FP64 add: off + 2^(52 - FIX_BITS_64) has its
// last bit at 2^-FIX_BITS_64 (off is in [0, 1))
__device__ __forceinline__ unsigned long long weight64(double off)
{
    constexpr double SHIFT = (double)(1ull << (52 - FIX_BITS_64));
    return (unsigned long long)(__double_as_longlong(off + SHIFT) - __double_as_longlong(SHIFT));
}
__device__ __forceinline__ void deposit4(unsigned long long *sAcc, unsigned *sCnt, int stride, const int dep[4],
                                         const double off[4])
{
    unsigned long long w1[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) w1[k] = dep[k] >= 0 ? weight64(off[k]) : 0ull;
    const bool same = dep[0] >= 0 && dep[1] == dep[0] && dep[2] == dep[0] && dep[3] == dep[0];
    const unsigned long long b = w1[0] + w1[1] + w1[2] + w1[3];
    const int c0 = __shfl_sync(0xffffffffu, dep[0], 0);
    const bool in = same && dep[0] == c0;
    const unsigned m = __ballot_sync(0xffffffffu, in);
    if (__popc(m) >= DEP_LANES) {
        // 32 lanes of at most 2^(FIX_BITS_64 + 2), summed in two 32-bit halves;
        // a third word of up to 20 bits is one add of 128 particles' weight
        const unsigned lo = __reduce_add_sync(0xffffffffu, in ? (unsigned)(b & 0xFFFFFFull) : 0u);
        const unsigned hi = __reduce_add_sync(0xffffffffu, in ? (unsigned)(b >> 24) : 0u);
        if ((threadIdx.x & 31) == 0)
            split_add64(sAcc, sCnt, stride, c0, ((unsigned long long)hi << 24) + lo, 4u * (unsigned)__popc(m));
        if (in) return;
    }
    if (same) {
        split_add64(sAcc, sCnt, stride, dep[0], b, 4u);
        return;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if (dep[k] >= 0) split_add64(sAcc, sCnt, stride, dep[k], w1[k], 1u);
}

// The push that also samples the diagnostics keeps its FP32 sums per NODE
// (both CIC weights of a particle, split words, four shared atomics per
// particle): its shared memory holds the histograms, and per-cell counts on
// top of them would leave room for fewer blocks per SM.
__device__ __forceinline__ void deposit4_nodes(unsigned long long *sAcc, const int dep[4], const float off[4])
{
    unsigned w0[4], w1[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        w1[k] = dep[k] >= 0 ? __float2uint_rn(off[k] * (float)(1 << FIX_BITS)) : 0u;
        w0[k] = dep[k] >= 0 ? (1u << FIX_BITS) - w1[k] : 0u;
    }
    const int lane = threadIdx.x & 31;
    const bool same = dep[0] >= 0 && dep[1] == dep[0] && dep[2] == dep[0] && dep[3] == dep[0];
    const unsigned a = w0[0] + w0[1] + w0[2] + w0[3];
    const unsigned b = w1[0] + w1[1] + w1[2] + w1[3];
    const int c0 = __shfl_sync(0xffffffffu, dep[0], 0);
    if (__all_sync(0xffffffffu, same && dep[0] == c0)) {
        const unsigned sa = __reduce_add_sync(0xffffffffu, a);
        const unsigned sb = __reduce_add_sync(0xffffffffu, b);
        if (lane == 0) {
            split_add(&sAcc[c0], sa);
            split_add(&sAcc[c0 + 1], sb);
        }
        return;
    }
    if (same) {
        split_add(&sAcc[dep[0]], a);
        split_add(&sAcc[dep[0] + 1], b);
        return;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        // an empty slot adds zero weights to node 0
        const int ck = dep[k] >= 0 ? dep[k] : 0;
        split_add(&sAcc[ck], w0[k]);
        split_add(&sAcc[ck + 1], w1[k]);
    }
}
__device__ __forceinline__ void deposit4_nodes(unsigned long long *sAcc, const int dep[4], const double off[4])
{
    constexpr unsigned long long ONE = 1ull << FIX_BITS_64;
    unsigned long long w1[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) w1[k] = dep[k] >= 0 ? weight64(off[k]) : 0ull;
    // as in the FP32 path: the lanes whose four slots sit in the first lane's
    // cell add their weights once for all, others add their own
    const bool same = dep[0] >= 0 && dep[1] == dep[0] && dep[2] == dep[0] && dep[3] == dep[0];
    const unsigned long long b = w1[0] + w1[1] + w1[2] + w1[3];
    const int c0 = __shfl_sync(0xffffffffu, dep[0], 0);
    const bool in = same && dep[0] == c0;
    const unsigned m = __ballot_sync(0xffffffffu, in);
    if (__popc(m) >= DEP_LANES) {
        // 32 lanes of at most 2^(FIX_BITS_64 + 2), summed in two 32-bit halves
        const unsigned lo = __reduce_add_sync(0xffffffffu, in ? (unsigned)(b & 0xFFFFFFull) : 0u);
        const unsigned hi = __reduce_add_sync(0xffffffffu, in ? (unsigned)(b >> 24) : 0u);
        if ((threadIdx.x & 31) == 0) {
            const unsigned long long sb = ((unsigned long long)hi << 24) + lo;
            atomicAdd(&sAcc[c0], 4ull * __popc(m) * ONE - sb);
            atomicAdd(&sAcc[c0 + 1], sb);
        }
        if (in) return;
    }
    if (same) {
        atomicAdd(&sAcc[dep[0]], 4ull * ONE - b);
        atomicAdd(&sAcc[dep[0] + 1], b);
        return;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (dep[k] >= 0) {
            atomicAdd(&sAcc[dep[k]], ONE - w1[k]);
            atomicAdd(&sAcc[dep[k] + 1], w1[k]);
        }
    }
}

// the species of (discharge, species) index ds has an energy-binned bound
__device__ __forceinline__ bool Dd_binned(const WsPtrs &W, int ds)
{
    return W.disc[ds / NSP].sp[ds % NSP].nbins > 0;
}

// Push arithmetic of a lane's four slots: E at the particle by linear
// interpolation, v + (q/m) E dt, offset + v dt / dx.  FP32: two slots per
// packed instruction (the same roundings as the scalar fused multiply-adds).
// Dead slots' cells are negative: their arithmetic is that of cell 0.
// The block's field table: E per node in FP32; in FP64 E and its step to the
// next node side by side, which takes the subtraction out of every particle.
template <typename Real> struct FieldT;
template <> struct FieldT<float> { using T = float; };
template <> struct FieldT<double> { using T = double2; };
__device__ __forceinline__ void push_arith(const double2 *sE, const int c[4], const double off[4], const double vx[4],
                                           double qm, double ks, double vn[4], double on[4])
{
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const double2 e = sE[max(c[k], 0)];
        vn[k] = vx[k] + qm * (e.x + off[k] * e.y);
        on[k] = off[k] + vn[k] * ks;
    }
}
__device__ __forceinline__ void push_arith(const float *sE, const int c[4], const float off[4],
                                                  const float vx[4], float qm, float ks, float vn[4], float on[4])
{
    const float2 qm2 = make_float2(qm, qm), ks2 = make_float2(ks, ks);
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        const int ca = max(c[2 * p], 0), cb = max(c[2 * p + 1], 0);
        const float2 e0 = make_float2(sE[ca], sE[cb]);
        const float2 e1 = make_float2(sE[ca + 1], sE[cb + 1]);
        const float2 of = make_float2(off[2 * p], off[2 * p + 1]);
        const float2 v0 = make_float2(vx[2 * p], vx[2 * p + 1]);
        const float2 de = __fadd2_rn(e1, make_float2(-e0.x, -e0.y));
        const float2 ep = __ffma2_rn(of, de, e0);
        const float2 v = __ffma2_rn(qm2, ep, v0);
        const float2 o = __ffma2_rn(v, ks2, of);
        vn[2 * p] = v.x;
        vn[2 * p + 1] = v.y;
        on[2 * p] = o.x;
        on[2 * p + 1] = o.y;
    }
}
// lab kinetic energy factor ke (v^2 + vy^2 + vz^2) of four slots
template <typename Real>
__device__ __forceinline__ void energy2(Real ke, const Real v[4], const Real vy[4], const Real vz[4], Real K[4])
{
#pragma unroll
    for (int k = 0; k < 4; ++k) K[k] = ke * (v[k] * v[k] + vy[k] * vy[k] + vz[k] * vz[k]);
}
template <>
__device__ __forceinline__ void energy2<float>(float ke, const float v[4], const float vy[4], const float vz[4],
                                               float K[4])
{
    const float2 ke2 = make_float2(ke, ke);
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        const float2 a = make_float2(v[2 * p], v[2 * p + 1]);
        const float2 y = make_float2(vy[2 * p], vy[2 * p + 1]);
        const float2 z = make_float2(vz[2 * p], vz[2 * p + 1]);
        float2 t = __fmul2_rn(a, a);
        t = __ffma2_rn(y, y, t);
        t = __ffma2_rn(z, z, t);
        t = __fmul2_rn(ke2, t);
        K[2 * p] = t.x;
        K[2 * p + 1] = t.y;
    }
}

// Cell and offset of four live slots after the move: fl = floor(on),
// cn = c + fl, o = on - fl.  Returns false when a slot left [0, N), when its
// offset rounded up to 1, or when the position is out of the range in which
// this is exact (NaN and infinities included); the caller then takes the
// general path from the same inputs.
//
// FP32: t = on + 1.5 2^23 rounded down is floor(on) + 1.5 2^23 for
// |on| < 2^22, its low bits are the integer, and t - 1.5 2^23 is exact: two
// packed adds instead of two conversions per slot (conversions run at a
// quarter of the rate).  Outside that range the integer read from t's bits is
// beyond any grid (or the sum wraps to one that is).
__device__ __forceinline__ bool cells4(const int c[4], const float on[4], int N, const double *, int cn[4], float o[4])
{
    constexpr float M = 12582912.0f;  // 1.5 2^23
    const float2 up = make_float2(M, M), dn = make_float2(-M, -M);
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        const float2 x = make_float2(on[2 * p], on[2 * p + 1]);
        const float2 t = __fadd2_rd(x, up);
        const float2 fl = __fadd2_rn(t, dn);
        const float2 r = __fadd2_rn(x, make_float2(-fl.x, -fl.y));
        cn[2 * p] = c[2 * p] + (__float_as_int(t.x) - 0x4B400000);
        cn[2 * p + 1] = c[2 * p + 1] + (__float_as_int(t.y) - 0x4B400000);
        o[2 * p] = r.x;
        o[2 * p + 1] = r.y;
    }
    const unsigned far = max(max((unsigned)cn[0], (unsigned)cn[1]), max((unsigned)cn[2], (unsigned)cn[3]));
    const float top = fmaxf(fmaxf(o[0], o[1]), fmaxf(o[2], o[3]));
    return far < (unsigned)N && top < 1.0f;
}

// FP64 runs on two units per SM here (an instruction takes a warp 64 cycles of
// its scheduler's unit), so the floor is kept off them: a slot that stays in
// its cell (the high word of on below 1.0's, sign included) needs no arithmetic
// at all, and when a lane of the warp has one that does not, the integer part
// comes from on's bits and its double from a table of -64 .. 63 (sT), for one
// FP64 instruction per slot.  Range checks are on the high words.
constexpr int FLOOR_MAX = 64;
__device__ __forceinline__ bool cells4(const int c[4], const double on[4], int N, const double *sT, int cn[4], double o[4])
{
    unsigned any = 0u, mag = 0u;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const unsigned hi = (unsigned)__double2hiint(on[k]);
        any = max(any, hi);
        mag = max(mag, hi & 0x7FFFFFFFu);
        cn[k] = c[k];
        o[k] = on[k];
    }
    if (!__any_sync(0xffffffffu, any >= 0x3FF00000u)) return true;  // c is in [0, N)
    unsigned far = 0u, top = 0u;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int h = __double2hiint(on[k]);
        const unsigned a = (unsigned)h & 0x7FFFFFFFu;
        const int e = max((int)(a >> 20) - 1023, -1);  // 2^e <= |on| (e = -1: below 1)
        const int ip = (int)(((a & 0xFFFFFu) | 0x100000u) >> ((20 - e) & 31));
        const bool frac = e < 0 || (((a << ((12 + e) & 31)) | (unsigned)__double2loint(on[k])) != 0u);
        // floor, in [-FLOOR_MAX, FLOOR_MAX) for |on| < FLOOR_MAX (others are sent back below)
        const int fl = h < 0 ? -(ip + (frac ? 1 : 0)) : ip;
        o[k] = on[k] - sT[(fl + FLOOR_MAX) & (2 * FLOOR_MAX - 1)];
        cn[k] = c[k] + fl;
        far = max(far, (unsigned)cn[k]);
        top = max(top, (unsigned)__double2hiint(o[k]));
    }
    // |on| < 64 (finite), every cell on the grid, every offset below 1
    return mag < 0x40500000u && far < (unsigned)N && top < 0x3FF00000u;
}

// Bins of the lab energies ke (v^2 + vy^2 + vz^2) of four slots.  FP64: the bin
// is the exponent and two mantissa bits, so an FP32 estimate (the values cut to
// 24 bits by moving bits, off the FP64 units) decides it unless it lies within
// 64 units of the last place of a bin's edge; its error is below 12 such units.
__device__ __forceinline__ void energy_bins(float ke, const float v[4], const float vy[4], const float vz[4], int nb,
                                            int bin[4])
{
    float K[4];
    energy2<float>(ke, v, vy, vz, K);
#pragma unroll
    for (int k = 0; k < 4; ++k) bin[k] = energy_bin(K[k], nb);
}
// |x| cut to an FP32 number (0 below FP32's normal range)
__device__ __forceinline__ float cut32(double x)
{
    const unsigned hi = (unsigned)__double2hiint(x) & 0x7FFFFFFFu;
    const unsigned b = __funnelshift_l((unsigned)__double2loint(x), hi - 0x38000000u, 3);
    return hi >= 0x38100000u && hi < 0x47E00000u ? __uint_as_float(b) : (hi < 0x38100000u ? 0.0f : 3e38f);
}
__device__ __forceinline__ void energy_bins(double ke, const double v[4], const double vy[4], const double vz[4], int nb,
                                            int bin[4])
{
    const float kf = cut32(ke);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float a = cut32(v[k]), b = cut32(vy[k]), c = cut32(vz[k]);
        const float K = kf * (a * a + b * b + c * c);
        const unsigned edge = (__float_as_uint(K) + 64u) & 0x1FFFFFu;
        bin[k] = energy_bin(K, nb);
        if (edge < 128u || !(K > 1e-20f && K < 1e20f))
            bin[k] = energy_bin(ke * (v[k] * v[k] + vy[k] * vy[k] + vz[k] * vz[k]), nb);
    }
}

// Launch shape of the push: NT threads per block, SPT slots per thread.  A
// warp takes SPT/4 consecutive sub-tiles of 128 slots per pass and lane l the
// four consecutive slots 4l .. 4l+3 of each (16-byte vectors, one Philox
// block); a block's pass covers NT SPT / 128 sub-tiles.  MINB is the blocks
// per SM the register allocation is sized for.
template <int NT, int SPT, int MINB>
struct PushShape {
    static constexpr int threads = NT;
    static constexpr int spt = SPT;
    static constexpr int minb = MINB;
    static constexpr int nw = NT / 32;
    static constexpr int groups = SPT / 4;                 // sub-tiles per warp and pass
    static constexpr int qcap = 32 + 32 * SPT;             // candidate queue: < 32 left + one pass
    static_assert(SPT % 4 == 0 && NT % 32 == 0, "shape");
    static_assert((TILES_PER_TICKET * SUBTILES) % (nw * groups) == 0, "a ticket holds whole passes");
};

template <typename Real, bool DIAG, typename SH>
__global__ void __launch_bounds__(SH::threads, SH::minb)
k_push(WsPtrs W, Pools<Real> P, int par, int Nmax, int eedf_max, int fm_max)
{
    pdl_wait();
    using Acc = typename AccT<Real>::T;
    constexpr int PUSH_THREADS = SH::threads, NW = SH::nw, G = SH::groups, QCAP = SH::qcap;
    // per-cell sums (counts + upper weights); the FP32 diagnostics push has no room for them
    constexpr bool FP64 = sizeof(Real) == 8;
    constexpr bool CELLS = !DIAG || FP64;
    using ET = typename FieldT<Real>::T;
    extern __shared__ __align__(16) unsigned char smem[];
    // FP32: sums, field; FP64: field, sums, the floors' doubles
    unsigned long long *sAcc = reinterpret_cast<unsigned long long *>(smem + (FP64 ? sizeof(ET) * (Nmax + 2) : 0));
    ET *sE = reinterpret_cast<ET *>(FP64 ? smem : smem + 8 * (size_t)(Nmax + 2));
    double *sT = reinterpret_cast<double *>(sAcc + (Nmax + 2));
    unsigned char *rest = FP64 ? reinterpret_cast<unsigned char *>(sT + 2 * FLOOR_MAX)
                               : reinterpret_cast<unsigned char *>(sE + (Nmax + 2));
    if (FP64)
        for (int i = threadIdx.x; i < 2 * FLOOR_MAX; i += SH::threads) sT[i] = (double)(i - FLOOR_MAX);
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    // per-warp list of collision candidates (slot, energy bin) before it is
    // written out, and the histograms
    int *qIdx = reinterpret_cast<int *>(rest) + w * QCAP;
    unsigned *sEedf = reinterpret_cast<unsigned *>(rest) + NW * QCAP;
    unsigned *sFm = sEedf + eedf_max;
    unsigned char *qBin = reinterpret_cast<unsigned char *>(sFm + fm_max) + w * QCAP;
    // particles per cell of the block's sums (FP64: and third words), after the queues' bins
    unsigned *sCnt = reinterpret_cast<unsigned *>(
        (reinterpret_cast<size_t>(reinterpret_cast<unsigned char *>(sFm + fm_max) + NW * QCAP) + 15) & ~size_t(15));

    __shared__ int s_ticket[2], s_stop, s_find;
    __shared__ unsigned s_cnt[C_NCOUNT];
    __shared__ unsigned s_btn[NUBIN_MAX];  // electron bounds per energy bin: thresholds

    Ctl *ctl = W.ctl;
    const int cur = ctl->cur;
    const unsigned long long step = ctl->step[par];
    const int total = ctl->total_chunks;
    // the state's buffer: slot i of an array sits at element b0 + i of its
    // first buffer, so that the arrays' addresses stay kernel parameters
    const unsigned b0 = cur ? P.stride : 0u;
    int *const cellA = P.cell[0];
    Real *const offA = P.off[0], *const vxA = P.vx[0], *const vyA = P.vy[0], *const vzA = P.vz[0];
    Acc *accG = acc_global<Real>(W);
    const unsigned lt_mask = (1u << lane) - 1u;

    int ds = -1, d = -1, run_tiles = 0;
    for (int q = tid; q < C_NCOUNT; q += PUSH_THREADS) s_cnt[q] = 0;
    auto flush = [&](int fds) {
        const int fd = fds / NSP, fs = fds % NSP;
        const Disc &Dd = W.disc[fd];
        __syncthreads();
        Acc *g = accG + (size_t)fs * W.total_nodes + Dd.gbase;
        for (int i = tid; i <= Dd.N; i += PUSH_THREADS) {
            const unsigned long long v = CELLS ? sacc_cells<Real>(sAcc, sCnt, Nmax + 2, i)
                                               : (sizeof(Real) == 4 ? split_value(sAcc[i]) : sAcc[i]);
            if (v != 0ull) acc_add(&g[i], sacc_value<Real>(v));
        }
        for (int q = tid; q < C_NCOUNT; q += PUSH_THREADS) {
            if (s_cnt[q]) atomicAdd(&W.counters[(size_t)fd * C_NCOUNT + q], (unsigned long long)s_cnt[q]);
        }
        if (DIAG) {
            if (fs == 0)
                for (int i = tid; i < Dd.eedf_bins; i += PUSH_THREADS)
                    if (sEedf[i]) atomicAdd(&W.eedf[Dd.eedf_base + i], sEedf[i]);
            if (fs == 1)
                for (int i = tid; i < Dd.fm_bins * Dd.fm_xbins; i += PUSH_THREADS)
                    if (sFm[i]) atomicAdd(&W.fm[Dd.fm_base + i], sFm[i]);
        }
        __syncthreads();
    };

    // ---- the warp's candidates go to the step's list (one reservation per
    // batch); the collision kernel takes them from there
    int qn = 0;  // warp-uniform
    auto list_out = [&]() {
        int base = 0;
        if (lane == 0) {
            base = (int)atomicAdd(&ctl->cand_n, (unsigned)qn);
            atomicAdd(&s_cnt[C_CANDS], (unsigned)qn);
            if (Dd_binned(W, ds)) atomicAdd(&s_cnt[C_BCANDS], (unsigned)qn);
            if ((long long)base + qn > W.cand_cap) set_status(ctl, ST_BIRTHBUF);
        }
        base = __shfl_sync(0xffffffffu, base, 0);
        for (int q = lane; q < qn; q += 32) {
            const long long at = (long long)base + q;
            if (at < W.cand_cap) W.cand[at] = make_int2(qIdx[q], (ds << 8) | qBin[q]);
        }
        __syncwarp();
        qn = 0;
    };

    // The block's tiles.  Few tiles per block (STATIC_TILES): one contiguous
    // share of all of them each, no ticket and no barrier between them.  Many:
    // tickets of TILES_PER_TICKET tiles, so that no block waits for a slower
    // one.  Both are worked off in stretches of one (discharge, species).
    const bool shared_out = total <= STATIC_TILES * (int)gridDim.x;
    int tcur = 0;
    if (shared_out) {
        tcur = (int)((long long)blockIdx.x * total / gridDim.x);
        if (tid == 0) s_stop = (int)((long long)(blockIdx.x + 1) * total / gridDim.x);
        __syncthreads();
    }
    for (int it = 0;; ++it) {
        if (shared_out) {
            if (tcur >= s_stop) break;
        } else {
            // two ticket buffers: a buffer is rewritten only after the barrier
            // that every reader of its previous value has passed
            if (tid == 0) s_ticket[it & 1] = (int)atomicAdd(&ctl->ticket, (unsigned)TILES_PER_TICKET);
            __syncthreads();
            tcur = s_ticket[it & 1];
            if (tcur >= total) break;
        }
        int nx = ds;
        if (ds < 0 || tcur < W.cnt[ds].chunk0 || tcur >= W.cnt[ds].chunk0 + W.cnt[ds].nchunk) {
            // the first (d, s) that ends after tile tcur: one thread finds it
            // (the ends never fall)
            __syncthreads();
            const int nds = W.D * NSP;
            for (int q = tid; q < nds; q += PUSH_THREADS) {
                const int eq = W.cnt[q].chunk0 + W.cnt[q].nchunk;
                const int ep = q > 0 ? W.cnt[q - 1].chunk0 + W.cnt[q - 1].nchunk : 0;
                if (eq > tcur && ep <= tcur) s_find = q;
            }
            __syncthreads();
            nx = s_find;
        }
        const int tbeg = max(tcur, W.cnt[nx].chunk0);  // padding tiles before it hold nothing
        const int tend = min(min(W.cnt[nx].chunk0 + W.cnt[nx].nchunk, tbeg + FLUSH_TILES),
                             shared_out ? s_stop : tcur + TILES_PER_TICKET);
        tcur = max(tbeg, tend);
        if (tbeg >= tend) continue;  // only padding, or a species without slots, up to here
        if (species_rests(W.disc[nx / NSP], nx % NSP, step)) {
            // a resting ion species: nothing to push
            continue;
        }
        // a new (d, s), or the block's integer sums at their bound: flush
        if (nx != ds || run_tiles + (tend - tbeg) > FLUSH_TILES) {
            if (qn > 0) list_out();
            if (ds >= 0) flush(ds);
            const int nd = nx / NSP;
            const Disc &Dn = W.disc[nd];
            if (nd != d) {
                const Real *Eg = reinterpret_cast<const Real *>(W.Ereal) + Dn.gbase;
                for (int i = tid; i <= Dn.N; i += PUSH_THREADS) {
                    if constexpr (FP64)
                        sE[i] = make_double2(Eg[i], i < Dn.N ? Eg[i + 1] - Eg[i] : 0.0);
                    else
                        sE[i] = Eg[i];
                }
                d = nd;
            }
            for (int i = tid; i <= Dn.N + 1; i += PUSH_THREADS) {
                sAcc[i] = 0ull;
                if (CELLS) sCnt[i] = 0u;
                if (CELLS && sizeof(Real) == 8) sCnt[Nmax + 2 + i] = 0u;
            }
            {
                const SpeciesC &Sn = Dn.sp[nx % NSP];
                for (int b = tid; b < Sn.nbins; b += PUSH_THREADS) {
                    const NuBin &nb = W.nubin[Sn.bin_off + b];
                    s_btn[b] = nb.tnull;
                }
            }
            for (int q = tid; q < C_NCOUNT; q += PUSH_THREADS) s_cnt[q] = 0;
            if (DIAG) {
                for (int i = tid; i < eedf_max; i += PUSH_THREADS) sEedf[i] = 0;
                for (int i = tid; i < fm_max; i += PUSH_THREADS) sFm[i] = 0;
            }
            ds = nx;
            run_tiles = 0;
            __syncthreads();
        }
        run_tiles += tend - tbeg;
        const int s = ds % NSP;
        const Disc &Dd = W.disc[d];
        const SpeciesC &S = Dd.sp[s];
        const Counts &C = W.cnt[ds];
        const int N = Dd.N;
        const int pb = Dd.pbase[s];
        const int end = pb + C.n_snap;
        // a sub-cycled ion species moves over ks steps per push
        const Real ks = Real(s > 0 ? Dd.ion_sub : 1);
        const Real qm = pick<Real>(S.qm, S.qm_f) * ks;
        const unsigned tnull = S.tnull;
        const int nbins = S.nbins;
        const bool binned = nbins > 0;  // electrons: bound per lab-energy bin
        const Real ke = pick<Real>(S.ke_eV, S.ke_eV_f);
        const float rN = 1.0f / (float)N;  // the diagnostics' x bins
        // the ticket's sub-tiles in rows of NW G: warp w takes sub-tiles
        // w G .. w G + G - 1 of every row
        constexpr int ROW = NW * G;
        const int st_beg = tbeg * SUBTILES, st_end = tend * SUBTILES;
        // the warp's first slot in the ticket
        const int wbase0 = pb + (tbeg - C.chunk0) * CHUNK + w * G * SUBTILE;
        unsigned tslots = 0, tlive = 0;  // the ticket's slot counts of this thread
        for (int r0 = st_beg; r0 < st_end; r0 += ROW) {
            if (O2_PUSH_L2_AHEAD > 0 && tid == 0) {
                // the row O2_PUSH_L2_AHEAD ahead in this ticket (on the first
                // row also those between): cell, offset and vx into L2
                const int ra = (r0 == st_beg) ? r0 + ROW : r0 + O2_PUSH_L2_AHEAD * ROW;
                const int rb = (r0 == st_beg) ? min(r0 + O2_PUSH_L2_AHEAD * ROW, st_end - ROW) : ra;
                for (int rp = ra; rp <= rb && rp < st_end; rp += ROW) {
                    const size_t sl = (size_t)b0 + (size_t)pb + (size_t)(rp - C.chunk0 * SUBTILES) * SUBTILE;
                    const unsigned n = (unsigned)min(ROW, st_end - rp) * SUBTILE;
                    l2_prefetch(cellA + sl, n * sizeof(int));
                    l2_prefetch(offA + sl, n * sizeof(Real));
                    l2_prefetch(vxA + sl, n * sizeof(Real));
                }
            }
#pragma unroll
            for (int g = 0; g < G; ++g) {
            const int sub = r0 + w * G + g;
            // a row of at most one tile fits the ticket's whole tiles; a
            // longer one can overhang its tail
            if (ROW > SUBTILES && sub >= st_end) break;
            const int i0 = wbase0 + (r0 - st_beg) * SUBTILE + g * SUBTILE + 4 * lane;

            // ---- phase A: push, absorb, null test, deposit, candidate queue
            int c[4];
            Real off[4], vx[4];
            const bool full = i0 + 3 < end;
            const unsigned ib = b0 + (unsigned)i0;
            if (full) {
                ld4(cellA + ib, c);
                ld4(offA + ib, off);
                ld4(vxA + ib, vx);
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const bool in = i0 + k < end;
                    c[k] = in ? cellA[ib + k] : -2;
                    off[k] = in ? offA[ib + k] : Real(0);
                    vx[k] = in ? vxA[ib + k] : Real(0);
                }
            }
            Real vyl[4], vzl[4];  // binned species only: the lab energy needs vy, vz
            if (binned) {
                if (full) {
                    ld4(vyA + ib, vyl);
                    ld4(vzA + ib, vzl);
                } else {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const bool in = i0 + k < end;
                        vyl[k] = in ? vyA[ib + k] : Real(0);
                        vzl[k] = in ? vzA[ib + k] : Real(0);
                    }
                }
            }
            const uint4 w4 = rng_block(Dd.seed, Dd.discharge, s, 0, 0, 0, step, (unsigned)((i0 - pb) >> 2));
            const unsigned wk[4] = {w4.x, w4.y, w4.z, w4.w};
            bool cchg = true;  // a cell index of the lane's slots changed
            unsigned candm = 0u, bins = 0u;
            int dep[4];  // cells after the move, -1 for a slot that holds no particle any more
            // the field at the particle, the new velocity and position (the
            // FP32 path takes two slots per packed instruction)
            Real vn[4], on[4];
            push_arith(sE, c, off, vx, qm, ks, vn, on);
            // null-collision thresholds; electrons: by the bin of the lab energy
            unsigned thr[4] = {tnull, tnull, tnull, tnull};
            if (binned) {
                int bin[4];
                energy_bins(ke, vn, vyl, vzl, nbins, bin);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    thr[k] = s_btn[bin[k]];
                    bins |= (unsigned)bin[k] << (8 * k);
                }
            }
            // Nearly every warp holds 128 live slots that all stay on the
            // grid: no masks, no selects (fast).  Any other case takes the
            // general path below from the same inputs.
            bool fast = full && (c[0] | c[1] | c[2] | c[3]) >= 0;
            fast = __all_sync(0xffffffffu, fast);
            if (fast) {
                Real o[4];
                fast = __all_sync(0xffffffffu, cells4(c, on, N, sT, dep, o));
                if (fast) {
                    cchg = ((c[0] ^ dep[0]) | (c[1] ^ dep[1]) | (c[2] ^ dep[2]) | (c[3] ^ dep[3])) != 0;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        c[k] = dep[k];
                        off[k] = o[k];
                        vx[k] = vn[k];
                        candm |= wk[k] < thr[k] ? 1u << k : 0u;
                    }
                    tslots += 4u;
                    tlive += 4u;
                }
            }
            bool live4 = true;  // the lane has something to write back
            if (!fast) {
                // each slot is pushed without branches; absorptions are noted in
                // a mask and handled after the four slots
                unsigned nslots = 0, nlive = 0, outm = 0, wallm = 0;
                bool nonfin = false;
                cchg = false;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int ck = c[k];
                    const bool was = ck >= 0;
                    nslots += ck >= -1 ? 1u : 0u;
                    nlive += was ? 1u : 0u;
                    const int cc = was ? ck : 0;
                    const Real v = vn[k];
                    Real o = on[k];
                    const Real fl = floor(o);
                    const bool bad = !(fl > Real(-2 * N - 4) && fl < Real(2 * N + 4));
                    // a non-finite velocity or position is an error, not an absorption
                    nonfin |= was && !isfinite(o);
                    int cn = bad ? (v < Real(0) ? -1 : N) : cc + (int)fl;
                    o -= fl;
                    const bool wrap = o >= Real(1);
                    o = wrap ? o - Real(1) : o;
                    cn += wrap ? 1 : 0;
                    const bool out = was && (cn < 0 || cn >= N);
                    const bool live = was && !out;
                    outm |= (out && isfinite(o)) ? 1u << k : 0u;
                    wallm |= cn >= N ? 1u << k : 0u;
                    vx[k] = was ? v : vx[k];
                    off[k] = live ? o : off[k];
                    const int cnew = was ? (out ? -1 : cn) : ck;
                    cchg |= cnew != ck;
                    c[k] = cnew;
                    dep[k] = live ? cn : -1;
                    candm |= live && wk[k] < thr[k] ? 1u << k : 0u;
                }
                if (nonfin) set_status(ctl, ST_NONFINITE);
                if (outm) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        if (!((outm >> k) & 1u)) continue;
                        const int wall = (wallm >> k) & 1u;
                        atomicAdd(&s_cnt[C_ABS + 2 * s + wall], 1u);
                        if (s == 2 && Dd.iedf_bins > 0) {
                            const Real v = vx[k], vy = vyA[ib + k], vz = vzA[ib + k];
                            const Real Ei = pick<Real>(S.ke_eV, S.ke_eV_f) * (v * v + vy * vy + vz * vz);
                            const Real bb = floor(Ei * pick<Real>(Dd.iedf_scale, Dd.iedf_scale_f));
                            if (bb >= Real(0) && bb < Real(Dd.iedf_bins))
                                atomicAdd(&W.iedf[Dd.iedf_base + wall * Dd.iedf_bins + (int)bb], 1u);
                        }
                    }
                }
                tslots += nslots;
                tlive += nlive;
                live4 = nlive != 0u;
            }
            // candidates are rare: one vote, and the queue only when a lane has one
            if (__any_sync(0xffffffffu, candm != 0u)) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const bool cand = (candm >> k) & 1u;
                    const unsigned m = __ballot_sync(0xffffffffu, cand);
                    if (cand) {
                        const int pos = qn + __popc(m & lt_mask);
                        qIdx[pos] = i0 + k;
                        qBin[pos] = (unsigned char)(bins >> (8 * k));
                    }
                    qn += __popc(m);
                }
            }
            if (DIAG) {
                // distributions after the free flight, before collisions
                if (s == 0 && Dd.eedf_bins > 0) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        if (dep[k] != N / 2) continue;
                        const Real v = vx[k], vy = vyA[ib + k], vz = vzA[ib + k];
                        const Real Ee = pick<Real>(S.ke_eV, S.ke_eV_f) * (v * v + vy * vy + vz * vz);
                        const Real bb = floor(Ee * pick<Real>(Dd.eedf_scale, Dd.eedf_scale_f));
                        if (bb >= Real(0) && bb < Real(Dd.eedf_bins)) atomicAdd(&sEedf[(int)bb], 1u);
                    }
                }
                if (s == 1 && Dd.fm_bins > 0) {
                    // cold, sorted O- of a warp fall into a few bins: the lanes
                    // of one bin add their count once (no 32-way conflicts)
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int cn = dep[k];
                        int fb = -1;
                        if (cn >= 0) {
                            const Real v = vx[k];
                            Real Es = pick<Real>(S.ke_eV, S.ke_eV_f) * v * v;
                            if (v < Real(0)) Es = -Es;
                            const Real bb = floor((Es + pick<Real>(Dd.fm_emax, Dd.fm_emax_f)) *
                                                  pick<Real>(Dd.fm_scale, Dd.fm_scale_f));
                            if (bb >= Real(0) && bb < Real(Dd.fm_bins)) {
                                // x bin floor(cn X / N) without an integer division: an
                                // estimate through 1/N in FP32 (off by at most one, as
                                // cn X <= 2^26), then corrected
                                const int pr = cn * Dd.fm_xbins;
                                int xb = (int)((float)pr * rN);
                                xb += (xb + 1) * N <= pr ? 1 : 0;
                                xb -= xb * N > pr ? 1 : 0;
                                fb = xb * Dd.fm_bins + (int)bb;
                            }
                        }
                        const unsigned peers = __match_any_sync(0xffffffffu, fb);
                        if (fb >= 0 && lane == __ffs(peers) - 1) atomicAdd(&sFm[fb], (unsigned)__popc(peers));
                    }
                }
            }
            if constexpr (CELLS)
                deposit4(sAcc, sCnt, Nmax + 2, dep, off);
            else
                deposit4_nodes(sAcc, dep, off);
            if (full) {
                // an unchanged value is not written back: slow ions keep
                // their cells for many steps, and a lane of dead slots
                // changes nothing (its DRAM sectors then stay clean)
                if (cchg) st4(cellA + ib, c);
                if (live4) {
                    st4(offA + ib, off);
                    st4(vxA + ib, vx);
                }
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (i0 + k < end) {
                        cellA[ib + k] = c[k];
                        offA[ib + k] = off[k];
                        vxA[ib + k] = vx[k];
                    }
                }
            }
            }
            __syncwarp();
            if (qn >= 32) list_out();
        }
        {
            const unsigned ws = __reduce_add_sync(0xffffffffu, tslots);
            const unsigned wl = __reduce_add_sync(0xffffffffu, tlive);
            if (lane == 0) {
                if (ws) atomicAdd(&s_cnt[C_SLOTS], ws);
                if (ws && binned) atomicAdd(&s_cnt[C_BSLOTS], ws);
                if (wl) atomicAdd(&s_cnt[C_LIVE], wl);
            }
        }
    }
    if (qn > 0) list_out();
    if (ds >= 0) flush(ds);
}


// Collisions of the step's candidates (null-collision method, Sec. III
// kinematics): one thread per candidate, in list order; a dying particle's
// charge leaves the global grid, births go to its sub-tile's records.  A
// candidate's cell and offset are read only when its collision has products
// or kills it, and its velocity is written back only after an event (a
// null event changes nothing): each field is a scattered access.
//
// What bounds it: the chain of dependent loads in FP32, the FP64 units in
// FP64 (about 500 FP64 instructions per warp of candidates, 16 cycles each on
// an SM's two units).  So the list is dealt out in batches of 32, one warp per
// block and SM first: a hundred FP64 candidates in one block took 28 us, on
// four SMs 15 us (FP32 8.8 -> 5.7 us; 1.3e5 candidates FP32 30 -> 26, FP64
// 140 -> 122 us, the latter from fewer FP64 instructions: uniforms from bits,
// comparisons of positive values as integers).  Blocks of 32, 64 or 128
// threads gave the same times.  The constants that a candidate needs are in its
// species' record, its table's ends included, one load level below the list.
// Event counts are summed per block for the discharge of the block's first
// candidate (the list holds runs of one discharge); lanes of another add
// theirs to the global counters, one add per warp and kind.
template <typename Real>
__global__ void __launch_bounds__(COLLIDE_THREADS)
k_collide(WsPtrs W, Pools<Real> P, int par)
{
    pdl_wait();
    using Acc = typename AccT<Real>::T;
    constexpr int NW = COLLIDE_THREADS / 32;
    __shared__ unsigned s_ev[C_NCOUNT];
    Ctl *ctl = W.ctl;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // the first batch's entry is loaded together with the list's length
    int q = (blockIdx.x + gridDim.x * warp) * 32 + lane;
    int2 e = q < W.cand_cap ? W.cand[q] : make_int2(0, 0);
    const int yblk = W.cand[min(blockIdx.x * 32u, (unsigned)W.cand_cap - 1u)].y;
    const int n = (int)min((long long)ctl->cand_n, (long long)W.cand_cap);
    const unsigned long long step = ctl->step[par];
    const unsigned b0 = ctl->cur ? P.stride : 0u;
    if ((int)blockIdx.x * 32 >= n) return;
    const int dblk = (yblk >> 8) / NSP;
    for (int k = threadIdx.x; k < C_NCOUNT; k += COLLIDE_THREADS) s_ev[k] = 0;
    __syncthreads();
    Acc *accG = acc_global<Real>(W);
    for (; q - lane < n; q += gridDim.x * COLLIDE_THREADS) {
        const int qn = q + gridDim.x * COLLIDE_THREADS;
        const int2 en = qn < n ? W.cand[qn] : make_int2(0, 0);
        int d = dblk, code = -1;  // what the lane counts: the reaction, its number + 32 with a violation
        if (q < n) {
            const int i = e.x, ds = e.y >> 8, bin = e.y & 0xFF;
            const unsigned ib = b0 + (unsigned)i;
            const int s = ds % NSP;
            d = ds / NSP;
            const Disc &Dd = W.disc[d];
            const SpeciesC &S = Dd.sp[s];
            const int rel = i - Dd.pbase[s];
            const int sub = (W.cnt[ds].chunk0 + rel / CHUNK) * SUBTILES + (rel % CHUNK) / SUBTILE;
            const int slot = rel % SUBTILE;
            int c = 0;
            Real off = Real(0);
            Real vx = P.vx[0][ib], vy = P.vy[0][ib], vz = P.vz[0][ib];
            const NuBin &nb = W.nubin[(size_t)d * NUBIN_MAX + (s == 0 ? bin : 0)];
            const Real nbin = pick<Real>(nb.numax_n, nb.numax_n_f);
            const Real nun = S.nbins > 0 ? nbin : pick<Real>(S.numax_n, S.numax_n_f);
            const BirthSink<Real> B = birth_sink<Real>(W, Dd, par, sub);
            const Outcome o = gas_collide<Real>(W, Dd, s, (unsigned)rel, step, nun, vx, vy, vz, P.cell[0] + ib,
                                                P.off[0] + ib, c, off, slot << 1, B);
            // a null event leaves the particle as it was: nothing to write
            if (o.alive) {
                if (o.reaction >= 0) {
                    P.vx[0][ib] = vx;
                    P.vy[0][ib] = vy;
                    P.vz[0][ib] = vz;
                }
            } else {
                P.cell[0][ib] = -1;
                deposit_global(accG + (size_t)s * W.total_nodes + Dd.gbase, c, off, -1);
            }
            if (o.reaction >= 0 || o.viol) code = (o.reaction >= 0 ? o.reaction : 31) + (o.viol ? 32 : 0);
        }
        if (code >= 0 && d == dblk) {
            if (code >= 32) atomicAdd(&s_ev[C_VIOL_GAS], 1u);
            if ((code & 31) < 31) atomicAdd(&s_ev[C_EVENTS + (code & 31)], 1u);
            code = -1;
        }
        if (__any_sync(0xffffffffu, code >= 0)) {
            const unsigned peers = __match_any_sync(0xffffffffu, code < 0 ? -1 : d * 64 + code);
            if (code >= 0 && lane == __ffs(peers) - 1) {
                unsigned long long *g = W.counters + (size_t)d * C_NCOUNT;
                const unsigned long long m = (unsigned long long)__popc(peers);
                if (code >= 32) atomicAdd(&g[C_VIOL_GAS], m);
                if ((code & 31) < 31) atomicAdd(&g[C_EVENTS + (code & 31)], m);
            }
        }
        e = en;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < C_NCOUNT; k += COLLIDE_THREADS)
        if (s_ev[k]) atomicAdd(&W.counters[(size_t)dblk * C_NCOUNT + k], (unsigned long long)s_ev[k]);
}

// Bound on P = n dx sigma u_n n1 of channel j of species S for a particle
// of speed |v|, over every gas molecule Box-Muller can give (|V| below 10
// thermal speeds): the prefix maximum of n dx sigma u_n over the table up
// to the centre-of-mass energy of |v| + 10 v_gas (beyond the table: the last
// value times that speed), times n1, with a 1e-3 margin for rounding.  A
// draw at or above it cannot collide, whatever the molecule.
// (The speed and its place on the species' energy grid are the same for all
// channels of the species: dsmc_locate once per particle and speed,
// dsmc_bound per channel.)
template <typename Real>
__device__ __forceinline__ void dsmc_locate(const WsPtrs &W, const SpeciesC &S, const Real v[3], Real &umax,
                                            int &k, int &region)
{
    umax = sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]) + Real(10) * pick<Real>(S.vgas_n, S.vgas_n_f);
    const XsPoint<Real> pm = xs_locate<Real>(S, Lut<Real>::E(W), pick<Real>(S.Ek, S.Ek_f) * umax * umax);
    k = pm.k;
    region = pm.region;
}

template <typename Real>
__device__ __forceinline__ Real dsmc_bound(const WsPtrs &W, const SpeciesC &S, int j, Real umax, int k, int region,
                                           Real n1)
{
    const Real *tb = GasTab<Real>::ptr(W) + S.gtab_off;
    const Real *pmr = GasTab<Real>::bound(W) + S.gtab_off;
    Real bnd;
    if (region == 0) {
        bnd = tb[j] * umax;
    } else if (region == 1) {
        bnd = pmr[(size_t)k * S.gtab_ld + j];
    } else {
        const Real last = tb[(size_t)(k + 1) * S.gtab_ld + j] * umax;
        const Real pmv = pmr[(size_t)k * S.gtab_ld + j];
        bnd = last > pmv ? last : pmv;
    }
    return bnd * n1 * Real(1.001);
}

// The paper's sequential scheme for the gas channels (Sec. II, Eq. 1),
// every n1 steps after the sort: part 0 walks the gas channels of the list
// numbered below (13), part 1 those above (14).  One block per tile of the
// table rebuilt after the sort; the tile's particles are held in shared
// memory.  For each channel of its species in turn a particle draws its test
// number and compares it with a bound on P (dsmc_bound); at the first one below
// it the particle is queued with that channel.  The block's threads take the
// queue one entry each (a gas molecule from the Maxwellian, P = n sigma(E) u n1
// dt clamped at 1 and counted, the test, the kinematics) and go on along the
// list with what the particle is then, into the next round's queue.  A particle
// that dies in (15), (16) or (17) is replaced by its product, which meets the
// later channels.  Random numbers: stream 6 of the chain's first particle,
// sub-stream = the channel's place in the list, draws 4g (molecule), 4g + 1
// (test, direction), 4g + 2 (second direction of (18)) in generation g.
// Products are recorded in the first particle's sub-tile: (18)'s with product
// bits 0 (electron) and 1 (O2+), the one that ends a chain with bit 1.  The
// decisions are those of walking each particle's chain in turn: a particle's
// channels stay in list order, and particles do not interact.
// What bounds it: latency and the Philox draw per particle and channel.  The
// rounds have a barrier each, and there are as many as one particle has
// candidates in a row; a queue and three barriers per channel, most of them
// with a few entries, took 160 us per part for 4e6 superparticles, 130 us so.
template <typename Real>
__global__ void __launch_bounds__(DSMC_THREADS, 3)
k_dsmc(WsPtrs W, Pools<Real> P, int par, int part)
{
    pdl_wait();
    __shared__ unsigned s_ev[C_NCOUNT];
    __shared__ Real sv[3][CHUNK];        // velocity of the chain's current particle
    __shared__ signed char ssp[CHUNK];   // its species, -1 for no particle
    __shared__ unsigned char sgen[CHUNK];
    __shared__ unsigned short sq[2][CHUNK];  // queues of this round and the next
    __shared__ unsigned char skk[CHUNK];     // place in the list of a queued particle's channel
    __shared__ Real sumax[CHUNK];        // speed bound and grid place of the particle (dsmc_locate)
    __shared__ unsigned short sk[CHUNK];
    __shared__ unsigned char sreg[CHUNK];
    __shared__ unsigned s_qn[3];
    Ctl *ctl = W.ctl;
    const int chunk = blockIdx.x;
    if (chunk >= ctl->total_chunks) return;
    int lo = 0, hi = W.D * NSP;  // (discharge, species) of the tile
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (W.cnt[mid].chunk0 <= chunk) lo = mid; else hi = mid;
    }
    const int ds = lo;
    const Counts &C = W.cnt[ds];
    if (chunk >= C.chunk0 + C.nchunk) return;  // padding between species
    const int d = ds / NSP, s = ds % NSP;
    const Disc &Dd = W.disc[d];
    const int tid = threadIdx.x;
    for (int q = tid; q < C_NCOUNT; q += DSMC_THREADS) s_ev[q] = 0;
    if (tid < 3) s_qn[tid] = 0u;
    const unsigned long long step = ctl->step[par];
    const int cur = ctl->cur;
    int *cellA = P.cell[cur];
    Real *offA = P.off[cur], *vxA = P.vx[cur], *vyA = P.vy[cur], *vzA = P.vz[cur];
    const Real *lutE = Lut<Real>::E(W);
    const Real n1 = Real(Dd.n1);
    const int rel0 = (chunk - C.chunk0) * CHUNK;
    const int pb = Dd.pbase[s];
    unsigned nlive = 0;
    for (int local = tid; local < CHUNK; local += DSMC_THREADS) {
        const int rel = rel0 + local;
        signed char sp = -1;
        if (rel < C.n) {
            const int i = pb + rel;
            if (cellA[i] >= 0) {
                sp = (signed char)s;
                const Real v[3] = {vxA[i], vyA[i], vzA[i]};
                sv[0][local] = v[0];
                sv[1][local] = v[1];
                sv[2][local] = v[2];
                Real um;
                int k, reg;
                dsmc_locate<Real>(W, Dd.sp[s], v, um, k, reg);
                sumax[local] = um;
                sk[local] = (unsigned short)k;
                sreg[local] = (unsigned char)reg;
                ++nlive;
            }
        }
        ssp[local] = sp;
        sgen[local] = 0;
    }
    if (nlive) atomicAdd(&s_ev[C_DSMC], nlive);
    __syncthreads();
    unsigned ntest = 0;  // Eq. 1 tests of this thread's particles
    // the part's stretch of the list (it is in the order of the reactions)
    int kbeg = 0, kend = Dd.ndsmc;
    while (kbeg < kend && part == 1 && Dd.dsmc[kbeg].reaction < 15) ++kbeg;
    while (kend > kbeg && part == 0 && Dd.dsmc[kend - 1].reaction > 12) --kend;
    // the test number of channel kk against the bound on P
    auto maybe = [&](int local, int kk, const DsmcCh &e) {
        const unsigned w = rng_block(Dd.seed, Dd.discharge, s, 6, kk, 4u * sgen[local] + 1u, step, (unsigned)(rel0 + local)).x;
        return unif<Real>(w) < dsmc_bound<Real>(W, Dd.sp[e.sp], e.j, sumax[local], sk[local], sreg[local], n1);
    };
    {
        // the first channel that may take each of the thread's particles, side
        // by side (independent chains)
        constexpr int PT = CHUNK / DSMC_THREADS;
        bool on[PT];
#pragma unroll
        for (int q = 0; q < PT; ++q) on[q] = ssp[tid + q * DSMC_THREADS] >= 0;
        for (int kk = kbeg; kk < kend; ++kk) {
            const DsmcCh e = Dd.dsmc[kk];
            if (e.sp != s) continue;  // no particle has changed its species yet
#pragma unroll
            for (int q = 0; q < PT; ++q) {
                const int local = tid + q * DSMC_THREADS;
                if (!on[q]) continue;
                ++ntest;
                if (maybe(local, kk, e)) {
                    on[q] = false;
                    skk[local] = (unsigned char)kk;
                    sq[0][atomicAdd(&s_qn[0], 1u)] = (unsigned short)local;
                }
            }
        }
    }
    for (int round = 0;; ++round) {
        __syncthreads();  // the round's queue is complete
        const int nq = (int)s_qn[round % 3];
        if (nq == 0) break;
        // the counter after the next: its last readers passed the barrier above
        if (tid == 0) s_qn[(round + 2) % 3] = 0u;
        const unsigned short *in = sq[round & 1];
        for (int qi = tid; qi < nq; qi += DSMC_THREADS) {
            const int local = in[qi];
            const int rel = rel0 + local;
            int kk = skk[local];
            {
                const DsmcCh e = Dd.dsmc[kk];
                const SpeciesC &S = Dd.sp[e.sp];
                const GasChan &ch = S.ch[e.j];
                const unsigned gen = sgen[local];
                Real v[3] = {sv[0][local], sv[1][local], sv[2][local]};
                const uint4 b = rng_block(Dd.seed, Dd.discharge, s, 6, kk, 4u * gen + 1u, step, (unsigned)rel);
                const uint4 a = rng_block(Dd.seed, Dd.discharge, s, 6, kk, 4u * gen, step, (unsigned)rel);
                Real n0, nn1, n2, n3;
                box_muller<Real>(a.x, a.y, n0, nn1);
                box_muller<Real>(a.z, a.w, n2, n3);
                const Real vg = pick<Real>(S.vgas_n, S.vgas_n_f);
                const Real V[3] = {vg * n0, vg * nn1, vg * n2};
                const Real g0 = v[0] - V[0], g1 = v[1] - V[1], g2 = v[2] - V[2];
                const Real u2 = g0 * g0 + g1 * g1 + g2 * g2;
                const Real u = sqrt(u2);
                const Real E = pick<Real>(S.Ek, S.Ek_f) * u2;
                // n_j dx sigma_j(E) from the species' node-major table
                const XsPoint<Real> pt = xs_locate<Real>(S, lutE, E);
                const Real *ra = GasTab<Real>::ptr(W) + S.gtab_off + (size_t)pt.k * S.gtab_ld;
                const Real xa = ra[e.j], xb = ra[S.gtab_ld + e.j];
                Real xs = pt.region == 2 ? xb : xa + pt.f * (xb - xa);
                xs = E < pick<Real>(ch.th, ch.th_f) ? Real(0) : xs;
                Real Pj = xs * u * n1;
                if (Pj > Real(1)) {
                    atomicAdd(&s_ev[C_VIOL_PAIR], 1u);
                    Pj = Real(1);
                }
                if (unif<Real>(b.x) < Pj) {
                    atomicAdd(&s_ev[C_EVENTS + ch.reaction], 1u);
                    Real nd[3], nd2[3] = {Real(0), Real(0), Real(1)};
                    iso_dir<Real>(unif<Real>(b.y), unif<Real>(b.z), nd);
                    if (ch.reaction == 18) {
                        const uint4 e2 = rng_block(Dd.seed, Dd.discharge, s, 6, kk, 4u * gen + 2u, step, (unsigned)rel);
                        iso_dir<Real>(unif<Real>(e2.x), unif<Real>(e2.y), nd2);
                    }
                    GasProducts<Real> pr;
                    Real vo[3];
                    Real um;
                    int bk, breg;
                    if (gas_event<Real>(W, Dd, S, ch, v, V, E, nd, nd2, vo, pr)) {
#pragma unroll
                        for (int q = 0; q < 3; ++q) sv[q][local] = vo[q];
                        dsmc_locate<Real>(W, S, vo, um, bk, breg);
                        if (pr.n > 0) {
                            const int i = pb + rel;
                            const int sub = chunk * SUBTILES + local / SUBTILE;
                            const BirthSink<Real> B = birth_sink<Real>(W, Dd, par, sub);
                            for (int q = 0; q < pr.n; ++q)
                                stage_birth<Real>(B, ((local % SUBTILE) << 1) | pr.prod[q], pr.sp[q], cellA[i], offA[i],
                                                  pr.v[q]);
                        }
                    } else {
                        ssp[local] = (signed char)pr.sp[0];
#pragma unroll
                        for (int q = 0; q < 3; ++q) sv[q][local] = pr.v[0][q];
                        sgen[local] = (unsigned char)(gen + 1u);
                        dsmc_locate<Real>(W, Dd.sp[pr.sp[0]], pr.v[0], um, bk, breg);
                    }
                    sumax[local] = um;
                    sk[local] = (unsigned short)bk;
                    sreg[local] = (unsigned char)breg;
                }
            }
            // on to the next channel that may take what the particle is now
            const int sp = ssp[local];
            for (++kk; kk < kend; ++kk) {
                const DsmcCh e = Dd.dsmc[kk];
                if (e.sp != sp) continue;
                ++ntest;
                if (maybe(local, kk, e)) {
                    skk[local] = (unsigned char)kk;
                    sq[(round + 1) & 1][atomicAdd(&s_qn[(round + 1) % 3], 1u)] = (unsigned short)local;
                    break;
                }
            }
        }
    }
    if (ntest) atomicAdd(&s_ev[C_PEVAL], ntest);
    // write back: the first particle's new velocity, or its removal and the
    // product that ends its chain; part 0 raises the species' recorded
    // largest speed (the particle-target pass that follows bounds P with it)
    Real m2 = Real(0);
    for (int local = tid; local < CHUNK; local += DSMC_THREADS) {
        const int rel = rel0 + local;
        if (rel >= C.n) break;
        const int i = pb + rel;
        const int c = cellA[i];
        if (c < 0) continue;
        const Real v[3] = {sv[0][local], sv[1][local], sv[2][local]};
        if (sgen[local] == 0) {
            vxA[i] = v[0];
            vyA[i] = v[1];
            vzA[i] = v[2];
            m2 = fmax(m2, Real(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]));
        } else {
            const Real off = offA[i];
            cellA[i] = -1;
            deposit_global(acc_global<Real>(W) + (size_t)s * W.total_nodes + Dd.gbase, c, off, -1);
            const int sub = chunk * SUBTILES + local / SUBTILE;
            const BirthSink<Real> B = birth_sink<Real>(W, Dd, par, sub);
            stage_birth<Real>(B, ((local % SUBTILE) << 1) | 1, ssp[local], c, off, v);
        }
    }
    if (part == 0) vmax_raise(W.vmax2, ds, (double)m2);
    __syncthreads();
    for (int k = tid; k < C_NCOUNT; k += DSMC_THREADS)
        if (s_ev[k]) atomicAdd(&W.counters[(size_t)d * C_NCOUNT + k], (unsigned long long)s_ev[k]);
}

template <typename Real>
static size_t push_smem_bytes(int Nmax, int eedf_max, int fm_max, int nw, int qcap, bool cells)
{
    size_t b = sizeof(unsigned long long) * (Nmax + 2) + sizeof(typename FieldT<Real>::T) * (Nmax + 2);
    if (sizeof(Real) == 8) b += sizeof(double) * 2 * FLOOR_MAX;
    b += sizeof(int) * nw * qcap;  // candidate slots
    b += sizeof(unsigned) * (eedf_max + fm_max);
    b += (size_t)nw * qcap;        // candidate energy bins
    b = (b + 15) & ~size_t(15);
    if (cells) b += sizeof(Real) * (Nmax + 2);  // particles per cell; FP64: and the third word
    return (b + 15) & ~size_t(15);
}

// The push's launch shapes (threads per block, slots per thread, blocks per
// SM the registers are sized for): the FP32 path has several for the
// autotuner, the FP64 path one.  Results do not depend on the shape (exact
// integer charge sums, births in parent order).
using PushF0 = PushShape<256, 4, 3>;
using PushF1 = PushShape<128, 4, 6>;
using PushF2 = PushShape<512, 4, 1>;
using PushF3 = PushShape<128, 8, 4>;
using PushF4 = PushShape<256, 8, 2>;
// (FP64: one block of 16 warps per SM, so that its field and sums are held once:
// 32 bytes per cell, with room for the histograms)
using PushD0 = PushShape<512, 4, 1>;
// Blocks per SM that callers may set in FP64.  One is resident and the default;
// of two the second follows the first (no block waits for another).
constexpr int PUSH_D_BLOCKS = 2;

template <typename Real, typename SH>
static cudaError_t push_shape_setup(LaunchCfg &L, int k)
{
    const size_t sm = push_smem_bytes<Real>(L.maxN, 0, 0, SH::nw, SH::qcap, true);
    const size_t smd = push_smem_bytes<Real>(L.maxN, L.eedf_max, L.fm_max, SH::nw, SH::qcap, sizeof(Real) == 8);
    cudaError_t e = allow_smem(k_push<Real, false, SH>, sm);
    if (e != cudaSuccess) return e;
    e = allow_smem(k_push<Real, true, SH>, smd);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_push<Real, false, SH>, SH::threads, sm);
    if (e != cudaSuccess) return e;
    L.shape_threads[k] = SH::threads;
    L.shape_spt[k] = SH::spt;
    L.shape_max_per_sm[k] = per_sm < 1 ? 1 : per_sm;
    L.shape_smem[k] = sm;
    L.shape_smem_diag[k] = smd;
    return cudaSuccess;
}

cudaError_t push_configure(bool fp64, LaunchCfg &L, int num_sms)
{
    cudaError_t e;
    if (fp64) {
        L.push_nshapes = 1;
        if ((e = push_shape_setup<double, PushD0>(L, 0))) return e;
        L.shape_max_per_sm[0] = std::max(L.shape_max_per_sm[0], PUSH_D_BLOCKS);
    } else {
        L.push_nshapes = 5;
        if ((e = push_shape_setup<float, PushF0>(L, 0))) return e;
        if ((e = push_shape_setup<float, PushF1>(L, 1))) return e;
        if ((e = push_shape_setup<float, PushF2>(L, 2))) return e;
        if ((e = push_shape_setup<float, PushF3>(L, 3))) return e;
        if ((e = push_shape_setup<float, PushF4>(L, 4))) return e;
    }
    L.num_sms = num_sms;
    L.push_shape = 0;
    L.push_max_per_sm = L.shape_max_per_sm[0];
    L.push_per_sm = fp64 ? 1 : L.push_max_per_sm;
    L.push_blocks = num_sms * L.push_per_sm;
    L.push_smem = L.shape_smem[0];
    L.push_smem_diag = L.shape_smem_diag[0];
    L.collide_blocks = num_sms * COLLIDE_PER_SM;
    return cudaSuccess;
}

template <typename Real, typename SH>
static void launch_push_shape(bool diag, const WsPtrs &W, const Pools<Real> &P, int par, const LaunchCfg &L,
                              cudaStream_t st)
{
    const int em = diag ? L.eedf_max : 0, fm = diag ? L.fm_max : 0;
    const size_t sm = diag ? L.push_smem_diag : L.push_smem;
    if (diag)
        launch_k(k_push<Real, true, SH>, L.push_blocks, SH::threads, sm, st, W, P, par, L.maxN, em, fm);
    else
        launch_k(k_push<Real, false, SH>, L.push_blocks, SH::threads, sm, st, W, P, par, L.maxN, em, fm);
}

cudaError_t launch_push(bool fp64, bool diag, const WsPtrs &W, const void *pools, int par,
                        const LaunchCfg &L, cudaStream_t st)
{
    if (fp64) {
        launch_push_shape<double, PushD0>(diag, W, *static_cast<const Pools<double> *>(pools), par, L, st);
    } else {
        const Pools<float> &P = *static_cast<const Pools<float> *>(pools);
        switch (L.push_shape) {
        case 1: launch_push_shape<float, PushF1>(diag, W, P, par, L, st); break;
        case 2: launch_push_shape<float, PushF2>(diag, W, P, par, L, st); break;
        case 3: launch_push_shape<float, PushF3>(diag, W, P, par, L, st); break;
        case 4: launch_push_shape<float, PushF4>(diag, W, P, par, L, st); break;
        default: launch_push_shape<float, PushF0>(diag, W, P, par, L, st); break;
        }
    }
    return cudaGetLastError();
}

cudaError_t launch_collide(bool fp64, const WsPtrs &W, const void *pools, int par, int blocks, cudaStream_t st)
{
    if (fp64)
        launch_k(k_collide<double>, blocks, COLLIDE_THREADS, 0, st, W, *static_cast<const Pools<double> *>(pools), par);
    else
        launch_k(k_collide<float>, blocks, COLLIDE_THREADS, 0, st, W, *static_cast<const Pools<float> *>(pools), par);
    return cudaGetLastError();
}

cudaError_t launch_dsmc(bool fp64, const WsPtrs &W, const void *pools, int par, int part, cudaStream_t st)
{
    if (fp64)
        launch_k(k_dsmc<double>, W.max_chunks, DSMC_THREADS, 0, st, W, *static_cast<const Pools<double> *>(pools), par,
                 part);
    else
        launch_k(k_dsmc<float>, W.max_chunks, DSMC_THREADS, 0, st, W, *static_cast<const Pools<float> *>(pools), par,
                 part);
    return cudaGetLastError();
}

} // namespace o2
