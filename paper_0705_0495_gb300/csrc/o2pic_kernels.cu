// o2pic_kernels.cu -- field solve, cell sort, particle-target pass, load and
// deposit kernels of libo2pic (GB300, sm_103a).
#include <cooperative_groups.h>

#include <climits>
#include <mutex>

#include "o2pic_launch.h"

namespace o2 {

constexpr double QE_ = 1.602176634e-19;

// ------------------------------------------------------------ helpers

template <typename Real> struct AccK;
template <> struct AccK<float> {
    using T = unsigned long long;
    static __device__ __forceinline__ T *ptr(const WsPtrs &W) { return W.acc_fix; }
};
template <> struct AccK<double> {
    using T = double;
    static __device__ __forceinline__ T *ptr(const WsPtrs &W) { return W.acc_dbl; }
};

__device__ __forceinline__ void dep_global(unsigned long long *acc, int c, float off, int sign)
{
    unsigned w1 = __float2uint_rn(off * (float)(1 << FIX_BITS));
    unsigned w0 = (1u << FIX_BITS) - w1;
    unsigned long long a = w0, b = w1;
    if (sign < 0) { a = 0ull - a; b = 0ull - b; }
    atomicAdd(&acc[c], a);
    atomicAdd(&acc[c + 1], b);
}
__device__ __forceinline__ void dep_global(double *acc, int c, double off, int sign)
{
    atomicAdd(&acc[c], sign * (1.0 - off));
    atomicAdd(&acc[c + 1], sign * off);
}

// exclusive scan of a[0..M) in shared memory by one block; returns the total
__device__ int block_scan_exclusive_int(int *a, int M, int *wsum)
{
    const int NT = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int per = (M + NT - 1) / NT;
    const int lo = tid * per, hi = min(M, lo + per);
    int run = 0;
    for (int i = lo; i < hi; ++i) {
        const int v = a[i];
        a[i] = run;
        run += v;
    }
    int v = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    if (lane == 31) wsum[warp] = v;
    __syncthreads();
    if (warp == 0) {
        int w = lane < NT / 32 ? wsum[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += t;
        }
        if (lane < NT / 32) wsum[lane] = w;
    }
    __syncthreads();
    const int excl = v - run + (warp > 0 ? wsum[warp - 1] : 0);
    for (int i = lo; i < hi; ++i) a[i] += excl;
    const int total = wsum[NT / 32 - 1];
    __syncthreads();
    return total;
}

// ------------------------------------------------------------ field

// Per discharge: densities from the accumulators, Poisson with
// phi_0 = U_rf sin(2 pi f t + phase), phi_N = 0, and the node field.
// The tridiagonal system (phi_{i-1} - 2 phi_i + phi_{i+1}) = -s_i,
// s_i = rho_i dx^2/eps0, is solved exactly by prefix sums.  With the net
// charge q_i of node i (interior nodes only), S1_i = sum_{k<=i} q_k and
// S2_i = sum_{m<=i} S1_m (i >= 1):
//   s_i = K dx q_i,  phi_i = phi_0 + i D0 - K dx S2_{i-1},
//   D0 = (K dx S2_{N-1} - phi_0)/N  (phi_N = 0),  S2_{N-1} = sum (N - i) q_i,
//   E_i = (K/2) T_i - D0/dx,  T_i = S1_i + S1_{i-1} inside,
//   T_0 = -2 q_0, T_N = 2 (S1_{N-1} + q_N)  (Gauss's law on the half cells),
// with K = e w / eps0 per unit of q.
//
// What bounds it: latency (a chain of a few loads, two scans and thread 0's
// FP64 divisions), and in FP64 the few FP64 units of the one SM that solved a
// discharge.  So a discharge of
// more than FIELD_ONE cells is solved by a cluster of FIELD_CLUSTER blocks,
// which exchange their two sums through distributed shared memory once; the
// weighted sum S2_{N-1} needs no prefix, so D0 is ready together with the
// prefixes; E comes from T_i alone, and densities, potential and FP64 field
// are formed only when they are asked for (diagnostics, pic_fields).  The tile
// table of the push (below) is built by one more block at the same time.
// Kernel time with one block and full sums always -> this: 4096 cells FP32
// 18.3 -> 8.3 us, FP64 62 -> 10.4 us; 128 cells FP64 13.5 -> 6.6 us; seven
// discharges FP32 12.6 -> 5.6 us, 64 discharges 55 -> 7.3 us.
// Why the line lies at 1024 cells (a whole time step, one block / a cluster, one
// discharge, FP32 and FP64): 256 cells 15.9 / 16.5 and 28.6 / 29.9 us, 512 cells
// 16.8 / 17.1 and 29.5 / 30.2, 1024 cells 17.8 / 17.3 and 31.5 / 30.4; seven
// discharges of 1024 cells 18.9 / 18.8 and 37.1 / 36.1, 64 of them 25.0 / 32.4 and
// 50.7 / 60.8.
constexpr int FIELD_THREADS = 256;
constexpr int FIELD_CLUSTER = 8;
constexpr int FIELD_ONE = 1024;  // nodes up to which one block per discharge is used
constexpr int FIELD_PER = 5;     // most nodes per thread
static_assert(FIELD_PER * FIELD_THREADS >= FIELD_ONE + 1 && FIELD_PER * FIELD_THREADS * FIELD_CLUSTER >= 4097, "");

// The sums of a block's nodes, in the units of the accumulators: exact
// integers (2^-FIX_BITS of a particle) in the FP32 path, doubles in the FP64
// path.  Sum1 holds S1 and q, Sum2 holds S2.
template <typename Real> struct FieldSum;
template <> struct FieldSum<float> {
    using S1 = long long;
    using S2 = __int128;
    static __device__ __forceinline__ S1 load(unsigned long long v) { return (long long)v; }
    static __device__ __forceinline__ S2 weigh(int w, S1 q) { return (S2)w * (S2)q; }
    static __device__ __forceinline__ S2 up(S2 v, int o)
    {
        const unsigned long long lo = __shfl_up_sync(0xffffffffu, (unsigned long long)v, o);
        const long long hi = __shfl_up_sync(0xffffffffu, (long long)(v >> 64), o);
        return ((S2)hi << 64) | (S2)lo;
    }
};
template <> struct FieldSum<double> {
    using S1 = double;
    using S2 = double;
    static __device__ __forceinline__ S1 load(double v) { return v; }
    static __device__ __forceinline__ S2 weigh(int w, S1 q) { return (double)w * q; }
    static __device__ __forceinline__ S2 up(S2 v, int o) { return __shfl_up_sync(0xffffffffu, v, o); }
};

template <typename Real>
__device__ __forceinline__ void field_block(const WsPtrs &W, int par, int diag, int mode, int csize, int d, int rank)
{
    namespace cg = cooperative_groups;
    using Acc = typename AccK<Real>::T;
    using F = FieldSum<Real>;
    using S1t = typename F::S1;
    using S2t = typename F::S2;
    constexpr int NW = FIELD_THREADS / 32;
    constexpr bool EXACT = sizeof(Real) == 4;
    __shared__ S1t w1[NW];                     // warp totals
    __shared__ S2t w2[NW], w3[NW];
    __shared__ S1t c1[FIELD_CLUSTER];          // block totals of the cluster
    __shared__ S2t c2[FIELD_CLUSTER], c3[FIELD_CLUSTER];
    __shared__ double s_phi0, s_D0, s_e0;
    __shared__ long long s_T0i;
    __shared__ float s_hKf, s_frf;
    __shared__ int s_intE;
    Ctl *ctl = W.ctl;
    const unsigned long long step = ctl->step[par];
    // every block of the cluster has started before another writes to its
    // shared memory (waited for there)
    if (csize > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    const Disc &Dd = W.disc[d];
    const int N = Dd.N, g = Dd.gbase, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tn = W.total_nodes;
    const double dx = Dd.dx;
    const bool full = diag || mode != 0;
    // nodes lo .. hi-1 of this thread: blocked, so that its prefix is local
    const int NC = (N + 1 + csize - 1) / csize;
    const int per = (NC + FIELD_THREADS - 1) / FIELD_THREADS;
    const int lo = min(rank * NC + tid * per, N + 1);
    const int hi = min(min(lo + per, (rank + 1) * NC), N + 1);
    Acc *acc = AccK<Real>::ptr(W) + g;
    Acc raw[NSP][FIELD_PER];
#pragma unroll
    for (int k = 0; k < FIELD_PER; ++k)
#pragma unroll
        for (int s = 0; s < NSP; ++s) raw[s][k] = lo + k < hi ? acc[(size_t)s * tn + lo + k] : Acc(0);
    // the drive's potential by one thread, of the warp with the fewest nodes,
    // while the loads are in flight (the FP64 sine takes about 1.5 us)
    if (tid == FIELD_THREADS - 1) s_phi0 = Dd.U_rf * sin(Dd.omega * ((double)step * Dd.dt) + Dd.phase);
    bool clear[NSP];
#pragma unroll
    for (int s = 0; s < NSP; ++s) clear[s] = mode == 0 && !species_rests(Dd, s, step);
    S1t q[FIELD_PER];     // net charge of the node
    S1t run = S1t(0);     // the thread's interior charge
    S2t part = S2t(0);    // sum of (N - i) q_i over the thread's interior nodes
#pragma unroll
    for (int k = 0; k < FIELD_PER; ++k) {
        const int i = lo + k;
        q[k] = S1t(0);
        if (i >= hi) continue;
        S1t a[NSP];
#pragma unroll
        for (int s = 0; s < NSP; ++s) {
            a[s] = F::load(raw[s][k]);
            if (clear[s]) acc[(size_t)s * tn + i] = Acc(0);
        }
        q[k] = a[2] - a[0] - a[1];
        if (i > 0 && i < N) {
            run += q[k];
            part += F::weigh(N - i, q[k]);
        }
        if (full) {
            if constexpr (EXACT) {
                const double sc = (i == 0 || i == N) ? Dd.dens_fix_wall : Dd.dens_fix;
#pragma unroll
                for (int s = 0; s < NSP; ++s) {
                    const size_t j = (size_t)s * tn + g + i;
                    if (diag) W.dens_sum_fix[j] += a[s];  // exact sums; scaled at read-out
                    W.dens[j] = (double)a[s] * sc;
                }
                W.rho[g + i] = QE_ * (double)q[k] * sc;
            } else {
                const double sc = Dd.weight / ((i == 0 || i == N) ? 0.5 * dx : dx);
                double dn[NSP];
#pragma unroll
                for (int s = 0; s < NSP; ++s) {
                    const size_t j = (size_t)s * tn + g + i;
                    dn[s] = a[s] * sc;
                    W.dens[j] = dn[s];
                    if (diag) W.dens_sum[j] += dn[s];
                }
                W.rho[g + i] = QE_ * (dn[2] - dn[0] - dn[1]);
            }
        }
    }
    // inclusive scan of the threads' charge, sum of their weighted charge
    S1t v = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const S1t x = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += x;
    }
    S2t r = part;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const S2t x = F::up(r, o);
        if (lane >= o) r += x;
    }
    if (lane == 31) {
        w1[warp] = v;
        w2[warp] = r;
    }
    __syncthreads();
    S1t excl = v - run;  // charge of the nodes before this thread's
    for (int w = 0; w < warp; ++w) excl += w1[w];
    if (csize > 1) {
        cg::cluster_group cl = cg::this_cluster();
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (tid < csize) {
            S1t t1 = w1[0];
            S2t t2 = w2[0];
            for (int w = 1; w < NW; ++w) {
                t1 += w1[w];
                t2 += w2[w];
            }
            *cl.map_shared_rank(&c1[rank], tid) = t1;
            *cl.map_shared_rank(&c2[rank], tid) = t2;
        }
        cl.sync();
        for (int c = 0; c < rank; ++c) excl += c1[c];
    }
    // K dx and D0, in the order of the formulas above
    const double K = EXACT ? Dd.Kfix : Dd.Kone;
    if (tid == 0) {
        S2t tot = S2t(0);
        if (csize > 1)
            for (int c = 0; c < csize; ++c) tot += c2[c];
        else
            for (int w = 0; w < NW; ++w) tot += w2[w];
        const double phi0 = s_phi0;
        const double D0 = (K * dx * (double)tot - phi0) / (double)N;
        s_D0 = D0;
        if constexpr (EXACT) {
            // E_i = (K/2) (T_i - T0) with T0 = 2 D0 / (K dx): T_i - round(T0) is
            // exact, so E leaves FP64 only through O(1) constants
            const double T0 = 2.0 * D0 / (K * dx);
            s_intE = (K > 0.0 && fabs(T0) < 4.0e18) ? 1 : 0;
            const long long T0i = s_intE ? llround(T0) : 0;
            s_T0i = T0i;
            s_hKf = (float)(0.5 * K);
            s_frf = (float)(T0 - (double)T0i);
        } else {
            s_e0 = D0 / dx;
        }
        if (diag && rank == 0) {
            if constexpr (EXACT) {
                W.phi0_sum[d] += phi0;
                W.D0_sum[d] += D0;
            }
            W.nsamp[d] += 1ull;
        }
    }
    __syncthreads();
    const double D0 = s_D0;
    Real *Er = reinterpret_cast<Real *>(W.Ereal) + g;
    S1t s1 = excl;
    S2t sum = S2t(0);  // the thread's share of S2
#pragma unroll
    for (int k = 0; k < FIELD_PER; ++k) {
        const int i = lo + k;
        if (i >= hi) break;
        S1t T;
        if (i == 0) T = -(q[k] + q[k]);
        else if (i == N) T = (s1 + q[k]) + (s1 + q[k]);
        else {
            T = s1 + s1 + q[k];
            s1 += q[k];
            sum += (S2t)s1;
        }
        if constexpr (EXACT) {
            if (s_intE) {
                const long long dT = T - s_T0i;
                Er[i] = s_hKf * (__ll2float_rn(dT) - s_frf);
                if (full) W.Efield[g + i] = 0.5 * K * ((double)dT - (double)s_frf);
            } else {  // no charge or an extreme field: evaluate in FP64
                const double E = -D0 / dx + 0.5 * K * (double)T;
                Er[i] = (Real)E;
                if (full) W.Efield[g + i] = E;
            }
        } else {
            const double E = (0.5 * K) * T - s_e0;
            Er[i] = E;
            if (full) W.Efield[g + i] = E;
        }
    }
    if (!full) return;
    // potential: the prefix of S2 over threads, warps and blocks, and its sums
    S2t pv = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const S2t x = F::up(pv, o);
        if (lane >= o) pv += x;
    }
    if (lane == 31) w3[warp] = pv;
    __syncthreads();
    S2t before = pv - sum;
    for (int w = 0; w < warp; ++w) before += w3[w];
    if (csize > 1) {
        cg::cluster_group cl = cg::this_cluster();
        if (tid < csize) {
            S2t t = w3[0];
            for (int w = 1; w < NW; ++w) t += w3[w];
            *cl.map_shared_rank(&c3[rank], tid) = t;
        }
        cl.sync();
        for (int c = 0; c < rank; ++c) before += c3[c];
    }
    const double phi0 = s_phi0;
    s1 = excl;
#pragma unroll
    for (int k = 0; k < FIELD_PER; ++k) {
        const int i = lo + k;
        if (i >= hi) break;
        double p;
        if (i == 0) p = phi0;
        else if (i == N) p = 0.0;
        else {
            // before = S2_{i-1}
            p = phi0 + (double)i * D0 - K * dx * (double)before;
            if constexpr (EXACT) {
                if (diag) W.phi_s2_sum[g + i] += before;
            }
            s1 += q[k];
            before += (S2t)s1;
        }
        W.phi[g + i] = p;
        if constexpr (!EXACT) {
            if (diag) W.phi_sum[g + i] += p;
        }
    }
}

// Births staged in the step of parity par, per (discharge, product species), for
// a whole block (in shared memory).
__device__ __forceinline__ const int *staged_births(const WsPtrs &W, int par)
{
    __shared__ int s_add[MAX_DISCHARGES * NSP];
    const Counts *tab = W.tab + (par ? W.D * NSP : 0);
    const int *words = birth_words(W, par);
    const int n = (W.ctl->tab_total[par] * SUBTILES + BIRTHS_TILES - 1) / BIRTHS_TILES * NSP;
    for (int k = threadIdx.x; k < W.D * NSP; k += blockDim.x) s_add[k] = 0;
    __syncthreads();
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        const int v = words[k];
        if (v == 0) continue;
        const int tile = k / NSP * TILE_ALIGN;
        int lo = 0, hi = W.D;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (tab[mid * NSP].chunk0 <= tile) lo = mid; else hi = mid;
        }
        atomicAdd(&s_add[lo * NSP + k % NSP], v);
    }
    __syncthreads();
    return s_add;
}

// Tile table for the step of parity par: tiles of each discharge start at a
// multiple of TILE_ALIGN, so that the birth-append blocks never span two, and
// those of each species at a multiple of TILES_PER_TICKET, so that a push
// ticket never spans two; the step's birth counts are cleared and the smallest
// room of a species is noted.  With `advance`
// the next step's counter is set and the candidate list emptied.  The counts
// are the current ones, or (after_births) those that the births of the step
// before will leave: its table's counts plus what staging has counted.
// One thread per discharge and a block scan over them (one thread walking the
// list took 0.25 us per entry: 50 us of every step of 64 discharges).
__device__ void tile_table(const WsPtrs &W, int par, unsigned long long step, bool advance, bool after_births)
{
    __shared__ int s_warp[32], s_room;
    Ctl *ctl = W.ctl;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NT = blockDim.x;
    constexpr int A = TILE_ALIGN, B = TILES_PER_TICKET;
    const Counts *old = W.tab + (par ? 0 : W.D * NSP);  // the table of the other parity
    Counts *keep = W.tab + (par ? W.D * NSP : 0);
    const int *add = after_births ? staged_births(W, par ^ 1) : nullptr;
    if (tid == 0) s_room = INT_MAX;
    int first = 0;  // tiles of the discharges before this pass
    for (int d0 = 0; d0 < W.D; d0 += NT) {
        const int d = d0 + tid;
        int n[NSP] = {0, 0, 0}, at[NSP], end = 0;
        if (d < W.D) {
#pragma unroll
            for (int s = 0; s < NSP; ++s)
                n[s] = after_births ? min(old[d * NSP + s].n_snap + add[d * NSP + s], W.disc[d].cap[s])
                                    : W.cnt[d * NSP + s].n;
        }
#pragma unroll
        for (int s = 0; s < NSP; ++s) {
            at[s] = (end + B - 1) / B * B;
            end = at[s] + (n[s] + CHUNK - 1) / CHUNK;
        }
        const int size = d < W.D ? (end + A - 1) / A * A : 0;
        int v = size;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += x;
        }
        __syncthreads();  // s_warp of the pass before has been read
        if (lane == 31) s_warp[warp] = v;
        int room = INT_MAX;
        if (d < W.D)
#pragma unroll
            for (int s = 0; s < NSP; ++s) room = min(room, W.disc[d].cap[s] - n[s]);
        room = __reduce_min_sync(0xffffffffu, room);
        if (lane == 0) atomicMin(&s_room, room);
        __syncthreads();
        int start = first + v - size;
        for (int w = 0; w < warp; ++w) start += s_warp[w];
        for (int w = 0; w < NT / 32; ++w) first += s_warp[w];
        if (d < W.D) {
#pragma unroll
            for (int s = 0; s < NSP; ++s) {
                const Counts c{n[s], n[s], start + at[s], (n[s] + CHUNK - 1) / CHUNK};
                W.cnt[d * NSP + s] = c;
                keep[d * NSP + s] = c;
            }
            if (d == W.D - 1) {
                int chunk = start + end;
                if (chunk > W.max_chunks) {
                    set_status(ctl, ST_CAPACITY);
                    chunk = 0;
                }
                ctl->total_chunks = chunk;
                ctl->tab_total[par] = chunk;
                ctl->ticket = 0u;
                ctl->room[par] = s_room;
                ctl->births[par] = 0;
                if (advance) {
                    ctl->cand_n = 0u;
                    ctl->step[par ^ 1] = step + 1ull;
                }
            }
        }
    }
    int *mine = birth_words(W, par);
    for (int k = tid; k < (W.max_chunks / TILE_ALIGN + 1) * NSP; k += NT) mine[k] = 0;
}

__global__ void __launch_bounds__(256) k_retile(WsPtrs W, int par)
{
    pdl_wait();
    tile_table(W, par, 0ull, false, false);
}

// The field of every discharge, and (mode 0) by one more cluster the step's
// tile table and the step counter.
template <typename Real>
__global__ void __launch_bounds__(FIELD_THREADS)
k_field(WsPtrs W, int par, int diag, int mode, int csize)
{
    pdl_wait();
    const int d = blockIdx.x / csize, rank = blockIdx.x % csize;
    if (d < W.D)
        field_block<Real>(W, par, diag, mode, csize, d, rank);
    else if (rank == 0)
        tile_table(W, par, W.ctl->step[par], true, false);
}

// Births of one step appended after the survivors, per discharge and
// product species in tile order (tiles are numbered in (parent species,
// slot) order), i.e. in parent order (staging has deposited their charge).  A
// block takes BIRTHS_TILES consecutive sub-tiles, two per thread.  Staging has
// counted the births of every block by product species (birth_blk), so a
// block's place among the blocks of its discharge is the sum of the earlier
// ones' counts: nothing waits, and a block without births ends at once (the
// one with the discharge's last sub-tile sets the slot counts).  When the
// blocks published totals and read those of their predecessors as these
// arrived: 5e7 superparticles 20 us, 9.7 us here; 4e6 8.5 us, 5.8 us here.
// The sub-tiles' record counts are cleared as they are read, for the next use.
template <typename Real>
__device__ __forceinline__ void births_block(const WsPtrs &W, const Pools<Real> &P, int par, int blk, bool set_counts)
{
    constexpr int NW = FIELD_THREADS / 32, TPT = BIRTHS_TILES / FIELD_THREADS;  // sub-tiles per thread
    __shared__ int wsum[NSP][NW];
    __shared__ int s_excl[NSP];
    __shared__ unsigned s_part[NSP][NW];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    Ctl *ctl = W.ctl;
    const Counts *tab = W.tab + (par ? W.D * NSP : 0);
    const int *words = birth_words(W, par);
    int own[NSP];  // the block's births
#pragma unroll
    for (int q = 0; q < NSP; ++q) own[q] = words[(size_t)blk * NSP + q];
    const int total = ctl->tab_total[par] * SUBTILES;  // sub-tiles
    if (blk * BIRTHS_TILES >= total) return;
    // discharge of the block: every discharge's tiles start at a multiple of
    // BIRTHS_TILES sub-tiles, so a block never spans two discharges
    int d = 0;
    {
        int lo = 0, hi = W.D;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (tab[mid * NSP].chunk0 * SUBTILES <= blk * BIRTHS_TILES) lo = mid; else hi = mid;
        }
        d = lo;
    }
    const Counts last_sp = tab[d * NSP + 2];
    const int T1 = (last_sp.chunk0 + last_sp.nchunk) * SUBTILES;  // end of the discharge's sub-tiles
    const bool last = set_counts && T1 > blk * BIRTHS_TILES && T1 <= (blk + 1) * BIRTHS_TILES;
    const int any = own[0] + own[1] + own[2];
    if (!last && any == 0) return;
    // births of the discharge's earlier blocks, three words each
    {
        const int first_blk = tab[d * NSP].chunk0 * SUBTILES / BIRTHS_TILES;
        const int npred = (blk - first_blk) * NSP;
        unsigned part[NSP] = {0u, 0u, 0u};
        for (int k = tid; k < npred; k += FIELD_THREADS) {
            const unsigned a = (unsigned)words[(size_t)first_blk * NSP + k];
            const int q = k % NSP;
#pragma unroll
            for (int r = 0; r < NSP; ++r) part[r] += r == q ? a : 0u;
        }
#pragma unroll
        for (int q = 0; q < NSP; ++q) {
            const unsigned v = __reduce_add_sync(0xffffffffu, part[q]);
            if (lane == 0) s_part[q][warp] = v;
        }
        __syncthreads();
        if (tid < NSP) {
            unsigned ex = 0;
            for (int w = 0; w < NW; ++w) ex += s_part[tid][w];
            s_excl[tid] = (int)ex;
            if (last) {
                const long long nn = (long long)tab[d * NSP + tid].n_snap + ex + words[(size_t)blk * NSP + tid];
                W.cnt[d * NSP + tid].n = (int)(nn < W.disc[d].cap[tid] ? nn : W.disc[d].cap[tid]);
            }
        }
    }
    if (any == 0) return;
    const BirthRec<Real> *rec0 = reinterpret_cast<const BirthRec<Real> *>(W.births);
    const int t0 = blk * BIRTHS_TILES + tid * TPT;
    int mine[NSP] = {0, 0, 0}, nrec[TPT];
#pragma unroll
    for (int j = 0; j < TPT; ++j) {
        const int t = t0 + j;
        nrec[j] = 0;  // records of the sub-tile (any order; the tag gives species and parent order)
        if (t < total && t < T1) {
            nrec[j] = min(W.tile_cnt[t], W.birth_cap);
            if (nrec[j]) W.tile_cnt[t] = 0;
            for (int r = 0; r < nrec[j]; ++r) ++mine[rec0[(size_t)t * W.birth_cap + r].tag & 3];
        }
    }
    int excl[NSP];
#pragma unroll
    for (int q = 0; q < NSP; ++q) {
        int v = mine[q];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += x;
        }
        if (lane == 31) wsum[q][warp] = v;
        excl[q] = v - mine[q];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NSP; ++q)
        for (int w = 0; w < warp; ++w) excl[q] += wsum[q][w];
    const Disc &Dd = W.disc[d];
    const unsigned b0 = ctl->cur ? P.stride : 0u;
    typename AccK<Real>::T *acc = AccK<Real>::ptr(W) + Dd.gbase;
#pragma unroll
    for (int j = 0; j < TPT; ++j) {
        const BirthRec<Real> *rec = rec0 + (size_t)(t0 + j) * W.birth_cap;
        // a record's place among its species: the number of that species'
        // records with a smaller tag (parent slot, then product)
        for (int r = 0; r < nrec[j]; ++r) {
            const BirthRec<Real> &b = rec[r];
            const int q = b.tag & 3;
            int rank = 0;
            for (int k = 0; k < nrec[j]; ++k) {
                const int tk = rec[k].tag;
                rank += (tk & 3) == q && tk < b.tag;
            }
            const long long dst = (long long)tab[d * NSP + q].n_snap + s_excl[q] + excl[q] + rank;
            if (dst >= Dd.cap[q]) {  // dropped, with the charge that staging deposited
                set_status(ctl, ST_CAPACITY);
                dep_global(acc + (size_t)q * W.total_nodes, b.c, b.off, -1);
                continue;
            }
            const size_t g = (size_t)b0 + Dd.pbase[q] + (size_t)dst;
            P.cell[0][g] = b.c;
            P.off[0][g] = b.off;
            P.vx[0][g] = b.vx;
            P.vy[0][g] = b.vy;
            P.vz[0][g] = b.vz;
        }
        for (int r = 0; r < nrec[j]; ++r) {
            const int q = rec[r].tag & 3;
#pragma unroll
            for (int p = 0; p < NSP; ++p) excl[p] += p == q ? 1 : 0;
        }
    }
}

template <typename Real>
__global__ void __launch_bounds__(FIELD_THREADS)
k_births(WsPtrs W, Pools<Real> P, int par)
{
    pdl_wait();
    births_block<Real>(W, P, par, blockIdx.x, true);
}

// The births of the step of parity par and, between two steps without a sort,
// the next step's field and tile table in the same launch: the field needs the
// births' charge (deposited when they were staged) and the table their numbers
// (counted then), not the append itself.  Both are chains of latencies: 5.5 and
// 5.6 us one after the other for seven small discharges, 6.2 us together; 9.7 and
// 8.3 us for one of 5e7 superparticles, 9.2 together.
// When a species has more births than room (an error that the call reports),
// the field has to wait for the append, which drops some and takes their charge
// back: the first cluster then does one after the other, for all discharges.
__device__ __noinline__ bool births_overflow(const WsPtrs &W, int par)
{
    const int *add = staged_births(W, par);
    const Counts *tab = W.tab + (par ? W.D * NSP : 0);
    bool over = false;
    for (int k = threadIdx.x; k < W.D * NSP; k += blockDim.x)
        over |= (long long)tab[k].n_snap + add[k] > W.disc[k / NSP].cap[k % NSP];
    return __syncthreads_or(over);
}
template <typename Real>
__device__ __noinline__ void births_then_field(const WsPtrs &W, const Pools<Real> &P, int par, int diag, int csize, int rank)
{
    for (int blk = rank; blk <= W.max_chunks / TILE_ALIGN; blk += csize) {
        births_block<Real>(W, P, par, blk, true);
        __syncthreads();
    }
    __threadfence();
    cooperative_groups::this_cluster().sync();
    for (int d = 0; d < W.D; ++d) {
        field_block<Real>(W, par ^ 1, diag, 0, csize, d, rank);
        __syncthreads();
    }
    if (rank == 0) tile_table(W, par ^ 1, W.ctl->step[par ^ 1], true, false);
}
template <typename Real>
__global__ void __launch_bounds__(FIELD_THREADS)
k_births_field(const __grid_constant__ WsPtrs W, const __grid_constant__ Pools<Real> P, int par, int diag, int csize)
{
    pdl_wait();
    const int d = blockIdx.x / csize, rank = blockIdx.x % csize;
    // counted per species only when all births together could be too many for one
    if (W.ctl->room[par] < W.ctl->births[par] && births_overflow(W, par)) {
        if (d == 0) births_then_field<Real>(W, P, par, diag, csize, rank);
        return;
    }
    if (d < W.D) {
        field_block<Real>(W, par ^ 1, diag, 0, csize, d, rank);
    } else if (d == W.D) {
        if (rank == 0) tile_table(W, par ^ 1, W.ctl->step[par ^ 1], true, true);
    } else {
        const int blk = blockIdx.x - (W.D + 1) * csize;
        if (blk <= W.max_chunks / TILE_ALIGN) births_block<Real>(W, P, par, blk, false);
    }
}

// ------------------------------------------------------------- sort

// block -> (ds, index of the block within ds) from a host-built table
__device__ __forceinline__ void sort_block(const int *tab, int &ds, int &bi)
{
    ds = tab[2 * blockIdx.x];
    bi = tab[2 * blockIdx.x + 1];
}

// Histogram of cells (dead slots in bucket N) of one block of SORT_CHUNK
// slots, one per warp (SORT_WARP_SLOTS slots, 16-bit counts): the warps'
// rows go to sort_whist for the scatter, their sum to row bi of the
// (block x bucket) count matrix of ds.  Each warp reads SORT_ILP slots per
// lane before counting, to keep loads in flight.
template <typename Real>
__global__ void __launch_bounds__(SORT_WARPS * 32)
k_sort_count(WsPtrs W, Pools<Real> P, const int *tab)
{
    pdl_wait();
    extern __shared__ __align__(16) unsigned short wsm[];
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        // the column scan that follows: its warp order and the tag of its words
        W.ctl->colscan_ticket = 0u;
        W.ctl->scatter_done = 0u;
        W.ctl->sort_epoch += 1u;
    }
    int ds, bi;
    sort_block(tab, ds, bi);
    const int d = ds / NSP, s = ds % NSP;
    const Disc &Dd = W.disc[d];
    const int N = Dd.N, n = W.cnt[ds].n;
    const int ws = sort_warp_slots(n, Dd.sort_gmax[s], N);
    const int G = (n + SORT_WARPS * ws - 1) / (SORT_WARPS * ws);
    if (bi == 0 && threadIdx.x == 0) W.vmax2[ds] = 0ull;  // raised by the scatter
    if (bi >= G) return;
    const int stride = (N + 2) & ~1;
    for (int i = threadIdx.x; i < SORT_WARPS * stride; i += blockDim.x) wsm[i] = 0;
    __syncthreads();
    const int *cell = P.cell[W.ctl->cur] + Dd.pbase[s];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    unsigned short *hw = wsm + (size_t)w * stride;
    const int lo = (bi * SORT_WARPS + w) * ws;
    const int hi = min(n, lo + ws);
    for (int i0 = lo; i0 < hi; i0 += 32 * SORT_ILP) {
        int b[SORT_ILP];
#pragma unroll
        for (int r = 0; r < SORT_ILP; ++r) {
            const int i = i0 + r * 32 + lane;
            b[r] = -1;
            if (i < hi) {
                const int c = cell[i];
                b[r] = c < 0 ? N : c;
            }
        }
#pragma unroll
        for (int r = 0; r < SORT_ILP; ++r) {
            // sorted runs: a whole row in one bucket needs no match
            const int b0 = __shfl_sync(0xffffffffu, b[r], 0);
            if (__all_sync(0xffffffffu, b[r] == b0)) {
                if (lane == 0 && b0 >= 0) hw[b0] += (unsigned short)32;
                __syncwarp();
                continue;
            }
            const unsigned peers = __match_any_sync(0xffffffffu, b[r]);
            if (b[r] >= 0 && lane == __ffs(peers) - 1) hw[b[r]] += (unsigned short)__popc(peers);
            __syncwarp();
        }
    }
    __syncthreads();
    int *row = W.sort_counts + Dd.sort_cbase[s] + (size_t)bi * (N + 1);
    unsigned short *wrow = W.sort_whist + ((size_t)Dd.sort_cbase[s] + (size_t)bi * (N + 1)) * SORT_WARPS;
    for (int i = threadIdx.x; i <= N; i += blockDim.x) {
        int t = 0;
#pragma unroll
        for (int q = 0; q < SORT_WARPS; ++q) {
            const unsigned short h = wsm[(size_t)q * stride + i];
            wrow[(size_t)q * (N + 1) + i] = h;
            t += h;
        }
        row[i] = t;
    }
}

// Column scan of the (block x bucket) count matrix: running sums down the
// sort blocks, so that each (block, bucket) entry becomes that block's first
// slot inside the bucket, and the bucket totals in sort_tot.  One warp per
// (d, s, 32 consecutive buckets, COLSCAN_SEG consecutive rows), in the order
// of a ticket: the warp loads its rows (each row's 32 buckets in one 128-byte
// load), publishes their column totals tagged with the sort, adds those of
// the earlier row segments of its buckets (warps with smaller tickets, so
// running or done, which publish before they wait) and writes each entry's
// exclusive prefix; the segment holding the last row writes the totals.
__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__global__ void __launch_bounds__(256)
k_sort_colscan(WsPtrs W, const int *unit_base)
{
    pdl_wait();
    const int lane = threadIdx.x & 31;
    Ctl *ctl = W.ctl;
    int u = 0;
    if (lane == 0) u = (int)atomicAdd(&ctl->colscan_ticket, 1u);
    u = __shfl_sync(0xffffffffu, u, 0);
    const int nds = W.D * NSP;
    if (u >= unit_base[nds]) return;
    int lo = 0, hi = nds;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (unit_base[mid] <= u) lo = mid; else hi = mid;
    }
    const int ds = lo;
    const int d = ds / NSP, s = ds % NSP;
    const Disc &Dd = W.disc[d];
    const int N = Dd.N;
    const int n = W.cnt[ds].n;
    const int chunk = SORT_WARPS * sort_warp_slots(n, Dd.sort_gmax[s], N);
    const int G = (n + chunk - 1) / chunk;
    const int nseg = (Dd.sort_gmax[s] + COLSCAN_SEG - 1) / COLSCAN_SEG;
    const int local = u - unit_base[ds];
    const int grp = local / nseg, sg = local % nseg;
    const int c = grp * 32 + lane;
    const bool valid = c <= N;
    int *cnt = W.sort_counts + Dd.sort_cbase[s];
    const int r0 = sg * COLSCAN_SEG;
    int v[COLSCAN_SEG];
    unsigned tot = 0;
#pragma unroll
    for (int k = 0; k < COLSCAN_SEG; ++k) {
        const int r = r0 + k;
        v[k] = (valid && r < G) ? cnt[(size_t)r * (N + 1) + c] : 0;
        tot += (unsigned)v[k];
    }
    const unsigned long long epoch = ctl->sort_epoch;
    // the words of segments 0 .. nseg-1 of this bucket group, 32 per segment
    unsigned long long *agg = W.colscan_agg + (size_t)(u - sg) * 32;
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(agg + (size_t)sg * 32 + lane),
                 "l"((epoch << 32) | tot) : "memory");
    unsigned pre = 0;
    long long spins = 0;
    bool late = false;
    for (int k0 = 0; k0 < sg && !late; k0 += 8) {
        unsigned long long w[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) w[k] = k0 + k < sg ? ld_relaxed_u64(agg + (size_t)(k0 + k) * 32 + lane) : 0ull;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (k0 + k >= sg) break;
            while ((w[k] >> 32) != (epoch & 0xFFFFFFFFull) && spins <= SPIN_LIMIT) {
                ++spins;
                __nanosleep(64);
                w[k] = ld_relaxed_u64(agg + (size_t)(k0 + k) * 32 + lane);
            }
            if ((w[k] >> 32) != (epoch & 0xFFFFFFFFull)) {
                set_status(ctl, ST_TIMEOUT);
                late = true;
                break;
            }
            pre += (unsigned)(w[k] & 0xFFFFFFFFull);
        }
    }
    unsigned run = pre;
#pragma unroll
    for (int k = 0; k < COLSCAN_SEG; ++k) {
        const int r = r0 + k;
        if (valid && r < G) cnt[(size_t)r * (N + 1) + c] = (int)run;
        run += (unsigned)v[k];
    }
    const int last = G > 0 ? (G - 1) / COLSCAN_SEG : 0;
    if (valid && sg == last) W.sort_tot[Dd.cs_base + s * (N + 2) + c] = (int)run;
}

// Per (d, s): bucket starts (cell_start) by a scan over the bucket totals.
__global__ void __launch_bounds__(512)
k_sort_cellscan(WsPtrs W)
{
    pdl_wait();
    extern __shared__ __align__(16) int isx[];
    __shared__ int wsum[32];
    const int ds = blockIdx.x;
    const int d = ds / NSP, s = ds % NSP;
    const Disc &Dd = W.disc[d];
    const int N = Dd.N, n = W.cnt[ds].n;
    const int *tot_g = W.sort_tot + Dd.cs_base + s * (N + 2);
    int *tot = isx;  // N+1
    for (int c = threadIdx.x; c <= N; c += blockDim.x) tot[c] = n > 0 ? tot_g[c] : 0;
    __syncthreads();
    block_scan_exclusive_int(tot, N + 1, wsum);
    int *cs = W.cell_start + Dd.cs_base + s * (N + 2);
    for (int c = threadIdx.x; c <= N; c += blockDim.x) cs[c] = tot[c];
    if (threadIdx.x == 0) {
        cs[N + 1] = n;
        W.sort_live[ds] = tot[N];  // live slots = start of the dead bucket
    }
}

// The scatter block that comes last makes the sorted buffer and its slot
// counts the current ones (every block has read the old ones by then; the
// count kernel has reset the counter).
__device__ __forceinline__ void sort_finish(const WsPtrs &W)
{
    __shared__ bool s_last;
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&W.ctl->scatter_done, 1u) == gridDim.x - 1u;
    __syncthreads();
    if (!s_last) return;
    for (int ds = threadIdx.x; ds < W.D * NSP; ds += blockDim.x) W.cnt[ds].n = W.sort_live[ds];
    if (threadIdx.x == 0) W.ctl->cur ^= 1;
}

// Stable scatter: warp w of block bi owns the slots from (bi SORT_WARPS + w) ws;
// the per-warp bucket counts (16-bit) that the count kernel kept give each
// warp its first slot per bucket relative to the block's, then each warp
// walks its slots in order, ranking equal buckets inside a 32-slot row by
// lane.  Dead slots (bucket N) are
// dropped.  SORT_ILP rows are loaded before they are ranked.
template <typename Real>
__global__ void __launch_bounds__(SORT_WARPS * 32)
k_sort_scatter(WsPtrs W, Pools<Real> P, const int *tab)
{
    pdl_wait();
    extern __shared__ __align__(16) unsigned short hsm[];
    int ds, bi;
    sort_block(tab, ds, bi);
    const int d = ds / NSP, s = ds % NSP;
    const Disc &Dd = W.disc[d];
    const int N = Dd.N, n = W.cnt[ds].n;
    const int ws = sort_warp_slots(n, Dd.sort_gmax[s], N);
    const int G = (n + SORT_WARPS * ws - 1) / (SORT_WARPS * ws);
    if (bi >= G) {
        sort_finish(W);
        return;
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int stride = (N + 2) & ~1;
    unsigned short *hw = hsm + (size_t)w * stride;
    const int cur = W.ctl->cur, nxt = cur ^ 1;
    const int pb = Dd.pbase[s];
    const int *cell = P.cell[cur] + pb;
    const int lo = (bi * SORT_WARPS + w) * ws;
    const int hi = min(n, lo + ws);
    // per bucket: warp offsets relative to the block's first slot in it, from
    // the warps' counts that the count kernel kept
    const unsigned short *wrow = W.sort_whist + ((size_t)Dd.sort_cbase[s] + (size_t)bi * (N + 1)) * SORT_WARPS;
    for (int c = threadIdx.x; c <= N; c += blockDim.x) {
        unsigned run = 0;
#pragma unroll
        for (int q = 0; q < SORT_WARPS; ++q) {
            const unsigned t = wrow[(size_t)q * (N + 1) + c];
            hsm[(size_t)q * stride + c] = (unsigned short)run;
            run += t;
        }
    }
    __syncthreads();
    const int *base = W.sort_counts + Dd.sort_cbase[s] + (size_t)bi * (N + 1);
    const int *cstart = W.cell_start + Dd.cs_base + s * (N + 2);
    const Real *offS = P.off[cur] + pb, *vxS = P.vx[cur] + pb, *vyS = P.vy[cur] + pb,
               *vzS = P.vz[cur] + pb;
    int *cellD = P.cell[nxt] + pb;
    Real *offD = P.off[nxt] + pb, *vxD = P.vx[nxt] + pb, *vyD = P.vy[nxt] + pb,
         *vzD = P.vz[nxt] + pb;
    const unsigned lt = (1u << lane) - 1u;
    // largest speed^2 of the live particles this lane moves, in the
    // particles' own precision (one conversion at the end: FP64 arithmetic
    // per particle is slow on this part)
    Real vm2 = Real(0);
    for (int i0 = lo; i0 < hi; i0 += 32 * SORT_ILP) {
        int b[SORT_ILP];
        int dst[SORT_ILP];
#pragma unroll
        for (int r = 0; r < SORT_ILP; ++r) {
            const int i = i0 + r * 32 + lane;
            b[r] = -1;
            if (i < hi) {
                const int c = cell[i];
                b[r] = c < 0 ? N : c;
            }
        }
        // every load of the rows' data (read-only path) before the ranks are
        // worked out, so that their latency overlaps that work; the source
        // and destination arrays never overlap
        Real ro[SORT_ILP], rx[SORT_ILP], ry[SORT_ILP], rz[SORT_ILP];
        int gb[SORT_ILP];
#pragma unroll
        for (int r = 0; r < SORT_ILP; ++r) {
            gb[r] = 0;
            if (b[r] >= 0 && b[r] < N) {
                const int i = i0 + r * 32 + lane;
                gb[r] = __ldg(&cstart[b[r]]) + __ldg(&base[b[r]]);
                ro[r] = __ldg(&offS[i]);
                rx[r] = __ldg(&vxS[i]);
                ry[r] = __ldg(&vyS[i]);
                rz[r] = __ldg(&vzS[i]);
            }
        }
#pragma unroll
        for (int r = 0; r < SORT_ILP; ++r) {
            dst[r] = -1;
            const int b0 = __shfl_sync(0xffffffffu, b[r], 0);
            if (__all_sync(0xffffffffu, b[r] == b0)) {
                // a whole row in one bucket: ranks are the lanes
                if (b0 >= 0 && b0 < N) dst[r] = (int)hw[b0] + lane;
                __syncwarp();
                if (lane == 0 && b0 >= 0) hw[b0] += (unsigned short)32;
                __syncwarp();
                continue;
            }
            const unsigned peers = __match_any_sync(0xffffffffu, b[r]);
            if (b[r] >= 0 && b[r] < N) dst[r] = (int)hw[b[r]] + __popc(peers & lt);
            __syncwarp();
            if (b[r] >= 0 && lane == __ffs(peers) - 1) hw[b[r]] += (unsigned short)__popc(peers);
            __syncwarp();
        }
#pragma unroll
        for (int r = 0; r < SORT_ILP; ++r) {
            if (dst[r] >= 0) {
                const int g = gb[r] + dst[r];
                vm2 = fmax(vm2, Real(rx[r] * rx[r] + ry[r] * ry[r] + rz[r] * rz[r]));
                cellD[g] = b[r];
                offD[g] = ro[r];
                vxD[g] = rx[r];
                vyD[g] = ry[r];
                vzD[g] = rz[r];
            }
        }
    }
    // speed bound of the species for the particle-target pass
    vmax_raise(W.vmax2, ds, (double)vm2);
    sort_finish(W);
}

// ------------------------------------------------------------ pair pass

template <typename Real>
struct PairBirth {
    int c;
    int pad;
    Real off, vx, vy, vz;
};

template <typename Real>
__device__ __forceinline__ Real pair_sigma(const WsPtrs &W, const TableDesc &T, Real E);

template <>
__device__ __forceinline__ float pair_sigma<float>(const WsPtrs &W, const TableDesc &T, float E)
{
    if (E < T.th_f) return 0.f;
    const float *nd = W.lutEf + T.off, *sv = W.lutSf + T.off;
    const int n = T.n;
    if (!(E > nd[0])) return sv[0];
    if (E >= nd[n - 1]) return sv[n - 1];
    int k = (int)((logf(E) - T.lnE0_f) * T.inv_dlog_f);
    k = k < 0 ? 0 : (k > n - 2 ? n - 2 : k);
    while (k > 0 && E < nd[k]) --k;
    while (k < n - 2 && E >= nd[k + 1]) ++k;
    const float f = (E - nd[k]) / (nd[k + 1] - nd[k]);
    return sv[k] + f * (sv[k + 1] - sv[k]);
}
template <>
__device__ __forceinline__ double pair_sigma<double>(const WsPtrs &W, const TableDesc &T, double E)
{
    if (E < T.th) return 0.0;
    const double *nd = W.lutE + T.off, *sv = W.lutS + T.off;
    const int n = T.n;
    if (!(E > nd[0])) return sv[0];
    if (E >= nd[n - 1]) return sv[n - 1];
    int k = (int)((log(E) - T.lnE0) * T.inv_dlog);
    k = k < 0 ? 0 : (k > n - 2 ? n - 2 : k);
    while (k > 0 && E < nd[k]) --k;
    while (k < n - 2 && E >= nd[k + 1]) ++k;
    const double f = (E - nd[k]) / (nd[k + 1] - nd[k]);
    return sv[k] + f * (sv[k + 1] - sv[k]);
}

template <typename Real>
__device__ __forceinline__ void iso_n(Real r1, Real r2, Real n[3])
{
    iso_dir<Real>(r1, r2, n);
}

// Particle-target reaction k by thinning (Eq. 1): no pair of the pass is
// faster than the sum of the two species' largest speeds (recorded at the
// sort and raised by the velocity changes since), so with u_cap that sum,
// rounded up to 5 significant bits in m/s (the same grid point whatever the
// rounding of the sum), B = n_target max sigma u tau over u <= u_cap bounds P
// for every pair; the cell's candidates are its projectiles at geometric
// gaps of rate B (a random stream per cell), and a candidate reacts with
// probability min(P, 1) / min(B, 1); with B >= 1 every projectile is a
// candidate.  Every projectile then reacts with probability min(P, 1).
__device__ __forceinline__ double round_up_5bits(double u)
{
    if (!(u > 0.0)) return 0.0;
    int e;
    const double m = frexp(u, &e);
    return ldexp(ceil(m * 32.0) / 32.0, e);
}
__device__ __forceinline__ double pair_bound_B(const WsPtrs &W, const Disc &Dd, int d, const PairC &pc, int liveT)
{
    const double vs = Dd.sp[0].vscale;  // cells per step -> m/s
    const double vp = sqrt(__longlong_as_double((long long)W.vmax2[d * NSP + pc.proj]));
    const double vt = sqrt(__longlong_as_double((long long)W.vmax2[d * NSP + pc.targ]));
    const double ucap_n = round_up_5bits((vp + vt) * vs) / vs;
    return (double)liveT * pc.coef * fmax(pc.bnd_g, pc.bnd_s * ucap_n);
}
// gap before the next candidate: floor(ln U / ln(1 - B)) for the draw-th word
// of the cell's stream (B < 1, lq = ln(1 - B)), at most 2^30
__device__ __forceinline__ long long pair_gap(const Disc &Dd, int ps, int rx, unsigned draw,
                                              unsigned long long step, int c, double lq)
{
    const uint4 g = rng_block(Dd.seed, Dd.discharge, ps, 4, rx, draw, step, (unsigned)c);
    const double G = floor(log(unif<double>(g.x)) / lq);
    return G < 1073741824.0 ? (long long)G : 1073741824LL;
}

// Sequential pass of reaction k over one cell by one warp; kills: the cell's
// particles killed by the reactions before it, per species, raised here.
template <typename Real>
__device__ __forceinline__ void pair_cell(const WsPtrs &W, const Pools<Real> &P, int cur, unsigned long long step, int gw,
                                          int k, int lane, int kills[NSP])
{
    const int d = W.cell_disc[gw];
    const Disc &Dd = W.disc[d];
    const int N = Dd.N, c = gw - Dd.ccell_base;
    const int *cs = W.cell_start + Dd.cs_base;
    const unsigned b0 = cur ? P.stride : 0u;
    int *cellA = P.cell[0] + b0;
    Real *offA = P.off[0] + b0, *vxA = P.vx[0] + b0, *vyA = P.vy[0] + b0, *vzA = P.vz[0] + b0;
    typename AccK<Real>::T *acc = AccK<Real>::ptr(W);
    PairBirth<Real> *births = reinterpret_cast<PairBirth<Real> *>(W.pair_births) + (size_t)gw * PAIR_BIRTH_CAP;
    unsigned long long *cnt = W.counters + (size_t)d * C_NCOUNT;
    int nb = W.pair_bcount[gw];
    const int rx = k == 0 ? 13 : (k == 1 ? 14 : 19);
    const PairC &pc = Dd.pair[k];
    const int ps = pc.proj, pt = pc.targ;
    const int p0 = cs[ps * (N + 2) + c], p1 = cs[ps * (N + 2) + c + 1];
    const int t0 = cs[pt * (N + 2) + c], t1 = cs[pt * (N + 2) + c + 1];
    const int range = t1 - t0;
    const int liveT = range - kills[pt];
    if (liveT <= 0 || p1 <= p0) return;
    const TableDesc &T = W.tables[pc.table];
    const Real coefP = Real(liveT) * pick<Real>(pc.coef, pc.coef_f);
    const int pbp = Dd.pbase[ps], pbt = Dd.pbase[pt];
    // candidates of the thinning, 32 at a time: each lane draws its gap, a
    // warp scan of (1 + gap) places them (the gaps do not depend on events)
    const double B = pair_bound_B(W, Dd, d, pc, liveT);
    const bool thin = B < 1.0;
    const double lq = thin ? log1p(-B) : 0.0;
    const Real Bc = thin ? Real(B) : Real(1);
    long long pos = p0 - 1;  // last candidate placed (warp-uniform)
    unsigned draw = 0;
    bool stop = false;
    unsigned nviol = 0, neval = 0;
    int nkp = 0, nkt = 0;
    while (!stop && pos + 1 < p1) {
        long long inc = 1 + (thin ? pair_gap(Dd, ps, rx, draw + (unsigned)lane, step, c, lq) : 0LL);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long x = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += x;
        }
        const long long ipos = pos + inc;
        const int i = ipos < p1 ? (int)ipos : p1;  // p1: no candidate for this lane
        pos = __shfl_sync(0xffffffffu, ipos, 31);
        draw += 32;
        int from = 0;
        for (;;) {
            bool ev = false, ex = false, viol = false, evald = false;
            int j = -1;
            uint4 d0 = make_uint4(0, 0, 0, 0);
            if (i < p1 && lane >= from && cellA[pbp + i] >= 0) {
                d0 = rng_block(Dd.seed, Dd.discharge, ps, 2, rx, 0, step, (unsigned)i);
                j = t0 + (int)__umulhi(d0.x, (unsigned)range);
                int walked = 0;
                while (cellA[pbt + j] < 0 && walked < range) {
                    j = (j + 1 < t1) ? j + 1 : t0;
                    ++walked;
                }
                if (cellA[pbt + j] < 0) {
                    ex = true;
                } else {
                    const Real g0 = vxA[pbp + i] - vxA[pbt + j];
                    const Real g1 = vyA[pbp + i] - vyA[pbt + j];
                    const Real g2 = vzA[pbp + i] - vzA[pbt + j];
                    const Real u2 = g0 * g0 + g1 * g1 + g2 * g2;
                    const Real u = sqrt(u2);
                    const Real E = pick<Real>(pc.Ek, pc.Ek_f) * u2;
                    Real Pc = coefP * pair_sigma<Real>(W, T, E) * u;
                    if (Pc > Real(1)) {  // Eq. 1 beyond 1: clamped and counted (R10)
                        viol = true;
                        Pc = Real(1);
                    }
                    ev = unif<Real>(d0.y) * Bc < Pc;
                    evald = true;
                }
            }
            const unsigned m = __ballot_sync(0xffffffffu, ev || ex);
            const int l = m ? __ffs(m) - 1 : 32;
            nviol += __popc(__ballot_sync(0xffffffffu, viol && lane <= l));
            neval += __popc(__ballot_sync(0xffffffffu, evald && lane <= l));
            if (!m) break;
            const bool exl = __shfl_sync(0xffffffffu, ex, l);
            if (exl) {
                stop = true;  // no live target left for this projectile
                break;
            }
            if (lane == l) {
                const int gi = pbp + i, gj = pbt + j;
                atomicAdd(&cnt[C_EVENTS + rx], 1ull);
                typename AccK<Real>::T *acc_p = acc + (size_t)ps * W.total_nodes + Dd.gbase;
                typename AccK<Real>::T *acc_t = acc + (size_t)pt * W.total_nodes + Dd.gbase;
                if (rx != 19) {
                    cellA[gi] = -1;
                    dep_global(acc_p, c, offA[gi], -1);
                } else {
                    uint4 d1 = rng_block(Dd.seed, Dd.discharge, ps, 2, 19, 1, step, (unsigned)i);
                    Real v[3] = {vxA[gi], vyA[gi], vzA[gi]};
                    Real V[3] = {vxA[gj], vyA[gj], vzA[gj]};
                    Real nd[3], n2[3], v1[3], Vo[3];
                    iso_n<Real>(unif<Real>(d0.z), unif<Real>(d0.w), nd);
                    const Real mf = pick<Real>(pc.mfrac, pc.mfrac_f), Mf = pick<Real>(pc.Mfrac, pc.Mfrac_f);
                    Real g0 = v[0] - V[0], g1 = v[1] - V[1], g2 = v[2] - V[2];
                    Real uu = g0 * g0 + g1 * g1 + g2 * g2 - pick<Real>(pc.dloss, pc.dloss_f);
                    Real up = uu > Real(0) ? sqrt(uu) : Real(0);
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        Real vcm = mf * v[q] + Mf * V[q];
                        v1[q] = vcm + Mf * up * nd[q];
                        Vo[q] = vcm - mf * up * nd[q];
                    }
                    iso_n<Real>(unif<Real>(d1.x), unif<Real>(d1.y), n2);
                    Real e2[3] = {Vo[0], Vo[1], Vo[2]};
                    Real a0 = v1[0] - e2[0], a1 = v1[1] - e2[1], a2 = v1[2] - e2[2];
                    Real ue = sqrt(a0 * a0 + a1 * a1 + a2 * a2);
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        Real cc = Real(0.5) * (v1[q] + e2[q]);
                        v1[q] = cc + Real(0.5) * ue * n2[q];
                        e2[q] = cc - Real(0.5) * ue * n2[q];
                    }
                    vxA[gi] = v1[0];
                    vyA[gi] = v1[1];
                    vzA[gi] = v1[2];
                    if (nb < PAIR_BIRTH_CAP) {
                        PairBirth<Real> &pbr = births[nb];
                        pbr.c = c;
                        pbr.off = offA[gi];
                        pbr.vx = e2[0];
                        pbr.vy = e2[1];
                        pbr.vz = e2[2];
                    } else {
                        set_status(W.ctl, ST_BIRTHBUF);
                    }
                }
                cellA[gj] = -1;
                dep_global(acc_t, c, offA[gj], -1);
            }
            __syncwarp();
            __threadfence_block();
            if (rx == 19) {
                ++nb;
                ++nkt;
            } else {
                ++nkp;
                ++nkt;
            }
            from = l + 1;
            if (from >= 32) break;
        }
    }
    if (lane == 0) {
        if (nviol) atomicAdd(&cnt[C_VIOL_PAIR], (unsigned long long)nviol);
        if (neval) atomicAdd(&cnt[C_PEVAL], (unsigned long long)neval);
        if (rx == 19) W.pair_bcount[gw] = nb < PAIR_BIRTH_CAP ? nb : PAIR_BIRTH_CAP;
    }
    kills[ps] += nkp;
    kills[pt] += nkt;
}

// May reaction k have a candidate in a cell with np projectiles and nt
// targets?  FP32 and on the safe side: u_cap is at most 17/16 of the sum of the
// largest speeds (round_up_5bits), B at most Bu, and the first gap
// floor(ln U / ln(1 - B)) reaches np when ln U <= -np Bu / (1 - Bu), as
// ln(1 - B) >= -B / (1 - B).  The margins cover the FP32 rounding.  (The FP64
// logarithms of the exact test cost more here than all else in the pass.)
__device__ __forceinline__ bool pair_maybe(const WsPtrs &W, const Disc &Dd, int d, int k, unsigned long long step, int c,
                                           int np, int nt)
{
    const PairC &pc = Dd.pair[k];
    if (pc.table < 0 || np <= 0 || nt <= 0) return false;
    const float vp = sqrtf((float)__longlong_as_double((long long)W.vmax2[d * NSP + pc.proj]));
    const float vt = sqrtf((float)__longlong_as_double((long long)W.vmax2[d * NSP + pc.targ]));
    const float Bu = (float)nt * pc.coef_f * fmaxf(pc.bnd_g_f, pc.bnd_s_f * (vp + vt) * 1.0626f) * 1.0001f;
    if (!(Bu < 0.999f)) return true;
    const int rx = k == 0 ? 13 : (k == 1 ? 14 : 19);
    const uint4 g = rng_block(Dd.seed, Dd.discharge, pc.proj, 4, rx, 0u, step, (unsigned)c);
    const float lnU = logf(((float)g.x + 0.5f) * (1.0f / 4294967296.0f));
    return !(lnU + 1e-5f - 1e-5f * lnU <= -(float)np * Bu / (1.0f - Bu) * 1.0001f);
}

// Particle-target reactions k0 .. k1-1 (0: (13), 1: (14), 2: (19)) of every
// cell, one launch.  A block takes PAIR_CELLS cells: one thread per cell and
// reaction sorts out those without a candidate (pair_maybe), then each warp
// takes the cells left, one at a time, and runs their reactions in order:
// projectiles in slot order, a batch of 32 candidates evaluated in parallel,
// the first accepting lane executed, the later lanes evaluated again.  Kills,
// (19)'s scattering and its births happen here; a cell's kills only lower the
// target counts of its later reactions, so a reaction that was sorted out
// stays so.  What bounds it: latency.  A test and a pass per reaction (six
// launches, FP64 logarithms in every cell): 37 us for seven small discharges,
// 51 us for 512 cells, 69 us for 4096; 6, 18 and 19 us here.
constexpr int PAIR_THREADS = 128, PAIR_CELLS = 16;
template <typename Real>
__global__ void __launch_bounds__(PAIR_THREADS)
k_pair(WsPtrs W, Pools<Real> P, int par, int k0, int k1)
{
    pdl_wait();
    __shared__ int s_flag[PAIR_CELLS];
    const int lane = threadIdx.x & 31, first = blockIdx.x * PAIR_CELLS;
    const unsigned long long step = W.ctl->step[par];
    const int cur = W.ctl->cur;
    if (threadIdx.x < PAIR_CELLS) s_flag[threadIdx.x] = 0;
    __syncthreads();
    if (threadIdx.x < PAIR_CELLS * NSP) {
        const int j = threadIdx.x % PAIR_CELLS, k = k0 + threadIdx.x / PAIR_CELLS, gw = first + j;
        if (gw < W.total_cells && k < k1) {
            const int d = W.cell_disc[gw];
            const Disc &Dd = W.disc[d];
            const int N = Dd.N, c = gw - Dd.ccell_base;
            const int *cp = W.cell_start + Dd.cs_base + Dd.pair[k].proj * (N + 2) + c;
            const int *ct = W.cell_start + Dd.cs_base + Dd.pair[k].targ * (N + 2) + c;
            if (pair_maybe(W, Dd, d, k, step, c, cp[1] - cp[0], ct[1] - ct[0])) atomicOr(&s_flag[j], 1 << k);
        }
    }
    __syncthreads();
    for (int j = threadIdx.x >> 5; j < PAIR_CELLS; j += PAIR_THREADS / 32) {
        const int flags = s_flag[j], gw = first + j;
        int kills[NSP] = {0, 0, 0};
        for (int k = k0; k < k1; ++k)
            if ((flags >> k) & 1) pair_cell<Real>(W, P, cur, step, gw, k, lane, kills);
    }
}

// ------------------------------------------------------------ Coulomb (1)-(3)

// Arithmetic of the Coulomb collision.  FP64: correctly rounded functions.
// FP32: the hardware approximations (rsqrtf, __fdividef, __logf, __sincosf,
// each documented within a few units of 2^-22), whose errors change a
// velocity by far less than the FP32 path's tolerance of 1e-5 of the thermal
// speed; sin and cos of 2 pi r come from pi (2 r - 1) in [-pi, pi) with the
// signs of both flipped.
template <typename Real> struct CoulMath;
template <> struct CoulMath<double> {
    static __device__ __forceinline__ double inv_u32(double kn_sqrt, double u2, double u)
    {
        (void)kn_sqrt;
        return 1.0 / (u2 * u);
    }
    static __device__ __forceinline__ double rcp(double x) { return 1.0 / x; }
    static __device__ __forceinline__ void normal2(unsigned a, unsigned b, double &n0, double &n1)
    {
        box_muller<double>(a, b, n0, n1);
    }
    static __device__ __forceinline__ void sincos2pi(double r, double *s, double *c) { sincospi(2.0 * r, s, c); }
    static __device__ __forceinline__ double sqrt_(double x) { return sqrt(x); }
};
template <> struct CoulMath<float> {
    static __device__ __forceinline__ float inv_u32(float, float u2, float u)
    {
        (void)u2;
        const float r = rsqrtf(u);
        return r * r * r * r * r * r;  // u^-3
    }
    static __device__ __forceinline__ float rcp(float x) { return __fdividef(1.0f, x); }
    static __device__ __forceinline__ void normal2(unsigned a, unsigned b, float &n0, float &n1)
    {
        const float x = -2.0f * __logf(unif<float>(a));
        const float r = x * rsqrtf(x);
        float s, c;
        __sincosf(3.14159265358979f * (2.0f * unif<float>(b) - 1.0f), &s, &c);
        n0 = -r * c;
        n1 = -r * s;
    }
    static __device__ __forceinline__ void sincos2pi(float r, float *s, float *c)
    {
        __sincosf(3.14159265358979f * (2.0f * r - 1.0f), s, c);
        *s = -*s;
        *c = -*c;
    }
    static __device__ __forceinline__ float sqrt_(float x) { return x * rsqrtf(x); }
};

// One binary Coulomb collision of two like particles i, j (Sec. III A, the
// model of Takizuka and Abe): tan(chi/2) = sqrt(kn / u^3) * xi with kn the
// Eq. 2 variance times u^3 for this cell, xi a standard normal; the azimuth
// phi = 2 pi r is measured from the plane of g and the z axis (the x-y plane
// when g is along z).  Each particle takes half of the change of g.
template <typename Real>
__device__ __forceinline__ void coulomb_pair(Real *vx, Real *vy, Real *vz, int i, int j, Real kn,
                                             Real xi, unsigned wphi)
{
    using M = CoulMath<Real>;
    const Real g0 = vx[i] - vx[j], g1 = vy[i] - vy[j], g2 = vz[i] - vz[j];
    const Real u2 = g0 * g0 + g1 * g1 + g2 * g2;
    if (!(u2 > Real(0))) return;
    const Real u = M::sqrt_(u2);
    const Real d = M::sqrt_(kn * M::inv_u32(Real(0), u2, u)) * xi;  // tan(chi/2)
    Real sn, om;                                                     // sin(chi), 1 - cos(chi)
    if (fabs(d) <= Real(1)) {
        const Real r = M::rcp(Real(1) + d * d);
        sn = Real(2) * d * r;
        om = Real(2) * d * d * r;
    } else {                                  // the same in 1/d (finite for any d)
        const Real e = M::rcp(d);
        const Real r = M::rcp(Real(1) + e * e);
        sn = Real(2) * e * r;
        om = Real(2) * r;
    }
    Real sp, cp;
    M::sincos2pi(unif<Real>(wphi), &sp, &cp);
    const Real up2 = g0 * g0 + g1 * g1;
    Real d0, d1, d2;
    if (up2 > Real(0)) {
        const Real up = M::sqrt_(up2), rp = M::rcp(up);
        const Real ex = g0 * rp, ey = g1 * rp;
        const Real a = g2 * sn * cp, b = u * sn * sp;
        d0 = ex * a - ey * b - g0 * om;
        d1 = ey * a + ex * b - g1 * om;
        d2 = -up * sn * cp - g2 * om;
    } else {
        d0 = u * sn * cp;
        d1 = u * sn * sp;
        d2 = -g2 * om;
    }
    vx[i] += Real(0.5) * d0;
    vy[i] += Real(0.5) * d1;
    vz[i] += Real(0.5) * d2;
    vx[j] -= Real(0.5) * d0;
    vy[j] -= Real(0.5) * d1;
    vz[j] -= Real(0.5) * d2;
}

// random numbers of collision k of a cell's pass: stream 5, the draw
// counter split over the sub-stream (high bits) and draw fields
__device__ __forceinline__ uint4 coulomb_rng(unsigned long long seed, int disc, int s,
                                             unsigned long long step, int c, unsigned k)
{
    return rng_block(seed, disc, s, 5, (int)(k >> 20), k & 0xFFFFFu, step, (unsigned)c);
}

// Copy n values of each component, COUL_COPY elements per thread in flight.
constexpr int COUL_COPY = 4;
// (T threads, this one number t)
template <typename Real, int T>
__device__ __forceinline__ void coulomb_copy(Real *dx, Real *dy, Real *dz, const Real *sx, const Real *sy,
                                             const Real *sz, int n, int t)
{
    for (int k0 = t; k0 < n; k0 += COUL_COPY * T) {
        Real ax[COUL_COPY], ay[COUL_COPY], az[COUL_COPY];
#pragma unroll
        for (int q = 0; q < COUL_COPY; ++q) {
            const int k = k0 + q * T;
            if (k < n) {
                ax[q] = sx[k];
                ay[q] = sy[k];
                az[q] = sz[k];
            }
        }
#pragma unroll
        for (int q = 0; q < COUL_COPY; ++q) {
            const int k = k0 + q * T;
            if (k < n) {
                dx[k] = ax[q];
                dy[k] = ay[q];
                dz[k] = az[q];
            }
        }
    }
}

// largest speed^2 among n velocities (a strided share per thread)
template <typename Real, int T>
__device__ __forceinline__ double speed2_max(const Real *x, const Real *y, const Real *z, int n, int t)
{
    Real m = Real(0);
    for (int k = t; k < n; k += T)
        m = fmax(m, Real(x[k] * x[k] + y[k] * y[k] + z[k] * z[k]));
    return (double)m;
}

// Collision k of a cell with the random numbers of draw 1 + k/2: the normal
// is the first (k even) or second (k odd) of the Box-Muller pair, the
// azimuth word 2 or 3.
template <typename Real>
__device__ __forceinline__ void coulomb_one(Real *vx, Real *vy, Real *vz, int i, int j, Real kn,
                                            unsigned long long seed, int disc, int s,
                                            unsigned long long step, int c, unsigned k)
{
    const uint4 w = coulomb_rng(seed, disc, s, step, c, 1u + (k >> 1));
    Real n0, n1;
    CoulMath<Real>::normal2(w.x, w.y, n0, n1);
    coulomb_pair<Real>(vx, vy, vz, i, j, kn, (k & 1u) ? n1 : n0, (k & 1u) ? w.w : w.z);
}

// The collisions of one cell.  Thread t takes collisions 2q and 2q + 1 for
// q = t, t + T, ..., which share one draw: pi(4q) = (b + q (4a mod n)) mod n,
// advanced by T (4a mod n) mod n per iteration; pi(4q+2) = pi(4q) + 2a mod
// n and pi(k+1) = pi(k) + a mod n.  prm holds a, b, 2a mod n and 4a mod n.
template <typename Real, int T>
__device__ __forceinline__ void coulomb_cell_pairs(Real *vx, Real *vy, Real *vz, unsigned un,
                                                   const unsigned *prm, Real kn, unsigned long long seed,
                                                   int disc, int s, unsigned long long step, int c, unsigned t)
{
    using M = CoulMath<Real>;
    const unsigned a = prm[0], b = prm[1], a2 = prm[2], a4 = prm[3];
    const unsigned pairs = (un & 1u) ? (un - 3u) / 2u : un / 2u;
    unsigned x = un <= (1u << 22) ? (b + (t * a4) % un) % un
                                  : (unsigned)(((unsigned long long)t * a4 + b) % un);
    const unsigned stepA = (unsigned)(((unsigned long long)T * a4) % un);
    for (unsigned q = t; 2u * q < pairs; q += T) {
        const uint4 w = coulomb_rng(seed, disc, s, step, c, 1u + q);
        Real n0, n1;
        M::normal2(w.x, w.y, n0, n1);
        unsigned y = x + a;
        if (y >= un) y -= un;
        coulomb_pair<Real>(vx, vy, vz, (int)x, (int)y, kn, n0, w.z);
        if (2u * q + 1u < pairs) {
            unsigned x1 = x + a2;
            if (x1 >= un) x1 -= un;
            unsigned y1 = x1 + a;
            if (y1 >= un) y1 -= un;
            coulomb_pair<Real>(vx, vy, vz, (int)x1, (int)y1, kn, n1, w.w);
        }
        x += stepA;
        if (x >= un) x -= un;
    }
    if ((un & 1u) && t == 0) {
        const int A = (int)(((unsigned long long)a * (un - 3u) + b) % un);
        const int B = (int)(((unsigned long long)a * (un - 2u) + b) % un);
        const int C = (int)(((unsigned long long)a * (un - 1u) + b) % un);
        const Real kh = Real(0.5) * kn;
        coulomb_one<Real>(vx, vy, vz, A, B, kh, seed, disc, s, step, c, pairs);
        coulomb_one<Real>(vx, vy, vz, B, C, kh, seed, disc, s, step, c, pairs + 1u);
        coulomb_one<Real>(vx, vy, vz, C, A, kh, seed, disc, s, step, c, pairs + 2u);
    }
}

// Coulomb collisions of one species in one cell by T threads (a block or a
// warp).  The n particles are paired by the affine permutation pi(k) = (a k +
// b) mod n, a coprime to n, from draw 0 of the cell's stream 5; collision m is
// (pi(2m), pi(2m+1)) with the random numbers of draw 1 + m/2 (two collisions
// per draw); for odd n thread 0 then runs the triangle of the last three, (A,
// B), (B, C), (C, A), with half the time each.  The pairs are disjoint, so no
// ordering is needed between threads.  A cell of at most `cap` particles is
// staged in shared memory sh (coalesced copies in and out); a larger one is
// worked on in place.  prm: four shared words of these threads.
template <typename Real, int T>
__device__ __forceinline__ void coulomb_cell(const WsPtrs &W, const Pools<Real> &P, int par, int gw, int s, int p0, int n,
                                             int t, Real *sh, int cap, unsigned *prm)
{
    auto sync = []() {
        if constexpr (T == 32) __syncwarp(); else __syncthreads();
    };
    const int d = W.cell_disc[gw];
    const Disc &Dd = W.disc[d];
    const int c = gw - Dd.ccell_base;
    if (n >= (1 << 29)) {
        if (t == 0) set_status(W.ctl, ST_BADSTATE);
        return;
    }
    if (t == 0) atomicAdd(&W.counters[(size_t)d * C_NCOUNT + C_COUL], (unsigned long long)n);
    const unsigned long long step = W.ctl->step[par];
    const unsigned long long seed = Dd.seed;
    const int disc = Dd.discharge;
    const unsigned b0 = W.ctl->cur ? P.stride : 0u;
    const size_t base = (size_t)b0 + Dd.pbase[s] + p0;
    Real *gx = P.vx[0] + base, *gy = P.vy[0] + base, *gz = P.vz[0] + base;
    const unsigned un = (unsigned)n;
    if (t == 0) {  // a, b, 2a mod n, 4a mod n of the cell's permutation
        const uint4 w0 = coulomb_rng(seed, disc, s, step, c, 0u);
        unsigned a = 1u + w0.x % (un - 1u);
        for (;;) {  // a -> a mod (n-1) + 1 until coprime; a = 1 always is
            unsigned x = a, y = un;
            while (y) {
                const unsigned r = x % y;
                x = y;
                y = r;
            }
            if (x == 1u) break;
            a = a % (un - 1u) + 1u;
        }
        prm[0] = a;
        prm[1] = w0.y % un;
        prm[2] = (unsigned)((2ull * a) % un);
        prm[3] = (unsigned)((4ull * a) % un);
    }
    const SpeciesC &S = Dd.sp[s];
    const Real kn = pick<Real>(S.coul_k, S.coul_k_f) * Real(n);
    // the new speeds raise the species' recorded largest speed, which bounds
    // P in a particle-target pass of the same step
    double m2;
    if (n <= cap) {
        Real *sx = sh, *sy = sx + cap, *sz = sy + cap;
        coulomb_copy<Real, T>(sx, sy, sz, gx, gy, gz, n, t);
        sync();
        coulomb_cell_pairs<Real, T>(sx, sy, sz, un, prm, kn, seed, disc, s, step, c, (unsigned)t);
        sync();
        coulomb_copy<Real, T>(gx, gy, gz, sx, sy, sz, n, t);
        m2 = speed2_max<Real, T>(sx, sy, sz, n, t);
    } else {
        sync();
        coulomb_cell_pairs<Real, T>(gx, gy, gz, un, prm, kn, seed, disc, s, step, c, (unsigned)t);
        sync();
        m2 = speed2_max<Real, T>(gx, gy, gz, n, t);
    }
    vmax_raise(W.vmax2, d * NSP + s, m2);
}

// Coulomb pass of every (species, cell), right after the sort (every slot of a
// cell is live), O2+ cells first, then O-, then electrons (the largest cells
// first).  GROUP = false: a block per cell.  GROUP = true: a block takes
// COUL_GROUP cells, a warp each those of at most COUL_WARP particles, and then
// the larger ones with all its warps.  What bounds small cells is latency (the
// permutation's greatest common divisor, the copies, a few collisions per
// thread): 2688 cells of about 150 particles took 56 us with a block each, in
// nine waves, and 11.7 us so (cells of 2000 to 4000 particles
// took 58 us with a block each and 131 us in groups).  Both forms handle every
// size and give the same bits; the host picks one by the particles that the
// cells hold (coulomb_groups).
constexpr int COUL_GROUP = COUL_THREADS / 32;
template <typename Real, bool GROUP>
__global__ void __launch_bounds__(COUL_THREADS, sizeof(Real) == 4 ? 2 : 1)
k_coulomb(WsPtrs W, Pools<Real> P, int par)
{
    pdl_wait();
    extern __shared__ __align__(16) unsigned char coul_smem[];
    __shared__ unsigned prm[COUL_GROUP][4];
    Real *sh = reinterpret_cast<Real *>(coul_smem);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto place = [&](int idx, int &gw, int &s, int &p0) {  // returns the cell's particles
        gw = idx % W.total_cells;
        s = NSP - 1 - idx / W.total_cells;
        const Disc &Dd = W.disc[W.cell_disc[gw]];
        const int *cs = W.cell_start + Dd.cs_base + s * (Dd.N + 2) + gw - Dd.ccell_base;
        p0 = cs[0];
        return cs[1] - cs[0];
    };
    int gw, s, p0;
    if constexpr (!GROUP) {
        const int n = place(blockIdx.x, gw, s, p0);
        if (n >= 2) coulomb_cell<Real, COUL_THREADS>(W, P, par, gw, s, p0, n, threadIdx.x, sh, COUL_STAGE, prm[0]);
    } else {
        __shared__ int s_n[COUL_GROUP];
        const int first = blockIdx.x * COUL_GROUP, end = NSP * W.total_cells;
        int n = 0;
        if (first + warp < end) n = place(first + warp, gw, s, p0);
        if (lane == 0) s_n[warp] = n;
        if (n >= 2 && n <= COUL_WARP)
            coulomb_cell<Real, 32>(W, P, par, gw, s, p0, n, lane, sh + (size_t)warp * 3 * COUL_WARP, COUL_WARP, prm[warp]);
        __syncthreads();
        for (int q = 0; q < COUL_GROUP; ++q) {
            if (s_n[q] <= COUL_WARP) continue;
            n = place(first + q, gw, s, p0);
            coulomb_cell<Real, COUL_THREADS>(W, P, par, gw, s, p0, n, threadIdx.x, sh, COUL_STAGE, prm[0]);
            __syncthreads();
        }
    }
}

#ifndef O2_INTER_CHAINS
#define O2_INTER_CHAINS 128
#endif
// Most chains (B particles) run on prepared random numbers.  256 cells of 2000 and
// 4000 ions, all three pairs, FP32 / FP64: 33 electrons a cell 143 / 2057 us with
// them, 180 / 3002 without, 64 129 / 1563 and 149 / 1959, 120 125 / 1344 and 131 /
// 1482, 200 123 / 1339 and 129 / 1467, 300 121 / 1323 and 123 / 1430.  The line
// could lie anywhere up to a block's 384 threads: 128 and 384 take the same time
// in a whole run (cfg2: 30.3 and 30.5 ms per 200 steps).
constexpr int INTER_CHAINS = O2_INTER_CHAINS;
constexpr int INTER_TILE = 1024;               // collisions prepared at a time

// The change of g = va - vb in one Coulomb collision of unlike particles (as
// coulomb_pair, with the pair's kn), from its random numbers: xi, and sp, cp =
// sin, cos of the azimuth.
template <typename Real>
__device__ __forceinline__ void coulomb_change(Real g0, Real g1, Real g2, Real kn, Real xi, Real sp, Real cp, Real dg[3])
{
    using M = CoulMath<Real>;
    dg[0] = dg[1] = dg[2] = Real(0);
    const Real u2 = g0 * g0 + g1 * g1 + g2 * g2;
    if (!(u2 > Real(0))) return;
    const Real u = M::sqrt_(u2);
    const Real d = M::sqrt_(kn * M::inv_u32(Real(0), u2, u)) * xi;
    Real sn, om;
    if (fabs(d) <= Real(1)) {
        const Real r = M::rcp(Real(1) + d * d);
        sn = Real(2) * d * r;
        om = Real(2) * d * d * r;
    } else {
        const Real e = M::rcp(d);
        const Real r = M::rcp(Real(1) + e * e);
        sn = Real(2) * e * r;
        om = Real(2) * r;
    }
    const Real up2 = g0 * g0 + g1 * g1;
    if (up2 > Real(0)) {
        const Real up = M::sqrt_(up2), rp = M::rcp(up);
        const Real ex = g0 * rp, ey = g1 * rp;
        const Real a = g2 * sn * cp, b = u * sn * sp;
        dg[0] = ex * a - ey * b - g0 * om;
        dg[1] = ey * a + ex * b - g1 * om;
        dg[2] = -up * sn * cp - g2 * om;
    } else {
        dg[0] = u * sn * cp;
        dg[1] = u * sn * sp;
        dg[2] = -g2 * om;
    }
}
// The whole collision: a takes fa of the change and b minus fb of it.
template <typename Real>
__device__ __forceinline__ void coulomb_pair_ab(Real va[3], Real vb[3], Real kn, Real fa, Real fb, Real xi,
                                                unsigned wphi)
{
    Real sp, cp, dg[3];
    CoulMath<Real>::sincos2pi(unif<Real>(wphi), &sp, &cp);
    coulomb_change<Real>(va[0] - vb[0], va[1] - vb[1], va[2] - vb[2], kn, xi, sp, cp, dg);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        va[q] += fa * dg[q];
        vb[q] -= fb * dg[q];
    }
}
__device__ __noinline__ float3 coulomb_change_any(float g0, float g1, float g2, float kn, float xi, float sp, float cp)
{
    float dg[3];
    coulomb_change<float>(g0, g1, g2, kn, xi, sp, cp, dg);
    return make_float3(dg[0], dg[1], dg[2]);
}
__device__ __forceinline__ float rsqrt_hw(float x)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rcp_hw(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// One link of a chain: what the inter-species pass waits for.  The FP32 link
// has no branch: the hardware's reciprocal and square root (equal to the
// guarded functions of CoulMath for the inputs accepted here, every one of
// them checked), the common small-angle form, and one check beside the chain
// that sends any other case through coulomb_change.  From about 470 to 320
// cycles a link (4e6 superparticles: one electron among 3900 ions, 970 -> 660
// us).
__device__ __forceinline__ void coulomb_link(float va[3], float vb[3], float kn, float fa, float fb, float xi, float sp,
                                             float cp)
{
    const float g0 = va[0] - vb[0], g1 = va[1] - vb[1], g2 = va[2] - vb[2];
    const float u2 = g0 * g0 + g1 * g1 + g2 * g2;
    const float u = u2 * rsqrt_hw(u2);
    const float q = rsqrt_hw(u);
    const float x = kn * (q * q * q * q * q * q);
    const float d = x * rsqrt_hw(x) * xi;
    const float r = rcp_hw(1.0f + d * d);
    const float sn = 2.0f * d * r, om = 2.0f * d * d * r;
    const float up2 = g0 * g0 + g1 * g1;
    const float up = up2 * rsqrt_hw(up2), rp = rcp_hw(up);
    const float ex = g0 * rp, ey = g1 * rp;
    const float a = g2 * sn * cp, b = u * sn * sp;
    float dg[3];
    dg[0] = ex * a - ey * b - g0 * om;
    dg[1] = ey * a + ex * b - g1 * om;
    dg[2] = -up * sn * cp - g2 * om;
    constexpr float LOW = 1.1754944e-38f, HIGH = 1e37f;  // normal, and far from overflow
    if (!(up2 >= LOW && u2 <= HIGH && x >= LOW && x <= HIGH && fabsf(d) <= 1.0f)) {
        const float3 t = coulomb_change_any(g0, g1, g2, kn, xi, sp, cp);
        dg[0] = t.x;
        dg[1] = t.y;
        dg[2] = t.z;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        va[k] += fa * dg[k];
        vb[k] -= fb * dg[k];
    }
}
__device__ __forceinline__ void coulomb_link(double va[3], double vb[3], double kn, double fa, double fb, double xi,
                                             double sp, double cp)
{
    double dg[3];
    coulomb_change<double>(va[0] - vb[0], va[1] - vb[1], va[2] - vb[2], kn, xi, sp, cp, dg);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        va[k] += fa * dg[k];
        vb[k] -= fb * dg[k];
    }
}

// Inter-species Coulomb collisions of one cell per block (Takizuka and Abe for
// unlike particles), after the intra-species pass, the species pairs e-O-,
// e-O2+, O- - O2+ in turn (cells do not meet, so one launch does all three and
// a cell with long chains does not hold up the others' next pair): the nA particles of the more numerous species (A) each collide once,
// those of the other (B) in turn; collision k joins A pi_A(k) with B
// pi_B(k mod nB) (affine permutations from draw 0 of the cell's stream 5
// with species field 3 + pair) with the random numbers of draw 1 + k/2.
// Thread t follows the B particles r = t, t + T, ...: particle pi_B(r) meets
// A pi_A(r), pi_A(r + nB), ... in that order, its velocity in registers; the
// A particles are disjoint across threads.  A is staged in shared memory
// when it has at most `cap` particles.
//
// What bounds it: the longest chain.  In the sheaths a handful of electrons
// meet thousands of ions one after the other, while the collisions of all
// other cells are done.  So with at most INTER_CHAINS chains the random
// numbers, normals and azimuths, which do not depend on the chain, are
// prepared by all threads, the next link's inputs are loaded ahead, and the
// cells at both walls start first.
template <typename Real>
__global__ void __launch_bounds__(COUL_THREADS, sizeof(Real) == 4 ? 2 : 1)
k_coulomb_inter(WsPtrs W, Pools<Real> P, int par, int cap)
{
    pdl_wait();
    extern __shared__ __align__(16) unsigned char coul_smem[];
    __shared__ unsigned prm[4];  // a, b of A's permutation, a, b of B's
    const int gw = (blockIdx.x & 1) ? W.total_cells - 1 - (int)(blockIdx.x >> 1) : (int)(blockIdx.x >> 1);
    const int d = W.cell_disc[gw];
    const Disc &Dd = W.disc[d];
    const int N = Dd.N, c = gw - Dd.ccell_base;
    for (int pair = 0; pair < 3; ++pair) {
        __syncthreads();  // the pair before is done with the shared memory and the velocities
        const int s0 = pair == 2 ? 1 : 0, s1 = pair == 0 ? 1 : 2;
        const int *cs = W.cell_start + Dd.cs_base;
        const int q0 = cs[s0 * (N + 2) + c], n0 = cs[s0 * (N + 2) + c + 1] - q0;
        const int q1 = cs[s1 * (N + 2) + c], n1 = cs[s1 * (N + 2) + c + 1] - q1;
        if (n0 <= 0 || n1 <= 0) continue;
        const bool zeroA = n0 >= n1;
        const int sA = zeroA ? s0 : s1, sB = zeroA ? s1 : s0;
        const int nA = zeroA ? n0 : n1, nB = zeroA ? n1 : n0;
        const int pA = zeroA ? q0 : q1, pB = zeroA ? q1 : q0;
        if (nA >= (1 << 29)) {
            if (threadIdx.x == 0) set_status(W.ctl, ST_BADSTATE);
            continue;
        }
        if (threadIdx.x == 0) atomicAdd(&W.counters[(size_t)d * C_NCOUNT + C_COUL], (unsigned long long)(nA + nB));
        const unsigned long long step = W.ctl->step[par];
        const unsigned long long seed = Dd.seed;
        const int disc = Dd.discharge;
        const int cur = W.ctl->cur;
        const int sfield = 3 + pair;
        if (threadIdx.x == 0) {
            const uint4 w0 = coulomb_rng(seed, disc, sfield, step, c, 0u);
            const unsigned w[4] = {w0.x, w0.y, w0.z, w0.w};
            const unsigned nn[2] = {(unsigned)nA, (unsigned)nB};
            for (int h = 0; h < 2; ++h) {
                const unsigned un = nn[h];
                unsigned a = 1u, b = 0u;
                if (un >= 2u) {
                    a = 1u + w[2 * h] % (un - 1u);
                    for (;;) {
                        unsigned x = a, y = un;
                        while (y) {
                            const unsigned t = x % y;
                            x = y;
                            y = t;
                        }
                        if (x == 1u) break;
                        a = a % (un - 1u) + 1u;
                    }
                    b = w[2 * h + 1] % un;
                }
                prm[2 * h] = a;
                prm[2 * h + 1] = b;
            }
        }
        Real *gax = P.vx[cur] + Dd.pbase[sA] + pA, *gay = P.vy[cur] + Dd.pbase[sA] + pA,
             *gaz = P.vz[cur] + Dd.pbase[sA] + pA;
        Real *gbx = P.vx[cur] + Dd.pbase[sB] + pB, *gby = P.vy[cur] + Dd.pbase[sB] + pB,
             *gbz = P.vz[cur] + Dd.pbase[sB] + pB;
        const bool staged = nA <= cap;
        Real *ax = gax, *ay = gay, *az = gaz;
        if (staged) {
            ax = reinterpret_cast<Real *>(coul_smem);
            ay = ax + cap;
            az = ay + cap;
            coulomb_copy<Real, COUL_THREADS>(ax, ay, az, gax, gay, gaz, nA, threadIdx.x);
        }
        __syncthreads();
        const unsigned aA = prm[0], bA = prm[1], aB = prm[2], bB = prm[3];
        const unsigned uA = (unsigned)nA, uB = (unsigned)nB;
        const Real kn = pick<Real>(Dd.ci_k[pair], Dd.ci_k_f[pair]) * Real(nB);
        const int ia = zeroA ? 0 : 1;  // index of A's share
        const Real fa = pick<Real>(Dd.ci_frac[pair][ia], Dd.ci_frac_f[pair][ia]);
        const Real fb = pick<Real>(Dd.ci_frac[pair][1 - ia], Dd.ci_frac_f[pair][1 - ia]);
        // indices advanced by additions mod n: j(r) = (aB r + bB) mod nB steps by
        // aB T mod nB, i(k) = (aA k + bA) mod nA by aA T mod nA over r and by
        // aA nB mod nA along a chain
        const unsigned t0 = threadIdx.x;
        unsigned j = (unsigned)(((unsigned long long)aB * t0 + bB) % uB);
        unsigned i0 = (unsigned)(((unsigned long long)aA * t0 + bA) % uA);
        const unsigned stepB = (unsigned)(((unsigned long long)aB * COUL_THREADS) % uB);
        const unsigned stepA = (unsigned)(((unsigned long long)aA * COUL_THREADS) % uA);
        const unsigned chainA = (unsigned)(((unsigned long long)aA * uB) % uA);
        Real m2b = Real(0);  // largest new speed^2 of this thread's B particles
        if (nB <= INTER_CHAINS) {
            // few, long chains: all threads prepare the random numbers of
            // INTER_TILE collisions, then the chains run through them
            Real *txi = reinterpret_cast<Real *>(coul_smem) + 3 * cap, *tsp = txi + INTER_TILE, *tcp = tsp + INTER_TILE;
            const bool mine = t0 < uB;
            Real vb[3] = {Real(0), Real(0), Real(0)};
            if (mine) {
                vb[0] = gbx[j];
                vb[1] = gby[j];
                vb[2] = gbz[j];
            }
            unsigned k = t0, i = i0;
            for (unsigned k0 = 0; k0 < uA; k0 += INTER_TILE) {
                const unsigned ke = min(k0 + (unsigned)INTER_TILE, uA);
                for (unsigned q = t0; 2 * q < INTER_TILE && k0 + 2 * q < ke; q += COUL_THREADS) {
                    const uint4 w = coulomb_rng(seed, disc, sfield, step, c, 1u + (k0 >> 1) + q);
                    CoulMath<Real>::normal2(w.x, w.y, txi[2 * q], txi[2 * q + 1]);
                    CoulMath<Real>::sincos2pi(unif<Real>(w.z), &tsp[2 * q], &tcp[2 * q]);
                    CoulMath<Real>::sincos2pi(unif<Real>(w.w), &tsp[2 * q + 1], &tcp[2 * q + 1]);
                }
                __syncthreads();
                if (mine && k < ke) {
                    // the next collision's inputs are loaded before the present one
                    Real va[3] = {ax[i], ay[i], az[i]};
                    Real xi = txi[k - k0], sp = tsp[k - k0], cp = tcp[k - k0];
                    for (;;) {
                        const unsigned k2 = k + uB;
                        unsigned i2 = i + chainA;
                        if (i2 >= uA) i2 -= uA;
                        const bool more = k2 < ke;
                        const unsigned in = more ? i2 : i, kn2 = more ? k2 - k0 : 0u;
                        const Real va2[3] = {ax[in], ay[in], az[in]};
                        const Real xi2 = txi[kn2], sp2 = tsp[kn2], cp2 = tcp[kn2];
                        coulomb_link(va, vb, kn, fa, fb, xi, sp, cp);
                        ax[i] = va[0];
                        ay[i] = va[1];
                        az[i] = va[2];
                        k = k2;
                        i = i2;
                        if (!more) break;
                        va[0] = va2[0];
                        va[1] = va2[1];
                        va[2] = va2[2];
                        xi = xi2;
                        sp = sp2;
                        cp = cp2;
                    }
                }
                __syncthreads();
            }
            if (mine) {
                gbx[j] = vb[0];
                gby[j] = vb[1];
                gbz[j] = vb[2];
                m2b = vb[0] * vb[0] + vb[1] * vb[1] + vb[2] * vb[2];
            }
        } else
        for (unsigned r = t0; r < uB; r += COUL_THREADS) {
            Real vb[3] = {gbx[j], gby[j], gbz[j]};
            unsigned i = i0;
            for (unsigned k = r; k < uA; k += uB) {
                const uint4 w = coulomb_rng(seed, disc, sfield, step, c, 1u + (k >> 1));
                Real n0r, n1r;
                CoulMath<Real>::normal2(w.x, w.y, n0r, n1r);
                Real va[3] = {ax[i], ay[i], az[i]};
                coulomb_pair_ab<Real>(va, vb, kn, fa, fb, (k & 1u) ? n1r : n0r, (k & 1u) ? w.w : w.z);
                ax[i] = va[0];
                ay[i] = va[1];
                az[i] = va[2];
                i += chainA;
                if (i >= uA) i -= uA;
            }
            gbx[j] = vb[0];
            gby[j] = vb[1];
            gbz[j] = vb[2];
            m2b = fmax(m2b, Real(vb[0] * vb[0] + vb[1] * vb[1] + vb[2] * vb[2]));
            j += stepB;
            if (j >= uB) j -= uB;
            i0 += stepA;
            if (i0 >= uA) i0 -= uA;
        }
        __syncthreads();
        if (staged) coulomb_copy<Real, COUL_THREADS>(gax, gay, gaz, ax, ay, az, nA, threadIdx.x);
        // the new speeds raise both species' recorded largest speeds
        vmax_raise(W.vmax2, d * NSP + sA, speed2_max<Real, COUL_THREADS>(ax, ay, az, nA, threadIdx.x));
        vmax_raise(W.vmax2, d * NSP + sB, (double)m2b);
    }
}

// Births of (19) appended to the electron array of each discharge in cell
// order (the order of the sequential pass).
template <typename Real>
__global__ void __launch_bounds__(256)
k_pair_append(WsPtrs W, Pools<Real> P)
{
    pdl_wait();
    extern __shared__ __align__(16) int pre[];
    __shared__ int wsum[32];
    const int d = blockIdx.x;
    const Disc &Dd = W.disc[d];
    const int N = Dd.N;
    int any = 0;
    for (int c = threadIdx.x; c < N; c += blockDim.x) {
        const int n = W.pair_bcount[Dd.ccell_base + c];
        pre[c] = n;
        any |= n;
    }
    if (!__syncthreads_or(any)) return;
    const int tot = block_scan_exclusive_int(pre, N, wsum);
    if (tot == 0) return;
    const int cur = W.ctl->cur;
    Counts &C = W.cnt[d * NSP + 0];
    const int n0 = C.n;
    typename AccK<Real>::T *acc = AccK<Real>::ptr(W) + Dd.gbase;  // species 0 block
    const PairBirth<Real> *births = reinterpret_cast<const PairBirth<Real> *>(W.pair_births);
    for (int c = threadIdx.x; c < N; c += blockDim.x) {
        const int nbc = W.pair_bcount[Dd.ccell_base + c];
        for (int r = 0; r < nbc; ++r) {
            const PairBirth<Real> &b = births[(size_t)(Dd.ccell_base + c) * PAIR_BIRTH_CAP + r];
            const int dst = n0 + pre[c] + r;
            if (dst >= Dd.cap[0]) {
                set_status(W.ctl, ST_CAPACITY);
                continue;
            }
            const int gidx = Dd.pbase[0] + dst;
            P.cell[cur][gidx] = b.c;
            P.off[cur][gidx] = b.off;
            P.vx[cur][gidx] = b.vx;
            P.vy[cur][gidx] = b.vy;
            P.vz[cur][gidx] = b.vz;
            dep_global(acc, b.c, b.off, 1);
        }
    }
    __syncthreads();
    for (int c = threadIdx.x; c < N; c += blockDim.x) W.pair_bcount[Dd.ccell_base + c] = 0;
    if (threadIdx.x == 0) C.n = min(n0 + tot, Dd.cap[0]);
}

// ------------------------------------------------------------ load / deposit

// Uniform positions in (0, L) and Maxwellian velocities from Philox stream 3
// (step 0, index = slot): draw 0 gives two Box-Muller pairs, draw 1 the
// position.  Computed in FP64 and rounded once to the storage precision.
template <typename Real>
__global__ void k_load(WsPtrs W, Pools<Real> P, const long long *n_init, const double *vt)
{
    const int ds = blockIdx.y;
    const int d = ds / NSP, s = ds % NSP;
    const Disc &Dd = W.disc[d];
    const int n = (int)n_init[ds];
    const int cur = W.ctl->cur;
    const double to_n = Dd.dt / Dd.dx;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const uint4 a = rng_block(Dd.seed, Dd.discharge, s, 3, 0, 0, 0ull, (unsigned)i);
        const uint4 b = rng_block(Dd.seed, Dd.discharge, s, 3, 0, 1, 0ull, (unsigned)i);
        double n0, n1, n2, n3;
        box_muller<double>(a.x, a.y, n0, n1);
        box_muller<double>(a.z, a.w, n2, n3);
        const double x = unif<double>(b.x) * Dd.L;
        const double xx = x / Dd.dx;
        int c = (int)floor(xx);
        if (c > Dd.N - 1) c = Dd.N - 1;
        if (c < 0) c = 0;
        Real off = (Real)(xx - c);
        if (off >= Real(1)) {
            if (c + 1 < Dd.N) {
                ++c;
                off = Real(0);
            } else {
                off = Real(0.99999994);
            }
        }
        const int g = Dd.pbase[s] + i;
        P.cell[cur][g] = c;
        P.off[cur][g] = off;
        P.vx[cur][g] = (Real)(vt[ds] * n0 * to_n);
        P.vy[cur][g] = (Real)(vt[ds] * n1 * to_n);
        P.vz[cur][g] = (Real)(vt[ds] * n2 * to_n);
    }
}

// ------------------------------------------------------------ state copies

// The state that a caller sets passes through the buffer that the next sort will
// write (free between steps): positions in its offsets, velocities in its
// velocities, alive flags in its cells; SI doubles there, so a chunk holds
// half the buffer's slots in the FP32 path.  Arithmetic as on a host: one
// division, floor, one product per value.  1e6 particles set: 4.2 ms when one
// host core converted them, 0.85 ms.

// does a live particle lie outside [0, L)?  *bad is set to 1
__global__ void __launch_bounds__(256) k_state_check(const double *x, const int *alive, int n, double L, unsigned *bad)
{
    bool out = false;
    for (int i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256)
        out |= (!alive || alive[i] != 0) && !(x[i] >= 0.0 && x[i] < L);
    if (out) *bad = 1u;
}

// chunk of n slots from slot g on
template <typename Real>
__global__ void __launch_bounds__(256)
k_state_in(Pools<Real> P, int cur, size_t g, int n, int N, double dx, double tdx, bool flags)
{
    const int nx = cur ^ 1;
    const double *x = reinterpret_cast<const double *>(P.off[nx]), *vx = reinterpret_cast<const double *>(P.vx[nx]),
                 *vy = reinterpret_cast<const double *>(P.vy[nx]), *vz = reinterpret_cast<const double *>(P.vz[nx]);
    for (int i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) {
        const bool al = !flags || P.cell[nx][i] != 0;
        const double xx = x[i] / dx;
        int c = al ? (int)floor(xx) : -1;
        if (c > N - 1) c = N - 1;
        const double off = al ? xx - c : 0.0;
        Real of = (Real)off;
        if (sizeof(Real) == 4 && al && of >= Real(1)) {
            if (c + 1 < N) {
                ++c;
                of = Real(0);
            } else {
                of = (Real)0x1.fffffep-1f;
            }
        }
        P.cell[cur][g + i] = c;
        P.off[cur][g + i] = of;
        P.vx[cur][g + i] = (Real)(vx[i] * tdx);
        P.vy[cur][g + i] = (Real)(vy[i] * tdx);
        P.vz[cur][g + i] = (Real)(vz[i] * tdx);
    }
}

// slots g .. g + n - 1 to the host's page-locked buffer: x, vx, vy, vz of ld
// doubles each, then ld alive flags
template <typename Real>
__global__ void __launch_bounds__(256)
k_state_out(Pools<Real> P, int cur, size_t g, int n, double *out, int ld, double dx, double vs)
{
    int *alive = reinterpret_cast<int *>(out + 4 * (size_t)ld);
    for (int i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) {
        const int c = P.cell[cur][g + i];
        out[i] = c >= 0 ? ((double)c + (double)P.off[cur][g + i]) * dx : 0.0;
        out[(size_t)ld + i] = (double)P.vx[cur][g + i] * vs;
        out[2 * (size_t)ld + i] = (double)P.vy[cur][g + i] * vs;
        out[3 * (size_t)ld + i] = (double)P.vz[cur][g + i] * vs;
        alive[i] = c >= 0 ? 1 : 0;
    }
}

static int state_blocks(int n) { return n <= 0 ? 1 : ((n + 255) / 256 < 1216 ? (n + 255) / 256 : 1216); }

cudaError_t launch_state_check(const double *x, const int *alive, int n, double L, unsigned *bad, cudaStream_t st)
{
    k_state_check<<<state_blocks(n), 256, 0, st>>>(x, alive, n, L, bad);
    return cudaGetLastError();
}

cudaError_t launch_state_in(bool fp64, const void *pools, int cur, size_t g, int n, int N, double dx, double tdx,
                            bool flags, cudaStream_t st)
{
    if (fp64)
        k_state_in<double><<<state_blocks(n), 256, 0, st>>>(*static_cast<const Pools<double> *>(pools), cur, g, n, N, dx,
                                                            tdx, flags);
    else
        k_state_in<float><<<state_blocks(n), 256, 0, st>>>(*static_cast<const Pools<float> *>(pools), cur, g, n, N, dx,
                                                           tdx, flags);
    return cudaGetLastError();
}

cudaError_t launch_state_out(bool fp64, const void *pools, int cur, size_t g, int n, double *out, int ld, double dx,
                             double vs, cudaStream_t st)
{
    if (fp64)
        k_state_out<double><<<state_blocks(n), 256, 0, st>>>(*static_cast<const Pools<double> *>(pools), cur, g, n, out, ld, dx, vs);
    else
        k_state_out<float><<<state_blocks(n), 256, 0, st>>>(*static_cast<const Pools<float> *>(pools), cur, g, n, out, ld, dx, vs);
    return cudaGetLastError();
}

// ------------------------------------------------------------ host reads

__global__ void __launch_bounds__(256) k_gather(GatherList g, unsigned *host)
{
    pdl_wait();
    const unsigned total = g.first[g.n];
    for (unsigned w = blockIdx.x * 256u + threadIdx.x; w < total; w += gridDim.x * 256u) {
        int k = 0;
        while (w >= g.first[k + 1]) ++k;
        const unsigned i = w - g.first[k];
        if (g.dst[k] != ~0u) host[g.dst[k] + i] = g.src[k][i];
        if (g.clear[k]) g.src[k][i] = 0u;
    }
}

cudaError_t launch_gather(const GatherList &g, unsigned *host, cudaStream_t st)
{
    const unsigned blocks = (g.first[g.n] + 255u) / 256u;
    launch_k(k_gather, blocks < 1u ? 1u : (blocks < 304u ? blocks : 304u), 256, 0, st, g, host);
    return cudaGetLastError();
}

// ------------------------------------------------------------ launchers

// the inter-species pass: A's velocities and one tile of random numbers
static size_t inter_smem_bytes(bool fp64)
{
    return coulomb_smem_bytes(fp64) + (size_t)INTER_TILE * 3 * (fp64 ? 8 : 4);
}

cudaError_t allow_smem(const void *kernel, size_t bytes)
{
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    cudaFuncAttributes a{};
    const cudaError_t e = cudaFuncGetAttributes(&a, kernel);
    if (e != cudaSuccess || (size_t)a.maxDynamicSharedSizeBytes >= bytes) return e;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

cudaError_t configure_kernels(bool fp64, LaunchCfg &L)
{
    cudaError_t e;
    L.sort_smem = sizeof(unsigned short) * SORT_WARPS * ((L.maxN + 2) & ~1);
    L.scatter_smem = sizeof(unsigned short) * SORT_WARPS * ((L.maxN + 2) & ~1);
    if (fp64) {
        e = allow_smem(k_sort_count<double>, L.sort_smem);
        if (e) return e;
        e = allow_smem(k_sort_scatter<double>, L.scatter_smem);
        if (e) return e;
        e = allow_smem(k_coulomb<double, false>, coulomb_smem_bytes(true));
        if (e) return e;
        e = allow_smem(k_coulomb<double, true>, coulomb_smem_bytes(true));
        if (e) return e;
        e = allow_smem(k_coulomb_inter<double>, inter_smem_bytes(true));
        if (e) return e;
    } else {
        e = allow_smem(k_sort_count<float>, L.sort_smem);
        if (e) return e;
        e = allow_smem(k_sort_scatter<float>, L.scatter_smem);
        if (e) return e;
        e = allow_smem(k_coulomb<float, false>, coulomb_smem_bytes(false));
        if (e) return e;
        e = allow_smem(k_coulomb<float, true>, coulomb_smem_bytes(false));
        if (e) return e;
        e = allow_smem(k_coulomb_inter<float>, inter_smem_bytes(false));
        if (e) return e;
    }
    return allow_smem(k_sort_cellscan, sizeof(int) * (L.maxN + 2));
}

cudaError_t launch_field(bool fp64, bool diag, int mode, const WsPtrs &W, int par, const LaunchCfg &L,
                         cudaStream_t st)
{
    const int csize = L.maxN + 1 > FIELD_ONE + 1 ? FIELD_CLUSTER : 1;
    const int grid = (W.D + (mode == 0 ? 1 : 0)) * csize;
    if (fp64)
        launch_cluster(k_field<double>, grid, FIELD_THREADS, csize, st, 0, W, par, diag ? 1 : 0, mode, csize);
    else
        launch_cluster(k_field<float>, grid, FIELD_THREADS, csize, st, 0, W, par, diag ? 1 : 0, mode, csize);
    return cudaGetLastError();
}

cudaError_t launch_births(bool fp64, const WsPtrs &W, const void *pools, int par, cudaStream_t st)
{
    const int blocks = W.max_chunks / TILE_ALIGN + 1;
    if (fp64)
        launch_k(k_births<double>, blocks, FIELD_THREADS, 0, st, W, *static_cast<const Pools<double> *>(pools), par);
    else
        launch_k(k_births<float>, blocks, FIELD_THREADS, 0, st, W, *static_cast<const Pools<float> *>(pools), par);
    return cudaGetLastError();
}

cudaError_t launch_births_field(bool fp64, bool diag, const WsPtrs &W, const void *pools, int par, const LaunchCfg &L,
                                cudaStream_t st)
{
    const int csize = L.maxN + 1 > FIELD_ONE + 1 ? FIELD_CLUSTER : 1;
    const int births = W.max_chunks / TILE_ALIGN + 1;
    const int grid = (W.D + 1) * csize + (births + csize - 1) / csize * csize;
    if (fp64)
        launch_cluster(k_births_field<double>, grid, FIELD_THREADS, csize, st, 0, W,
                       *static_cast<const Pools<double> *>(pools), par, diag ? 1 : 0, csize);
    else
        launch_cluster(k_births_field<float>, grid, FIELD_THREADS, csize, st, 0, W,
                       *static_cast<const Pools<float> *>(pools), par, diag ? 1 : 0, csize);
    return cudaGetLastError();
}

int kernels_per_sort() { return 4; }
int kernels_per_pair() { return 2; }

cudaError_t launch_sort(bool fp64, const WsPtrs &W, const void *pools, const int *tab, const LaunchCfg &L,
                        cudaStream_t st)
{
    const size_t scan_smem = sizeof(int) * (L.maxN + 2);
    const int cs_blocks = (L.sort_col_warps * 32 + 255) / 256;
    if (fp64) {
        const Pools<double> &P = *static_cast<const Pools<double> *>(pools);
        launch_k(k_sort_count<double>, L.sort_blocks, SORT_WARPS * 32, L.sort_smem, st, W, P, tab);
        launch_k(k_sort_colscan, cs_blocks, 256, 0, st, W, L.sort_warp_base);
        launch_k(k_sort_cellscan, W.D * NSP, 512, scan_smem, st, W);
        launch_k(k_sort_scatter<double>, L.sort_blocks, SORT_WARPS * 32, L.scatter_smem, st, W, P, tab);
    } else {
        const Pools<float> &P = *static_cast<const Pools<float> *>(pools);
        launch_k(k_sort_count<float>, L.sort_blocks, SORT_WARPS * 32, L.sort_smem, st, W, P, tab);
        launch_k(k_sort_colscan, cs_blocks, 256, 0, st, W, L.sort_warp_base);
        launch_k(k_sort_cellscan, W.D * NSP, 512, scan_smem, st, W);
        launch_k(k_sort_scatter<float>, L.sort_blocks, SORT_WARPS * 32, L.scatter_smem, st, W, P, tab);
    }
    return cudaGetLastError();
}

size_t coulomb_smem_bytes(bool fp64) { return (size_t)COUL_STAGE * 3 * (fp64 ? 8 : 4); }

template <typename Real>
static void launch_coulomb_real(const WsPtrs &W, const Pools<Real> &P, int par, bool groups, size_t smem, cudaStream_t st)
{
    const int cells = W.total_cells * NSP;
    if (groups)
        launch_k(k_coulomb<Real, true>, (cells + COUL_GROUP - 1) / COUL_GROUP, COUL_THREADS, smem, st, W, P, par);
    else
        launch_k(k_coulomb<Real, false>, cells, COUL_THREADS, smem, st, W, P, par);
}

cudaError_t launch_coulomb(bool fp64, const WsPtrs &W, const void *pools, int par, const LaunchCfg &L, cudaStream_t st)
{
    const size_t smem = coulomb_smem_bytes(fp64);
    if (fp64)
        launch_coulomb_real<double>(W, *static_cast<const Pools<double> *>(pools), par, L.coul_groups, smem, st);
    else
        launch_coulomb_real<float>(W, *static_cast<const Pools<float> *>(pools), par, L.coul_groups, smem, st);
    return cudaGetLastError();
}

cudaError_t launch_coulomb_inter(bool fp64, const WsPtrs &W, const void *pools, int par, cudaStream_t st)
{
    const size_t smem = inter_smem_bytes(fp64);
    if (fp64)
        launch_k(k_coulomb_inter<double>, W.total_cells, COUL_THREADS, smem, st, W,
                 *static_cast<const Pools<double> *>(pools), par, COUL_STAGE);
    else
        launch_k(k_coulomb_inter<float>, W.total_cells, COUL_THREADS, smem, st, W,
                 *static_cast<const Pools<float> *>(pools), par, COUL_STAGE);
    return cudaGetLastError();
}

cudaError_t launch_pair_reactions(bool fp64, const WsPtrs &W, const void *pools, int par, int k0, int k1, cudaStream_t st)
{
    const int blocks = (W.total_cells + PAIR_CELLS - 1) / PAIR_CELLS;
    if (fp64)
        launch_k(k_pair<double>, blocks, PAIR_THREADS, 0, st, W, *static_cast<const Pools<double> *>(pools), par, k0, k1);
    else
        launch_k(k_pair<float>, blocks, PAIR_THREADS, 0, st, W, *static_cast<const Pools<float> *>(pools), par, k0, k1);
    return cudaGetLastError();
}

cudaError_t launch_pair_append(bool fp64, const WsPtrs &W, const void *pools, const LaunchCfg &L, cudaStream_t st)
{
    if (fp64)
        launch_k(k_pair_append<double>, W.D, 256, sizeof(int) * (L.maxN + 1), st, W,
                 *static_cast<const Pools<double> *>(pools));
    else
        launch_k(k_pair_append<float>, W.D, 256, sizeof(int) * (L.maxN + 1), st, W,
                 *static_cast<const Pools<float> *>(pools));
    return cudaGetLastError();
}

cudaError_t launch_pair(bool fp64, const WsPtrs &W, const void *pools, int par, const LaunchCfg &L,
                        cudaStream_t st)
{
    const cudaError_t e = launch_pair_reactions(fp64, W, pools, par, 0, 3, st);
    if (e) return e;
    return launch_pair_append(fp64, W, pools, L, st);
}

cudaError_t launch_retile(const WsPtrs &W, int par, cudaStream_t st)
{
    launch_k(k_retile, 1, 256, 0, st, W, par);
    return cudaGetLastError();
}

cudaError_t launch_load(bool fp64, const WsPtrs &W, const void *pools, const long long *d_ninit,
                        const double *d_vt, int max_n, cudaStream_t st)
{
    dim3 grid((max_n + 255) / 256 > 0 ? ((max_n + 255) / 256 < 4096 ? (max_n + 255) / 256 : 4096) : 1,
              W.D * NSP);
    if (fp64)
        k_load<double><<<grid, 256, 0, st>>>(W, *static_cast<const Pools<double> *>(pools), d_ninit, d_vt);
    else
        k_load<float><<<grid, 256, 0, st>>>(W, *static_cast<const Pools<float> *>(pools), d_ninit, d_vt);
    return cudaGetLastError();
}

} // namespace o2
