// o2pic_static.cu -- charge deposit and field solve of one discharge from
// particle arrays the caller owns, with no memory allocation anywhere.
//
// Some callers cannot allocate device memory at all: code running inside a
// framework that owns every allocation, code that must not trigger a
// cudaMalloc (which can synchronise the device) in the middle of its own
// work, or code with a fixed memory budget checked up front.  For them the
// charge accumulators live in one file-scope __device__ array of fixed size
// (STATIC_MAX_CELLS + 1 nodes per species), which every GPU that loads this
// library reserves until the process exits.  The caller passes the particle
// arrays and the output arrays; this file never calls cudaMalloc, cudaFree
// or an allocating library routine.
#include <cooperative_groups.h>

#include <algorithm>
#include <mutex>
#include <string>

#include "../../include/o2pic.h"
#include "o2pic_dev.cuh"
#include "o2pic_launch.h"

namespace {

namespace cg = cooperative_groups;
using i128 = __int128;

constexpr int STATIC_MAX_CELLS = 4096;
constexpr int STATIC_NODES = STATIC_MAX_CELLS + 1;
constexpr double QE_S = 1.602176634e-19;
constexpr double EPS0_S = 8.8541878128e-12;
constexpr int MAX_DEVICES = 64;

// Per-species charge accumulators shared by every call on a device: fixed
// point (weight * 2^FIX_BITS) in the FP32 path, FP64 in the FP64 path; both
// 8 bytes per node.  3 * 4097 * 8 bytes = 98,328 bytes per device.
static __device__ __align__(256) unsigned long long g_static_acc[3 * STATIC_NODES];

std::mutex g_mu;
void *g_acc_ptr[MAX_DEVICES] = {};

// The three particle arrays of a call.
template <typename Real>
struct Particles {
    const int *cell[3];
    const Real *off[3];
    long long n[3];
    bool vec[3];  // both arrays start on a 16-byte (offsets: 4 elements) boundary
};

// Sums of a block, per CELL and in 32-bit words of shared memory: the number
// of particles in the cell and the sum of their upper weights w1 = offset in
// fixed point, cut into words small enough that every sum is exact.  Node i is
// then count_i - W_i + W_(i-1): the integer that adding both weights of every
// particle gives.  (64-bit shared atomics are several times slower than
// 32-bit ones on this part, and double ones slower still.)
//   FP32: w1 = rn(offset 2^24), words of 12 and 13 bits, 2^18 particles.
//   FP64: w1 = rn(offset 2^63), four words of 16 bits, 2^14 particles: exact for
//         offsets from 2^-11 on, rounded at 2^-64 of a particle below.  (With
//         2^-52 and three words, a node that held one small weight was further
//         from 64 bits than a double sum: 2000 particles in 4096 cells, rho off
//         by 1.4e-15 of a node's value against 7e-16; 1.3e-16 so.)
// The sums of all species may go into the same words, electrons and O- negative
// (modulo 2^32).
template <typename Real> struct Sums;
template <> struct Sums<float> {
    static constexpr int WORDS = 2, BITS = o2::FIX_BITS, SPLIT = 12;
    static constexpr long long MOST = 1ll << 18;  // slots between two flushes
    static constexpr bool RANGE = false;          // a flush is rare: it looks at every cell
    using Acc = unsigned long long;
    static __device__ __forceinline__ void weigh(float off, unsigned w[WORDS])
    {
        // an offset outside [0, 1] (or NaN) is clamped into it, so that the
        // two weights stay within [0, 2^FIX_BITS] and add up to one particle
        const unsigned v = __float2uint_rn(fminf(fmaxf(off, 0.0f), 1.0f) * (float)(1 << BITS));
        w[0] = v & ((1u << SPLIT) - 1u);
        w[1] = v >> SPLIT;
    }
    static __device__ __forceinline__ long long value(const unsigned w[WORDS])
    {
        return (long long)(int)w[1] * (1 << SPLIT) + (int)w[0];
    }
    // a node's sum, from the words of its cell and of the cell before it
    static __device__ __forceinline__ i128 node(int cnt, const unsigned w[WORDS], const unsigned p[WORDS])
    {
        return (i128)((long long)cnt * (1 << BITS) - value(w) + value(p));
    }
    static __device__ __forceinline__ void flush(Acc *a, i128 v) { atomicAdd(a, (Acc)(long long)v); }
    static __device__ __forceinline__ i128 read(Acc v) { return (i128)(long long)v; }
};
template <> struct Sums<double> {
    static constexpr int WORDS = 4, BITS = 63;
    static constexpr long long MOST = 1ll << 14;
    static constexpr bool RANGE = true;  // a flush is frequent: it looks at the cells between the lowest and highest
    using Acc = double;
    static __device__ __forceinline__ void weigh(double off, unsigned w[WORDS])
    {
        // outside [0, 1): clamped as in the FP32 path; the weight's bits come from
        // the offset's (integer units throughout: FP64 has two units per SM here)
        if ((unsigned)__double2hiint(off) >= 0x3FF00000u) off = fmin(fmax(off, 0.0), 1.0);
        const unsigned long long b = (unsigned long long)__double_as_longlong(off) & 0x7FFFFFFFFFFFFFFFull;
        const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
        const int sh = (int)(b >> 52) - 1012;  // off = m 2^(sh - 63)
        const unsigned long long v =
            sh >= 0 ? m << sh : (sh >= -53 ? (m + (1ull << (-sh - 1))) >> -sh : 0ull);
#pragma unroll
        for (int j = 0; j < WORDS; ++j) w[j] = (unsigned)(v >> (16 * j)) & 0xFFFFu;
    }
    static __device__ __forceinline__ i128 value(const unsigned w[WORDS])
    {
        i128 v = (int)w[WORDS - 1];
#pragma unroll
        for (int j = WORDS - 2; j >= 0; --j) v = v * 65536 + (int)w[j];
        return v;
    }
    static __device__ __forceinline__ i128 node(int cnt, const unsigned w[WORDS], const unsigned p[WORDS])
    {
        return (i128)cnt * ((i128)1 << BITS) - value(w) + value(p);
    }
    static __device__ __forceinline__ void flush(Acc *a, i128 v)
    {
        atomicAdd(a, (double)v * (1.0 / 9223372036854775808.0));
    }
    // a sum of multiples of 2^-63 (any rounding of the atomics is coarser)
    static __device__ __forceinline__ i128 read(Acc v)
    {
        const double hi = floor(v);
        return (i128)(long long)hi * ((i128)1 << BITS) + (i128)(long long)((v - hi) * 9223372036854775808.0);
    }
};

constexpr int UNIT_THREADS = 512;         // threads of a deposit block
constexpr int UNIT = 4 * UNIT_THREADS;    // slots a block takes at a time, four consecutive ones per thread
constexpr int STATIC_CLUSTER = 8;

// Four consecutive slots of one species into the block's sums (cnt and the
// words, each an array of `stride` cells).  As in the push: lanes whose four
// slots sit in the first lane's cell (ordered particles) sum over the warp and
// one lane adds for all; a lane whose four share a cell adds them once.
// Every lane of the warp calls it; cells are -1 for nothing.  neg: subtracted.
template <typename Real>
__device__ __forceinline__ void add4(unsigned *cnt, int stride, const int c[4], const Real off[4], bool neg)
{
    using S = Sums<Real>;
    auto add = [neg](unsigned *p, unsigned v) { atomicAdd(p, neg ? 0u - v : v); };
    unsigned w[4][S::WORDS], sum[S::WORDS];
#pragma unroll
    for (int k = 0; k < 4; ++k) S::weigh(off[k], w[k]);
    const bool same = c[0] >= 0 && c[1] == c[0] && c[2] == c[0] && c[3] == c[0];
    const int c0 = __shfl_sync(0xffffffffu, c[0], 0);
    const bool in = same && c[0] == c0;
    const unsigned m = __ballot_sync(0xffffffffu, in);
#pragma unroll
    for (int j = 0; j < S::WORDS; ++j) sum[j] = w[0][j] + w[1][j] + w[2][j] + w[3][j];
    if (__popc(m) >= 4) {
        unsigned all[S::WORDS];
#pragma unroll
        for (int j = 0; j < S::WORDS; ++j) all[j] = __reduce_add_sync(0xffffffffu, in ? sum[j] : 0u);
        if ((threadIdx.x & 31) == 0) {
            add(&cnt[c0], 4u * (unsigned)__popc(m));
#pragma unroll
            for (int j = 0; j < S::WORDS; ++j) add(&cnt[(j + 1) * stride + c0], all[j]);
        }
        if (in) return;
    }
    if (same) {
        add(&cnt[c[0]], 4u);
#pragma unroll
        for (int j = 0; j < S::WORDS; ++j) add(&cnt[(j + 1) * stride + c[0]], sum[j]);
        return;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (c[k] < 0) continue;
        add(&cnt[c[k]], 1u);
#pragma unroll
        for (int j = 0; j < S::WORDS; ++j) add(&cnt[(j + 1) * stride + c[k]], w[k][j]);
    }
}

__device__ __forceinline__ void load4(const int *p, int v[4])
{
    const int4 t = __ldcs(reinterpret_cast<const int4 *>(p));
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void load4(const float *p, float v[4])
{
    const float4 t = __ldcs(reinterpret_cast<const float4 *>(p));
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void load4(const double *p, double v[4])
{
    const double2 a = __ldcs(reinterpret_cast<const double2 *>(p));
    const double2 b = __ldcs(reinterpret_cast<const double2 *>(p) + 1);
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}

// slots i .. i+3 of species s; a cell outside the grid counts as empty
template <typename Real>
__device__ __forceinline__ void fetch4(const Particles<Real> &P, int s, long long i, int N, int c[4], Real off[4])
{
    if (P.vec[s] && i + 4 <= P.n[s]) {
        load4(P.cell[s] + i, c);
        load4(P.off[s] + i, off);
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const bool in = i + k < P.n[s];
            c[k] = in ? P.cell[s][i + k] : -1;
            off[k] = in ? P.off[s][i + k] : Real(0);
        }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) c[k] = (unsigned)c[k] < (unsigned)N ? c[k] : -1;
}

template <typename Real>
__device__ __forceinline__ i128 node_of(const unsigned *cnt, int stride, int i)
{
    using S = Sums<Real>;
    unsigned w[S::WORDS], p[S::WORDS];
#pragma unroll
    for (int j = 0; j < S::WORDS; ++j) {
        w[j] = cnt[(j + 1) * stride + i];
        p[j] = i > 0 ? cnt[(j + 1) * stride + i - 1] : 0u;
    }
    return S::node((int)cnt[i], w, p);
}

// Charge deposit of many particles.  What bounds it: the particles' bytes
// (5e7 FP32 particles in 4096 cells: 400 MB, 59 us at the copy rate; 94 us
// here, 65 us without the additions) and the shared atomics.  Each block takes
// one contiguous share of the three species' units, sums it per cell in shared
// memory (one species at a time) and adds the cells it touched to the global
// accumulators.  Global atomics for every particle took 3900 us.
// Two blocks per SM with the next slots in flight: 94 us; three without: 103.
// (species s's accumulators start at acc + s * anodes)
template <typename Real>
__device__ __forceinline__ void deposit_share(typename Sums<Real>::Acc *acc, size_t anodes, const Particles<Real> &P, int N)
{
    using S = Sums<Real>;
    extern __shared__ __align__(16) unsigned ssum[];
    __shared__ int s_lo, s_hi;
    const int tid = threadIdx.x, stride = N + 1;
    long long units = 0;
#pragma unroll
    for (int s = 0; s < 3; ++s) units += (P.n[s] + UNIT - 1) / UNIT;
    // the block's share of the units, numbered through the three species
    const long long ub = units / gridDim.x * blockIdx.x + units % gridDim.x * blockIdx.x / gridDim.x;
    const long long ue = units / gridDim.x * (blockIdx.x + 1) + units % gridDim.x * (blockIdx.x + 1) / gridDim.x;
    for (int k = tid; k < (S::WORDS + 1) * stride; k += UNIT_THREADS) ssum[k] = 0u;
    if (tid == 0) {
        s_lo = N;
        s_hi = -1;
    }
    __syncthreads();
    long long u0 = 0;  // first unit of species s
#pragma unroll 1
    for (int s = 0; s < 3; ++s) {
        const long long u1 = u0 + (P.n[s] + UNIT - 1) / UNIT;
        long long a = max(ub, u0);
        const long long e = min(ue, u1);
        while (a < e) {
            const long long b = min(e, a + S::MOST / UNIT);
            int lo = N, hi = -1;
            // the next four slots are loaded before these are added up
            int c[4], cx[4];
            Real off[4], ox[4];
            fetch4<Real>(P, s, (a - u0) * UNIT + 4 * tid, N, c, off);
            for (long long q = a; q < b; ++q) {
                if (q + 1 < b) fetch4<Real>(P, s, (q + 1 - u0) * UNIT + 4 * tid, N, cx, ox);
                add4<Real>(ssum, stride, c, off, false);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (S::RANGE) {
                        hi = max(hi, c[k]);
                        lo = min(lo, c[k] >= 0 ? c[k] : N);
                    }
                    c[k] = cx[k];
                    off[k] = ox[k];
                }
            }
            if (S::RANGE) {
                lo = __reduce_min_sync(0xffffffffu, lo);
                hi = __reduce_max_sync(0xffffffffu, hi);
                if ((tid & 31) == 0 && hi >= 0) {
                    atomicMin(&s_lo, lo);
                    atomicMax(&s_hi, hi);
                }
            }
            __syncthreads();
            lo = S::RANGE ? s_lo : 0;
            hi = S::RANGE ? s_hi : N - 1;
            for (int i = lo + tid; i <= hi + 1; i += UNIT_THREADS) {
                const i128 v = node_of<Real>(ssum, stride, i);
                if (v != 0) S::flush(&acc[s * anodes + i], v);
            }
            __syncthreads();
            for (int i = lo + tid; i <= hi; i += UNIT_THREADS)
#pragma unroll
                for (int j = 0; j <= S::WORDS; ++j) ssum[j * stride + i] = 0u;
            if (tid == 0) {
                s_lo = N;
                s_hi = -1;
            }
            __syncthreads();
            a = b;
        }
        u0 = u1;
    }
}

template <typename Real>
__global__ void __launch_bounds__(UNIT_THREADS, 2)
k_static_deposit(typename Sums<Real>::Acc *acc, Particles<Real> P, int N)
{
    o2::pdl_wait();
    deposit_share<Real>(acc, STATIC_NODES, P, N);
}

// The same for the state of a handle's discharges (one, or blockIdx.y of all):
// after the load and after a state was replaced.  The caller has cleared the
// accumulators.  With two global atomics per particle it took 215 us for 1e6
// FP32 particles in 501 cells, 7 us here.
__device__ __forceinline__ unsigned long long *acc_of(const o2::WsPtrs &W, float) { return W.acc_fix; }
__device__ __forceinline__ double *acc_of(const o2::WsPtrs &W, double) { return W.acc_dbl; }
template <typename Real>
__global__ void __launch_bounds__(UNIT_THREADS, 2)
k_deposit_disc(o2::WsPtrs W, o2::Pools<Real> P, int only)
{
    const int d = only >= 0 ? only : (int)blockIdx.y;
    const o2::Disc &Dd = W.disc[d];
    const unsigned b0 = W.ctl->cur ? P.stride : 0u;
    Particles<Real> A{};
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        const size_t at = (size_t)b0 + Dd.pbase[s];  // a multiple of the tile size
        A.cell[s] = P.cell[0] + at;
        A.off[s] = P.off[0] + at;
        A.n[s] = W.cnt[d * o2::NSP + s].n;
        A.vec[s] = true;
    }
    deposit_share<Real>(acc_of(W, Real(0)) + Dd.gbase, (size_t)W.total_nodes, A, Dd.N);
}

// What the solve needs of the discharge.  The constants are formed on the
// host: an FP64 division by every thread costs more here than the whole solve.
struct SolveC {
    int N;
    double dx, phi0;
    double c;   // e weight dx / eps0 per unit of charge (K dx)
    double h;   // c / (2 dx)
    double rs;  // e weight / dx per unit of charge
    double *rho, *phi, *E;
};

__device__ __forceinline__ i128 shfl_up128(i128 v, int o)
{
    const unsigned long long lo = __shfl_up_sync(0xffffffffu, (unsigned long long)v, o);
    const long long hi = __shfl_up_sync(0xffffffffu, (long long)(v >> 64), o);
    return ((i128)hi << 64) | (i128)lo;
}

// The Dirichlet problem (phi_{i-1} - 2 phi_i + phi_{i+1}) = -rho_i dx^2 / eps0,
// phi_0 = U(t), phi_N = 0, by two prefix sums over the nodes' net charge q_i,
// both exact (integers): S1_i = sum q, S2_i = sum S1 over the interior,
// phi_i = phi_0 + i D0 - c S2_{i-1}, E_i = (c / 2dx) (S1_i + S1_{i-1}) - D0/dx,
// with Gauss's law on the half cells at the walls.  Thread t of block `rank`
// of a cluster of `csize` holds nodes lo .. hi-1.
template <int NT, int PER>
__device__ void static_solve(const SolveC &C, int csize, int rank, int lo, int hi, const i128 q[PER])
{
    constexpr int NW = NT / 32;
    __shared__ i128 w1[NW], w2[NW], c1[STATIC_CLUSTER], c2[STATIC_CLUSTER];
    // warps that can hold nodes
    const int NC = (C.N + csize) / csize, per = (NC + NT - 1) / NT, nw = ((NC + per - 1) / per + 31) / 32;
    const int N = C.N, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // S2_i = (S1 of the threads before) x (nodes so far) + the thread's own,
    // so both prefixes come from one exchange of (charge, own S2, nodes)
    i128 run = 0, own = 0;
    int m = 0;  // the thread's interior nodes
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int i = lo + k;
        if (i < hi && i > 0 && i < N) {
            run += q[k];
            own += run;
            ++m;
        }
    }
    // fold a later stretch (r, o, m') into an earlier one (R, O): charge R + r,
    // S2 of both O + o + m' R
    i128 R = run, O = own;
    int M = m;
    if (warp < nw)  // (the other warps hold no nodes)
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const i128 r = shfl_up128(R, o), p = shfl_up128(O, o);
        const int mm = __shfl_up_sync(0xffffffffu, M, o);
        if (lane >= o) {
            O += p + (i128)M * r;
            R += r;
            M += mm;
        }
    }
    __shared__ int wm[NW], cm[STATIC_CLUSTER];
    if (lane == 31) {
        w1[warp] = R;
        w2[warp] = O;
        wm[warp] = M;
    }
    // the prefix before this thread within its warp
    i128 pr = shfl_up128(R, 1), po = shfl_up128(O, 1);
    int pm = __shfl_up_sync(0xffffffffu, M, 1);
    if (lane == 0) {
        pr = 0;
        po = 0;
        pm = 0;
    }
    __syncthreads();
    auto fold = [](i128 &r, i128 &o, i128 r2, i128 o2, int m2) {  // (r, o) then (r2, o2, m2)
        o += o2 + (i128)m2 * r;
        r += r2;
    };
    i128 br = 0, bo = 0;  // everything before this thread
    i128 tr = 0, to = 0;  // everything (the first warp)
    if (csize > 1) {
        cg::cluster_group cl = cg::this_cluster();
        if (tid < csize) {
            i128 r = 0, o = 0;
            int mm = 0;
            for (int w = 0; w < nw; ++w) {
                fold(r, o, w1[w], w2[w], wm[w]);
                mm += wm[w];
            }
            *cl.map_shared_rank(&c1[rank], tid) = r;
            *cl.map_shared_rank(&c2[rank], tid) = o;
            *cl.map_shared_rank(&cm[rank], tid) = mm;
        }
        cl.sync();
        if (warp < nw) {
            for (int b = 0; b < rank; ++b) fold(br, bo, c1[b], c2[b], cm[b]);
            if (warp == 0) {
                tr = br;
                to = bo;
                for (int b = rank; b < csize; ++b) fold(tr, to, c1[b], c2[b], cm[b]);
            }
        }
    } else if (warp == 0) {
        for (int w = 0; w < nw; ++w) fold(tr, to, w1[w], w2[w], wm[w]);
    }
    if (warp < nw) {
        for (int w = 0; w < warp; ++w) fold(br, bo, w1[w], w2[w], wm[w]);
        fold(br, bo, pr, po, pm);
    }
    __shared__ double s_D0, s_e0;
    if (tid == 0) {
        s_D0 = (C.c * (double)to - C.phi0) / (double)N;
        s_e0 = s_D0 / C.dx;
    }
    __syncthreads();
    const double D0 = s_D0, e0 = s_e0;
    i128 s1 = br, s2 = bo;  // S1_{i-1}, S2_{i-1}
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int i = lo + k;
        if (i >= hi) break;
        i128 T;
        double p;
        if (i == 0) {
            T = -2 * q[k];
            p = C.phi0;
        } else if (i == N) {
            T = 2 * (s1 + q[k]);
            p = 0.0;
        } else {
            T = 2 * s1 + q[k];
            p = C.phi0 + (double)i * D0 - C.c * (double)s2;
            s1 += q[k];
            s2 += s1;
        }
        C.rho[i] = (double)q[k] * ((i == 0 || i == N) ? 2.0 * C.rs : C.rs);
        C.phi[i] = p;
        C.E[i] = C.h * (double)T - e0;
    }
}

// The solve from the global accumulators: one block up to SOLVE_ONE cells, a
// cluster of 8 beyond.  Whole call for 1.8e5 slots, one block / a cluster, FP32
// and FP64: 128 cells 7.7 / 8.5 and 10.3 / 10.9 us, 256 cells 8.3 / 8.5 and 11.4 /
// 11.1, 512 cells 9.2 / 8.7 and 13.8 / 11.6, 1024 cells 10.9 / 9.3 and 17.8 / 12.6.
constexpr int SOLVE_THREADS = 256, SOLVE_PER = 5, SOLVE_ONE = 256;
template <typename Real>
__global__ void __launch_bounds__(SOLVE_THREADS)
k_static_solve(const typename Sums<Real>::Acc *acc, SolveC C, int csize)
{
    using S = Sums<Real>;
    o2::pdl_wait();
    if (csize > 1) cg::this_cluster().sync();  // every block has started
    const int rank = blockIdx.x, tid = threadIdx.x, NC = (C.N + csize) / csize;
    const int per = (NC + SOLVE_THREADS - 1) / SOLVE_THREADS;
    const int lo = min(rank * NC + tid * per, C.N + 1);
    const int hi = min(min(lo + per, (rank + 1) * NC), C.N + 1);
    i128 q[SOLVE_PER];
#pragma unroll
    for (int k = 0; k < SOLVE_PER; ++k) {
        q[k] = 0;
        if (lo + k < hi)
            q[k] = S::read(acc[2 * STATIC_NODES + lo + k]) - S::read(acc[lo + k]) - S::read(acc[STATIC_NODES + lo + k]);
    }
    static_solve<SOLVE_THREADS, SOLVE_PER>(C, csize, rank, lo, hi, q);
}

// Deposit and solve of few particles in one launch: a cluster of 8 blocks,
// each with the net sums of its share of the particles (all three species) in
// its own shared memory; block r then collects its nodes from all eight and
// solves them.  What bounds it: the latency of its stages (4e4 FP64 particles
// in 128 cells: 12.4 us; the five launches it replaces with one thread's sums
// 53 us).  Divisions stay off the threads: FP64 runs on few units here.  Sums per
// species, three times the words to clear and to collect: the same time in up to
// 256 cells, 2000 FP64 particles in 4096 cells 46 us, 25 so.
constexpr int SMALL_PER = 2;  // nodes per thread: (4097 / 8) / 512
constexpr long long SMALL_MOST = 1ll << 17;  // slots: 2^14 per block (the FP64 sums' limit) and species units
static_assert(SMALL_MOST / STATIC_CLUSTER <= Sums<double>::MOST && SMALL_MOST / STATIC_CLUSTER <= Sums<float>::MOST, "");
template <typename Real>
__global__ void __launch_bounds__(UNIT_THREADS)
k_static_small(Particles<Real> P, SolveC C)
{
    using S = Sums<Real>;
    extern __shared__ __align__(16) unsigned ssum[];
    o2::pdl_wait();
    cg::cluster_group cl = cg::this_cluster();
    const int rank = blockIdx.x, tid = threadIdx.x, N = C.N, stride = N + 1;
    for (int k = tid; k < (S::WORDS + 1) * stride; k += UNIT_THREADS) ssum[k] = 0u;
    __syncthreads();
    // warps of 128 slots, dealt out block by block, so that the blocks' shares differ by one at most
    int u[4] = {0, 0, 0, 0};
#pragma unroll
    for (int s = 0; s < 3; ++s) u[s + 1] = u[s] + (int)((P.n[s] + 127) / 128);
    for (int q = rank + STATIC_CLUSTER * (tid >> 5); q < u[3]; q += STATIC_CLUSTER * (UNIT_THREADS / 32)) {
        const int s = q < u[1] ? 0 : (q < u[2] ? 1 : 2);
        int c[4];
        Real off[4];
        fetch4<Real>(P, s, (long long)(q - (s == 0 ? 0 : (s == 1 ? u[1] : u[2]))) * 128 + 4 * (tid & 31), N, c, off);
        add4<Real>(ssum, stride, c, off, s != 2);
    }
    cl.sync();
    const int NC = (N + STATIC_CLUSTER) / STATIC_CLUSTER;
    const int per = (NC + UNIT_THREADS - 1) / UNIT_THREADS;
    const int lo = min(rank * NC + tid * per, N + 1);
    const int hi = min(min(lo + per, (rank + 1) * NC), N + 1);
    // the block's nodes from the words of all eight blocks: eight lanes per
    // node, one block each (all their loads in flight at once), then summed
    __shared__ i128 s_q[STATIC_NODES / STATIC_CLUSTER + 2];
    {
        const int first = rank * NC, count = min(NC, N + 1 - first);
        const unsigned *o = cl.map_shared_rank(ssum, tid % STATIC_CLUSTER);
        for (int j0 = 0; j0 < count; j0 += UNIT_THREADS / STATIC_CLUSTER) {
            const int j = j0 + tid / STATIC_CLUSTER, i = first + j;
            i128 v = j < count ? node_of<Real>(o, stride, i) : (i128)0;
#pragma unroll
            for (int b = 1; b < STATIC_CLUSTER; b <<= 1) {
                const unsigned long long lo64 = __shfl_xor_sync(0xffffffffu, (unsigned long long)v, b);
                const long long hi64 = __shfl_xor_sync(0xffffffffu, (long long)(v >> 64), b);
                v += ((i128)hi64 << 64) | (i128)lo64;
            }
            if (j < count && tid % STATIC_CLUSTER == 0) s_q[j] = v;
        }
        __syncthreads();
    }
    i128 q[SMALL_PER];
#pragma unroll
    for (int k = 0; k < SMALL_PER; ++k) q[k] = lo + k < hi ? s_q[lo + k - rank * NC] : (i128)0;
    // the solve's exchange synchronises the cluster after these reads, before any block can end
    static_solve<UNIT_THREADS, SMALL_PER>(C, STATIC_CLUSTER, rank, lo, hi, q);
}

pic_status static_fail(pic_status s, const std::string &m)
{
    o2::set_last_error(m.c_str());
    return s;
}

// Reaches every kernel that a call may launch, whatever the first call's size
// and precision: asking for a kernel's attributes loads it.
template <typename Real>
cudaError_t static_setup()
{
    constexpr int most = (int)sizeof(unsigned) * (Sums<Real>::WORDS + 1) * STATIC_NODES;
    cudaError_t e = o2::allow_smem(k_static_deposit<Real>, most);
    if (e == cudaSuccess) e = o2::allow_smem(k_static_small<Real>, most);
    if (e == cudaSuccess) e = o2::allow_smem(k_static_solve<Real>, 0);
    return e;
}

template <typename Real>
cudaError_t static_run(void *acc, const int *const *cell, const void *const *off, const long long *n, const SolveC &C,
                       int num_sms, cudaStream_t st)
{
    using S = Sums<Real>;
    Particles<Real> P{};
    long long all = 0;
    for (int s = 0; s < 3; ++s) {
        P.cell[s] = cell[s];
        P.off[s] = static_cast<const Real *>(off[s]);
        P.n[s] = n[s];
        P.vec[s] = (reinterpret_cast<size_t>(cell[s]) & 15) == 0 && (reinterpret_cast<size_t>(off[s]) & 15) == 0;
        all += n[s];
    }
    const size_t sm = sizeof(unsigned) * (S::WORDS + 1) * (C.N + 1);
    if (all <= SMALL_MOST - 3 * 128 * STATIC_CLUSTER)  // a block's 128-slot shares stay within SMALL_MOST / 8
        return o2::launch_cluster(k_static_small<Real>, STATIC_CLUSTER, UNIT_THREADS, STATIC_CLUSTER, st, sm, P, C);
    // the array keeps the previous call's sums: clear it first
    cudaError_t e = cudaMemsetAsync(acc, 0, sizeof(unsigned long long) * 3 * STATIC_NODES, st);
    if (e != cudaSuccess) return e;
    typename S::Acc *a = static_cast<typename S::Acc *>(acc);
    // what fits on an SM by threads and shared memory; not more blocks than units
    const long long units = all / UNIT + 3;
    const int per_sm = (int)std::min<size_t>(2, (224u << 10) / (sm + 1024));
    const int grid = (int)std::min<long long>(units, (long long)num_sms * per_sm);
    e = o2::launch_k(k_static_deposit<Real>, grid, UNIT_THREADS, sm, st, a, P, C.N);
    if (e != cudaSuccess) return e;
    const int csize = C.N > SOLVE_ONE ? STATIC_CLUSTER : 1;
    return o2::launch_cluster(k_static_solve<Real>, csize, SOLVE_THREADS, csize, st, 0, a, C, csize);
}

} // namespace

namespace {
template <typename Real>
size_t deposit_smem(int maxN)
{
    return sizeof(unsigned) * (Sums<Real>::WORDS + 1) * (maxN + 1);
}
template <typename Real>
cudaError_t deposit_discs(const o2::WsPtrs &W, const o2::Pools<Real> &P, int disc, int maxN, long long max_slots,
                          int num_sms, cudaStream_t st)
{
    const size_t sm = deposit_smem<Real>(maxN);
    const int blocks = (int)std::min<long long>(max_slots / UNIT + 3, 2ll * num_sms);
    k_deposit_disc<Real><<<dim3(blocks, disc >= 0 ? 1 : W.D), UNIT_THREADS, sm, st>>>(W, P, disc);
    return cudaGetLastError();
}
} // namespace

cudaError_t o2::deposit_configure(bool fp64, const LaunchCfg &L)
{
    return fp64 ? allow_smem(k_deposit_disc<double>, deposit_smem<double>(L.maxN))
                : allow_smem(k_deposit_disc<float>, deposit_smem<float>(L.maxN));
}

cudaError_t o2::launch_deposit_all(bool fp64, const WsPtrs &W, const void *pools, int disc, long long max_slots,
                                   const LaunchCfg &L, cudaStream_t st)
{
    if (fp64)
        return deposit_discs<double>(W, *static_cast<const Pools<double> *>(pools), disc, L.maxN, max_slots, L.num_sms, st);
    return deposit_discs<float>(W, *static_cast<const Pools<float> *>(pools), disc, L.maxN, max_slots, L.num_sms, st);
}

extern "C" pic_status pic_field_solve_static(const pic_config *cfg, long long step, const int *const *d_cell,
                                             const void *const *d_off, const long long *n, double *d_rho,
                                             double *d_phi, double *d_E, void *cuda_stream)
{
    if (!cfg || !d_cell || !d_off || !n || !d_rho || !d_phi || !d_E)
        return static_fail(PIC_EINVAL, "pic_field_solve_static: NULL argument");
    const int N = cfg->n_cells;
    if (N < 2 || N > STATIC_MAX_CELLS)
        return static_fail(PIC_EINVAL, "pic_field_solve_static: n_cells must be in [2, 4096] (the size of "
                                       "its fixed scratch array)");
    if (!(cfg->L_m > 0) || !(cfg->dt_s > 0) || !(cfg->weight_m2 >= 0) || step < 0)
        return static_fail(PIC_EINVAL, "pic_field_solve_static: need L > 0, dt > 0, weight >= 0, step >= 0");
    if (cfg->precision != PIC_FP64 && cfg->precision != PIC_FP32_MIXED)
        return static_fail(PIC_EINVAL, "pic_field_solve_static: bad precision");
    for (int s = 0; s < 3; ++s)
        if (n[s] < 0 || (n[s] > 0 && (!d_cell[s] || !d_off[s])))
            return static_fail(PIC_EINVAL, "pic_field_solve_static: bad particle arrays");
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= MAX_DEVICES)
        return static_fail(PIC_ECUDA, std::string("pic_field_solve_static: cudaGetDevice: ") + cudaGetErrorString(e));
    void *acc = nullptr;
    static int num_sms[MAX_DEVICES];  // guarded by g_mu
    int sms = 0;
    {
        // set-up, once per device, with that device current: the device
        // address of the scratch array (its host-side name is only a handle)
        // and the kernels' shared-memory limits
        std::lock_guard<std::mutex> lock(g_mu);
        if (!g_acc_ptr[dev]) {
            void *p = nullptr;
            e = cudaGetSymbolAddress(&p, g_static_acc);
            if (e != cudaSuccess || !p)
                return static_fail(PIC_ECUDA, std::string("pic_field_solve_static: cudaGetSymbolAddress: ") +
                                                  cudaGetErrorString(e));
            e = cudaDeviceGetAttribute(&num_sms[dev], cudaDevAttrMultiProcessorCount, dev);
            if (e == cudaSuccess) e = static_setup<float>();
            if (e == cudaSuccess) e = static_setup<double>();
            if (e != cudaSuccess)
                return static_fail(PIC_ECUDA, std::string("pic_field_solve_static: ") + cudaGetErrorString(e));
            g_acc_ptr[dev] = p;
        }
        acc = g_acc_ptr[dev];
        sms = num_sms[dev];
    }
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const bool fp64 = cfg->precision == PIC_FP64;
    const double PI_S = 3.14159265358979323846;
    const double t = (double)step * cfg->dt_s;
    SolveC C{};
    C.N = N;
    C.dx = cfg->L_m / N;
    C.phi0 = cfg->U_rf_V * sin(2.0 * PI_S * cfg->f_rf_Hz * t + cfg->rf_phase);
    const double unit = fp64 ? 1.0 / 9223372036854775808.0 : 1.0 / (double)(1 << o2::FIX_BITS);
    C.c = QE_S * cfg->weight_m2 * unit * C.dx / EPS0_S;
    C.h = C.c / (2.0 * C.dx);
    C.rs = QE_S * cfg->weight_m2 * unit / C.dx;
    C.rho = d_rho;
    C.phi = d_phi;
    C.E = d_E;
    e = fp64 ? static_run<double>(acc, d_cell, d_off, n, C, sms, st) : static_run<float>(acc, d_cell, d_off, n, C, sms, st);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess)
        return static_fail(PIC_ECUDA, std::string("pic_field_solve_static: launch: ") + cudaGetErrorString(e));
    return PIC_OK;
}
