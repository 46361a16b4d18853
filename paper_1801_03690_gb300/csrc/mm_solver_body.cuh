// Persistent solver kernel: Algorithm 4 (projected preconditioned NCG) with
// its two inner solvers (Algorithm 1 on the scalar-potential stiffness and
// on the approximate Hessian of Eq. precond), run entirely on the device.
//
// One cooperative launch covers a whole minimisation.  The blocks form a
// team that moves through phases separated by team barriers; every phase is
// a pass over rows (one thread per SELL-32 row) that also writes per-block
// partial sums.  After a barrier every block reduces the same
// partials in the same fixed order, so all blocks hold bit-identical scalars
// and take the same branch at every decision (potential-solve convergence,
// li1-li3, line-search branches, beta*ZA, t1-t3) without host round trips or
// atomics on floating-point data.  Barrier waits are bounded: a wait that
// runs out sets the device error flag and every block leaves the kernel.
#pragma once
#include <cuda_runtime.h>
#include <math.h>

#include "mm_internal.cuh"

// MM_LARGE 1: the form for plain FP64 on meshes of many rows (mm_kern_s*_large.cu),
// where a potential step waits for memory rather than for the FP64 pipe.  There
// the branches that skip the multiply-adds of padding, and the registers that
// the minimiser's own state takes once it is inlined around the phases, keep
// loads from being issued early: 8.7 M unknowns took 368 us a CG step in the
// other form and 332 us in this one (without the branches or with the minimiser
// a function of its own alone: 366 and 367), 3.2 M 146 and 135 (1024 threads).  Below, the pipe
// and the fixed costs of a phase count: the other form is faster on 250,047
// unknowns (field step 26.1 against 27.9 ms) and on 29,791 (9.4 against 10.0).
#ifndef MM_LARGE
#define MM_LARGE 0
#endif
#if MM_LARGE
#define MM_OUTLINE __noinline__
#else
#define MM_OUTLINE
#endif

namespace mm {

namespace {

constexpr unsigned long long kBarrierTimeoutNs = 5000000000ull;  // 5 s per wait
constexpr int kWarps = MM_BLOCK / 32;
constexpr int kFlat = 4;         // team_reduce: values summed through shared memory at most

// A block's share of `items` (32-row slices, or rows that take a whole warp):
// full rounds, in which the team's warps take items in turn, and its part of
// the last, partial round, `count` items from `tail` on.  Turns spread the
// expensive rows (magnet surface, grain boundaries) over all blocks:
// contiguous ranges left a block waiting 7 to 9 us at the barriers of a step on
// 3.2 M unknowns.  Splitting the last round evenly keeps every SM at work on a
// mesh with fewer rows than threads (29,791 rows: 6 or 7 warps on each of
// the 152 SMs instead of 16 on 58 of them).
struct Share {
    int full, tail, count;
};

// Scalars of the running CG solve (Algorithm 1), kept by the lanes that fold
// the team's values.  Each is one lane's work: an FP64 instruction of every
// warp occupies the SM's FP64 pipe for 19 cycles a warp, and with the step
// length, beta and the stopping tests evaluated by all 16 (32) warps of a block
// the direction and update phases took 6.3 and 5.1 us at 512 threads (29,791
// rows) and 51.5 and 15.8 us at 1024 (3.2 M rows, FP32); now 5.9, 4.5, 49.3
// and 14.0.
struct CgScalars {
    double rz, rz_old;               // r.z, and before the last step
    double a, beta;                  // step length, beta
    double rmax;                     // FP32 solve: largest |r|^2 since the last update
    float af, betaf;
    double eps;                      // preconditioner solve: limit of |r| (li3)
    int stop;                        // the residual meets the solve's (or the update's) limit
};

struct TeamSmem {
    CgScalars cg;
    double v[kFlat][MM_BLOCK];       // one value per thread
    double w[MM_MAXRED][kWarps];     // one value per warp
    double res[MM_MAXRED];           // the team's values
    Share phi, nm, phi4;             // slices of the potential rows, magnetic rows, float4 groups of the former
    Share rows[MM_MAXLEV], coarse[MM_MAXLEV], dense;   // multigrid: slices of a level, its restriction's items, dense rows
    int dead;
};

struct Team {
    int nb;
    int rank;
    unsigned long long* count;   // arrival counter (barrier words [0..1])
    unsigned long long target;   // its value once the last barrier is complete
    int* err;
    double* part;
    TeamSmem* sm;
    int epoch;
    bool dead;
};

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Arrival and wait of one thread per block.  The 64-bit counter only grows
// (zeroed by the host before each launch): the k-th barrier is complete once
// it reaches k * nb.  A release-add publishes the block's writes (those of
// its other threads are ordered before it by the block barrier) and an
// acquire-load that sees the target makes every other block's visible.  The
// wait is bounded: it ends with the device error flag set, which the other
// blocks' waits look at now and then.  What bounds it is the chain of L2
// round trips (write drain, add, load), so there is nothing else in it:
// an atomic with its result, two full fences, a sleep and a look at the
// error flag on each side took 1.91 us per empty barrier at 304 blocks of
// 256 threads and 2.35 us at 608; this form takes 1.25 us at 152 x 512 and
// 1.29 us at 152 x 1024 (one block per SM) and 1.42 / 2.28 us at the old
// grids.  An all-gather of tagged values without a counter took 3.2 us and
// more (every block polls every other's line).
__device__ __forceinline__ bool team_arrive_wait(Team& t) {
    asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(t.count), "l"(1ull) : "memory");
    unsigned long long seen;
    unsigned spin = 0;
    unsigned long long t0 = 0;
    while (true) {
        asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(seen) : "l"(t.count) : "memory");
        if (seen >= t.target) return true;
        if ((++spin & 1023u) == 0) {
            if (*(volatile int*)t.err) return false;
            const unsigned long long now = global_ns();
            if (t0 == 0) t0 = now;
            if (now - t0 > kBarrierTimeoutNs) {
                atomicCAS(t.err, 0, (int)ST_TIMEOUT);
                return false;
            }
        }
    }
}

// Team barrier with a bounded wait: the writes of every block before it are
// visible to every block after it.
__device__ bool team_sync(Team& t) {
    t.target += (unsigned long long)t.nb;
    __syncthreads();
    if (threadIdx.x == 0 && !team_arrive_wait(t)) t.sm->dead = 1;
    __syncthreads();
    t.dead = t.sm->dead != 0;
    return !t.dead;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Sum (or maximum) of N values in a fixed order, as a tree: the FP64 adder
// answers after 64 cycles and takes a warp every 19, so depth counts.
template <int N>
__device__ __forceinline__ double fold_tree(double (&a)[N], bool sum) {
#pragma unroll
    for (int h = 1; h < N; h *= 2) {
#pragma unroll
        for (int i = 0; i + h < N; i += 2 * h) a[i] = sum ? a[i] + a[i + h] : fmax(a[i], a[i + h]);
    }
    return a[0];
}

// Over the lanes of a warp; the result is lane 0's.
__device__ __forceinline__ double warp_fold(double v, bool sum) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double u = __shfl_down_sync(0xffffffffu, v, o);
        v = sum ? v + u : fmax(v, u);
    }
    return v;
}

// Sums of KP (a power of two, at most 32) values over the lanes of a warp in
// KP - 1 + log2(32 / KP) additions: a pair of lanes shares each round's work,
// one keeping the lower half of the values and the other the upper half.
// The sum of value k ends in lane (32 / KP) * k.
template <int KP>
__device__ __forceinline__ double warp_sums_shared(double (&v)[KP]) {
    const int lane = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int n = KP / 2; n >= 1; n /= 2) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const double give = up ? v[i] : v[i + n];
            const double keep = up ? v[i + n] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
        o >>= 1;
    }
#pragma unroll
    for (int r = 16 / KP; r > 0; r >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], r);
    return v[0];
}

// Second half of a team reduction: the block's partial values of K
// quantities (the first NS sums, the others maxima) are in `part`; after the
// barrier every block folds all partials identically, one warp per quantity,
// into t.sm->res.  fin(k, value) runs on the lane that folded value k; what it
// writes to shared memory every thread may read afterwards.
struct NoFinish {
    __device__ void operator()(int, double) const {}
};
template <int K, int NS, class Fin>
__device__ __forceinline__ bool team_combine(Team& t, const double* part, Fin fin) {
    if (!team_sync(t)) return false;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k = warp; k < K; k += kWarps) {
        const double* pk = part + (size_t)k * t.nb;
        const bool sum = k < NS;
        double s = 0.0;                       // the maxima are of values >= 0
        for (int j0 = 0; j0 < t.nb; j0 += 5 * 32) {
            double a[5];
#pragma unroll
            for (int u = 0; u < 5; ++u) {
                const int j = j0 + 32 * u + lane;
                a[u] = j < t.nb ? pk[j] : 0.0;
            }
            const double f = fold_tree<5>(a, sum);
            s = j0 == 0 ? f : sum ? s + f : fmax(s, f);
        }
        s = warp_fold(s, sum);
        if (lane == 0) {
            t.sm->res[k] = s;
            fin(k, s);
        }
    }
    __syncthreads();
    return true;
}

// Partials of this reduction (double buffered: a block may enter the next
// reduction while others still fold this one).
__device__ __forceinline__ double* team_partials(Team& t) {
    double* p = t.part + (size_t)(t.epoch & 1) * MM_MAXRED * t.nb;
    t.epoch++;
    return p;
}

// Reduce NS sums and NX maxima (of values >= 0) over the team, in FP64 and in
// a fixed order.  FP64 additions are what it costs: a full shuffle tree in
// every warp for every value issues 5 additions a warp, 80 per block and
// value pair, and took 7.6 us for two values (5.3 us for one) with the serial
// folds that followed.  Up to kFlat values therefore go through shared
// memory, where one warp per value sums MM_BLOCK / 32 of them per lane before
// its only tree; more values share their trees (warp_sums_shared).
template <int NS, int NX, class Fin = NoFinish>
__device__ bool team_reduce(Team& t, double (&s)[NS > 0 ? NS : 1], double (&x)[NX > 0 ? NX : 1], Fin fin = Fin()) {
    constexpr int K = NS + NX;
    static_assert(K <= MM_MAXRED, "too many reduction values");
    TeamSmem& sm = *t.sm;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double* part = team_partials(t);
    if constexpr (K <= kFlat) {
#pragma unroll
        for (int k = 0; k < NS; ++k) sm.v[k][threadIdx.x] = s[k];
#pragma unroll
        for (int k = 0; k < NX; ++k) sm.v[NS + k][threadIdx.x] = x[k];
        __syncthreads();
        if (warp < K) {
            const bool sum = warp < NS;
            double f = 0.0;
#pragma unroll 1
            for (int h = 0; h < kWarps; h += 8) {
                double a[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) a[u] = sm.v[warp][32 * (h + u) + lane];
                const double g = fold_tree<8>(a, sum);
                f = h == 0 ? g : sum ? f + g : fmax(f, g);
            }
            f = warp_fold(f, sum);
            if (lane == 0) part[(size_t)warp * t.nb + t.rank] = f;
        }
    } else {
        constexpr int KP = NS > 8 ? 16 : NS > 4 ? 8 : NS > 2 ? 4 : NS > 1 ? 2 : 1;
        double v[KP];
#pragma unroll
        for (int k = 0; k < KP; ++k) v[k] = k < NS ? s[k < NS ? k : 0] : 0.0;
        const double f = warp_sums_shared<KP>(v);
        constexpr int step = 32 / KP;
        if (lane % step == 0 && lane / step < NS) sm.w[lane / step][warp] = f;
#pragma unroll
        for (int k = 0; k < NX; ++k) {
            const double m = warp_fold(x[k], false);
            if (lane == 0) sm.w[NS + k][warp] = m;
        }
        __syncthreads();
        for (int k = warp; k < K; k += kWarps) {
            const double f2 = warp_fold(lane < kWarps ? sm.w[k][lane] : 0.0, k < NS);
            if (lane == 0) part[(size_t)k * t.nb + t.rank] = f2;
        }
    }
    if (!team_combine<K, NS>(t, part, fin)) return false;
#pragma unroll
    for (int k = 0; k < NS; ++k) s[k] = sm.res[k];
#pragma unroll
    for (int k = 0; k < NX; ++k) x[k] = sm.res[NS + k];
    return true;
}

// Team sums accumulated in FP32 per thread and warp (the FP32 phases, whose
// sums are all of positive terms), in FP64 across warps and blocks.
template <int NS, class Fin>
__device__ bool team_sum_f32(Team& t, float (&s)[NS], Fin fin) {
    TeamSmem& sm = *t.sm;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double* part = team_partials(t);
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        const float v = warp_sum(s[k]);
        if (lane == 0) sm.w[k][warp] = (double)v;
    }
    __syncthreads();
    if (warp < NS) {
        const double f = warp_fold(lane < kWarps ? sm.w[warp][lane] : 0.0, true);
        if (lane == 0) part[(size_t)warp * t.nb + t.rank] = f;
    }
    return team_combine<NS, NS>(t, part, fin);
}

// Team values of a CG step: d.q of the direction step gives the step length,
// r.z of the update gives beta and takes the old value's place.
__device__ __forceinline__ void cg_length(CgScalars& g, double dq) {
    g.a = g.rz / dq;
    g.af = (float)g.a;
}
__device__ __forceinline__ void cg_beta(CgScalars& g, double rz) {
    g.beta = rz / g.rz;
    g.betaf = (float)g.beta;
    g.rz_old = g.rz;
    g.rz = rz;
}
__device__ __forceinline__ bool is_zero(double v) { return (__double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFll) == 0; }

// What the team values of an FP32 solve's preconditioned residual are for: the
// first (mode INIT_FIRST), one after a reliable update (INIT_NEXT), one of a CG
// step (STEP).
enum CgMode { CG_INIT_FIRST, CG_INIT_NEXT, CG_STEP };
struct CgResidual {
    CgScalars& g;
    CgMode mode;
    double upd2, tol2;
    __device__ void operator()(int k, double s) const {
        if (k == 0) {
            if (mode == CG_INIT_FIRST) g.rz = s;
            else cg_beta(g, s);
        } else if (mode != CG_STEP) {
            g.rmax = s;
        } else {
            g.stop = s < upd2 * g.rmax || s < tol2;
            g.rmax = fmax(g.rmax, s);
        }
    }
};

struct Row {
    long long base;
    int width;
};

__device__ __forceinline__ Row sell_row(const long long* sptr, int r) {
    const int s = r >> 5;
    const long long b = sptr[s];
    return {b + (r & 31), (int)((sptr[s + 1] - b) >> 5)};
}

__device__ __forceinline__ Share make_share(const Team& t, int items) {
    const int stride = t.nb * kWarps, full = items / stride, left = items - full * stride;
    const int q = left / t.nb, m = left - q * t.nb;
    return {full, full * stride + q * t.rank + min(t.rank, m), q + (t.rank < m ? 1 : 0)};
}

// Item of this warp in round k = 0 .. full (-1: none).
__device__ __forceinline__ int team_item(const Team& t, const Share& h, int k) {
    const int warp = (int)(threadIdx.x >> 5);
    if (k < h.full) return (k * t.nb + t.rank) * kWarps + warp;
    return warp < h.count ? h.tail + warp : -1;
}

// Loop over this warp's items of a share (warp-uniform), and over this
// thread's rows r < n of a share of slices.
#define ITEMS(i, share)                                                       \
    for (int i##_k = 0, i##_f = (share).full; i##_k <= i##_f; ++i##_k)        \
        if (const int i = team_item(t, (share), i##_k); i >= 0)
#define ROWS(r, share, n)                                                     \
    ITEMS(r##_s, share)                                                       \
        if (const int r = 32 * r##_s + ((int)threadIdx.x & 31); r < (n))

// Row dot products over a SELL-32 row.  All column indices and values of a
// chunk are loaded before any gather, so each thread keeps a whole row's
// worth of independent loads in flight: measured on GB300 this lifts an FP32
// SpMV from 3.8 to 6.6 TB/s inside the persistent kernel.  The matrix
// entries are read once per product, so they are loaded with the
// evict-first (streaming) policy, which leaves L2 to the gathered vectors
// (+1.5% NCG iterations/s on the 8.7 M-unknown polycrystal).
// Entries past the slice's width (the same for the whole warp) gather x[pad]
// (pad = r for square matrices, 0 for rectangular ones whose row index may
// exceed the columns) and skip the FP64 multiply-add, which would occupy the
// SM's FP64 pipe for 19 cycles to add zero.
template <int CH, typename T, typename VT, typename XT>
__device__ __forceinline__ T sell_dot_row(const Row& A, const int* __restrict__ col, const VT* __restrict__ val,
                                          const XT* x, int pad) {
    T s = T(0);
    for (int k0 = 0; k0 < A.width; k0 += CH) {
        int c[CH];
        VT v[CH];
#pragma unroll
        for (int u = 0; u < CH; ++u) {
            const bool ok = k0 + u < A.width;
            const long long e = A.base + 32ll * (k0 + u);
            c[u] = ok ? __ldcs(col + e) : pad;
            v[u] = ok ? __ldcs(val + e) : VT(0);
        }
#pragma unroll
        for (int u = 0; u < CH; ++u) {
            const T g = (T)x[c[u]];
            if (MM_LARGE || sizeof(T) == 4 || k0 + u < A.width) s += (T)v[u] * g;
        }
    }
    return s;
}

template <int CH, typename T, typename VT, typename XT>
__device__ __forceinline__ T sell_dot(const long long* __restrict__ sptr, const int* __restrict__ col,
                                      const VT* __restrict__ val, const XT* x, int r, int pad) {
    return sell_dot_row<CH, T>(sell_row(sptr, r), col, val, x, pad);
}
template <int CH, typename T, typename VT, typename XT>
__device__ __forceinline__ T sell_dot(const long long* __restrict__ sptr, const int* __restrict__ col,
                                      const VT* __restrict__ val, const XT* x, int r) {
    return sell_dot<CH, T>(sptr, col, val, x, r, r);
}

// f(p, s, v) for the team's potential rows p with s = (K_phi x)_p in FP64 and
// v = pre(p), the row's vector operands.  A round is a chain of slice pointers,
// entries and gathers, each an L2 round trip, then the FP64 pipe: the pointers
// are read one round ahead and the vector operands before the product (left to
// the compiler they came after it: 26.1 against 22.2 us for a direction step on
// 250,047 rows of 15 entries).
template <typename XT, class Pre, class F>
__device__ __forceinline__ void phi_products(const Problem& P, const Team& t, const XT* x, Pre pre, F f) {
#if MM_LARGE
    for (int p = t.rank * MM_BLOCK + (int)threadIdx.x; p < P.nphi; p += t.nb * MM_BLOCK) {
        const double s = sell_dot_row<8, double>(sell_row(P.p_sptr, p), P.p_col, P.Kp, x, p);
        f(p, s, pre(p));
    }
#else
    const Share h = t.sm->phi;
    const int lane = threadIdx.x & 31;
    auto item = [&](int k) { return k <= h.full ? team_item(t, h, k) : -1; };
    auto slice = [&](int i) { return i < 0 ? Row{0, 0} : sell_row(P.p_sptr, 32 * i + lane); };
    int i = item(0);
    Row A = slice(i);
    for (int k = 0; k <= h.full; ++k) {
        const int ni = item(k + 1);
        const Row N = slice(ni);
        const int p = 32 * i + lane;
        if (i >= 0 && p < P.nphi) {
            const auto v = pre(p);
            f(p, sell_dot_row<8, double>(A, P.p_col, P.Kp, x, p), v);
        }
        i = ni;
        A = N;
    }
#endif
}
struct NoOperands {};
struct Operands {
    double a, b, c;
};

// Same for a scalar matrix applied to a SoA 3-vector (stride n); T the
// type of the sums and of the values (FP64, or FP32 in the precision form's
// preconditioner).
template <int CH, typename T>
__device__ __forceinline__ void sell_dot3(const long long* __restrict__ sptr, const int* __restrict__ col,
                                          const T* __restrict__ val, const T* x, int n, int r,
                                          T& s0, T& s1, T& s2) {
    const Row A = sell_row(sptr, r);
    s0 = s1 = s2 = T(0);
    for (int k0 = 0; k0 < A.width; k0 += CH) {
        int c[CH];
        T v[CH];
#pragma unroll
        for (int u = 0; u < CH; ++u) {
            const bool ok = k0 + u < A.width;
            const long long e = A.base + 32ll * (k0 + u);
            c[u] = ok ? __ldg(col + e) : r;
            v[u] = ok ? __ldg(val + e) : T(0);
        }
#pragma unroll
        for (int u = 0; u < CH; ++u) {
            const T g0 = x[c[u]], g1 = x[n + c[u]], g2 = x[2 * n + c[u]];
            if (sizeof(T) == 4 || k0 + u < A.width) {
                s0 += v[u] * g0;
                s1 += v[u] * g1;
                s2 += v[u] * g2;
            }
        }
    }
}

// Two SELL-32 rows r0 and r1 of different slices (two: r1 exists) per thread,
// CH entries of both rows loaded before any gather: twice the loads in
// flight of the one-row form at the register cost of CH = 16.  Used by the
// FP32 direction step and the level-0 products of the multigrid cycle,
// whose rows hold a handful of entries.  Lanes past a row's width read
// x[pad].
template <int CH, typename VT>
__device__ __forceinline__ void sell_dot_2rows(const long long* __restrict__ sptr, const int* __restrict__ col,
                                               const VT* __restrict__ val, const VT* x, int r0, int r1,
                                               bool two, int pad, VT& s0, VT& s1) {
    const Row A = sell_row(sptr, r0);
    const Row B = two ? sell_row(sptr, r1) : Row{0, 0};
    s0 = VT(0);
    s1 = VT(0);
    const int w = A.width > B.width ? A.width : B.width;
    for (int k0 = 0; k0 < w; k0 += CH) {
        int c0[CH], c1[CH];
        VT v0[CH], v1[CH];
#pragma unroll
        for (int u = 0; u < CH; ++u) {
            const bool ok0 = k0 + u < A.width, ok1 = k0 + u < B.width;
            c0[u] = ok0 ? __ldcs(col + A.base + 32ll * (k0 + u)) : pad;
            v0[u] = ok0 ? __ldcs(val + A.base + 32ll * (k0 + u)) : VT(0);
            c1[u] = ok1 ? __ldcs(col + B.base + 32ll * (k0 + u)) : pad;
            v1[u] = ok1 ? __ldcs(val + B.base + 32ll * (k0 + u)) : VT(0);
        }
#pragma unroll
        for (int u = 0; u < CH; ++u) {
            s0 += v0[u] * x[c0[u]];
            s1 += v1[u] * x[c1[u]];
        }
    }
}

// The offset table of the slice of row r (MM_NO_TAB in entry 0: the slice
// keeps its column array), two 16-byte loads that every lane of the warp
// makes at the same address.
struct SliceTab {
    int d[8];
};
__device__ __forceinline__ SliceTab slice_tab(const int* __restrict__ tab, int r) {
    const int4* t4 = reinterpret_cast<const int4*>(tab) + 2 * (r >> 5);
    const int4 a = __ldg(t4), b = __ldg(t4 + 1);
    return {{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w}};
}

// sell_dot_2rows for the FP32 K_phi layout with slice offset tables: when
// both rows' slices have a table (at most 8 entries per row), entry u of row
// r is column r + tab[u] and only the values are loaded; otherwise both rows
// go through sell_dot_2rows on the layout's columns.  The entries of a table
// slice are the row's couplings in column order with zeros for the offsets
// it lacks, so the sums are those of the plain layout.  Square matrices
// only (lanes past a row's width read x[r0]).
__device__ __forceinline__ void sell_dot_2rows_tab(const long long* __restrict__ sptr, const int* __restrict__ col,
                                                   const float* __restrict__ val, const int* __restrict__ tab,
                                                   const float* x, int r0, int r1, bool two, float& s0, float& s1) {
    const SliceTab ta = slice_tab(tab, r0);
    const SliceTab tb = slice_tab(tab, two ? r1 : r0);
    if (ta.d[0] == MM_NO_TAB || tb.d[0] == MM_NO_TAB) {
        sell_dot_2rows<8>(sptr, col, val, x, r0, r1, two, r0, s0, s1);
        return;
    }
    const Row A = sell_row(sptr, r0);
    const Row B = two ? sell_row(sptr, r1) : Row{0, 0};
    float v0[8], v1[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        v0[u] = u < A.width ? __ldcs(val + A.base + 32ll * u) : 0.0f;
        v1[u] = u < B.width ? __ldcs(val + B.base + 32ll * u) : 0.0f;
    }
    s0 = 0.0f;
    s1 = 0.0f;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        s0 += v0[u] * x[u < A.width ? r0 + ta.d[u] : r0];
        s1 += v1[u] * x[u < B.width ? r1 + tb.d[u] : r0];
    }
}

// One row of the same layout (sell_dot's one-row form, 16 entries per chunk).
__device__ __forceinline__ float sell_dot_tab(const long long* __restrict__ sptr, const int* __restrict__ col,
                                              const float* __restrict__ val, const int* __restrict__ tab,
                                              const float* x, int r) {
    const SliceTab ta = slice_tab(tab, r);
    if (ta.d[0] == MM_NO_TAB) return sell_dot<16, float>(sptr, col, val, x, r);
    const Row A = sell_row(sptr, r);
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = u < A.width ? __ldcs(val + A.base + 32ll * u) : 0.0f;
    float s = 0.0f;
#pragma unroll
    for (int u = 0; u < 8; ++u) s += v[u] * x[u < A.width ? r + ta.d[u] : r];
    return s;
}

// Loop over row pairs (r, r2): the rows of two rounds per thread; two: r2
// exists.
#define ROWS2(r, r2, two, share, n)                                                                          \
    for (int r##_k = 0, r##_f = (share).full, r2 = 0; r##_k <= r##_f; r##_k += 2)                            \
        if (const int r##_s = team_item(t, (share), r##_k); r##_s >= 0)                                      \
            if (const int r = 32 * r##_s + ((int)threadIdx.x & 31); r < (n))                                 \
                if (const int r##_t = r##_k < r##_f ? team_item(t, (share), r##_k + 1) : -1; true)           \
                    if (const bool two = r##_t >= 0 && (r2 = 32 * r##_t + ((int)threadIdx.x & 31)) < (n); true)

// The FP32 products of level 0 (K_phi and the smoothed prolongation) over the
// team's rows in the tile shape P.tile_rows selects; f(r, s, v) takes row r,
// its sum s and v = pre(r), the row's vector operands, which pre loads before
// the product's loads are issued: the vector loads then overlap the matrix
// loads and the gathers instead of following them.  Both shapes visit a
// thread's rows in the same order (its rows of the rounds), so
// per-thread sums f accumulates come out in the same order too.  tab: the
// slice offset tables of the FP32 K_phi (nullptr for other matrices).
// pad_self: lanes past a row's width gather x[r] (square matrices) rather
// than x[0].
template <class Pre, class F>
__device__ __forceinline__ void level0_products(const Problem& P, const Team& t, const long long* __restrict__ sptr,
                                                const int* __restrict__ col, const float* __restrict__ val,
                                                const int* __restrict__ tab, const float* x, int n, bool pad_self,
                                                Pre pre, F f) {
    if (P.tile_rows != 1) {
        ROWS2(r, r2, two, t.sm->phi, n) {
            const auto v0 = pre(r);
            const auto v1 = pre(two ? r2 : r);
            float s0, s1;
            if (tab) sell_dot_2rows_tab(sptr, col, val, tab, x, r, r2, two, s0, s1);
            else sell_dot_2rows<8>(sptr, col, val, x, r, r2, two, pad_self ? r : 0, s0, s1);
            f(r, s0, v0);
            if (two) f(r2, s1, v1);
        }
    } else {
        ROWS(r, t.sm->phi, n) {
            const auto v0 = pre(r);
            f(r, tab ? sell_dot_tab(sptr, col, val, tab, x, r) : sell_dot<16, float>(sptr, col, val, x, r, pad_self ? r : 0),
              v0);
        }
    }
}

// ---- row kernels of the three operators of Eq. (energy) on the magnetic
// graph, shared by the solver phases and the operator entry point.

// (D x)_p of a magnetic row p (Sec. 3.1: the right-hand side of the
// potential equation), x a SoA 3-vector over the magnetic nodes.
__device__ __forceinline__ double row_div(const Problem& P, const double* x, int p) {
    const int nm = P.nm;
    const long long nz = P.nnzm;
    const Row mr = sell_row(P.m_sptr, p);
    double bp = 0.0;
    for (int k0 = 0; k0 < mr.width; k0 += 8) {
        int c[8];
        double b0[8], b1[8], b2[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const bool ok = k0 + u < mr.width;
            const long long e = mr.base + 32ll * (k0 + u);
            c[u] = ok ? __ldg(P.m_col + e) : p;
            b0[u] = ok ? __ldg(P.B + e) : 0.0;
            b1[u] = ok ? __ldg(P.B + nz + e) : 0.0;
            b2[u] = ok ? __ldg(P.B + 2 * nz + e) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const double g0 = x[c[u]], g1 = x[nm + c[u]], g2 = x[2 * nm + c[u]];
            if (k0 + u < mr.width) bp += b0[u] * g0 + b1[u] * g1 + b2[u] * g2;
        }
    }
    return bp;
}

// (D^T phi)_i of a magnetic node i (the magnetostatic part of the gradient).
__device__ __forceinline__ void row_divT(const Problem& P, const double* phi, int i, double& t0, double& t1,
                                         double& t2) {
    const long long nz = P.nnzm;
    const Row rw = sell_row(P.m_sptr, i);
    t0 = t1 = t2 = 0.0;
    for (int k0 = 0; k0 < rw.width; k0 += 8) {
        int c[8];
        double q0[8], q1[8], q2[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const bool ok = k0 + u < rw.width;
            const long long e = rw.base + 32ll * (k0 + u);
            c[u] = ok ? __ldg(P.m_col + e) : i;
            q0[u] = ok ? __ldg(P.G + e) : 0.0;
            q1[u] = ok ? __ldg(P.G + nz + e) : 0.0;
            q2[u] = ok ? __ldg(P.G + 2 * nz + e) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (k0 + u < rw.width) {
                const double ph = phi[c[u]];
                t0 += q0[u] * ph;
                t1 += q1[u] * ph;
                t2 += q2[u] * ph;
            }
    }
}

// The local operators at node i: c = K_A x (exchange stiffness on each
// component; C_A x = 2 c) and a = C_K x (the lumped anisotropy block).
__device__ __forceinline__ void row_local(const Problem& P, const double* x, int i, double& c0, double& c1,
                                          double& c2, double& a0, double& a1, double& a2) {
    const int nm = P.nm;
    sell_dot3<8>(P.m_sptr, P.m_col, P.KA, x, nm, i, c0, c1, c2);
    const double x0 = x[i], x1 = x[nm + i], x2 = x[2 * nm + i];
    const double kxx = P.CK[i], kxy = P.CK[nm + i], kxz = P.CK[2 * nm + i];
    const double kyy = P.CK[3 * nm + i], kyz = P.CK[4 * nm + i], kzz = P.CK[5 * nm + i];
    a0 = kxx * x0 + kxy * x1 + kxz * x2;
    a1 = kxy * x0 + kyy * x1 + kyz * x2;
    a2 = kxz * x0 + kyz * x1 + kzz * x2;
}

struct SlotScalars {
    double F, terms[4], gmax, dphi, xdiff, xmax, M[3];
};

struct Ctx {
    const Problem* P;
    Team t;
    long long evals, nli, li, mi, ls_extra, mr;
    long long li2, li2_first, restarts, steepest;
    double h[3];
    SlotScalars sl[MM_NSLOT];
    int y_is_g;
    double ptol;             // relative residual the potential solves stop at
    double gy_prev;          // g_j . y_j of the last direction (beta*FR, beta*PRP)
};

// ---------------------------------------------------------------- phases

// x_s = N(x_c + a d), |x_c + a d| kept for Eq. (opt2); max|x_s - x_c|, max|x_s|.
__device__ bool ph_trial(Ctx& C, int c, int s, double a) {
    const Problem& P = *C.P;
    Team& t = C.t;
    const int nm = P.nm;
    double mx[2] = {0.0, 0.0};
    double dummy[1] = {0.0};
    const double* xc = P.X[c];
    double* xs = P.X[s];
    ROWS(i, t.sm->nm, nm) {
        double u0 = xc[i] + a * P.d[i];
        double u1 = xc[nm + i] + a * P.d[nm + i];
        double u2 = xc[2 * nm + i] + a * P.d[2 * nm + i];
        double n = sqrt(u0 * u0 + u1 * u1 + u2 * u2);
        double v0 = u0 / n, v1 = u1 / n, v2 = u2 / n;
        xs[i] = v0;
        xs[nm + i] = v1;
        xs[2 * nm + i] = v2;
        P.unorm[i] = n;
        mx[0] = fmax(mx[0], fmax(fabs(v0 - xc[i]), fmax(fabs(v1 - xc[nm + i]), fabs(v2 - xc[2 * nm + i]))));
        mx[1] = fmax(mx[1], fmax(fabs(v0), fmax(fabs(v1), fabs(v2))));
    }
    if (!team_reduce<0, 2>(t, dummy, mx)) return false;
    C.sl[s].xdiff = mx[0];
    C.sl[s].xmax = mx[1];
    return true;
}

// Potential-solve set-up: rhs = D x_s on the magnetic rows, r = rhs - K phi,
// z = diag(K)^-1 r.  Sums: |rhs|^2, r.z, |r|^2.
__device__ bool ph_pinit(Ctx& C, int s, double& bb, double& rz, double& rr) {
    const Problem& P = *C.P;
    Team& t = C.t;
    const int nm = P.nm;
    const double* x = P.X[s];
    double acc[3] = {0.0, 0.0, 0.0};
    double dummy[1] = {0.0};
    auto pre = [](int) { return NoOperands{}; };
    phi_products(P, t, P.phi, pre, [&](int p, double kphi, NoOperands) {
        double bp = 0.0;
        if (p < nm) {
            bp = row_div(P, x, p);
            P.rhs[p] = bp;
        }
        const double r = bp - kphi;
        const double z = r * P.dinvP[p];
        P.pres[p] = r;
        P.pprec[p] = z;
        acc[0] += bp * bp;
        acc[1] += r * z;
        acc[2] += r * r;
    });
    if (!team_reduce<3, 0>(t, acc, dummy)) return false;
    bb = acc[0];
    rz = acc[1];
    rr = acc[2];
    return true;
}

// Plain product q = K v (no reduction).
__device__ bool ph_pmatvec(Ctx& C, const double* v, double* q) {
    const Problem& P = *C.P;
    Team& t = C.t;
    phi_products(P, t, v, [](int) { return NoOperands{}; }, [&](int p, double s, NoOperands) { q[p] = s; });
    return team_sync(t);
}

// CG direction step of Algorithm 1 with the product formed by recurrence:
// w = K z, d = z + beta d, q = w + beta q (= K d), in place.  Sum: d . q.
__device__ bool ph_pdirection(Ctx& C, const double* z, double beta, double* d, double* q) {
    const Problem& P = *C.P;
    Team& t = C.t;
    double acc[1] = {0.0};
    double dummy[1] = {0.0};
    const bool first = is_zero(beta);
    auto pre = [&](int p) { return first ? Operands{z[p], 0.0, 0.0} : Operands{z[p], d[p], q[p]}; };
    phi_products(P, t, z, pre, [&](int p, double s, const Operands& v) {
        const double dn = first ? v.a : v.a + beta * v.b;
        const double qn = first ? s : s + beta * v.c;
        d[p] = dn;
        q[p] = qn;
        acc[0] += dn * qn;
    });
    CgScalars& g = t.sm->cg;
    return team_reduce<1, 0>(t, acc, dummy, [&g](int, double s) { cg_length(g, s); });
}

// phi += a v; r -= a q; z = diag^-1 r.  Sums: r.z, |r|^2 (against tol2).
__device__ bool ph_pupdate(Ctx& C, const double* v, double a, double tol2) {
    const Problem& P = *C.P;
    Team& t = C.t;
    double acc[2] = {0.0, 0.0};
    double dummy[1] = {0.0};
    ROWS(p, t.sm->phi, P.nphi) {
        P.phi[p] += a * v[p];
        const double r = P.pres[p] - a * P.pq[p];
        const double z = r * P.dinvP[p];
        P.pres[p] = r;
        P.pprec[p] = z;
        acc[0] += r * z;
        acc[1] += r * r;
    }
    CgScalars& g = t.sm->cg;
    return team_reduce<2, 0>(t, acc, dummy, [&g, tol2](int k, double s) {
        if (k == 0) cg_beta(g, s);
        else g.stop = !(s >= tol2);
    });
}

__device__ bool ph_pzero(Ctx& C) {
    const Problem& P = *C.P;
    Team& t = C.t;
    ROWS(p, t.sm->phi, P.nphi) {
        P.phi[p] = 0.0;
        P.pres[p] = 0.0;
    }
    return team_sync(t);
}

// ---- precision form of the potential solve: the correction equation
// K delta = r (r the FP64 residual) is solved by Algorithm 1 in FP32 (FP32
// operator, vectors and products; FP64 reductions); then phi += delta and
// r -= K delta in FP64 (iterative refinement of the FP64 residual).

// Compensated FP32 accumulation (Ogita, Rump and Oishi, "Accurate sum and
// dot product", SIAM J. Sci. Comput. 26 (2005), algorithm Dot2): the
// rounding error of every product (by FMA) and of every addition (by the
// two-sum transformation) is collected in a second FP32 word, so the result
// is as accurate as if computed in twice the working precision.  The
// restriction rows of the smoothed aggregates sum a few hundred terms that
// largely cancel; their rounding would otherwise enter the coarse
// correction amplified by the coarse inverse.
struct Dot2 {
    float p, s;
};

// (The _rn intrinsics keep the compiler from contracting the transformations
// into FMAs, which would break their exactness.)
__device__ __forceinline__ float two_sum(float a, float b, float& err) {
    const float x = __fadd_rn(a, b);
    const float z = __fsub_rn(x, a);
    err = __fadd_rn(__fsub_rn(a, __fsub_rn(x, z)), __fsub_rn(b, z));
    return x;
}

__device__ __forceinline__ void dot2_add(Dot2& d, float a, float b) {
    const float h = __fmul_rn(a, b);
    const float r = __fmaf_rn(a, b, -h);     // exact: a b = h + r
    float q;
    d.p = two_sum(d.p, h, q);
    d.s = __fadd_rn(d.s, __fadd_rn(q, r));
}

__device__ __forceinline__ void dot2_merge(Dot2& d, float p, float s) {
    float q;
    d.p = two_sum(d.p, p, q);
    d.s = __fadd_rn(d.s, __fadd_rn(s, q));
}

// The dot product of CSR row `row` (< 0: an empty row) with x, computed by a
// group of G consecutive lanes (G divides 32): lane gl of the group takes
// entries gl, gl + G, ..., CH per pass with all of a pass's loads issued
// before any gather, accumulates them compensated, and the group combines
// its lanes with a G-lane xor reduction (every lane of the warp takes part).
template <int G, int CH, class XF>
__device__ __forceinline__ float group_csr_dot2(const long long* __restrict__ ptr, const int* __restrict__ col,
                                                const float* __restrict__ val, XF x, int row, int gl) {
    const long long b = row >= 0 ? ptr[row] : 0, e = row >= 0 ? ptr[row + 1] : 0;
    Dot2 s = {0.0f, 0.0f};
    for (long long o = b + gl; o < e; o += (long long)G * CH) {
        int c[CH];
        float v[CH];
#pragma unroll
        for (int u = 0; u < CH; ++u) {
            const long long k = o + (long long)G * u;
            const bool ok = k < e;
            c[u] = ok ? __ldcs(col + k) : 0;
            v[u] = ok ? __ldcs(val + k) : 0.0f;
        }
#pragma unroll
        for (int u = 0; u < CH; ++u) dot2_add(s, v[u], x(c[u]));
    }
#pragma unroll
    for (int off = G / 2; off > 0; off >>= 1) {
        const float p = __shfl_xor_sync(0xffffffffu, s.p, off);
        const float q = __shfl_xor_sync(0xffffffffu, s.s, off);
        dot2_merge(s, p, q);
    }
    return s.p + s.s;
}

// ---- smoothed-aggregation multigrid V-cycle (the FP32 solve's
// preconditioner when a hierarchy exists and prm.amg is set); operators as
// in struct Level.  A down phase computes rpre = b - A x on the rows of its
// level (one thread per row), then, after a team barrier, b_{l+1} = P^T rpre
// and x_{l+1} = omega D^-1 b_{l+1} on the rows of the next level (a group of
// lanes per row).

// Restriction rows of a down phase: b_{l+1} = P^T r with r(j) given by bx,
// x_{l+1} = omega D^-1 b_{l+1}.  A group of G lanes per coarse row, so a
// warp works on 32 / G rows at once: at the fine end the rows of P^T hold
// tens of entries (2.9 per fine row on the lattice meshes), and a whole warp
// per row spent its time in the 5-level shuffle reduction.
template <int G, class XF>
__device__ __forceinline__ void amg_restrict_g(const Problem& P, const Team& t, const Level& V, int l, XF bx) {
    constexpr int RPW = 32 / G;
    const bool last = (l + 1 == P.nlev);
    float* bn = last ? P.bco : P.lev[l + 1].b;
    float* xn = last ? nullptr : P.lev[l + 1].x;
    const float* dn = last ? nullptr : P.lev[l + 1].dinv;
    const float on = last ? 0.0f : P.lev[l + 1].omega;
    const int lane = threadIdx.x & 31, grp = lane / G, gl = lane % G;
    ITEMS(I0, t.sm->coarse[l]) {
        const int I = I0 * RPW + grp;
        const float s = group_csr_dot2<G, 12>(V.t_ptr, V.t_col, V.t_val, bx, I < V.nc ? I : -1, gl);
        if (gl == 0 && I < V.nc) {
            bn[I] = s;
            if (!last) xn[I] = on * dn[I] * s;
        }
    }
}

// Lanes per restriction row.  Levels with long rows (the coarse end of the
// hierarchy: hundreds of entries) or with no more rows than the team has
// warps take a whole warp per row, whatever P.restrict_lanes says: with 8 lanes
// three quarters of the warps had no rows on the latter (field steps: 12
// platelets 37.9 ms, 36.9 now; 3.2 M-unknown polycrystal 97.0, 96.6 now).  The
// others take P.restrict_lanes lanes, 8 by default (measured on the
// 8.7 M-unknown polycrystal: 8 lanes 190 us, 4 lanes 211, 16 lanes 225 for the
// level-0 down phase).
__device__ __forceinline__ int restrict_group(const Problem& P, const Team& t, int l) {
    const Level& V = P.lev[l];
    if (V.wide || V.nc <= t.nb * kWarps) return 32;
    return P.restrict_lanes == 4 || P.restrict_lanes == 16 ? P.restrict_lanes : 8;
}

template <class XF>
__device__ __forceinline__ void amg_restrict(const Problem& P, const Team& t, const Level& V, int l, XF bx) {
    const int g = restrict_group(P, t, l);
    if (g == 32) amg_restrict_g<32>(P, t, V, l, bx);
    else if (g == 4) amg_restrict_g<4>(P, t, V, l, bx);
    else if (g == 16) amg_restrict_g<16>(P, t, V, l, bx);
    else amg_restrict_g<8>(P, t, V, l, bx);
}

// Down phase of level l; at level 0, b is the FP32 residual and x = omega
// D^-1 b has been written with it by the update step.  The pre-smoothed
// residual rpre is restricted after a team barrier with P^T, which holds
// half the entries of U^T (U^T b, the same vector, needs no barrier:
// measured on the 8.7 M-unknown polycrystal, the U^T restriction took 205
// of the phase's 323 us).
// rpre = b - A x on the rows of level 0 (K_phi, a handful of entries per
// row), a function of its own so that its registers are allocated apart
// from the restriction's.
__device__ __noinline__ void amg_down0_rows(const Problem& P, const Team& t) {
    const Level& V = P.lev[0];
    const float* b = P.pres32;
    level0_products(P, t, V.sptr, V.col, V.val, V.tab, P.amg_x0, V.n, true, [&](int r) { return b[r]; },
                    [&](int r, float s, float br) { V.rpre[r] = br - s; });
}

__device__ __noinline__ bool ph_amg_down(Ctx& C, int l) {
    const Problem& P = *C.P;
    Team& t = C.t;
    const Level& V = P.lev[l];
    if (l == 0) {
        amg_down0_rows(P, t);
    } else {
        ROWS(r, t.sm->rows[l], V.n) V.rpre[r] = V.b[r] - sell_dot<16, float>(V.sptr, V.col, V.val, V.x, r);
    }
    if (!team_sync(t)) return false;
    const float* rp = V.rpre;
    amg_restrict(P, t, V, l, [=](int j) { return rp[j]; });
    return team_sync(t);
}

// Coarsest level: y = A_c^-1 b, one warp per row of the dense inverse.
__device__ __noinline__ bool ph_amg_dense(Ctx& C) {
    const Problem& P = *C.P;
    Team& t = C.t;
    const int n = P.nco, lane = threadIdx.x & 31;
    ITEMS(row, t.sm->dense) {
        const float* a = P.ainv + (size_t)row * n;
        float s = 0.0f;
#pragma unroll 8
        for (int j = lane; j < n; j += 32) s += a[j] * P.bco[j];
        s = warp_sum(s);
        if (lane == 0) P.yco[row] = s;
    }
    return team_sync(t);
}

// Up phase of level l: y = omega D^-1 (b + rpre) + U y_{l+1}.  At level 0,
// y is the preconditioned residual z; sums r.z and |r|^2.
__device__ __noinline__ bool ph_amg_up(Ctx& C, int l, const CgResidual& fin) {
    const Problem& P = *C.P;
    Team& t = C.t;
    const Level& V = P.lev[l];
    const float* yc = (l + 1 == P.nlev) ? P.yco : P.lev[l + 1].y;
    const float* bv = (l == 0) ? P.pres32 : V.b;
    float acc[2] = {0.0f, 0.0f};
    // per row: b and omega D^-1 (b + rpre), loaded ahead of the product
    auto pre = [&](int r) {
        const float b = bv[r];
        return make_float2(b, V.omega * V.dinv[r] * (b + V.rpre[r]));
    };
    auto row = [&](int r, float s, float2 v) {
        const float y = v.y + s;
        V.y[r] = y;
        acc[0] += v.x * y;
        acc[1] += v.x * v.x;
    };
    if (l == 0) {
        level0_products(P, t, V.u_sptr, V.u_col, V.u_val, nullptr, yc, V.n, false, pre, row);
    } else {
        ROWS(r, t.sm->rows[l], V.n) {
            const float2 v = pre(r);
            row(r, sell_dot<16, float>(V.u_sptr, V.u_col, V.u_val, yc, r, 0), v);
        }
    }
    if (l > 0) return team_sync(t);
    return team_sum_f32<2>(t, acc, fin);
}

// z = V-cycle(r) for r = pres32, whose smoothed iterate amg_x0 = omega
// D^-1 r has been written (and a barrier passed) by the caller.  Sums r.z,
// |r|^2.
__device__ bool amg_vcycle(Ctx& C, const CgResidual& fin) {
    const Problem& P = *C.P;
    for (int l = 0; l < P.nlev; ++l)
        if (!ph_amg_down(C, l)) return false;
    if (!ph_amg_dense(C)) return false;
    for (int l = P.nlev - 1; l >= 0; --l)
        if (!ph_amg_up(C, l, fin)) return false;
    return true;
}

__device__ __forceinline__ bool use_amg(const Problem& P) { return P.prm.amg != 0 && P.nlev > 0; }

// r32 = r, z32 = M^-1 r32 (Jacobi or the V-cycle), delta = 0.  Sums: r.z, |r|^2.
__device__ bool ph_p32_init(Ctx& C, const CgResidual& fin) {
    const Problem& P = *C.P;
    Team& t = C.t;
    if (use_amg(P)) {
        ROWS(p, t.sm->phi, P.nphi) {
            const float r = (float)P.pres[p];
            P.pres32[p] = r;
            P.amg_x0[p] = P.amg_omega * P.dinvP32[p] * r;
            P.pdelta32[p] = 0.0f;
        }
        if (!team_sync(t)) return false;
        return amg_vcycle(C, fin);
    }
    float acc[2] = {0.0f, 0.0f};
    ROWS(p, t.sm->phi, P.nphi) {
        const float r = (float)P.pres[p];
        const float z = r * P.dinvP32[p];
        P.pres32[p] = r;
        P.pprec32[p] = z;
        P.pdelta32[p] = 0.0f;
        acc[0] += r * z;
        acc[1] += r * r;
    }
    return team_sum_f32<2>(t, acc, fin);
}

// FP32 direction step: d = z + beta d, q = K32 z + beta q.  Sum: d . q.
__device__ bool ph_p32_direction(Ctx& C, float beta) {
    const Problem& P = *C.P;
    Team& t = C.t;
    float acc[1] = {0.0f};
    const bool first = (beta == 0.0f);
    const float* z = P.pprec32;
    // per row: the new direction z + beta d and beta q, loaded ahead of the product
    auto pre = [&](int p) {
        return first ? make_float2(z[p], 0.0f) : make_float2(z[p] + beta * P.pdir32[p], beta * P.pq32[p]);
    };
    auto row = [&](int p, float s, float2 v) {
        const float qn = s + v.y;
        P.pdir32[p] = v.x;
        P.pq32[p] = qn;
        acc[0] += v.x * qn;
    };
    level0_products(P, t, P.k_sptr, P.k_col, P.Kp32, P.k_tab, z, P.nphi, true, pre, row);
    CgScalars& g = t.sm->cg;
    return team_sum_f32<1>(t, acc, [&g](int, double s) { cg_length(g, s); });
}

// delta += a d; r -= a q; z = M^-1 r.  Sums: r.z, |r|^2.
__device__ bool ph_p32_update(Ctx& C, float a, const CgResidual& fin) {
    const Problem& P = *C.P;
    Team& t = C.t;
    // Streaming pass in float4 (four rows per load; the FP32 vectors are
    // 256-byte aligned allocations), the n_phi % 4 tail in scalar form.
    // Measured on GB300 inside the solver kernel: 5.2 vs 8.1 us for a
    // three-vector pass over the bench mesh.
    const int n4 = P.nphi >> 2;
    float4* __restrict__ res4 = reinterpret_cast<float4*>(P.pres32);
    float4* __restrict__ del4 = reinterpret_cast<float4*>(P.pdelta32);
    const float4* __restrict__ dir4 = reinterpret_cast<const float4*>(P.pdir32);
    const float4* __restrict__ q4 = reinterpret_cast<const float4*>(P.pq32);
    const float4* __restrict__ dv4 = reinterpret_cast<const float4*>(P.dinvP32);
    if (use_amg(P)) {
        // no sums here: r.z and |r|^2 come with z from the V-cycle
        float4* __restrict__ x04 = reinterpret_cast<float4*>(P.amg_x0);
        const float om = P.amg_omega;
        ROWS(i, t.sm->phi4, n4) {
            const float4 d = dir4[i], q = q4[i], r = res4[i], e = del4[i], w = dv4[i];
            const float4 nr = make_float4(r.x - a * q.x, r.y - a * q.y, r.z - a * q.z, r.w - a * q.w);
            del4[i] = make_float4(e.x + a * d.x, e.y + a * d.y, e.z + a * d.z, e.w + a * d.w);
            res4[i] = nr;
            x04[i] = make_float4(om * w.x * nr.x, om * w.y * nr.y, om * w.z * nr.z, om * w.w * nr.w);
        }
        if (const int j = (int)threadIdx.x; t.rank == t.nb - 1 && j < P.nphi - 4 * n4) {
            const int p = 4 * n4 + j;
            P.pdelta32[p] += a * P.pdir32[p];
            const float r = P.pres32[p] - a * P.pq32[p];
            P.pres32[p] = r;
            P.amg_x0[p] = om * P.dinvP32[p] * r;
        }
        if (!team_sync(t)) return false;
        return amg_vcycle(C, fin);
    }
    float acc[2] = {0.0f, 0.0f};
    float4* __restrict__ z4 = reinterpret_cast<float4*>(P.pprec32);
    ROWS(i, t.sm->phi4, n4) {
        const float4 d = dir4[i], q = q4[i], r = res4[i], e = del4[i], w = dv4[i];
        const float4 nr = make_float4(r.x - a * q.x, r.y - a * q.y, r.z - a * q.z, r.w - a * q.w);
        const float4 z = make_float4(nr.x * w.x, nr.y * w.y, nr.z * w.z, nr.w * w.w);
        del4[i] = make_float4(e.x + a * d.x, e.y + a * d.y, e.z + a * d.z, e.w + a * d.w);
        res4[i] = nr;
        z4[i] = z;
        acc[0] += (nr.x * z.x + nr.y * z.y) + (nr.z * z.z + nr.w * z.w);
        acc[1] += (nr.x * nr.x + nr.y * nr.y) + (nr.z * nr.z + nr.w * nr.w);
    }
    if (const int j = (int)threadIdx.x; t.rank == t.nb - 1 && j < P.nphi - 4 * n4) {
        const int p = 4 * n4 + j;
        P.pdelta32[p] += a * P.pdir32[p];
        const float r = P.pres32[p] - a * P.pq32[p];
        const float z = r * P.dinvP32[p];
        P.pres32[p] = r;
        P.pprec32[p] = z;
        acc[0] += r * z;
        acc[1] += r * r;
    }
    return team_sum_f32<2>(t, acc, fin);
}

// FP64 refinement: phi += delta; r -= K delta (FP64 operator).  Sum: |r|^2.
__device__ bool ph_p64_refine(Ctx& C, double& rr) {
    const Problem& P = *C.P;
    Team& t = C.t;
    double acc[1] = {0.0};
    double dummy[1] = {0.0};
    const float* dl = P.pdelta32;
    auto pre = [&](int p) { return Operands{(double)dl[p], P.phi[p], P.pres[p]}; };
    phi_products(P, t, dl, pre, [&](int p, double s, const Operands& v) {
        P.phi[p] = v.b + v.a;
        const double r = v.c - s;
        P.pres[p] = r;
        acc[0] += r * r;
    });
    if (!team_reduce<1, 0>(t, acc, dummy)) return false;
    rr = acc[0];
    return true;
}

// Precision form of the potential solve: Algorithm 1 runs in FP32 on the
// correction equation K delta = r and keeps its direction across
// "reliable updates" (Clark et al., Comput. Phys. Commun. 181 (2010)):
// whenever the FP32 residual has dropped by inner_tol relative to its
// largest value since the last update (or below the target), the
// correction is folded into phi in FP64, the FP64 residual is recomputed
// from it (r -= K delta), and FP32 continues from that residual with the
// same direction.  Stops when the FP64 residual meets poisson_tol.
__device__ bool solve_potential_mixed(Ctx& C, double bb, double rr) {
    const Problem& P = *C.P;
    const double tol2 = C.ptol * C.ptol * bb;
    const double upd2 = P.prm.inner_tol * P.prm.inner_tol;
    if (rr < tol2) return true;
    CgScalars& g = C.t.sm->cg;
    if (!ph_p32_init(C, {g, CG_INIT_FIRST, upd2, tol2})) return false;
    float beta = 0.0f;
    long long k = 0;
    int updates = 0;
    while (k < P.prm.poisson_max_iter) {
        if (!ph_p32_direction(C, beta)) return false;
        if (!ph_p32_update(C, g.af, {g, CG_STEP, upd2, tol2})) return false;
        ++k;
        beta = g.betaf;
        if (g.stop) {
            // reliable update; beta is that of the true residual to the one
            // before this step, so the scalar r.z goes back to it
            const double rz = g.rz_old;
            if (!ph_p64_refine(C, rr)) return false;
            C.mr++;
            ++updates;
            if (rr < tol2 || updates >= P.prm.max_refine) {
                C.mi += k + updates;
                return true;
            }
            if (threadIdx.x == 0) g.rz = rz;
            if (!ph_p32_init(C, {g, CG_INIT_NEXT, upd2, tol2})) return false;
            beta = g.betaf;
        }
    }
    // iteration cap: fold the pending correction into phi
    if (!ph_p64_refine(C, rr)) return false;
    C.mr++;
    C.mi += k + updates + 1;
    return true;
}

// Algorithm 1 on K_phi phi = D m (Sec. 3.1), warm-started from phi.
__device__ bool solve_potential(Ctx& C, int s) {
    const Problem& P = *C.P;
    double bb, rz, rr;
    if (!ph_pinit(C, s, bb, rz, rr)) return false;
    if (bb == 0.0) return ph_pzero(C);
    if (P.prm.precision == 1) return solve_potential_mixed(C, bb, rr);
    const double tol2 = C.ptol * C.ptol * bb;
    CgScalars& g = C.t.sm->cg;
    if (threadIdx.x == 0) g.rz = rz;             // (thread 0 also folds r.z and d.q)
    double beta = 0.0;
    long long k = 0;
    bool stop = !(rr >= tol2);
    while (!stop && k < P.prm.poisson_max_iter) {
        if (!ph_pdirection(C, P.pprec, beta, P.pdir[0], P.pq)) return false;
        if (!ph_pupdate(C, P.pdir[0], g.a, tol2)) return false;
        beta = g.beta;
        stop = g.stop != 0;
        ++k;
    }
    C.mi += k;
    return true;
}

// Energy and gradient pass (Eq. energy, nablaLF, proj, opt2) at slot s:
// grad = C_A x + C_K x + D^T phi - w h; lambda = x . grad; g = grad - lambda x.
__device__ bool ph_gradient(Ctx& C, int s, bool trial) {
    const Problem& P = *C.P;
    Team& t = C.t;
    const int nm = P.nm;
    const double* x = P.X[s];
    double* gr = P.GR[s];
    double* gp = P.GP[s];
    double* lamv = P.LAM[s];
    const double h0 = C.h[0], h1 = C.h[1], h2 = C.h[2];
    // sums: exchange, anisotropy, Zeeman, phi.rhs, phi.r, dphi, M0, M1, M2, sum w
    double acc[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    double mx[1] = {0.0};
    ROWS(p, t.sm->phi, P.nphi) {
        acc[4] += P.phi[p] * P.pres[p];
        P.PHI[s][p] = P.phi[p];
        if (p < nm) {
            const int i = p;
            acc[3] += P.phi[i] * P.rhs[i];
            double c0, c1, c2, a0, a1, a2, t0, t1, t2;
            row_local(P, x, i, c0, c1, c2, a0, a1, a2);
            row_divT(P, P.phi, i, t0, t1, t2);
            const double x0 = x[i], x1 = x[nm + i], x2 = x[2 * nm + i];
            const double wi = P.w[i];
            const double g0 = 2.0 * c0 + a0 + t0 - wi * h0;
            const double g1 = 2.0 * c1 + a1 + t1 - wi * h1;
            const double g2 = 2.0 * c2 + a2 + t2 - wi * h2;
            acc[0] += x0 * c0 + x1 * c1 + x2 * c2;
            acc[1] += 0.5 * (x0 * a0 + x1 * a1 + x2 * a2);
            acc[2] -= wi * (h0 * x0 + h1 * x1 + h2 * x2);
            const double lam = x0 * g0 + x1 * g1 + x2 * g2;
            const double p0 = g0 - lam * x0, p1 = g1 - lam * x1, p2 = g2 - lam * x2;
            gr[i] = g0;
            gr[nm + i] = g1;
            gr[2 * nm + i] = g2;
            gp[i] = p0;
            gp[nm + i] = p1;
            gp[2 * nm + i] = p2;
            lamv[i] = lam;
            mx[0] = fmax(mx[0], fmax(fabs(p0), fmax(fabs(p1), fabs(p2))));
            if (trial)
                acc[5] += (p0 * P.d[i] + p1 * P.d[nm + i] + p2 * P.d[2 * nm + i]) / P.unorm[i];
            acc[6] += wi * x0;
            acc[7] += wi * x1;
            acc[8] += wi * x2;
            acc[9] += wi;
        }
    }
    if (!team_reduce<10, 1>(t, acc, mx)) return false;
    SlotScalars& S = C.sl[s];
    S.terms[0] = acc[0];
    S.terms[1] = acc[1];
    S.terms[2] = 0.5 * (acc[3] + acc[4]);   // phi.b - 1/2 phi.K phi, K phi = b - r
    S.terms[3] = acc[2];
    S.F = ((S.terms[0] + S.terms[1]) + S.terms[2]) + S.terms[3];
    S.dphi = acc[5];
    S.gmax = mx[0];
    S.M[0] = acc[6] / acc[9];
    S.M[1] = acc[7] / acc[9];
    S.M[2] = acc[8] / acc[9];
    return true;
}

// One function evaluation at slot s: at x_c + a d (trial) or at x_s as is.
// Warm start of a trial evaluation: phi is linear in m and the trial point
// is x_c + a d to first order, so phi(a) ~ PHI[c] + theta (PHI[ref] - PHI[c])
// with theta = a / a_ref (theta = 0: start from the current state's phi).
__device__ bool ph_phi_start(Ctx& C, int c, int ref, double theta) {
    const Problem& P = *C.P;
    Team& t = C.t;
    const double* a = P.PHI[c];
    const double* b = P.PHI[ref];
    ROWS(p, t.sm->phi, P.nphi) P.phi[p] = (theta == 0.0) ? a[p] : a[p] + theta * (b[p] - a[p]);
    return team_sync(t);
}

__device__ bool ph_phi_restore(Ctx& C, int c) {
    const Problem& P = *C.P;
    Team& t = C.t;
    ROWS(p, t.sm->phi, P.nphi) P.phi[p] = P.PHI[c][p];
    return team_sync(t);
}

// One function evaluation at slot s: at x_c + a d (trial, potential warm
// start from the slots c and ref, see ph_phi_start) or at x_s as is (warm
// start from the last potential).
__device__ bool evaluate(Ctx& C, int c, int s, bool trial, double a, int ref = 0, double theta = 0.0) {
    if (trial && !ph_trial(C, c, s, a)) return false;
    if (trial && !ph_phi_start(C, c, ref, theta)) return false;
    if (!solve_potential(C, s)) return false;
    if (!ph_gradient(C, s, trial)) return false;
    C.evals++;
    return true;
}

// Team values of the preconditioner's solve: of a direction step (step length,
// li2), of the initial residual (|b| and li3's limit) and of an update (beta,
// li3).
struct InnerLength {
    CgScalars& g;
    __device__ void operator()(int, double dHd) const {
        cg_length(g, dHd);
        g.stop = dHd <= 0.0;
    }
};
struct InnerResidual {
    CgScalars& g;
    bool initial;
    __device__ void operator()(int k, double s) const {
        if (k == 0) {
            if (initial) g.rz = s;
            else cg_beta(g, s);
        } else {
            const double r = sqrt(s);
            if (initial) g.eps = fmin(0.5, sqrt(r)) * r;
            g.stop = r < g.eps;
        }
    }
};

// w = H(m) v (Eq. precond, magnetostatics dropped; last term only if
// keep_last_term).  With d given, the inner CG direction step follows by
// recurrence: d = ca v + beta d and hd = ca w + beta hd (= H d), in place,
// sum d . hd (step length and li2's sign).  Without d, w is written to hd.
__device__ bool ph_hess(Ctx& C, int s, const double* v, double ca, double beta, double* d,
                        double* hd) {
    const Problem& P = *C.P;
    Team& t = C.t;
    const int nm = P.nm;
    const double* m = P.X[s];
    const double* lamv = P.LAM[s];
    const double* gr = P.GR[s];
    const bool keep = P.prm.keep_last_term != 0;
    const bool first = is_zero(beta);
    double acc[1] = {0.0};
    double dummy[1] = {0.0};
    ROWS(i, t.sm->nm, nm) {
        double c0, c1, c2, k0, k1, k2;
        row_local(P, v, i, c0, c1, c2, k0, k1, k2);
        const double v0 = v[i], v1 = v[nm + i], v2 = v[2 * nm + i];
        const double Cv0 = 2.0 * c0 + k0;
        const double Cv1 = 2.0 * c1 + k1;
        const double Cv2 = 2.0 * c2 + k2;
        const double m0 = m[i], m1 = m[nm + i], m2 = m[2 * nm + i];
        const double mc = m0 * Cv0 + m1 * Cv1 + m2 * Cv2;
        const double lam = lamv[i];
        double w0 = Cv0 - mc * m0 - lam * v0;
        double w1 = Cv1 - mc * m1 - lam * v1;
        double w2 = Cv2 - mc * m2 - lam * v2;
        if (keep) {
            const double vg = v0 * gr[i] + v1 * gr[nm + i] + v2 * gr[2 * nm + i];
            w0 -= vg * m0;
            w1 -= vg * m1;
            w2 -= vg * m2;
        }
        if (d) {
            double dn[3] = {ca * v0, ca * v1, ca * v2};
            double hn[3] = {ca * w0, ca * w1, ca * w2};
            if (!first) {
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    dn[c] += beta * d[c * nm + i];
                    hn[c] += beta * hd[c * nm + i];
                }
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                d[c * nm + i] = dn[c];
                hd[c * nm + i] = hn[c];
                acc[0] += dn[c] * hn[c];
            }
        } else {
            hd[i] = w0;
            hd[nm + i] = w1;
            hd[2 * nm + i] = w2;
        }
    }
    return team_reduce<1, 0>(t, acc, dummy, InnerLength{t.sm->cg});
}

// One application of an operator of Eq. (energy) (the operator entry
// point): MODE_DIV q = D v (v: idir[0], 3 x nm; q: pq, n_phi, zero on the
// air rows), MODE_DIVT w = D^T phi (phi: pdir[0]; w: ihd), MODE_LOCAL
// w = (C_A + C_K) v (v: idir[0]; w: ihd).
__device__ bool ph_operator(Ctx& C, int mode) {
    const Problem& P = *C.P;
    Team& t = C.t;
    const int nm = P.nm;
    if (mode == MODE_DIV) {
        ROWS(p, t.sm->phi, P.nphi) P.pq[p] = (p < nm) ? row_div(P, P.idir[0], p) : 0.0;
    } else if (mode == MODE_DIVT) {
        ROWS(i, t.sm->nm, nm) {
            double t0, t1, t2;
            row_divT(P, P.pdir[0], i, t0, t1, t2);
            P.ihd[i] = t0;
            P.ihd[nm + i] = t1;
            P.ihd[2 * nm + i] = t2;
        }
    } else {
        ROWS(i, t.sm->nm, nm) {
            double c0, c1, c2, a0, a1, a2;
            row_local(P, P.idir[0], i, c0, c1, c2, a0, a1, a2);
            P.ihd[i] = 2.0 * c0 + a0;
            P.ihd[nm + i] = 2.0 * c1 + a1;
            P.ihd[2 * nm + i] = 2.0 * c2 + a2;
        }
    }
    return team_sync(t);
}

// Algorithm 1 for H(m_s) y = g_s, y_0 = 0, Jacobi diag(C_A), exits li1-li3.
__device__ bool precond_solve(Ctx& C, int s) {
    const Problem& P = *C.P;
    Team& t = C.t;
    const int nm = P.nm;
    const int jmax = P.prm.jmax;
    if (jmax <= 0) {
        C.y_is_g = 1;
        return true;
    }
    const double* gp = P.GP[s];
    // residual gr = H*0 + b with b = -g; preconditioned yv; direction -yv
    double acc[2] = {0.0, 0.0};
    double dummy[1] = {0.0};
    ROWS(i, t.sm->nm, nm) {
        const double di = P.dinvA[i];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double r = -gp[c * nm + i];
            const double z = di * r;
            P.ires[c * nm + i] = r;
            P.iprec[c * nm + i] = z;
            P.isol[c * nm + i] = 0.0;
            acc[0] += r * z;
            acc[1] += r * r;
        }
    }
    CgScalars& g = t.sm->cg;
    if (!team_reduce<2, 0>(t, acc, dummy, InnerResidual{g, true})) return false;
    C.y_is_g = 0;
    if (g.stop) return true;                    // y = 0 (only when g = 0 ... eps = 0)
    double beta = 0.0;
    int steps = 0;
    while (steps < jmax) {
        // direction d = -yv + beta d and H d, by recurrence
        if (!ph_hess(C, s, P.iprec, -1.0, beta, P.idir[0], P.ihd)) return false;
        ++steps;
        C.li++;
        if (g.stop) {                           // li2
            C.li2++;
            if (steps == 1) {
                C.y_is_g = 1;
                C.li2_first++;
            }
            return true;
        }
        const double a = g.a;
        const double* dv = P.idir[0];
        double a2[2] = {0.0, 0.0};
        ROWS(i, t.sm->nm, nm) {
            const double di = P.dinvA[i];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int q = c * nm + i;
                P.isol[q] += a * dv[q];
                const double r = P.ires[q] + a * P.ihd[q];
                const double z = di * r;
                P.ires[q] = r;
                P.iprec[q] = z;
                a2[0] += r * z;
                a2[1] += r * r;
            }
        }
        if (!team_reduce<2, 0>(t, a2, dummy, InnerResidual{g, false})) return false;
        if (g.stop) return true;                // li3
        beta = g.beta;
    }
    return true;                                // li1
}

// The precision form's preconditioner apply: precond_solve with H's
// products and the residual, preconditioned-residual, direction and
// H-direction vectors in FP32 (K_A, C_K and diag(C_A)^-1 as FP32 copies);
// m, lambda and the gradient are read from the FP64 state, the dots are
// FP32 products summed in FP64, the step length and beta stay FP64 scalars
// and the solution y accumulates in FP64 (the search direction is built from
// it).  The exits li1-li3 and their counters are those of precond_solve.
__device__ bool ph_hess32(Ctx& C, int s, const float* v, float beta, float* d, float* hd) {
    const Problem& P = *C.P;
    Team& t = C.t;
    const int nm = P.nm;
    const double* m = P.X[s];
    const double* lamv = P.LAM[s];
    const double* gr = P.GR[s];
    const bool keep = P.prm.keep_last_term != 0;
    const bool first = (beta == 0.0f);
    double acc[1] = {0.0};
    double dummy[1] = {0.0};
    ROWS(i, t.sm->nm, nm) {
        float c0, c1, c2;
        sell_dot3<8>(P.m_sptr, P.m_col, P.KA32, v, nm, i, c0, c1, c2);
        const float v0 = v[i], v1 = v[nm + i], v2 = v[2 * nm + i];
        const float kxx = P.CK32[i], kxy = P.CK32[nm + i], kxz = P.CK32[2 * nm + i];
        const float kyy = P.CK32[3 * nm + i], kyz = P.CK32[4 * nm + i], kzz = P.CK32[5 * nm + i];
        const float Cv0 = 2.0f * c0 + (kxx * v0 + kxy * v1 + kxz * v2);
        const float Cv1 = 2.0f * c1 + (kxy * v0 + kyy * v1 + kyz * v2);
        const float Cv2 = 2.0f * c2 + (kxz * v0 + kyz * v1 + kzz * v2);
        const float m0 = (float)m[i], m1 = (float)m[nm + i], m2 = (float)m[2 * nm + i];
        const float mc = m0 * Cv0 + m1 * Cv1 + m2 * Cv2;
        const float lam = (float)lamv[i];
        float w[3] = {Cv0 - mc * m0 - lam * v0, Cv1 - mc * m1 - lam * v1, Cv2 - mc * m2 - lam * v2};
        if (keep) {
            const float vg = v0 * (float)gr[i] + v1 * (float)gr[nm + i] + v2 * (float)gr[2 * nm + i];
            w[0] -= vg * m0;
            w[1] -= vg * m1;
            w[2] -= vg * m2;
        }
        const float vv[3] = {v0, v1, v2};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            // d = -v + beta d, hd = -H v + beta hd (= H d)
            float dn = -vv[c], hn = -w[c];
            if (!first) {
                dn += beta * d[c * nm + i];
                hn += beta * hd[c * nm + i];
            }
            d[c * nm + i] = dn;
            hd[c * nm + i] = hn;
            acc[0] += (double)(dn * hn);
        }
    }
    return team_reduce<1, 0>(t, acc, dummy, InnerLength{t.sm->cg});
}

__device__ bool precond_solve32(Ctx& C, int s) {
    const Problem& P = *C.P;
    Team& t = C.t;
    const int nm = P.nm;
    const int jmax = P.prm.jmax;
    if (jmax <= 0) {
        C.y_is_g = 1;
        return true;
    }
    const double* gp = P.GP[s];
    double acc[2] = {0.0, 0.0};
    double dummy[1] = {0.0};
    ROWS(i, t.sm->nm, nm) {
        const float di = P.dinvA32[i];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float r = (float)(-gp[c * nm + i]);
            const float z = di * r;
            P.ires32[c * nm + i] = r;
            P.iprec32[c * nm + i] = z;
            P.isol[c * nm + i] = 0.0;
            acc[0] += (double)(r * z);
            acc[1] += (double)(r * r);
        }
    }
    CgScalars& g = t.sm->cg;
    if (!team_reduce<2, 0>(t, acc, dummy, InnerResidual{g, true})) return false;
    C.y_is_g = 0;
    if (g.stop) return true;
    float beta = 0.0f;
    int steps = 0;
    while (steps < jmax) {
        if (!ph_hess32(C, s, P.iprec32, beta, P.idir32, P.ihd32)) return false;
        ++steps;
        C.li++;
        if (g.stop) {                           // li2
            C.li2++;
            if (steps == 1) {
                C.y_is_g = 1;
                C.li2_first++;
            }
            return true;
        }
        const double a = g.a;
        const float af = g.af;
        double a2[2] = {0.0, 0.0};
        ROWS(i, t.sm->nm, nm) {
            const float di = P.dinvA32[i];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int q = c * nm + i;
                P.isol[q] += a * (double)P.idir32[q];
                const float r = P.ires32[q] + af * P.ihd32[q];
                const float z = di * r;
                P.ires32[q] = r;
                P.iprec32[q] = z;
                a2[0] += (double)(r * z);
                a2[1] += (double)(r * r);
            }
        }
        if (!team_reduce<2, 0>(t, a2, dummy, InnerResidual{g, false})) return false;
        if (g.stop) return true;                // li3
        beta = g.betaf;
    }
    return true;                                // li1
}

// The preconditioner apply of the configured form.
__device__ bool precond_apply(Ctx& C, int s) {
    return C.P->prm.precision ? precond_solve32(C, s) : precond_solve(C, s);
}

// beta*ZA dots between slot a (new gradient gn) and slot c (old gradient go)
// with y the preconditioned gn and d the previous direction:
//   y.gn, y.go, (gn-go).y, (gn-go).d, gn.d, gn.gn, gn.go, (gn-go).gn
__device__ bool ph_dir_dots(Ctx& C, int a, int c, double (&dots)[8]) {
    const Problem& P = *C.P;
    Team& t = C.t;
    const int nm = P.nm;
    const double* y = C.y_is_g ? P.GP[a] : P.isol;
    const double* gn = P.GP[a];
    const double* go = P.GP[c];
    double dummy[1] = {0.0};
    for (int k = 0; k < 8; ++k) dots[k] = 0.0;
    ROWS(i, t.sm->nm, nm) {
#pragma unroll
        for (int q3 = 0; q3 < 3; ++q3) {
            const int q = q3 * nm + i;
            const double yy = y[q], n = gn[q], o = go[q], dd = P.d[q];
            const double dg = n - o;
            dots[0] += yy * n;
            dots[1] += yy * o;
            dots[2] += dg * yy;
            dots[3] += dg * dd;
            dots[4] += n * dd;
            dots[5] += n * n;
            dots[6] += n * o;
            dots[7] += dg * n;
        }
    }
    return team_reduce<8, 0>(t, dots, dummy);
}

// d = -v + beta d (kind 1: v = y; kind 2: v = g; kind 3: d = -g), max_i |d_i|.
__device__ bool ph_dir_write(Ctx& C, int a, int kind, double beta, double& dmax) {
    const Problem& P = *C.P;
    Team& t = C.t;
    const int nm = P.nm;
    const double* y = C.y_is_g ? P.GP[a] : P.isol;
    const double* v = (kind == 1) ? y : P.GP[a];
    const double b = (kind == 3) ? 0.0 : beta;   // b == 0: d_old is not read
    double mx[1] = {0.0};
    double dummy[1] = {0.0};
    ROWS(i, t.sm->nm, nm) {
        double n2 = 0.0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const int q = c * nm + i;
            const double dn = (b == 0.0) ? -v[q] : -v[q] + b * P.d[q];
            P.d[q] = dn;
            n2 += dn * dn;
        }
        mx[0] = fmax(mx[0], sqrt(n2));
    }
    if (!team_reduce<0, 1>(t, dummy, mx)) return false;
    dmax = mx[0];
    return true;
}

__device__ __forceinline__ double beta_za(double y_gn, double y_go, double dg_y, double dg_d) {
    if (y_gn > y_go) return (dg_d == 0.0) ? 0.0 : dg_y / dg_d;
    return 0.0;
}

// The direction update of Algorithm 3/4 with y the preconditioned new
// gradient: beta*ZA (restarted Hestenes-Stiefel), beta*FR = g+.y+ / g.y
// (Eq. FRstar), beta*PRP = (g+ - g).y+ / g.y (Eq. PRPstar), g.y = gy_prev
// of the last direction (0 gives beta = 0).
__device__ __forceinline__ double beta_rule(int rule, double y_gn, double y_go, double dg_y, double dg_d,
                                            double gy_prev) {
    if (rule == 1) return (gy_prev == 0.0) ? 0.0 : y_gn / gy_prev;
    if (rule == 2) return (gy_prev == 0.0) ? 0.0 : dg_y / gy_prev;
    return beta_za(y_gn, y_go, dg_y, dg_d);
}

// New direction with beta*ZA and the descent safeguard; returns g.d.
__device__ bool direction(Ctx& C, int a, int c, bool initial, double& dmax, double& gd) {
    double dots[8];
    if (!ph_dir_dots(C, a, c, dots)) return false;
    const double y_gn = dots[0], y_go = dots[1], dg_y = dots[2], dg_d = dots[3];
    const double gn_d = dots[4], gn_gn = dots[5], gn_go = dots[6], dg_gn = dots[7];
    const int rule = C.P->prm.beta_rule;
    int kind = 1;
    double beta = 0.0;
    if (initial) {
        gd = -y_gn;
        if (gd >= 0.0) {
            kind = 3;
            gd = -gn_gn;
            C.steepest++;
        }
    } else {
        beta = beta_rule(rule, y_gn, y_go, dg_y, dg_d, C.gy_prev);
        gd = -y_gn + beta * gn_d;
        if (gd >= 0.0) {
            beta = beta_rule(rule, gn_gn, gn_go, dg_gn, dg_d, C.gy_prev);
            kind = 2;
            gd = -gn_gn + beta * gn_d;
            C.restarts++;
            if (gd >= 0.0) {
                kind = 3;
                beta = 0.0;
                gd = -gn_gn;
                C.steepest++;
            }
        }
    }
    C.gy_prev = (kind == 1) ? y_gn : gn_gn;     // g.y of the direction built (y = g after the safeguard)
    return ph_dir_write(C, a, kind, beta, dmax);
}

__device__ __forceinline__ bool cubic_step(double f0, double g0, double a, double f1, double g1,
                                           double& out) {
    const double d1 = g0 + g1 - 3.0 * (f1 - f0) / a;
    const double disc = d1 * d1 - g0 * g1;
    if (!(disc > 0.0)) return false;
    const double d2 = sqrt(disc);
    const double den = g1 - g0 + 2.0 * d2;
    if (den == 0.0) return false;
    out = a - a * (g1 + d2 - d1) / den;
    return isfinite(out);
}

// Algorithm 4 at the current field from slot C.cur.
__device__ MM_OUTLINE int minimize(Ctx& C, int& cur) {
    const Problem& P = *C.P;
    const Params& prm = P.prm;
    int c = cur;
    if (!evaluate(C, c, c, false, 0.0)) return ST_TIMEOUT;
    if (!precond_apply(C, c)) return ST_TIMEOUT;
    double dmax, gd;
    if (!direction(C, c, c, true, dmax, gd)) return ST_TIMEOUT;
    double a_prev = 1.0;
    int status = ST_RUNNING;
    if (!isfinite(C.sl[c].F)) status = ST_NONFINITE;
    else if (C.sl[c].gmax == 0.0) status = ST_OK;
    const double sq_tau = sqrt(prm.tau_F);
    const double cb_tau = cbrt(prm.tau_F);
    double dF_prev = -1.0;                      // last accepted decrease (none yet)
    while (status == ST_RUNNING && C.nli < prm.max_iter) {
        const double F0 = C.sl[c].F;
        // potential tolerance of this iteration's evaluations (poisson_sched):
        // loosened while the last decrease is far above the t1 threshold, so
        // that the energy error (quadratic in the potential error) stays far
        // below the decrease the line search resolves
        C.ptol = prm.poisson_tol;
        if (prm.poisson_sched && dF_prev > 0.0) {
            const double q = dF_prev / (prm.tau_F * (1.0 + fabs(F0)));
            if (q > 100.0) C.ptol = fmin(prm.poisson_tol_max, fmax(prm.poisson_tol, prm.poisson_tol * sqrt(q) / 10.0));
        }
        const double dphi0 = gd;
        const double a_max = prm.theta_max / dmax;
        const double a_t = fmin(a_prev, a_max);
        const int ts = (c + 1) % MM_NSLOT, ss = (c + 2) % MM_NSLOT;
        if (!evaluate(C, c, ts, true, a_t, c, 0.0)) return ST_TIMEOUT;
        double a_s;
        if (!cubic_step(F0, dphi0, a_t, C.sl[ts].F, C.sl[ts].dphi, a_s))
            a_s = (C.sl[ts].dphi < 0.0) ? 4.0 * a_t : 0.5 * a_t;
        a_s = fmin(fmax(a_s, 0.1 * a_t), fmin(4.0 * a_t, a_max));
        if (!evaluate(C, c, ss, true, a_s, ts, a_s / a_t)) return ST_TIMEOUT;
        int b;
        double a_b;
        if (C.sl[ss].F <= C.sl[ts].F) {
            b = ss;
            a_b = a_s;
        } else {
            b = ts;
            a_b = a_t;
        }
        if (!(C.sl[b].F <= F0 + prm.c1 * a_b * dphi0)) {
            bool found = false;
            double a = 0.5 * fmin(a_t, a_s);
            for (int k = 0; k < prm.max_backtrack; ++k) {
                if (!evaluate(C, c, ts, true, a, ss, a / a_s)) return ST_TIMEOUT;
                C.ls_extra++;
                if (C.sl[ts].F <= F0 + prm.c1 * a * dphi0) {
                    b = ts;
                    a_b = a;
                    found = true;
                    break;
                }
                a *= 0.5;
            }
            if (!found) {
                status = ST_STALLED;
                break;
            }
        }
        C.nli++;
        const SlotScalars& S = C.sl[b];
        dF_prev = F0 - S.F;
        if (!isfinite(S.F)) {
            status = ST_NONFINITE;
            break;
        }
        const bool t1 = F0 - S.F < prm.tau_F * (1.0 + fabs(S.F));
        const bool t2 = S.xdiff < sq_tau * (1.0 + S.xmax);
        const bool t3 = S.gmax < cb_tau * (1.0 + fabs(S.F));
        if (!precond_apply(C, b)) return ST_TIMEOUT;
        if (!direction(C, b, c, false, dmax, gd)) return ST_TIMEOUT;
        c = b;
        a_prev = a_b;
        if (t1 && t2 && t3) status = ST_OK;
    }
    if (status == ST_RUNNING) status = ST_NOT_CONVERGED;
    // leave the accepted state's potential as the working one (the next
    // field step starts from it; the host reads it)
    if (!ph_phi_restore(C, c)) return ST_TIMEOUT;
    cur = c;
    return status;
}

}  // namespace

// The solver on one team of nb blocks (this block is number rank).
__device__ __forceinline__ void solver_body(const Problem& P, int nb, int rank) {
    __shared__ TeamSmem team_smem;
    Ctx C;
    C.P = &P;
    C.t.sm = &team_smem;
    C.t.target = 0;
    C.t.nb = nb;
    C.t.rank = rank;
    C.t.count = reinterpret_cast<unsigned long long*>(P.bar);
    C.t.err = P.err;
    C.t.part = P.partials;
    C.t.epoch = 0;
    C.t.dead = false;
    if (threadIdx.x == 0) {
        TeamSmem& sm = team_smem;
        sm.dead = 0;
        sm.phi = make_share(C.t, (P.nphi + 31) >> 5);
        sm.nm = make_share(C.t, (P.nm + 31) >> 5);
        sm.phi4 = make_share(C.t, ((P.nphi >> 2) + 31) >> 5);
        for (int l = 0; l < P.nlev; ++l) {
            const int rpw = 32 / restrict_group(P, C.t, l);
            sm.rows[l] = make_share(C.t, (P.lev[l].n + 31) >> 5);
            sm.coarse[l] = make_share(C.t, (P.lev[l].nc + rpw - 1) / rpw);
        }
        sm.dense = make_share(C.t, P.nco);
    }
    __syncthreads();
    C.evals = C.nli = C.li = C.mi = C.ls_extra = C.mr = 0;
    C.li2 = C.li2_first = C.restarts = C.steepest = 0;
    C.y_is_g = 0;
    C.ptol = P.prm.poisson_tol;
    C.gy_prev = 0.0;
    int cur = P.state->cur;
    C.h[0] = P.state->h[0];
    C.h[1] = P.state->h[1];
    C.h[2] = P.state->h[2];
    int status = ST_OK;
    switch (P.mode) {
        case MODE_MINIMIZE:
            status = minimize(C, cur);
            break;
        case MODE_EVAL:
            if (!evaluate(C, cur, cur, false, 0.0)) status = ST_TIMEOUT;
            break;
        case MODE_PRECOND:
            if (!precond_apply(C, cur)) status = ST_TIMEOUT;
            break;
        case MODE_HESS: {
            // input v in idir[0], output in ihd
            if (!ph_hess(C, cur, P.idir[0], 1.0, 0.0, nullptr, P.ihd)) status = ST_TIMEOUT;
            break;
        }
        case MODE_KPHI: {
            // input in pdir[0], output in pq
            if (!ph_pmatvec(C, P.pdir[0], P.pq)) status = ST_TIMEOUT;
            break;
        }
        case MODE_DIV:
        case MODE_DIVT:
        case MODE_LOCAL:
            if (!ph_operator(C, P.mode)) status = ST_TIMEOUT;
            break;
        default:
            status = ST_TIMEOUT;
    }
    if (C.t.dead) status = ST_TIMEOUT;
    if (rank == 0 && threadIdx.x == 0) {
        DevState* st = P.state;
        st->cur = cur;
        st->status = status;
        st->evals = C.evals;
        st->nli = C.nli;
        st->li = C.li;
        st->mi = C.mi;
        st->ls_extra = C.ls_extra;
        st->mr = C.mr;
        st->li2 = C.li2;
        st->li2_first = C.li2_first;
        st->restarts = C.restarts;
        st->steepest = C.steepest;
        if (P.mode == MODE_MINIMIZE || P.mode == MODE_EVAL) {
            const SlotScalars& S = C.sl[cur];
            st->F = S.F;
            for (int k = 0; k < 4; ++k) st->terms[k] = S.terms[k];
            for (int k = 0; k < 3; ++k) st->M[k] = S.M[k];
            st->gmax = S.gmax;
        }
        st->y_is_g = C.y_is_g;
    }
}

// One instantiation per occupancy target (MINB x 256 resident threads per
// SM), each compiled in its own translation unit (mm_kern_*.cu); the host
// picks one through solver_kernel() / solver_batch_kernel().  The single form
// runs them as one block per SM (MM_BLOCK = MINB x 256, set by its unit): a
// barrier of 152 blocks costs 1.25 us where one of 304 costs 1.42 us and one
// of 608 2.28 us, and a reduction folds 152 partials.  Batches keep blocks of
// 256 threads, so that small members can have a fraction of an SM.
template <int MINB, int LARGE = MM_LARGE>
__global__ void __launch_bounds__(MM_BLOCK, MINB * 256 / MM_BLOCK) k_solver(const __grid_constant__ Problem P) {
    solver_body(P, (int)gridDim.x, (int)blockIdx.x);
}

// Batched form: the grid is split into teams, team j = blocks
// [team_first[j], team_first[j+1]) runs the solver on problem j.  Teams only
// synchronise internally, so problems of different sizes and iteration
// counts proceed independently inside one launch.
template <int MINB>
__global__ void __launch_bounds__(MM_BLOCK, MINB) k_solver_batch(const Problem* __restrict__ probs,
                                                                  const int* __restrict__ team_first, int nteams) {
    int lo = 0, hi = nteams;                 // team_first[lo] <= blockIdx.x < team_first[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (team_first[mid] <= (int)blockIdx.x) lo = mid;
        else hi = mid;
    }
    const int first = team_first[lo];
    solver_body(probs[lo], team_first[lo + 1] - first, (int)blockIdx.x - first);
}

}  // namespace mm
