// Forward pass and training pass of the warm-start network on the
// 5th-generation tensor cores (tcgen05): BF16 operands staged in shared
// memory, FP32 accumulators in tensor memory (TMEM), M = 128 per MMA (one
// TMEM lane per row).  Included by mm_mlp.cu (it uses that file's layer
// sizes and parameter layout).
//
// Per tile of 128 rows (a group of 4 warps, thread t owns row t of the tile):
//   x   = bf16((X - mean) / std)                  -> shared memory
//   h1  = relu(x W1^T + b1)   1 MMA  (K = 16)     TMEM -> registers -> bf16 -> shared
//   h2  = relu(h1 W2^T + b2)  8 MMAs (K = 8 x 16)
//   h3  = relu(h2 W3^T + b3)  8 MMAs
//   y   = h3 W4^T + b4        8 MMAs, N = 16 (outputs 4..15 are zero weights)
// One thread issues the MMAs of a layer and commits them to an mbarrier;
// every thread waits on it (bounded: a wait that runs out sets the error
// flag, and the block leaves after freeing its TMEM), then reads its row of
// the accumulator with tcgen05.ld.  The rounding points (input, weights,
// hidden activations to BF16; FP32 accumulation) are those of the mma.sync
// path, so both paths compute the same network.
//
// Operand layout in shared memory: "no swizzle, K-major" core matrices of
// 8 rows x 16 bytes (8 bf16 along K); element (r, k) of an R x K operand at
// byte (r / 8) * (16 K) + (k / 8) * 128 + (r % 8) * 16 + (k % 8) * 2, i.e.
// core matrices 128 B apart along K (the descriptor's leading-dimension
// offset) and 16 K bytes apart along R (its stride-dimension offset).  The
// weights W_l [out][in] are the B operands as stored (K = in contiguous).
// The same bytes are an MN-major operand whose MN runs along the columns and
// K along the rows: core matrices 128 B apart along MN and 16 x columns bytes
// apart along K.  The training pass needs no transposed copy for that reason.
#pragma once

namespace tc {

constexpr int TM = 128;      // rows per tile = the MMA's M = TMEM lanes
constexpr int N4 = 16;       // the last layer's N, padded
constexpr int TCOLS = 128;   // TMEM columns allocated (one N = 128 accumulator)
constexpr unsigned long long kWaitNs = 2000000000ull;   // 2 s per MMA wait (mm_mlp_set_wait_limit)

constexpr int GROUPS = 4;    // forward pass: tiles in flight per SM, 128 threads each

struct __align__(128) Smem {
    __nv_bfloat16 w1[NH * NIN];
    __nv_bfloat16 w2[NH * NH];
    __nv_bfloat16 w3[NH * NH];
    __nv_bfloat16 w4[N4 * NH];
    __nv_bfloat16 x[GROUPS][TM * NIN];
    __nv_bfloat16 h[GROUPS][TM * NH];
    float b[3 * NH + N4];
    float mean[NIN], istd[NIN];
    unsigned long long bar[GROUPS];
    unsigned tmem;
};

__device__ __forceinline__ unsigned core_off(int r, int k, int K) {
    return (unsigned)((r >> 3) * (K * 16) + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2);
}

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor of a tile of `cols` columns in the layout
// above: start address, leading-dimension offset (next core matrix along K),
// stride-dimension offset (next core matrix along MN), the descriptor version
// bits 46-48 = 0b001, no swizzle.
__device__ __forceinline__ unsigned long long sdesc(const void* p, int cols, bool mn_major = false) {
    const unsigned long long a = (smem_u32(p) & 0x3FFFFu) >> 4;
    const unsigned long long dc = 128u >> 4, dr = (unsigned)(cols * 16) >> 4;   // along columns, along rows
    return a | ((mn_major ? dr : dc) << 16) | ((mn_major ? dc : dr) << 32) | (1ull << 46);
}

// Instruction descriptor of kind::f16: D FP32 (bits 4-5 = 1), A and B BF16
// (bits 7-9 and 10-12 = 1), A and B MN-major (bits 15, 16; 0: K-major), N >> 3
// at bits 17-22, M >> 4 at bits 24-28.
__host__ __device__ constexpr unsigned idesc_bf16(int M, int N, bool a_mn = false, bool b_mn = false) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)a_mn << 15) | ((unsigned)b_mn << 16) |
           ((unsigned)(N >> 3) << 17) | ((unsigned)(M >> 4) << 24);
}

__device__ __forceinline__ void mma(unsigned tmem, unsigned long long a, unsigned long long b, unsigned id,
                                    unsigned accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
        "l"(a), "l"(b), "r"(id), "r"(accumulate));
}

__device__ __forceinline__ void commit(unsigned long long* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ unsigned long long now_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Wait for the completion of the mbarrier phase with the given parity;
// false if it did not complete within `limit` ns (limit 0: without a look).
__device__ __forceinline__ bool wait_phase(unsigned long long* bar, unsigned parity,
                                           unsigned long long limit = kWaitNs) {
    if (limit == 0) return false;
    const unsigned a = smem_u32(bar);
    const unsigned long long t0 = now_ns();
    while (true) {
        unsigned ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(ok)
            : "r"(a), "r"(parity)
            : "memory");
        if (ok) return true;
        if (now_ns() - t0 > limit) return false;
    }
}

__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }

// 32 consecutive FP32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld32(unsigned taddr, float (&v)[32]) {
    unsigned r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_ld16(unsigned taddr, float (&v)[16]) {
    unsigned r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// A row-major [rows][COLS] BF16 matrix (16-byte aligned) into the tile layout,
// 16 bytes per thread and step; eight lanes take the eight rows of a core
// matrix, so that a warp's stores are contiguous.
template <int COLS>
__device__ __forceinline__ void stage_tile(__nv_bfloat16* dst, const __nv_bfloat16* __restrict__ src, int rows, int have,
                                           int tid, int nthreads) {
    unsigned char* d = reinterpret_cast<unsigned char*>(dst);
    for (int i = tid; i < rows * (COLS / 8); i += nthreads) {
        const int r = (i / COLS) * 8 + (i & 7), k = ((i >> 3) % (COLS / 8)) * 8;
        const uint4 v = r < have ? *reinterpret_cast<const uint4*>(src + r * COLS + k) : make_uint4(0, 0, 0, 0);
        *reinterpret_cast<uint4*>(d + core_off(r, k, COLS)) = v;
    }
}

// Four consecutive floats; vec: the array is 16-byte aligned.
__device__ __forceinline__ float4 load4(const float* p, bool vec) {
    return vec ? *reinterpret_cast<const float4*>(p) : make_float4(p[0], p[1], p[2], p[3]);
}

// Barriers of one group of 128 threads (hardware barriers 1 .. GROUPS).
__device__ __forceinline__ void group_sync(int g) { asm volatile("bar.sync %0, 128;" ::"r"(g + 1) : "memory"); }
__device__ __forceinline__ bool group_and(int g, bool v) {
    unsigned r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %1, 0;\n\tbar.red.and.pred p, %2, 128, q;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(r)
        : "r"((unsigned)v), "r"(g + 1)
        : "memory");
    return r != 0;
}

// relu(a + b) of two columns as packed BF16.  The maximum is taken after the
// rounding, which keeps its sign (a NaN gives 0 either way).
__device__ __forceinline__ unsigned bias_relu2(float a0, float a1, float b0, float b1) {
    unsigned long long a, b, s;
    asm("mov.b64 %0, {%1, %2};" : "=l"(a) : "f"(a0), "f"(a1));
    asm("mov.b64 %0, {%1, %2};" : "=l"(b) : "f"(b0), "f"(b1));
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(s) : "l"(a), "l"(b));
    float s0, s1;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(s0), "=f"(s1) : "l"(s));
    const __nv_bfloat162 r = __hmax2(__floats2bfloat162_rn(s0, s1), __floats2bfloat162_rn(0.0f, 0.0f));
    return *reinterpret_cast<const unsigned*>(&r);
}

// Hidden-layer epilogue of this thread's row: h = relu(acc + b) to BF16,
// into the next layer's A operand (shared).
__device__ __forceinline__ void hidden_epilogue(unsigned char* hb, unsigned tlane, const float* b, int row) {
#pragma unroll 1
    for (int j = 0; j < NH / 32; ++j) {
        float v[32];
        tmem_ld32(tlane + 32 * j, v);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 b0 = *reinterpret_cast<const float4*>(b + 32 * j + 8 * q);
            const float4 b1 = *reinterpret_cast<const float4*>(b + 32 * j + 8 * q + 4);
            const float* u = v + 8 * q;
            *reinterpret_cast<uint4*>(hb + core_off(row, 32 * j + 8 * q, NH)) =
                make_uint4(bias_relu2(u[0], u[1], b0.x, b0.y), bias_relu2(u[2], u[3], b0.z, b0.w),
                           bias_relu2(u[4], u[5], b1.x, b1.y), bias_relu2(u[6], u[7], b1.z, b1.w));
        }
    }
}

// One CTA per SM: the weights once in shared memory (72 KB) and GROUPS groups
// of 128 threads, each taking tiles of its own through the four layers with an
// input tile, an activation tile (36 KB) and 128 TMEM columns of its own.  A
// tile is a chain of four dependent products with an epilogue each; while one
// group waits for its product or runs its epilogue, the others' products keep
// the tensor core at work.  Two CTAs of 128 threads, each with weights of its
// own, element-wise staging and two-byte stores took 61 us a call at 20,011
// rows and 615 us at 3,375,000; this form takes 41 and 350 (the tensor rate
// would allow 123).
__global__ void __launch_bounds__(GROUPS * TM, 1) k_mlp_forward_tc(long long n, const float* __restrict__ X, int vec,
                                                                   const __nv_bfloat16* __restrict__ wb,
                                                                   const float* __restrict__ p,
                                                                   const float* __restrict__ norm,
                                                                   float* __restrict__ Y, int* err,
                                                                   unsigned long long limit) {
    extern __shared__ __align__(1024) unsigned char tc_smem[];
    Smem& s = *reinterpret_cast<Smem*>(tc_smem);
    constexpr int NT = GROUPS * TM;
    const int tid = threadIdx.x, warp = tid >> 5, g = tid / TM, row = tid % TM;
    const long long ntiles = (n + TM - 1) / TM, stride = (long long)gridDim.x * GROUPS;
    long long tile = blockIdx.x + (long long)gridDim.x * g;
    float4 xv[NIN / 4];                          // this thread's row of the group's next tile
    auto fetch = [&](long long t) {
        const long long r = t * TM + row;
        if (r < n) {
#pragma unroll
            for (int q = 0; q < NIN / 4; ++q) xv[q] = load4(X + r * NIN + 4 * q, vec);
        }
    };
    fetch(tile);
    stage_tile<NIN>(s.w1, wb + OFF_W1, NH, NH, tid, NT);
    stage_tile<NH>(s.w2, wb + OFF_W2, NH, NH, tid, NT);
    stage_tile<NH>(s.w3, wb + OFF_W3, NH, NH, tid, NT);
    stage_tile<NH>(s.w4, wb + OFF_W4, N4, NOUT, tid, NT);
    if (tid < NH) {
        s.b[tid] = p[OFF_B1 + tid];
        s.b[NH + tid] = p[OFF_B2 + tid];
        s.b[2 * NH + tid] = p[OFF_B3 + tid];
    }
    if (tid < N4) s.b[3 * NH + tid] = (tid < NOUT) ? p[OFF_B4 + tid] : 0.0f;
    if (tid < NIN) {
        s.mean[tid] = norm[tid];
        s.istd[tid] = norm[NIN + tid];
    }
    if (tid < GROUPS) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s.bar[tid])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s.tmem)),
                     "r"(GROUPS * TCOLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_async_smem();
    before_sync();
    __syncthreads();
    after_sync();
    const unsigned tbase = s.tmem + (unsigned)(g * TCOLS);                // the group's accumulator
    const unsigned tlane = tbase + ((unsigned)((warp & 3) * 32) << 16);   // this warp's 32 TMEM lanes
    const unsigned long long dx = sdesc(s.x[g], NIN), dh = sdesc(s.h[g], NH);
    constexpr unsigned id128 = idesc_bf16(TM, NH), id16 = idesc_bf16(TM, N4);
    // one K step of 16 bf16 = two core matrices = 256 B = 16 in the address field
    constexpr unsigned long long KSTEP = 256 >> 4;
    unsigned char* xb = reinterpret_cast<unsigned char*>(s.x[g]);
    unsigned char* hb = reinterpret_cast<unsigned char*>(s.h[g]);
    unsigned parity = 0;
    bool ok = true;
    // A layer's MMAs, issued by one thread of the group once all its writes are in place ...
    auto issue = [&](unsigned long long a, const __nv_bfloat16* w, int k_in, unsigned id) {
        fence_async_smem();
        before_sync();
        group_sync(g);
        after_sync();
        if (row == 0) {
            const unsigned long long dw = sdesc(w, k_in);
#pragma unroll 8
            for (int k = 0; k < k_in / 16; ++k) mma(tbase, a + k * KSTEP, dw + k * KSTEP, id, k > 0);
            commit(&s.bar[g]);
        }
    };
    // ... and their completion (the whole group agrees).
    auto done = [&]() -> bool {
        const bool all = group_and(g, wait_phase(&s.bar[g], parity, limit));
        if (all) parity ^= 1u;
        after_sync();
        return all;
    };
    for (; tile < ntiles; tile += stride) {
        const long long r = tile * TM + row;
        {
            __align__(16) __nv_bfloat16 o[NIN];
#pragma unroll
            for (int q = 0; q < NIN / 4; ++q) {
                const float u[4] = {xv[q].x, xv[q].y, xv[q].z, xv[q].w};
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    o[4 * q + c] = __float2bfloat16(r < n ? (u[c] - s.mean[4 * q + c]) * s.istd[4 * q + c] : 0.0f);
            }
            *reinterpret_cast<uint4*>(xb + core_off(row, 0, NIN)) = reinterpret_cast<const uint4*>(o)[0];
            *reinterpret_cast<uint4*>(xb + core_off(row, 8, NIN)) = reinterpret_cast<const uint4*>(o)[1];
        }
        issue(dx, s.w1, NIN, id128);
        fetch(tile + stride);
        if (!(ok = done())) break;
        hidden_epilogue(hb, tlane, s.b, row);
        issue(dh, s.w2, NH, id128);
        if (!(ok = done())) break;
        hidden_epilogue(hb, tlane, s.b + NH, row);
        issue(dh, s.w3, NH, id128);
        if (!(ok = done())) break;
        hidden_epilogue(hb, tlane, s.b + 2 * NH, row);
        issue(dh, s.w4, NH, id16);
        if (!(ok = done())) break;
        float v[16];
        tmem_ld16(tlane, v);         // (the next tile's first product follows the group's next barrier)
        if (r < n) {
            float y[NOUT];
#pragma unroll
            for (int c = 0; c < NOUT; ++c) y[c] = v[c] + s.b[3 * NH + c];
            if (vec) {
                *reinterpret_cast<float4*>(Y + r * NOUT) = make_float4(y[0], y[1], y[2], y[3]);
            } else {
#pragma unroll
                for (int c = 0; c < NOUT; ++c) Y[r * NOUT + c] = y[c];
            }
        }
    }
    if (!ok) {
        if (row == 0) atomicExch(err, 1);
        wait_phase(&s.bar[g], parity);    // the phase that did not complete: let it finish (bounded)
    }
    before_sync();
    __syncthreads();
    after_sync();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s.tmem), "r"(GROUPS * TCOLS)
                     : "memory");
}

// ---- training pass: forward, loss, activation gradients and all weight and
// bias gradients of a tile of 128 rows without leaving the SM.  The tile's
// input, its three hidden activations and the weights stay in shared memory
// (184 KB, one CTA per SM); a layer's dZ overwrites the activation whose sign
// masked it.  Every tile is used in both directions (K-major for the layer
// products, MN-major for dZ W and dZ^T A, see the layout above), and the
// gradients accumulate in TMEM over the CTA's tiles:
//   columns   0 .. 127  the layer's product      128 .. 255  dW3 (lane = out)
//           256 .. 383  dW2 (lane = out)          384 .. 399  dW1 (lane = out)
//           400 .. 415  dW4^T (lane = in)         416 .. 463  db3, db2, db1
// (bias gradients: products with a column of ones).  A CTA leaves one set of
// partials, written column by column so that a warp stores 128 contiguous
// bytes; k_mlp_reduce sums them.  After 8 tiles the accumulators are added to
// the partials in FP32 and start again, so that no sum in TMEM runs over more
// than 1,024 rows.
// What bounds it: at a tile or two per SM the chain of 8 dependent products
// with an epilogue each, then the 143 KB of partials per CTA.  Through
// separate kernels (forward, backward, and per layer a weight-gradient, a
// reduction and a bias kernel, activations and dZ in HBM, two-byte strided
// loads, the loss by one block) a training step took 222 / 333 / 957 us at
// 64 / 16,384 / 65,536 rows; it takes 73 / 76 / 110 us now, with the
// caller's reads of the loss and the parameters (31 us at 16,384 rows in a
// loop that reads neither).
constexpr int TT = 256;              // threads: two per row, each with half the columns
constexpr int TRAIN_COLS = 512;      // TMEM columns allocated
constexpr int C_G3 = 128, C_G2 = 256, C_G1 = 384, C_G4 = 400, C_B = 416;
constexpr int FLUSH_TILES = 8;
constexpr int PSTRIDE = (NPARAM + 63) / 64 * 64;   // floats of one CTA's partials

struct __align__(128) TrainSmem {
    __nv_bfloat16 w4[N4 * NH];
    __nv_bfloat16 w3[NH * NH];
    __nv_bfloat16 w2[NH * NH];
    __nv_bfloat16 h[3][TM * NH];
    __nv_bfloat16 w1[NH * NIN];
    __nv_bfloat16 x[TM * NIN];
    __nv_bfloat16 dz[TM * N4];       // dZ4, columns 4 .. 15 zero
    __nv_bfloat16 ones[TM * N4];     // column 0 one, the others zero
    float b[3 * NH + N4];
    float mean[NIN], istd[NIN];
    float red[4], b4[4][NOUT];
    unsigned long long bar;
    unsigned tmem;
};

__global__ void __launch_bounds__(TT, 1) k_mlp_train_tc(long long n, const float* __restrict__ X,
                                                         const float* __restrict__ T, int vec,
                                                         const __nv_bfloat16* __restrict__ wb,
                                                         const float* __restrict__ p, const float* __restrict__ norm,
                                                         float* __restrict__ partial, float* __restrict__ tiles,
                                                         int* err, unsigned long long limit) {
    extern __shared__ __align__(1024) unsigned char tc_tsmem[];
    TrainSmem& s = *reinterpret_cast<TrainSmem*>(tc_tsmem);
    const int tid = threadIdx.x, warp = tid >> 5, row = tid & (TM - 1), half = tid / TM;
    stage_tile<NIN>(s.w1, wb + OFF_W1, NH, NH, tid, TT);
    stage_tile<NH>(s.w2, wb + OFF_W2, NH, NH, tid, TT);
    stage_tile<NH>(s.w3, wb + OFF_W3, NH, NH, tid, TT);
    stage_tile<NH>(s.w4, wb + OFF_W4, N4, NOUT, tid, TT);
    for (int i = tid; i < NH; i += TT) {
        s.b[i] = p[OFF_B1 + i];
        s.b[NH + i] = p[OFF_B2 + i];
        s.b[2 * NH + i] = p[OFF_B3 + i];
    }
    if (tid < N4) s.b[3 * NH + tid] = (tid < NOUT) ? p[OFF_B4 + tid] : 0.0f;
    if (tid < NIN) {
        s.mean[tid] = norm[tid];
        s.istd[tid] = norm[NIN + tid];
    }
    {   // half 0: columns 0 .. 7 of the ones, half 1: columns 8 .. 15 of both
        const uint4 zero = make_uint4(0, 0, 0, 0), one = make_uint4(0x3F80u, 0, 0, 0);
        *reinterpret_cast<uint4*>(reinterpret_cast<unsigned char*>(s.ones) + core_off(row, 8 * half, N4)) =
            half == 0 ? one : zero;
        *reinterpret_cast<uint4*>(reinterpret_cast<unsigned char*>(s.dz) + core_off(row, 8 * half, N4)) = zero;
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s.bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s.tmem)),
                     "r"(TRAIN_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_async_smem();
    before_sync();
    __syncthreads();
    after_sync();
    const unsigned tbase = s.tmem;
    const unsigned tlane = tbase + ((unsigned)((warp & 3) * 32) << 16);   // a warp reads lanes 32 (warp % 4) ..
    constexpr unsigned id128 = idesc_bf16(TM, NH), id16 = idesc_bf16(TM, N4);
    constexpr unsigned id128_b = idesc_bf16(TM, NH, false, true);         // dZ W
    constexpr unsigned id128_ab = idesc_bf16(TM, NH, true, true), id16_ab = idesc_bf16(TM, N4, true, true);   // dZ^T A
    // one K step of 16: along the columns of a tile (two core matrices), along its rows
    constexpr unsigned long long KC = 256 >> 4, KR = (2 * NH * 16) >> 4, KR16 = (2 * 16 * 16) >> 4;
    unsigned parity = 0;
    bool ok = true;
    // the step's MMAs, issued by one thread once every thread's writes are in place, and their completion
    auto product = [&](auto issue) -> bool {
        fence_async_smem();
        before_sync();
        __syncthreads();
        after_sync();
        if (tid == 0) {
            issue();
            commit(&s.bar);
        }
        const bool mine = wait_phase(&s.bar, parity, limit);
        const bool all = __syncthreads_and(mine) != 0;
        if (all) parity ^= 1u;
        after_sync();
        return all;
    };
    auto layer = [&](const __nv_bfloat16* a, const __nv_bfloat16* w, unsigned id) {   // a w^T, K = 128
        const unsigned long long da = sdesc(a, NH), dw = sdesc(w, NH);
#pragma unroll
        for (int k = 0; k < NH / 16; ++k) mma(tbase, da + k * KC, dw + k * KC, id, k > 0);
    };
    auto layer_back = [&](const __nv_bfloat16* dz, const __nv_bfloat16* w) {          // dz w
        const unsigned long long da = sdesc(dz, NH), dw = sdesc(w, NH, true);
#pragma unroll
        for (int k = 0; k < NH / 16; ++k) mma(tbase, da + k * KC, dw + k * KR, id128_b, k > 0);
    };
    // dst (+)= a^T b over the tile's rows; a 128 columns, b NB columns
    auto outer = [&](int dst, const __nv_bfloat16* a, const __nv_bfloat16* b, int nb, bool fresh) {
        const unsigned long long da = sdesc(a, NH, true), db = sdesc(b, nb, true);
        const unsigned id = nb == NH ? id128_ab : id16_ab;
        const unsigned long long kb = nb == NH ? KR : KR16;
#pragma unroll
        for (int k = 0; k < TM / 16; ++k) mma(tbase + dst, da + k * KR, db + k * kb, id, !fresh || k > 0);
    };
    // activation epilogue: h = relu(acc + b) (rows past n: 0, so that they add nothing to a gradient)
    auto forward_rows = [&](__nv_bfloat16* h, const float* b, bool valid) {
        unsigned char* hb = reinterpret_cast<unsigned char*>(h);
#pragma unroll
        for (int j = 2 * half; j < 2 * half + 2; ++j) {
            float v[32];
            tmem_ld32(tlane + 32 * j, v);
            __align__(16) __nv_bfloat16 o[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) o[i] = __float2bfloat16(valid ? fmaxf(v[i] + b[32 * j + i], 0.0f) : 0.0f);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                *reinterpret_cast<uint4*>(hb + core_off(row, 32 * j + 8 * q, NH)) = reinterpret_cast<const uint4*>(o)[q];
        }
    };
    // gradient epilogue: h (an activation) becomes dZ = acc [h > 0]
    auto backward_rows = [&](__nv_bfloat16* h, bool valid) {
        unsigned char* hb = reinterpret_cast<unsigned char*>(h);
#pragma unroll
        for (int j = 2 * half; j < 2 * half + 2; ++j) {
            float v[32];
            tmem_ld32(tlane + 32 * j, v);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint4* at = reinterpret_cast<uint4*>(hb + core_off(row, 32 * j + 8 * q, NH));
                __align__(16) __nv_bfloat16 o[8];
                *reinterpret_cast<uint4*>(o) = *at;
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    o[i] = __float2bfloat16(valid && __bfloat162float(o[i]) > 0.0f ? v[8 * q + i] : 0.0f);
                *at = *reinterpret_cast<const uint4*>(o);
            }
        }
    };
    const float scale = 2.0f / ((float)n * (float)NOUT);
    const long long ntiles = (n + TM - 1) / TM;
    float* out = partial + (size_t)blockIdx.x * PSTRIDE;
    float b4[NOUT] = {0.0f, 0.0f, 0.0f, 0.0f};           // (half 0) bias gradient of the last layer
    int held = 0;                                        // tiles in the accumulators
    bool first = true;                                   // no partials written yet
    auto put = [&](int e, float v) { out[e] = first ? v : out[e] + v; };
    auto flush = [&]() {
#pragma unroll 1
        for (int j = 2 * half; j < 2 * half + 2; ++j) {
            float v[32];
            tmem_ld32(tlane + C_G3 + 32 * j, v);
#pragma unroll
            for (int i = 0; i < 32; ++i) put(OFF_W3 + (32 * j + i) * NH + row, v[i]);
            tmem_ld32(tlane + C_G2 + 32 * j, v);
#pragma unroll
            for (int i = 0; i < 32; ++i) put(OFF_W2 + (32 * j + i) * NH + row, v[i]);
        }
        float v[16];
        if (half == 0) {
            tmem_ld16(tlane + C_G1, v);
#pragma unroll
            for (int i = 0; i < NIN; ++i) put(OFF_W1 + i * NH + row, v[i]);
        } else {
            tmem_ld16(tlane + C_G4, v);
#pragma unroll
            for (int i = 0; i < NOUT; ++i) put(OFF_W4 + i * NH + row, v[i]);
            tmem_ld16(tlane + C_B, v);
            put(OFF_B3 + row, v[0]);
            tmem_ld16(tlane + C_B + 16, v);
            put(OFF_B2 + row, v[0]);
            tmem_ld16(tlane + C_B + 32, v);
            put(OFF_B1 + row, v[0]);
        }
        first = false;
        held = 0;
    };
    for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const long long r = tile * TM + row;
        const bool valid = r < n;
        float4 t4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        {
            __align__(16) __nv_bfloat16 o[8];
            float v[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
            if (valid) {
                const float4 u0 = load4(X + r * NIN + 8 * half, vec), u1 = load4(X + r * NIN + 8 * half + 4, vec);
                const float u[8] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
#pragma unroll
                for (int c = 0; c < 8; ++c) v[c] = (u[c] - s.mean[8 * half + c]) * s.istd[8 * half + c];
                if (half == 0) t4 = load4(T + r * NOUT, vec);
            }
#pragma unroll
            for (int c = 0; c < 8; ++c) o[c] = __float2bfloat16(v[c]);
            *reinterpret_cast<uint4*>(reinterpret_cast<unsigned char*>(s.x) + core_off(row, 8 * half, NIN)) =
                *reinterpret_cast<const uint4*>(o);
        }
        const bool fresh = held == 0;
        if (!(ok = product([&] { mma(tbase, sdesc(s.x, NIN), sdesc(s.w1, NIN), id128, 0u); }))) break;
        forward_rows(s.h[0], s.b, valid);
        if (!(ok = product([&] { layer(s.h[0], s.w2, id128); }))) break;
        forward_rows(s.h[1], s.b + NH, valid);
        if (!(ok = product([&] { layer(s.h[1], s.w3, id128); }))) break;
        forward_rows(s.h[2], s.b + 2 * NH, valid);
        if (!(ok = product([&] { layer(s.h[2], s.w4, id16); }))) break;
        float lo = 0.0f;
        if (half == 0) {
            float v[16];
            tmem_ld16(tlane, v);
            const float t[NOUT] = {t4.x, t4.y, t4.z, t4.w};
            float y[NOUT];
            __align__(16) __nv_bfloat16 o[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) o[c] = __float2bfloat16(0.0f);
#pragma unroll
            for (int c = 0; c < NOUT; ++c) {
                y[c] = valid ? v[c] + s.b[3 * NH + c] : 0.0f;
                o[c] = __float2bfloat16(valid ? scale * (y[c] - t[c]) : 0.0f);
                b4[c] += __bfloat162float(o[c]);
            }
            lo = row_loss(y, t);
            *reinterpret_cast<uint4*>(reinterpret_cast<unsigned char*>(s.dz) + core_off(row, 0, N4)) =
                *reinterpret_cast<const uint4*>(o);
        }
        lo = tile_loss(lo, s.red);
        if (tid == 0) tiles[tile] = lo;
        if (!(ok = product([&] {
                  mma(tbase, sdesc(s.dz, N4), sdesc(s.w4, NH, true), id128_b, 0u);
                  outer(C_G4, s.h[2], s.dz, N4, fresh);
              })))
            break;
        backward_rows(s.h[2], valid);
        if (!(ok = product([&] {
                  layer_back(s.h[2], s.w3);
                  outer(C_G3, s.h[2], s.h[1], NH, fresh);
                  outer(C_B, s.h[2], s.ones, N4, fresh);
              })))
            break;
        backward_rows(s.h[1], valid);
        if (!(ok = product([&] {
                  layer_back(s.h[1], s.w2);
                  outer(C_G2, s.h[1], s.h[0], NH, fresh);
                  outer(C_B + 16, s.h[1], s.ones, N4, fresh);
              })))
            break;
        backward_rows(s.h[0], valid);
        if (!(ok = product([&] {
                  outer(C_G1, s.h[0], s.x, NIN, fresh);
                  outer(C_B + 32, s.h[0], s.ones, N4, fresh);
              })))
            break;
        if (++held == FLUSH_TILES) flush();
    }
    if (ok) {
        if (held > 0) flush();
        if (half == 0) {
#pragma unroll
            for (int c = 0; c < NOUT; ++c) {
                float v = b4[c];
                for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
                if ((tid & 31) == 0) s.b4[warp][c] = v;
            }
        }
        __syncthreads();
        if (tid < NOUT) out[OFF_B4 + tid] = (s.b4[0][tid] + s.b4[1][tid]) + (s.b4[2][tid] + s.b4[3][tid]);
    } else {
        if (tid == 0) atomicExch(err, 1);
        wait_phase(&s.bar, parity);       // the phase that did not complete: let it finish (bounded)
    }
    before_sync();
    __syncthreads();
    after_sync();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "r"(TRAIN_COLS) : "memory");
}

// Gradients from the CTAs' partials in a fixed order, with the Adam update if
// `update`; the last block folds the loss.  No gradient or weight is written once a wait of
// this or an earlier pass has run out: a CTA that gave up left its partials
// incomplete (its loss is not read either).  64 parameters per block, four
// threads per parameter (each a quarter of the partials, eight loads in
// flight): one thread per parameter over 128 partials leaves a thread with 16
// dependent rounds of loads.
__global__ void __launch_bounds__(256) k_mlp_reduce(long long n, int nparts, const float* __restrict__ partial,
                                                    const float* __restrict__ tiles, float* __restrict__ g,
                                                    float* __restrict__ loss, const int* err, int update,
                                                    const Adam a) {
    const int failed = *err;
    if (blockIdx.x == gridDim.x - 1) {
        if (update && !failed && threadIdx.x == 0) *a.steps = a.step;
        fold_loss(n, tiles, loss);
        return;
    }
    __shared__ float sh[4][64];
    const int lane = threadIdx.x & 63, q = threadIdx.x >> 6, e = blockIdx.x * 64 + lane;
    float s = 0.0f;
    if (e < NPARAM) {
        for (int c0 = q; c0 < nparts; c0 += 32) {
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = c0 + 4 * u < nparts ? partial[(size_t)(c0 + 4 * u) * PSTRIDE + e] : 0.0f;
            s += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
        }
    }
    sh[q][lane] = s;
    __syncthreads();
    if (q != 0 || e >= NPARAM || failed) return;
    s = (sh[0][lane] + sh[1][lane]) + (sh[2][lane] + sh[3][lane]);
    // dW1, dW2 and dW3 come transposed ([in][out])
    int i = e;
    if (e < OFF_B1) i = (e % NH) * NIN + e / NH;
    else if (e >= OFF_W2 && e < OFF_B2) i = OFF_W2 + ((e - OFF_W2) % NH) * NH + (e - OFF_W2) / NH;
    else if (e >= OFF_W3 && e < OFF_B3) i = OFF_W3 + ((e - OFF_W3) % NH) * NH + (e - OFF_W3) / NH;
    g[i] = s;
    if (update) adam_update(a, i, s);
}

}  // namespace tc
