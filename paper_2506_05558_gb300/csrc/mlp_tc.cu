// Tensor-core path (sm_100-family tcgen05) of the MLP's "TN" GEMM:
// C[m][n] = sum_k A[m][k] B[n][k], bf16 operands (K-major), FP32 accumulator
// in tensor memory.
//
// One CTA (4 warps) computes a 128 x Nt tile (Nt = N rounded up to 16, at most
// 256) of one K split. Per 64-wide K stage all threads copy the A (128 x 64)
// and B (Nt x 64) tiles into shared memory in the canonical no-swizzle K-major
// layout (8-row x 16-byte core matrices, K-adjacent cores 128 B apart, 8-row
// groups 1024 B apart), fence the async proxy, and one elected thread issues
// four tcgen05.mma (K = 16 each) into the TMEM accumulator and commits them to
// an mbarrier. The epilogue reads the accumulator back with tcgen05.ld (each
// warp its 32 TMEM lanes) and stores FP32 rows. Every wait on the mbarrier is
// bounded; on timeout the kernel records an error code, frees its TMEM and
// returns.
#include <cuda_bf16.h>

#include "common.cuh"
#include "mlp_train.cuh"

namespace gs {

constexpr int kTcM = 128;
constexpr int kTcBK = 64;
constexpr int kTcMaxN = 256;
constexpr uint32_t kTcSpinLimit = 1u << 22;

__device__ int g_tc_error;  // 0 = ok, otherwise the line of the failing wait

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// Shared-memory matrix descriptor (tcgen05): start address, leading (K) and
// stride (M/N) byte offsets in 16-byte units, descriptor version 1, no swizzle.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// Instruction descriptor, kind::f16: D f32, A and B bf16, both K-major, N, M.
__host__ __device__ constexpr uint32_t instr_desc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

__global__ void __launch_bounds__(128) k_gemm_tn_tc(const __nv_bfloat16* __restrict__ A, int64_t lda,
                                                    const __nv_bfloat16* __restrict__ B, int64_t ldb,
                                                    float* __restrict__ C, int64_t ldc, int64_t M, int N, int Nt,
                                                    int64_t K, int64_t k_per_split, int64_t c_split_stride,
                                                    uint32_t tmem_cols) {
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ __align__(8) uint64_t s_bar;
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail;
    uint8_t* sA = smem;  // two buffers of A (128 x 64 bf16) followed by B (Nt x 64 bf16)
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t m0 = (int64_t)blockIdx.x * kTcM;
    const int64_t kb = (int64_t)blockIdx.z * k_per_split;
    const int64_t ke = min(K, kb + k_per_split);
    const uint32_t bar = smem_u32(&s_bar);

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&s_tmem)),
                     "r"(tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(bar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        s_fail = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = s_tmem;
    const uint32_t idesc = instr_desc_bf16(kTcM, Nt);
    uint32_t phase = 0;
    bool first = true;
    const int rows_total = kTcM + Nt;
    const uint32_t buf_bytes = (uint32_t)rows_total * kTcBK * 2;
    // stage k0 into buffer b: 16-byte cp.async copies (zero-filled outside the matrix), one commit group
    auto issue_stage = [&](int64_t k0, int b) {
        uint8_t* sAb = sA + b * buf_bytes;
        uint8_t* sBb = sAb + kTcM * kTcBK * 2;
        for (int i = tid; i < rows_total * (kTcBK / 8); i += 128) {
            const int r = i / (kTcBK / 8), kc = i % (kTcBK / 8);
            const bool isA = r < kTcM;
            const int rr = isA ? r : r - kTcM;
            const int64_t grow = isA ? m0 + rr : rr;
            const int64_t gk = k0 + kc * 8;
            const bool row_ok = isA ? grow < M : grow < N;
            uint8_t* dst = (isA ? sAb : sBb) + (uint32_t)(((rr >> 3) * (kTcBK / 8) + kc) * 128 + (rr & 7) * 16);
            if (row_ok && gk < ke && gk + 8 > ke) {  // a K tail inside the chunk: element by element
                __nv_bfloat16 tmp[8];
                const __nv_bfloat16* src = (isA ? A + grow * lda : B + grow * ldb);
                for (int e = 0; e < 8; e++) tmp[e] = (gk + e < ke) ? src[gk + e] : __float2bfloat16_rn(0.f);
                *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<uint4*>(tmp);
                continue;
            }
            const bool ok = row_ok && gk + 8 <= ke;
            const __nv_bfloat16* src = ok ? (isA ? A + grow * lda : B + grow * ldb) + gk : A;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_u32(dst)), "l"(src),
                         "r"(ok ? 16 : 0)
                         : "memory");
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };

    // double-buffered: the copies of slice s + 1 are in flight while slice s is
    // waited for and multiplied; a buffer is refilled only after the MMA that
    // read it has completed (the mbarrier wait at the end of its iteration)
    if (kb < ke) issue_stage(kb, 0);
    int buf = 0;
    for (int64_t k0 = kb; k0 < ke; k0 += kTcBK) {
        const bool more = k0 + kTcBK < ke;
        if (more) issue_stage(k0 + kTcBK, buf ^ 1);
        if (more) asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        else asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        __syncthreads();
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const uint32_t a0 = smem_u32(sA + buf * buf_bytes), b0 = a0 + kTcM * kTcBK * 2;
#pragma unroll
            for (int s = 0; s < kTcBK / 16; s++) {
                const uint64_t ad = smem_desc(a0 + s * 256, 128, 1024);
                const uint64_t bd = smem_desc(b0 + s * 256, 128, 1024);
                const uint32_t acc = (first && s == 0) ? 0u : 1u;
                asm volatile(
                    "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                    "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
                    "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
                    : "memory");
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar)
                         : "memory");
            uint32_t spins = 0;
            while (!mbar_try_wait(bar, phase)) {
                if (++spins > kTcSpinLimit) {
                    s_fail = 1;
                    break;
                }
            }
        }
        first = false;
        phase ^= 1u;
        buf ^= 1;
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        if (s_fail) {
            asm volatile("cp.async.wait_group 0;\n" ::: "memory");  // no copy may land after the exit
            break;
        }
    }

    if (!s_fail && !first) {
        // epilogue: warp w reads TMEM lanes 32w..32w+31 (rows of the tile), 16 columns at a time
        const int64_t row = m0 + 32 * warp + lane;
        float* Cz = C + (int64_t)blockIdx.z * c_split_stride;
        for (int c0 = 0; c0 < Nt; c0 += 16) {
            uint32_t r[16];
            const uint32_t taddr = tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)c0;
            asm volatile(
                "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
                "[%16];\n"
                : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                  "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                  "=r"(r[15])
                : "r"(taddr));
            asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
            if (row < M && c0 < N) {  // N and ldc are multiples of 16: whole 16-column groups, 128-bit stores
                float4* dst = reinterpret_cast<float4*>(Cz + row * ldc + c0);
#pragma unroll
                for (int j = 0; j < 4; j++)
                    dst[j] = make_float4(__uint_as_float(r[4 * j]), __uint_as_float(r[4 * j + 1]),
                                         __uint_as_float(r[4 * j + 2]), __uint_as_float(r[4 * j + 3]));
            }
        }
    } else if (s_fail && tid == 0) {
        atomicCAS(&g_tc_error, 0, __LINE__);
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(tmem_cols) : "memory");
    }
}

int gemm_tn_tc(const __nv_bfloat16* A, int64_t lda, const __nv_bfloat16* B, int64_t ldb, float* C, int64_t ldc,
               int64_t M, int N, int64_t K, int64_t k_per_split, int64_t c_split_stride, cudaStream_t s) {
    const int Nt = (int)ceil_div(N, 16) * 16;
    if (Nt > kTcMaxN || M <= 0 || K <= 0) return GS_ERR_INVALID_ARG;
    uint32_t cols = 32;
    while (cols < (uint32_t)Nt) cols <<= 1;
    const size_t smem = 2 * (size_t)(kTcM + Nt) * kTcBK * 2;  // two stages
    static bool attr_set = false;
    if (!attr_set) {
        // at most ~115 KB of the SM's shared memory per CTA so that at most two
        // CTAs (2 x 256 TMEM columns) share an SM
        cudaFuncSetAttribute(k_gemm_tn_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
        attr_set = true;
    }
    const size_t smem_launch = smem < 80 * 1024 ? 80 * 1024 : smem;
    const int64_t splits = ceil_div(K, k_per_split);
    dim3 grid((unsigned)ceil_div(M, kTcM), 1, (unsigned)splits);
    k_gemm_tn_tc<<<grid, 128, smem_launch, s>>>(A, lda, B, ldb, C, ldc, M, N, Nt, K, k_per_split, c_split_stride,
                                                 cols);
    count_launch();
    return GS_OK;
}

}  // namespace gs

extern "C" int gs_mlp_tc_error(int32_t* out) {
    if (!out) return GS_ERR_INVALID_ARG;
    int v = 0;
    if (cudaMemcpyFromSymbol(&v, gs::g_tc_error, sizeof(int)) != cudaSuccess) {
        (void)cudaGetLastError();
        return GS_ERR_CUDA;
    }
    *out = v;
    return GS_OK;
}

namespace gs {

// ---------------------------------------------------------------------------
// Fused inference of the whole MLP on tensor cores (tcgen05).
//
// Persistent CTAs of 512 threads, one per SM (about 206 KB of shared memory):
// each converts the four weight matrices to bfloat16 once, in the canonical
// no-swizzle K-major layout (K-adjacent 8x16-byte core matrices 128 B apart,
// 8-row groups (K/8) * 128 B apart), then walks 128-patch tiles. Per tile the
// threads gather the patch features straight from the image into the same
// layout (X, 128 x 208), and for each layer one elected thread issues the
// K/16 tcgen05.mma (M = 128 patches, N = 128 or 16, bf16 in, FP32 in a
// 128-column TMEM accumulator) and commits them to an mbarrier; the sixteen
// warps then read the accumulator back (warps w, w + 4, w + 8 and w + 12 share TMEM
// lane quarter w % 4 and split the columns), add the bias, apply GELU and write the
// bf16 activations over the previous layer's buffer (that product has
// completed) as the next layer's A operand. The last layer writes (logit,
// depth, log-scale) in FP32. Every mbarrier wait is bounded; on timeout the
// kernel records the failing line in g_tc_error, frees its TMEM and returns.
// ---------------------------------------------------------------------------
constexpr int kFM = 128, kFIn = 194, kFInPad = 208, kFHid = 128, kFOut = 3, kFOutPad = 16;
constexpr int kFThreads = 512;
constexpr uint32_t kFOffW1 = 0;
constexpr uint32_t kFOffW2 = kFOffW1 + kFHid * kFInPad * 2;     // 53248
constexpr uint32_t kFOffW3 = kFOffW2 + kFHid * kFHid * 2;       // 86016
constexpr uint32_t kFOffW4 = kFOffW3 + kFHid * kFHid * 2;       // 118784
constexpr uint32_t kFOffX = kFOffW4 + kFOutPad * kFHid * 2;     // 122880
constexpr uint32_t kFOffH = kFOffX + kFM * kFInPad * 2;         // 176128
constexpr uint32_t kFOffB = kFOffH + kFM * kFHid * 2;           // 208896: biases, FP32
constexpr uint32_t kFSmem = kFOffB + (3 * kFHid + kFOutPad) * 4;

// Byte offset of element (r, k) of a K-major [rows][K] bf16 matrix, K % 8 == 0.
__device__ __forceinline__ uint32_t kmajor_off(int r, int k, int K) {
    return (uint32_t)((((r >> 3) * (K >> 3) + (k >> 3)) << 7) + ((r & 7) << 4) + ((k & 7) << 1));
}

__device__ __forceinline__ uint4 pack8_bf16(const float* v) {
    uint4 u;
    uint32_t* w = reinterpret_cast<uint32_t*>(&u);
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
        w[i] = *reinterpret_cast<const uint32_t*>(&h);
    }
    return u;
}

// Element j (0..7) of eight packed bfloat16 values (j a compile-time constant in
// unrolled loops, so the value stays in registers).
__device__ __forceinline__ __nv_bfloat16 bf16_at(const uint4& u, int j) {
    const uint32_t w = j < 2 ? u.x : j < 4 ? u.y : j < 6 ? u.z : u.w;
    return __ushort_as_bfloat16((unsigned short)((j & 1) ? (w >> 16) : (w & 0xFFFFu)));
}

__device__ __forceinline__ float gelu_erf(float z) { return 0.5f * z * (1.f + erff(z * 0.70710678118654752f)); }

// W [rows_valid][cols_valid] FP32 (nn.Linear layout) -> bf16 [rows][K] K-major at dst, zero padded.
__device__ void stage_weight(const float* __restrict__ Wm, int rows_valid, int cols_valid, int rows, int K,
                             uint8_t* dst) {
    const int chunks = rows * (K >> 3);
#pragma unroll 4
    for (int q = threadIdx.x; q < chunks; q += blockDim.x) {
        const int r = q / (K >> 3), kc = q % (K >> 3);
        float v[8];
#pragma unroll
        for (int e = 0; e < 8; e++) {
            const int k = kc * 8 + e;
            v[e] = (r < rows_valid && k < cols_valid) ? Wm[(int64_t)r * cols_valid + k] : 0.f;
        }
        *reinterpret_cast<uint4*>(dst + kmajor_off(r, kc * 8, K)) = pack8_bf16(v);
    }
}

// What the training step's backward needs from the forward, written by the
// TRAIN instantiation: the features transposed (Xt [208][Mp], bf16), the derivative of
// the activation at the pre-activations (G[l] [128][Mp] FP32, l < 3: the error function
// is at hand here) and the activations, both transposed (Ht[l] [128][Mp], bf16), the output
// layer before its bias (Z3 [Mp][16] FP32), rows up to Mp; and the weights transposed
// (Wt[l - 1] [in][out padded], bf16, l = 1..3).
struct TrainFwdOut {
    __nv_bfloat16* Xt;
    float* G[3];
    __nv_bfloat16* Ht[3];
    float* Z3;
    __nv_bfloat16* Wt[3];
    int64_t Mp;
};

// GELU and its derivative, the values of gelu_f and gelu_grad_f.
__device__ __forceinline__ void gelu_both(float z, float& f, float& g) {
    const float e = 1.f + erff(z * 0.70710678118654752f);
    f = 0.5f * z * e;
    g = 0.5f * e + z * 0.39894228040143268f * expf(-0.5f * z * z);
}

template <bool TRAIN>
__global__ void __launch_bounds__(kFThreads, 1) k_mlp_forward_tc(
    const float* __restrict__ image, int W, int H, const float* __restrict__ w1, const float* __restrict__ b1,
    const float* __restrict__ w2, const float* __restrict__ b2, const float* __restrict__ w3,
    const float* __restrict__ b3, const float* __restrict__ w4, const float* __restrict__ b4,
    float* __restrict__ out, TrainFwdOut to) {
    extern __shared__ __align__(1024) uint8_t sm[];
    __shared__ __align__(8) uint64_t s_bar;
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nx = W >> 3, ny = H >> 3;
    const int64_t M = (int64_t)nx * ny;
    const int64_t n_tiles = TRAIN ? to.Mp / kFM : (M + kFM - 1) / kFM;
    const uint32_t bar = smem_u32(&s_bar);
    float* s_b = reinterpret_cast<float*>(sm + kFOffB);  // b1 | b2 | b3 | b4 (padded to 16)

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&s_tmem)),
                     "r"(128)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(bar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        s_fail = 0;
    }
    stage_weight(w1, kFHid, kFIn, kFHid, kFInPad, sm + kFOffW1);
    stage_weight(w2, kFHid, kFHid, kFHid, kFHid, sm + kFOffW2);
    stage_weight(w3, kFHid, kFHid, kFHid, kFHid, sm + kFOffW3);
    stage_weight(w4, kFOut, kFHid, kFOutPad, kFHid, sm + kFOffW4);
    for (int i = tid; i < 3 * kFHid + kFOutPad; i += kFThreads) {
        const int l = i / kFHid, j = i % kFHid;
        s_b[i] = l == 0 ? b1[j] : l == 1 ? b2[j] : l == 2 ? b3[j] : (j < kFOut ? b4[j] : 0.f);
    }
    if (TRAIN) {
        for (int i = blockIdx.x * kFThreads + tid; i < kFHid * (2 * kFHid + kFOutPad); i += gridDim.x * kFThreads) {
            const int l = i / (kFHid * kFHid), j = i % (kFHid * kFHid), ro = l < 2 ? kFHid : kFOutPad;
            const int c = j / ro, r = j % ro;
            const float* wl = l == 0 ? w2 : l == 1 ? w3 : w4;
            __nv_bfloat16* wt = l == 0 ? to.Wt[0] : l == 1 ? to.Wt[1] : to.Wt[2];
            wt[j] = __float2bfloat16_rn(l < 2 || r < kFOut ? wl[r * kFHid + c] : 0.f);
        }
    }
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = s_tmem;
    const uint32_t sbase = smem_u32(sm);
    uint32_t phase = 0;

    for (int64_t tile = blockIdx.x; tile < n_tiles && !s_fail; tile += gridDim.x) {
        // 1. features: chunk q = (row r, 8-column group kc); a warp covers 32 patches of one group
        const int64_t p0 = tile * kFM;
#pragma unroll 4
        for (int q = tid; q < kFM * (kFInPad >> 3); q += kFThreads) {
            const int r = q % kFM, kc = q / kFM;
            const int64_t p = p0 + r;
            float v[8];
            if (p < M) {
                const int py = (int)(p / nx), px = (int)(p % nx);
                if (kc < 24) {  // 3 channels x 8 rows of 8 pixels
                    const int c = kc >> 3, dy = kc & 7;
                    const float4* src =
                        reinterpret_cast<const float4*>(image + ((int64_t)c * H + 8 * py + dy) * W + 8 * px);
                    const float4 a = src[0], b = src[1];
                    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
                } else {
#pragma unroll
                    for (int e = 0; e < 8; e++) v[e] = 0.f;
                    if (kc == 24) {  // patch centre in [-1, 1]^2, x first
                        v[0] = (px + 0.5f) / nx * 2.f - 1.f;
                        v[1] = (py + 0.5f) / ny * 2.f - 1.f;
                    }
                }
            } else {
#pragma unroll
                for (int e = 0; e < 8; e++) v[e] = 0.f;
            }
            const uint4 pk = pack8_bf16(v);
            *reinterpret_cast<uint4*>(sm + kFOffX + kmajor_off(r, kc * 8, kFInPad)) = pk;
            if (TRAIN) {  // X^T: for each of the 8 columns, consecutive threads write consecutive patches
#pragma unroll
                for (int e = 0; e < 8; e++) to.Xt[(int64_t)(kc * 8 + e) * to.Mp + p] = bf16_at(pk, e);
            }
        }
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        __syncthreads();

        for (int l = 0; l < 4; l++) {
            const int K = l == 0 ? kFInPad : kFHid;
            const int N = l == 3 ? kFOutPad : kFHid;
            if (tid == 0) {
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                const uint32_t a0 = sbase + (l == 0 ? kFOffX : kFOffH);
                const uint32_t b0 = sbase + (l == 0 ? kFOffW1 : l == 1 ? kFOffW2 : l == 2 ? kFOffW3 : kFOffW4);
                const uint32_t sbo = (uint32_t)(K >> 3) * 128u;
                const uint32_t idesc = instr_desc_bf16(kFM, N);
                for (int s = 0; s < K / 16; s++) {
                    const uint64_t ad = smem_desc(a0 + s * 256, 128, sbo);
                    const uint64_t bd = smem_desc(b0 + s * 256, 128, sbo);
                    const uint32_t acc = s > 0 ? 1u : 0u;
                    asm volatile(
                        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
                        "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
                        : "memory");
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                                 bar)
                             : "memory");
                uint32_t spins = 0;
                while (!mbar_try_wait(bar, phase)) {
                    if (++spins > kTcSpinLimit) {
                        s_fail = __LINE__;
                        break;
                    }
                }
            }
            phase ^= 1u;
            __syncthreads();
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            if (s_fail) break;
            // 2. epilogue: row r of the tile = TMEM lane 32 (warp % 4) + lane
            const int quarter = warp & 3, cols = warp >> 2;
            const int r = 32 * quarter + lane;
            const uint32_t trow = tmem + ((uint32_t)(32 * quarter) << 16);
            if (l < 3) {
                for (int c0 = 32 * cols; c0 < 32 * cols + 32; c0 += 16) {
                    uint32_t u[16];
                    asm volatile(
                        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
                        "%15}, [%16];\n"
                        : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]),
                          "=r"(u[7]), "=r"(u[8]), "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]),
                          "=r"(u[14]), "=r"(u[15])
                        : "r"(trow + (uint32_t)c0));
                    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
                    float v[16];
                    if (TRAIN) {
                        const int64_t p = p0 + r;
                        float zr[16];
#pragma unroll
                        for (int j = 0; j < 16; j++) zr[j] = __uint_as_float(u[j]) + s_b[l * kFHid + c0 + j];
                        float* Gl = l == 0 ? to.G[0] : l == 1 ? to.G[1] : to.G[2];  // no dynamic index into the param
#pragma unroll
                        for (int j = 0; j < 16; j++) gelu_both(zr[j], v[j], zr[j]);
#pragma unroll
                        for (int j = 0; j < 16; j++) Gl[(int64_t)(c0 + j) * to.Mp + p] = zr[j];
                    } else {
#pragma unroll
                        for (int j = 0; j < 16; j++) v[j] = gelu_erf(__uint_as_float(u[j]) + s_b[l * kFHid + c0 + j]);
                    }
                    const uint4 h0 = pack8_bf16(v), h1 = pack8_bf16(v + 8);
                    *reinterpret_cast<uint4*>(sm + kFOffH + kmajor_off(r, c0, kFHid)) = h0;
                    *reinterpret_cast<uint4*>(sm + kFOffH + kmajor_off(r, c0 + 8, kFHid)) = h1;
                    if (TRAIN) {  // H^T: per column, the warp's 32 consecutive patches
                        const int64_t p = p0 + r;
                        __nv_bfloat16* Hl = l == 0 ? to.Ht[0] : l == 1 ? to.Ht[1] : to.Ht[2];
#pragma unroll
                        for (int j = 0; j < 8; j++) {
                            Hl[(int64_t)(c0 + j) * to.Mp + p] = bf16_at(h0, j);
                            Hl[(int64_t)(c0 + 8 + j) * to.Mp + p] = bf16_at(h1, j);
                        }
                    }
                }
            } else if (cols == 0) {
                uint32_t u[16];
                asm volatile(
                    "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
                    "%15}, [%16];\n"
                    : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]),
                      "=r"(u[8]), "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]),
                      "=r"(u[15])
                    : "r"(trow));
                asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
                const int64_t p = p0 + r;
                if (TRAIN) {  // the output layer before its bias, all 16 padded columns, every row up to Mp
                    float4* zd = reinterpret_cast<float4*>(to.Z3 + p * kFOutPad);
#pragma unroll
                    for (int j = 0; j < 4; j++)
                        zd[j] = make_float4(__uint_as_float(u[4 * j]), __uint_as_float(u[4 * j + 1]),
                                            __uint_as_float(u[4 * j + 2]), __uint_as_float(u[4 * j + 3]));
                } else if (p < M) {
#pragma unroll
                    for (int j = 0; j < kFOut; j++) out[p * kFOut + j] = __uint_as_float(u[j]) + s_b[3 * kFHid + j];
                }
            }
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
            __syncthreads();
        }
    }
    if (s_fail && tid == 0) atomicCAS(&g_tc_error, 0, s_fail);
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(128) : "memory");
    }
}

// ---------------------------------------------------------------------------
// Loss and backward pass of one training step in one launch (tcgen05).
//
// CTA b takes the 256 patches of split b: the loss and its gradient from the output
// layer, then per layer, from the last, on dZ (bf16, held in shared memory as rows for
// dH and transposed for dW): dH = dZ W (two M = 128 products, operands in shared
// memory), this split's share of dW = dZ^T H (M = 128, K = 256 patches, H^T staged in
// four slices), both accumulated in the 512 columns of TMEM; then dZ of the layer below =
// dH * G, element by element from TMEM. Two more warps add the columns of the FP32 dZ,
// row after row (the bias gradients), from copies of 16 columns while the other eight
// form the next 16. The shares go to part [split][kBwStride]; k_mlp_reduce
// adds them in split order.
// A 1080p frame (32400 patches, 127 CTAs): 56 us against 340 for 18 launches of 15-22 us
// (products, GELU, split and column sums, each bound by latency). Bound by latency here
// too (24% of issue slots): a layer is 7000 cycles of slices and products and 11000 of
// dZ and sums. Shares written neuron by neuron (32 lines a store) and column sums by
// one warp, eight loads ahead, took 86 us.
// Every mbarrier wait is bounded, as above.
// ---------------------------------------------------------------------------
constexpr int kBwRows = 256, kBwThreads = 320;
constexpr uint32_t kBwOffZ = 0;                                    // dZ [2][128][K <= 128]
constexpr uint32_t kBwOffZt = kBwOffZ + kBwRows * kFHid * 2;       // dZ^T [128][256]
constexpr uint32_t kBwOffW = kBwOffZt + kFHid * kBwRows * 2;       // W^T [in 128][out]
constexpr uint32_t kBwOffB = kBwOffW + kFHid * kFHid * 2;          // H^T slices [in <= 208][64], FP32 columns
constexpr uint32_t kBwSlice = kFHid * kTcBK * 2, kBwSlice0 = kFInPad * kTcBK * 2;
constexpr uint32_t kBwColBuf = kBwRows * 17 * 4;                   // 16 columns, one word of padding a row
constexpr uint32_t kBwSmem = kBwOffB + 2 * kBwColBuf + 2 * kBwSlice;  // 231,424 bytes
static_assert(2 * kBwSlice <= 2 * kBwColBuf && kBwSlice0 <= 2 * kBwSlice && kBwSmem <= 232448, "buffers fit");
// Slices 0 and 1 lie behind the column buffers and are fetched while these are in use,
// 2 and 3 over them; of the first layer's wider ones, two are in flight.
__device__ __forceinline__ uint32_t bw_slice(int l, int sl) {
    if (l == 0) return kBwOffB + (sl & 1 ? 0 : 2 * kBwColBuf);
    return kBwOffB + (sl < 2 ? 2 * kBwColBuf + sl * kBwSlice : (sl - 2) * kBwSlice);
}

__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void bar_arrive(int id, int n) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t addr, float (&v)[16]) {
    uint32_t u[16];
    __syncwarp();
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]), "=r"(u[8]),
          "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]), "=r"(u[15])
        : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int j = 0; j < 16; j++) v[j] = __uint_as_float(u[j]);
}

// A run of K / 16 products into the accumulator at d, from K-major operands with
// core-matrix rows sbo bytes apart; keep: add to what is there.
__device__ __forceinline__ void mma_run(uint32_t d, uint32_t a, uint32_t a_sbo, uint32_t b, uint32_t b_sbo, int steps,
                                        uint32_t idesc, bool keep) {
    for (int s = 0; s < steps; s++) {
        const uint64_t ad = smem_desc(a + s * 256, 128, a_sbo), bd = smem_desc(b + s * 256, 128, b_sbo);
        asm volatile(
            "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
            "l"(ad), "l"(bd), "r"(idesc), "r"((keep || s > 0) ? 1u : 0u)
            : "memory");
    }
}

struct BwdIn {
    const float* Z3;
    const float* b4;
    const float* targets;
    const float* G[3];
    const __nv_bfloat16* Hin_t[4];  // X^T, H_0^T, H_1^T, H_2^T
    const __nv_bfloat16* Wt[3];     // of layers 1, 2, 3
    int64_t M, Mp;
    float w_depth, w_scale;
    float* out;        // [M][3] or null
    float* part;       // [splits][kMlpPart]
    float* loss_part;  // [splits]
};

__global__ void __launch_bounds__(kBwThreads, 1) k_mlp_backward_tc(const __grid_constant__ BwdIn in) {
    extern __shared__ __align__(1024) uint8_t sm[];
    __shared__ __align__(8) uint64_t s_bar;
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail;
    __shared__ float s_red[8];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool maker = tid < 256;  // the last two warps add columns
    const int64_t k0 = (int64_t)blockIdx.x * kBwRows, ke = min(k0 + kBwRows, in.Mp);
    const uint32_t bar = smem_u32(&s_bar), sbase = smem_u32(sm);
    float* part = in.part + (int64_t)blockIdx.x * kMlpPart;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&s_tmem)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(bar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        s_fail = 0;
    }
    // W^T of layer l (in rows of `out` values) to shared memory
    auto load_w = [&](int l) {
        const int K = l == 3 ? kFOutPad : kFHid;
        const __nv_bfloat16* wt = l == 3 ? in.Wt[2] : l == 2 ? in.Wt[1] : in.Wt[0];
        for (int q = tid; q < kFHid * (K >> 3); q += 256) {
            const int r = q / (K >> 3), kc = q % (K >> 3);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sbase + kBwOffW + kmajor_off(r, kc * 8, K)),
                         "l"(wt + r * K + kc * 8)
                         : "memory");
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    // the loss: thread t, patch k0 + t (as k_mlp_loss)
    float* col3 = reinterpret_cast<float*>(sm + kBwOffZ + kBwRows * kFOutPad * 2);  // behind the last layer's dZ
    if (maker) {
        load_w(3);
        for (int i = tid; i < kFHid * kBwRows * 2 / 16; i += 256)
            reinterpret_cast<uint4*>(sm + kBwOffZt)[i] = make_uint4(0u, 0u, 0u, 0u);
        const int64_t m = k0 + tid;
        float l = 0.f, g[3] = {0.f, 0.f, 0.f};
        if (m < in.M) {
            const float4 z = *reinterpret_cast<const float4*>(in.Z3 + m * kFOutPad);
            const float logit = z.x + in.b4[0], depth = z.y + in.b4[1], ls = z.z + in.b4[2];
            if (in.out) {
                in.out[m * 3 + 0] = logit;
                in.out[m * 3 + 1] = depth;
                in.out[m * 3 + 2] = ls;
            }
            const float t = in.targets[m * 4 + 0], zt = in.targets[m * 4 + 1], st = in.targets[m * 4 + 2];
            const float mask = in.targets[m * 4 + 3];
            const float inv = 1.f / (float)in.M;
            // softplus(x) - t x, computed stably
            l = fmaxf(logit, 0.f) + log1pf(expf(-fabsf(logit))) - t * logit;
            l += in.w_depth * mask * fabsf(depth - zt) + in.w_scale * mask * fabsf(ls - st);
            l *= inv;
            auto sg = [](float x) { return x > 0.f ? 1.f : (x < 0.f ? -1.f : 0.f); };
            g[0] = (1.f / (1.f + expf(-logit)) - t) * inv;
            g[1] = in.w_depth * mask * sg(depth - zt) * inv;
            g[2] = in.w_scale * mask * sg(ls - st) * inv;
        }
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (lane == 0) s_red[warp] = l;
        bar_sync(1, 256);  // the zeros are in place
        const float v[8] = {g[0], g[1], g[2], 0.f, 0.f, 0.f, 0.f, 0.f};
        const uint4 pk = pack8_bf16(v);
        uint8_t* z = sm + kBwOffZ + (tid >> 7) * (128 * kFOutPad * 2);
        *reinterpret_cast<uint4*>(z + kmajor_off(tid & 127, 0, kFOutPad)) = pk;
        *reinterpret_cast<uint4*>(z + kmajor_off(tid & 127, 8, kFOutPad)) = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int c = 0; c < 3; c++) {
            *reinterpret_cast<__nv_bfloat16*>(sm + kBwOffZt + kmajor_off(c, tid, kBwRows)) = bf16_at(pk, c);
            col3[tid * 17 + c] = g[c];
        }
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    }
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = s_tmem;
    // a column's sum, row after row
    auto add_column = [&](const float* col, float* dst) {
        float a = 0.f;
#pragma unroll 32
        for (int r = 0; r < kBwRows; r++) a += col[r * 17];
        *dst = a;
    };
    if (warp == 8) {
        if (lane < 3) add_column(col3 + lane, part + kMlpPartB3 + lane);
        if (lane == 31) {
            float a = 0.f;
            for (int k = 0; k < 8; k++) a += s_red[k];
            in.loss_part[blockIdx.x] = a;
        }
    }
    auto load_slice = [&](int l, int sl) {  // 64 patches of the layer's H^T, zeros past the split
        const int n_in = l == 0 ? kFInPad : kFHid;
        const __nv_bfloat16* ht = l == 0 ? in.Hin_t[0] : l == 1 ? in.Hin_t[1] : l == 2 ? in.Hin_t[2] : in.Hin_t[3];
        const uint32_t dst = sbase + bw_slice(l, sl);
        for (int q = tid; q < n_in * (kTcBK / 8); q += 256) {
            const int r = q / (kTcBK / 8), kc = q % (kTcBK / 8);
            const int64_t gk = k0 + sl * kTcBK + kc * 8;
            const bool ok = gk + 8 <= ke;  // Mp is a multiple of 128
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst + kmajor_off(r, kc * 8, kTcBK)),
                         "l"(ht + (ok ? (int64_t)r * in.Mp + gk : 0)), "r"(ok ? 16 : 0)
                         : "memory");
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    if (maker) {
        load_slice(3, 0);
        load_slice(3, 1);
    }
    uint32_t phase = 0;

    for (int l = 3; l >= 0; l--) {
        const int n_in = l == 0 ? kFInPad : kFHid;
        constexpr int kSlices = kBwRows / kTcBK;
        // slices 0 and 1 (of the first layer, 0) are on their way
        if (maker) {
            if (l == 0) {
                load_slice(0, 1);
            } else {
                load_slice(l, 2);
                load_slice(l, 3);
            }
        }
        for (int sl = 0; sl < kSlices; sl++) {
            if (maker) {
                if (l == 0) {
                    if (sl < kSlices - 1) asm volatile("cp.async.wait_group 1;\n" ::: "memory");
                    else asm volatile("cp.async.wait_group 0;\n" ::: "memory");
                } else {
                    if (sl == 0) asm volatile("cp.async.wait_group 3;\n" ::: "memory");
                    else if (sl == 1) asm volatile("cp.async.wait_group 2;\n" ::: "memory");
                    else if (sl == 2) asm volatile("cp.async.wait_group 1;\n" ::: "memory");
                    else asm volatile("cp.async.wait_group 0;\n" ::: "memory");
                }
                asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
            }
            __syncthreads();
            const bool wait = l == 0 || sl == kSlices - 1;
            if (tid == 0) {
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                if (sl == 0 && l > 0) {
                    const int K = l == 3 ? kFOutPad : kFHid;
                    const uint32_t sbo = (uint32_t)(K >> 3) * 128u;
                    for (int t = 0; t < 2; t++)
                        mma_run(tmem + 256 + 128 * t, sbase + kBwOffZ + t * (128 * K * 2), sbo, sbase + kBwOffW, sbo, K / 16,
                                instr_desc_bf16(kFM, kFHid), false);
                }
                mma_run(tmem, sbase + kBwOffZt + sl * (kTcBK / 16) * 256, (kBwRows >> 3) * 128, sbase + bw_slice(l, sl),
                        (kTcBK >> 3) * 128, kTcBK / 16, instr_desc_bf16(kFM, n_in), sl > 0);
                if (wait) {
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar)
                                 : "memory");
                    uint32_t spins = 0;
                    while (!mbar_try_wait(bar, phase)) {
                        if (++spins > kTcSpinLimit) {
                            s_fail = __LINE__;
                            break;
                        }
                    }
                }
            }
            if (!wait) continue;
            phase ^= 1u;
            __syncthreads();
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            if (s_fail) break;
            if (maker && l == 0 && sl + 2 < kSlices) load_slice(0, sl + 2);
        }
        if (s_fail) {
            asm volatile("cp.async.wait_group 0;\n" ::: "memory");  // no copy may land after the exit
            break;
        }
        const int quarter = warp & 3;
        if (maker) {
            if (l > 1) load_w(l - 1);
            if (l > 0) load_slice(l - 1, 0);
            if (l > 1) load_slice(l - 1, 1);
            // this split's dW: output neuron = TMEM lane
            float* pw = part + (l == 0 ? kMlpPartW0 : l == 1 ? kMlpPartW1 : l == 2 ? kMlpPartW2 : kMlpPartW3);
            const int n = 32 * quarter + lane;
            if (l < 3 || quarter == 0) {
                const int n_out = l < 3 ? kFHid : kFOutPad;
                for (int c0 = 16 * (warp >> 2); c0 < n_in; c0 += 32) {
                    float v[16];
                    tmem_ld16(tmem + ((uint32_t)(32 * quarter) << 16) + (uint32_t)c0, v);
                    if (n < n_out) {
#pragma unroll
                        for (int j = 0; j < 16; j++) pw[(c0 + j) * n_out + n] = v[j];
                    }
                }
            }
        }
        if (l > 0) {
            // dZ of the layer below
            const float* Gl = l == 1 ? in.G[0] : l == 2 ? in.G[1] : in.G[2];
            float* pb = part + (l == 1 ? kMlpPartB0 : l == 2 ? kMlpPartB1 : kMlpPartB2);
            if (maker) {
                const int t = warp >> 2, rt = 32 * quarter + lane, r = 128 * t + rt;
                const int64_t m = k0 + r;
                const uint32_t trow = tmem + 256 + 128 * t + ((uint32_t)(32 * quarter) << 16);
                float gx[2][16];  // two chunks ahead
                auto load_g = [&](int c, float (&g)[16]) {
#pragma unroll
                    for (int j = 0; j < 16; j++) g[j] = m < in.Mp ? Gl[(int64_t)(16 * c + j) * in.Mp + m] : 0.f;
                };
                load_g(0, gx[0]);
                load_g(1, gx[1]);
#pragma unroll 2
                for (int c = 0; c < 8; c++) {
                    float d[16];
                    tmem_ld16(trow + 16 * c, d);
#pragma unroll
                    for (int j = 0; j < 16; j++) d[j] *= gx[c & 1][j];
                    if (c < 6) load_g(c + 2, gx[c & 1]);
                    const uint4 h0 = pack8_bf16(d), h1 = pack8_bf16(d + 8);
                    if (l > 1) {  // rows for the next dH
                        uint8_t* z = sm + kBwOffZ + t * (128 * kFHid * 2);
                        *reinterpret_cast<uint4*>(z + kmajor_off(rt, 16 * c, kFHid)) = h0;
                        *reinterpret_cast<uint4*>(z + kmajor_off(rt, 16 * c + 8, kFHid)) = h1;
                    }
#pragma unroll
                    for (int j = 0; j < 8; j++) {
                        *reinterpret_cast<__nv_bfloat16*>(sm + kBwOffZt + kmajor_off(16 * c + j, r, kBwRows)) = bf16_at(h0, j);
                        *reinterpret_cast<__nv_bfloat16*>(sm + kBwOffZt + kmajor_off(16 * c + 8 + j, r, kBwRows)) =
                            bf16_at(h1, j);
                    }
                    if (c >= 2) bar_sync(4 + (c & 1), 256 + 32);  // the buffer's columns have been added
                    float* col = reinterpret_cast<float*>(sm + kBwOffB + (c & 1) * kBwColBuf) + r * 17;
#pragma unroll
                    for (int j = 0; j < 16; j++) col[j] = d[j];
                    bar_arrive(2 + (c & 1), 256 + 32);
                }
                // the next layer's W^T, all but the newest one or two groups
                if (l > 1) asm volatile("cp.async.wait_group 2;\n" ::: "memory");
            } else {
                for (int c = warp & 1; c < 8; c += 2) {  // a buffer each
                    bar_sync(2 + (c & 1), 256 + 32);
                    if (lane < 16)
                        add_column(reinterpret_cast<const float*>(sm + kBwOffB + (c & 1) * kBwColBuf) + lane, pb + 16 * c + lane);
                    __syncwarp();
                    if (c < 6) bar_arrive(4 + (c & 1), 256 + 32);
                }
            }
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
            __syncthreads();
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        }
    }
    if (s_fail && tid == 0) atomicCAS(&g_tc_error, 0, s_fail);
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(512) : "memory");
    }
}

static int fused_sms() {
    static int n_sm = 0;
    if (n_sm == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
        cudaFuncSetAttribute(k_mlp_forward_tc<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFSmem);
        cudaFuncSetAttribute(k_mlp_forward_tc<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFSmem);
        cudaFuncSetAttribute(k_mlp_backward_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBwSmem);
    }
    return n_sm > 0 ? n_sm : 1;
}

int mlp_forward_fused(const float* const* w, const float* const* b, const float* image, int W, int H, float* out,
                      cudaStream_t s) {
    const int n_sm = fused_sms();
    const int64_t M = (int64_t)(W / 8) * (H / 8);
    const int64_t n_tiles = (M + kFM - 1) / kFM;
    if (n_tiles == 0) return GS_OK;
    const int grid = (int)(n_tiles < n_sm ? n_tiles : n_sm);
    TrainFwdOut none{};
    k_mlp_forward_tc<false><<<grid, kFThreads, kFSmem, s>>>(image, W, H, w[0], b[0], w[1], b[1], w[2], b[2], w[3],
                                                            b[3], out, none);
    count_launch();
    return GS_OK;
}

// The training step's forward and its loss and backward, a launch each: the split
// shares of the gradients in part ([ceil(Mp / 256)][kMlpPart]) and of the loss in
// loss_part. Mp = patches rounded up to a multiple of 128; image 16-byte aligned.
int mlp_train_fused(const float* const* w, const float* const* b, const float* image, int W, int H,
                    const MlpTrainBufs& t, int64_t M, int64_t Mp, const float* targets, float w_depth, float w_scale,
                    float* out, cudaStream_t s) {
    const int n_sm = fused_sms();
    const int64_t n_tiles = Mp / kFM;
    const int grid = (int)(n_tiles < n_sm ? n_tiles : n_sm);
    const TrainFwdOut to{t.Xt, {t.G[0], t.G[1], t.G[2]}, {t.Ht[0], t.Ht[1], t.Ht[2]}, t.Z3,
                         {t.Wt[0], t.Wt[1], t.Wt[2]}, Mp};
    k_mlp_forward_tc<true><<<grid, kFThreads, kFSmem, s>>>(image, W, H, w[0], b[0], w[1], b[1], w[2], b[2], w[3],
                                                           b[3], nullptr, to);
    count_launch();
    const BwdIn bi{t.Z3, b[3], targets, {t.G[0], t.G[1], t.G[2]}, {t.Xt, t.Ht[0], t.Ht[1], t.Ht[2]},
                   {t.Wt[0], t.Wt[1], t.Wt[2]}, M, Mp, w_depth, w_scale, out, t.part, t.loss_part};
    k_mlp_backward_tc<<<(unsigned)ceil_div(Mp, kBwRows), kBwThreads, kBwSmem, s>>>(bi);
    count_launch();
    return GS_OK;
}

}  // namespace gs
