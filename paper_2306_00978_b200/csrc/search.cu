// Scale search of the method (Sec. 3.2): for each alpha of a caller-given list, s = s_X^alpha
// (Eq. 5), quantize W diag(s) with the library's own quantizer, run the library's own layer on
// diag(s)^-1 X, and measure the output error against the fp16 layer W X (Eq. 4).  Everything
// that the search evaluates is therefore exactly what deployment will run.  The reference product
// W X is a plain dense fp16 GEMM with fp32 accumulation and output; it runs once per search, on
// a tcgen05 kernel of this file (no library call, no allocation).
#include "tcgen05.cuh"

namespace awq {

namespace {

constexpr int kLossBlocks = 296;

// xs[b][m][k] = fp16_rne(fp32(X[m][k]) / s[b][k]): the caller's side of Eq. 4, one IEEE division and
// one rounding per element; eight elements per thread (K is a multiple of 128), which divides them by every gridDim.y-th of the
// scale arrays.
__global__ void divide_by_scale_kernel(const __half* __restrict__ X, const float* __restrict__ s, int count,
                                       __half* __restrict__ xs, size_t chunks, size_t block_chunks, int K) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= chunks) return;
    const int k0 = (int)((i * 8) % (size_t)K);
    const uint4 h = reinterpret_cast<const uint4*>(X)[i];
    const uint32_t w[4] = {h.x, h.y, h.z, h.w};
    float x[8];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[e]));
        x[2 * e] = f.x; x[2 * e + 1] = f.y;
    }
    for (int b = blockIdx.y; b < count; b += gridDim.y) {
        const float4 s0 = *reinterpret_cast<const float4*>(s + (size_t)b * K + k0), s1 = *reinterpret_cast<const float4*>(s + (size_t)b * K + k0 + 4);
        const float sk[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
        uint32_t o[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const __half2 r = __floats2half2_rn(__fdiv_rn(x[2 * e], sk[2 * e]), __fdiv_rn(x[2 * e + 1], sk[2 * e + 1]));
            o[e] = *reinterpret_cast<const uint32_t*>(&r);
        }
        reinterpret_cast<uint4*>(xs)[b * block_chunks + i] = make_uint4(o[0], o[1], o[2], o[3]);
    }
}

// xs[m][k] = fp16_rne(fp32(X[m][k]) * inv_s[k]): what awq_linear_scaled computes inside the layer,
// as a kernel of its own for the shapes whose kernel cannot fold it.
__global__ void multiply_by_inverse_kernel(const __half* __restrict__ X, const float* __restrict__ inv_s,
                                           __half* __restrict__ xs, size_t chunks, int K) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= chunks) return;
    const int k0 = (int)((i * 8) % (size_t)K);
    const uint4 h = reinterpret_cast<const uint4*>(X)[i];
    const uint32_t w[4] = {h.x, h.y, h.z, h.w};
    uint32_t o[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[e]));
        const __half2 r = __floats2half2_rn(__fmul_rn(f.x, inv_s[k0 + 2 * e]), __fmul_rn(f.y, inv_s[k0 + 2 * e + 1]));
        o[e] = *reinterpret_cast<const uint32_t*>(&r);
    }
    reinterpret_cast<uint4*>(xs)[i] = make_uint4(o[0], o[1], o[2], o[3]);
}
__global__ void inverse_scale_kernel(const float* __restrict__ s, float* __restrict__ inv_s, int K) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < K) inv_s[k] = __frcp_rn(s[k]);
}

// Sums of (y_q - y_ref)^2, one y_q per blockIdx.y: every block adds a fixed, interleaved share of the elements in fp64
// (eight at a time: N is a multiple of 128) and the last kernel adds the blocks' sums in a fixed tree, so the loss is
// reproducible.  (One element at a time and one thread for the last step: 30 us of a grid point's 85.)
__device__ __forceinline__ double block_sum(double acc) {
    __shared__ double s_sum[256];
    s_sum[threadIdx.x] = acc;
    __syncthreads();
    for (int off = 128; off >= 1; off >>= 1) {
        if ((int)threadIdx.x < off) s_sum[threadIdx.x] += s_sum[threadIdx.x + off];
        __syncthreads();
    }
    return s_sum[0];
}
__global__ void __launch_bounds__(256)
sqdiff_partial_kernel(const __half* __restrict__ yq, const float* __restrict__ yref, size_t chunks, size_t block_chunks,
                      double* __restrict__ partials) {
    const uint4* y = reinterpret_cast<const uint4*>(yq) + blockIdx.y * block_chunks;
    double acc = 0.0;
    for (size_t i = (size_t)blockIdx.x * 256 + threadIdx.x; i < chunks; i += (size_t)gridDim.x * 256) {
        const uint4 h = y[i];
        const float4 r0 = reinterpret_cast<const float4*>(yref)[2 * i], r1 = reinterpret_cast<const float4*>(yref)[2 * i + 1];
        const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&h.x)), b = __half22float2(*reinterpret_cast<const __half2*>(&h.y));
        const float2 c = __half22float2(*reinterpret_cast<const __half2*>(&h.z)), d = __half22float2(*reinterpret_cast<const __half2*>(&h.w));
        const float e[8] = {a.x - r0.x, a.y - r0.y, b.x - r0.z, b.y - r0.w, c.x - r1.x, c.y - r1.y, d.x - r1.z, d.y - r1.w};
#pragma unroll
        for (int k = 0; k < 8; ++k) acc += (double)e[k] * (double)e[k];
    }
    const double sum = block_sum(acc);
    if (threadIdx.x == 0) partials[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = sum;
}
__global__ void __launch_bounds__(256)
sqdiff_final_kernel(const double* partials, int blocks, double inv_count, float* __restrict__ out) {
    start_behind_predecessor();
    double t = 0.0;
    for (int i = threadIdx.x; i < blocks; i += 256) t += __ldcg(partials + (size_t)blockIdx.x * blocks + i);
    const double sum = block_sum(t);
    if (threadIdx.x == 0) out[blockIdx.x] = (float)(sum * inv_count);
}

size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

// Scratch of `batch` grid points at a time.  One needs no more than its own arrays, in rows as they come; several are stacked, each
// product's rows padded to what one store of the SM-pair kernel covers.
SearchPlan carve(void* base, int M, int N, int K, int group, int batch) {
    SearchPlan r;
    size_t off = 0;
    auto take = [&](size_t bytes) { const size_t o = off; off += align256(bytes); return static_cast<unsigned char*>(base) + o; };
    r.batch = batch;
    r.rows = batch > 1 ? (M + 31) / 32 * 32 : M;
    const size_t b = (size_t)r.batch;
    r.s = reinterpret_cast<float*>(take(b * K * 4));
    r.xs = reinterpret_cast<__half*>(take(b * r.rows * K * 2));
    r.qweight = take(b * N * K / 2);
    r.scales = take(b * (K / group) * N * 2);
    r.zeros = take(b * (K / group) * N / 2);
    r.yq = reinterpret_cast<__half*>(take(b * r.rows * N * 2));
    r.yref = reinterpret_cast<float*>(take((size_t)M * N * 4));
    r.partials = reinterpret_cast<double*>(take(b * kLossBlocks * 8));
    r.losses = reinterpret_cast<float*>(take((size_t)kMaxSearchAlphas * 4));
    r.total = off;
    return r;
}

// ---------------------------------------------------------------- dense reference product
// C[m][n] = sum_k X[m][k] * W[n][k]: both operands have K contiguous.  A block takes 128 channels (A, the lanes of tensor
// memory) x 128 tokens: one warp copies 64 input channels of both per stage (128-byte swizzle), one issues the products, four
// store the accumulator, a lane a channel, so that a token's 32 channels are one 128-byte store.  Three stages, two blocks per
// SM: one block's start and stores run under the other's products.  4096 channels x 4096 x 512 tokens: 28.6 us; 94 us on warp-level
// m16n8k16 products of 128 x 128 x 32 tiles in two shared-memory buffers.
constexpr int kRefTile = 128, kRefStages = 3, kRefOperand = kRefTile * kBK * 2, kRefThreads = 192;
constexpr int kRefSmem = kRefStages * 2 * kRefOperand + 1024;

__device__ __forceinline__ void umma_f16_smem(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}

__global__ void __launch_bounds__(kRefThreads)
reference_product_kernel(const __grid_constant__ CUtensorMap w_map, const __grid_constant__ CUtensorMap x_map, float* __restrict__ C,
                         int M, int N, int K, unsigned int* status_word) {
    extern __shared__ unsigned char smem_dyn[];
    __shared__ __align__(8) unsigned long long s_bars[2 * kRefStages + 1];
    __shared__ unsigned int s_abort;
    __shared__ uint32_t s_tmem_base;
    const uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u, bars = smem_u32(s_bars);
    auto full = [&](uint32_t s) { return bars + 8u * s; };
    auto empty = [&](uint32_t s) { return bars + 8u * (uint32_t)(kRefStages + s); };
    const uint32_t acc_full = bars + 16u * (uint32_t)kRefStages;
    const int warp = __shfl_sync(0xFFFFFFFFu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int n0 = blockIdx.x * kRefTile, m0 = blockIdx.y * kRefTile, steps = K / kBK;
    if (threadIdx.x == 0) {
        s_abort = 0u;
        for (uint32_t s = 0; s < (uint32_t)kRefStages; ++s) { mbar_init(full(s), 1); mbar_init(empty(s), 1); }
        mbar_init(acc_full, 1);
        mbar_fence_init();
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem_base)), "r"(128u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = s_tmem_base;
    const WaitCtl ctl{status_word, &s_abort};
    if (warp == 0) {
        const bool lead = elect_one();
        uint32_t stage = 0, phase = 0;
        int i = 0;
        for (; i < steps; ++i) {
            if (!mbar_wait_warp(empty(stage), phase ^ 1u, ctl)) break;
            if (lead) {
                mbar_arrive_expect_tx(full(stage), 2 * kRefOperand);
                tma_load_2d(base + stage * (2 * kRefOperand), &w_map, i * kBK, n0, full(stage));
                tma_load_2d(base + stage * (2 * kRefOperand) + kRefOperand, &x_map, i * kBK, m0, full(stage));   // rows past M: zeros
            }
            __syncwarp();
            if (++stage == kRefStages) { stage = 0; phase ^= 1u; }
        }
        if (i < steps)                                               // giving up: the copies in flight land first
            for (int q = 0; q < kRefStages && q < i; ++q) {
                if (stage == 0) { stage = kRefStages - 1; phase ^= 1u; } else { --stage; }
                const unsigned long long t0 = global_ns();
                while (!mbar_try_wait(full(stage), phase) && global_ns() - t0 < drain_limit_ns(ctl)) {}
            }
    } else if (warp == 1) {
        const bool lead = elect_one();
        constexpr uint32_t idesc = instr_desc(kRefTile);
        uint32_t stage = 0, phase = 0;
        int i = 0;
        for (; i < steps; ++i) {
            if (!mbar_wait_warp(full(stage), phase, ctl)) break;
            tc_fence_after();
            const uint64_t a = smem_desc_sw128(base + stage * (2 * kRefOperand)), b = smem_desc_sw128(base + stage * (2 * kRefOperand) + kRefOperand);
            if (lead) {
#pragma unroll
                for (int k = 0; k < kBK / 16; ++k)
                    umma_f16_smem(tmem_base, a + (uint64_t)(2 * k), b + (uint64_t)(2 * k), idesc, (i > 0 || k > 0) ? 1u : 0u);
                umma_commit(empty(stage));
                if (i + 1 == steps) umma_commit(acc_full);
            }
            __syncwarp();
            if (++stage == kRefStages) { stage = 0; phase ^= 1u; }
        }
    } else if (mbar_wait_warp(acc_full, 0u, ctl)) {
        tc_fence_after();
        const int quad = warp & 3, n = n0 + quad * 32 + lane;
#pragma unroll 1
        for (int c = 0; c < kRefTile; c += 32) {
            uint32_t r[32];
            tmem_ld_32cols(tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)c, r);
            tmem_ld_wait(r);
#pragma unroll
            for (int i = 0; i < 32; ++i)
                if (m0 + c + i < M) C[(size_t)(m0 + c + i) * N + n] = __uint_as_float(r[i]);
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(128u) : "memory");
    }
}

}  // namespace

// Grid points evaluated together: those asked for, as many as 384 MB hold beside the reference product (twenty of 4096 -> 4096 with
// 512 tokens), and as many as the scratch at hand holds; at least one.
SearchPlan search_plan(void* scratch, size_t scratch_bytes, int M, int N, int K, int group, int points) {
    const size_t most = ((size_t)384 << 20) + (size_t)M * N * 4;
    int batch = 1;
    while (batch < points && carve(nullptr, M, N, K, group, batch + 1).total <= most) ++batch;
    while (batch > 1 && carve(nullptr, M, N, K, group, batch).total > scratch_bytes) --batch;
    return carve(scratch, M, N, K, group, batch);
}

// y_ref[m][n] = sum_k X[m][k] W[n][k], fp32 [M][N] row-major.
cudaError_t launch_reference_product(const void* W, const void* X, float* yref, int M, int N, int K, unsigned int* status_word,
                                     cudaStream_t st) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return cudaErrorNotSupported;
    CUtensorMap maps[2];
    for (int i = 0; i < 2; ++i) {
        const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)(i ? M : N)}, strides[1] = {(cuuint64_t)K * 2};
        const cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)kRefTile}, estr[2] = {1, 1};
        if (enc(&maps[i], CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void*>(i ? X : W), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    const cudaError_t e = cudaFuncSetAttribute(reference_product_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kRefSmem);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)(N / kRefTile), (unsigned)((M + kRefTile - 1) / kRefTile));
    reference_product_kernel<<<grid, kRefThreads, kRefSmem, st>>>(maps[0], maps[1], yref, M, N, K, status_word);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_divide_by_scale(const void* X, const float* s, int count, void* xs, int M, int rows, int K, cudaStream_t st) {
    const size_t chunks = (size_t)M * K / 8;
    const unsigned blocks = (unsigned)((chunks + 255) / 256);
    // X is loaded and widened once per thread where that leaves blocks enough
    const unsigned share = blocks >= 1024 ? 1u : blocks >= 256 ? 4u : 16u;
    divide_by_scale_kernel<<<dim3(blocks, share < (unsigned)count ? share : (unsigned)count), 256, 0, st>>>(
        reinterpret_cast<const __half*>(X), s, count, reinterpret_cast<__half*>(xs), chunks, (size_t)rows * K / 8, K);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_multiply_by_inverse(const void* X, const float* inv_s, void* xs, int M, int K, cudaStream_t st) {
    const size_t chunks = (size_t)M * K / 8;
    multiply_by_inverse_kernel<<<(unsigned)((chunks + 255) / 256), 256, 0, st>>>(
        reinterpret_cast<const __half*>(X), inv_s, reinterpret_cast<__half*>(xs), chunks, K);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_inverse_scale(const float* s, float* inv_s, int K, cudaStream_t st) {
    inverse_scale_kernel<<<(K + 255) / 256, 256, 0, st>>>(s, inv_s, K);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_squared_difference(const void* yq, const float* yref, int count, int M, int rows, int N, double* partials, cudaStream_t st) {
    sqdiff_partial_kernel<<<dim3(kLossBlocks, (unsigned)count), 256, 0, st>>>(reinterpret_cast<const __half*>(yq), yref, (size_t)M * N / 8,
                                                                             (size_t)rows * N / 8, partials);
    count_launch();
    return cudaGetLastError();
}
cudaError_t launch_losses(const double* partials, int count, size_t n, float* losses, cudaStream_t st) {
    const cudaError_t e = launch_behind(sqdiff_final_kernel, (unsigned)count, 256, 0, st, partials, kLossBlocks, 1.0 / (double)n, losses);
    if (e != cudaSuccess) return e;
    count_launch();
    return cudaGetLastError();
}
}  // namespace awq
