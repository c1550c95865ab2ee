// Offline step of the layer: channel scale (Eq. 5), fold into W (Eq. 3), group-wise
// asymmetric 4-bit round-to-nearest (Eq. 2) and the packed tile layout (Sec. 4.2).
//
// 2 bytes read and ~0.52 bytes written per weight; the issue of instructions sets the time.  One warp takes a band of 16
// rows x 128 columns; lane (g, t) holds rows g and g+8, columns 16j+4t..+3 (j = 0..3) of both 64-column
// blocks, which is exactly the data of the two 16-byte packed pieces it writes.  Every
// rounding point is an explicit IEEE operation (no contraction); the per-weight division is
// replaced by a multiplication only where that provably rounds to the same integer.
#include <algorithm>
#include <mutex>
#include <type_traits>

#include "common.cuh"

namespace awq {

__device__ __forceinline__ float channel_scale_one(float a, float alpha, int mode) {
    if (mode == kAlphaZero) return 1.0f;
    const bool ok = isfinite(a) && a > 0.0f;
    if (!ok) return 1.0f;
    if (mode == kAlphaOne) return a;
    if (mode == kAlphaHalf) return __fsqrt_rn(a);
    return (float)pow((double)a, (double)alpha);
}

__global__ void channel_scale_kernel(const float* __restrict__ a, float alpha, int mode,
                                     float* __restrict__ s, int K) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < K) s[k] = channel_scale_one(mode == kAlphaZero ? 1.0f : a[k], alpha, mode);
}

// s of several alphas: blockIdx.y counts them
struct Alphas {
    float v[kMaxSearchAlphas];
    int mode[kMaxSearchAlphas];
};
__global__ void channel_scales_kernel(const float* a, const __grid_constant__ Alphas alphas, float* __restrict__ s, int K) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x, i = blockIdx.y, mode = alphas.mode[i];
    start_behind_predecessor();
    if (k < K) s[(size_t)i * K + k] = channel_scale_one(mode == kAlphaZero ? 1.0f : __ldcg(a + k), alphas.v[i], mode);
}

// Delta (fp16) and zero point of a group from its min and max; `top` is the largest code
// (15 for 4-bit, 7 for 3-bit grids).
__device__ __forceinline__ void group_params(float mn, float mx, float top, __half& d16, float& d, float& z) {
    const float d32 = __fdiv_rn(__fsub_rn(mx, mn), top);
    d16 = __float2half_rn(d32);
    const unsigned short bits = __half_as_ushort(d16);
    if ((bits & 0x7FFFu) == 0u || (bits & 0x7C00u) == 0x7C00u) d16 = __ushort_as_half(0x3C00u);
    d = __half2float(d16);
    z = fminf(fmaxf(rintf(__fdiv_rn(-mn, d)), 0.0f), top);
}

// q = clamp(rne(w / d) + z, 0, 15) with w / d the IEEE-rounded fp32 quotient.  `rd` = 1 / d
// (rounded).  w * rd is within 2.5e-7 |w / d| of the quotient, so it rounds to the same integer
// unless it lies within 1e-3 of a half-integer (or is large): only then is the division done.
__device__ __forceinline__ uint32_t code_of(float w, float d, float rd, float z, float top) {
    const float t = __fmul_rn(w, rd);
    float r = rintf(t);
    if (!(fabsf(t - r) < 0.499f && fabsf(t) < 1024.0f)) r = rintf(__fdiv_rn(w, d));
    return (uint32_t)fminf(fmaxf(__fadd_rn(r, z), 0.0f), top);
}
__device__ __forceinline__ float min3(float a, float b, float c) {
    float d; asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c)); return d;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
    float d; asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c)); return d;
}
__device__ __forceinline__ float max3_nan(float a, float b, float c) {      // a NaN stays
    float d; asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c)); return d;
}

// Two floats in a register pair; fma, add and sub round each half as the scalar instructions do.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
    f32x2 d; asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi)); return d;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c)); return d;
}
// (nothing may be added to a packed product: about one such sum in 10^5 came out as if the two instructions were fused)
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 d; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b)); return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b)); return d;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
    f32x2 d; asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b)); return d;
}


// One warp per band (16 rows) and 128 columns.  A thread block covers a group's columns (two groups for G = 64); up to
// G = 128 its warps take bands of their own and never meet, above the warps of a band exchange their min / max through shared memory.
// Scales and zero points are stored per 128 columns for G > 128 (each group's entry G / 128 times), so that the
// layer kernels need no variant for them.
template <int G> struct QCfg {
    static constexpr int kCols = G < 128 ? 128 : G;                 // columns per thread block
    static constexpr int kColWarps = kCols / 128;
    static constexpr int kBands = kColWarps <= 4 ? 4 / kColWarps : 1;
    static constexpr int kWarps = kColWarps * kBands, kThreads = kWarps * 32;
    static constexpr int kSets = G == 64 ? 4 : 2;                   // (row, group) pairs of a lane
    static constexpr int kStored = G < 128 ? G : 128;               // columns per stored scale / zero point
    static constexpr int kBlocks = 16 / kWarps;                     // thread blocks per SM: 128 registers per thread
};
// A warp's tile of W in shared memory: 16 rows of 256 bytes, 32 bytes apart so that the eight-byte loads of four rows meet all banks.
constexpr int kQRowBytes = 256 + 32, kQTileBytes = 16 * kQRowBytes, kQStages = 2;

// What a launch covers: items of (array part, column block, band step) in that order; blocks take equal contiguous ranges.
struct QuantizeCut {
    int N, K;
    int col_blocks, band_steps;              // column blocks of kCols, steps of kBands bands
    int items, share, longer;                // all items; items / blocks, items % blocks
    int arrays, per_part;                    // scale arrays (1 unless the scale search), arrays per part
};

// Group-wise round-to-nearest and the packed layout.  Lane (g, t) of a warp holds rows g and g + 8, columns 16j + 4t .. +3 of both
// 64-column blocks, which is the data of the two packed pieces that it writes; the products w' = w * s stay in registers (64),
// formed once.  The division w' / Delta is done only where it can matter: w' * (1 / Delta) rounds to the same integer unless it
// lies within the group's own error bound of a half-integer; the largest such distance of a packed word decides, and a
// word that fails is redone element by element with the division (code_of).  Rounding is by adding 1.5 * 2^23;
// clamping to [0, top] is compiled in only for the warps one of whose groups can leave the range.
// What bounds it is issue: per scheduler and cycle count, a packed multiply-add takes 2 cycles for two weights, a three-input
// min / max and a conversion fp16 -> fp32 2, a conversion to an integer 8.  So the four nibbles' sum ends in 2^23 + the
// nibbles, which is read as bits (no conversion), all fp32 steps are packed in pairs of columns, and a lane has 64 weights, so that the
// three IEEE divisions of a group's parameters, formed once per row by different lanes of the four that share it, weigh little.
// W comes through shared memory, each warp's next tiles by asynchronous copies while it works on the one before.
// 4096 -> 11008 (113.6 MB), calls among others: 31.3 us with 32 weights per lane, scalar steps and four conversions per packed word pair,
// 29.2 us so, 27.3 with the launch set up behind the call in front (a single launch 32.2); 20 arrays on 4096 x 4096 157 -> 133 us.  16 warps per SM issue in 60 % of the cycles (fma pipe 47 %, alu 43 %): the
// warps' own dependencies are what is left.  Blocks per SM 3 / 4 / 5: 150 / 137 / 146 us (five spill); W widened once per item in
// shared memory: 144 us (spills); a third tile in flight: 12 % slower; columns before bands in the order of items: 5 % slower.
// MANY (the scale search): `a` is `arrays` arrays of K scales; W is quantized with each and the packed arrays follow one another.
template <int G, int BITS, bool CLIP, bool SYM, bool MANY = false>
__global__ void __launch_bounds__(QCfg<G>::kThreads, QCfg<G>::kBlocks)
quantize_pack_tile_kernel(const __half* W, const float* a, float alpha,
                          int mode, const float* clip,
                          uint32_t* __restrict__ qweight, __half* __restrict__ scales,
                          uint8_t* __restrict__ zeros, const __grid_constant__ QuantizeCut cut) {
    using Cfg = QCfg<G>;
    constexpr float top = (float)((1 << BITS) - 1);       // largest code
    constexpr int kSets = Cfg::kSets, kColWarps = Cfg::kColWarps;
    extern __shared__ __align__(16) unsigned char q_smem[];
    __shared__ float2 s_mm[kColWarps > 1 ? 2 : 1][kColWarps][Cfg::kBands * 16];   // G > 128: [step parity][column warp][row] (min, max)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int bw = warp % Cfg::kBands, cw = warp / Cfg::kBands;
    const int g = lane >> 2, t = lane & 3;
    const int K = cut.K, bands = cut.N / 16;
    unsigned char* tiles = q_smem + warp * (kQStages * kQTileBytes);
    float* s_sm = reinterpret_cast<float*>(q_smem + Cfg::kWarps * (kQStages * kQTileBytes));   // [arrays of the part][kCols]

    start_behind_predecessor();
    const int block = (int)blockIdx.x;
    const int first = block * cut.share + min(block, cut.longer), last = first + cut.share + (block < cut.longer ? 1 : 0);
    const int per_part_items = cut.col_blocks * cut.band_steps;

    // this warp's tile of an item, eight 16-byte pieces per lane
    auto fetch = [&](int item) {
        if (item < last) {
            const int in_part = item % per_part_items, cb = in_part / cut.band_steps, band = (in_part - cb * cut.band_steps) * Cfg::kBands + bw;
            const __half* src = W + (size_t)(band * 16 + (lane >> 4)) * K + cb * Cfg::kCols + cw * 128 + (lane & 15) * 8;
            const uint32_t dst = (uint32_t)__cvta_generic_to_shared(tiles + (item % kQStages) * kQTileBytes + (lane >> 4) * kQRowBytes + (lane & 15) * 16);
#pragma unroll
            for (int i = 0; i < 8; ++i)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + i * 2 * kQRowBytes), "l"(src + (size_t)(2 * i) * K) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    fetch(first);
    fetch(first + 1);

    const f32x2 big2 = pack2(12582912.0f, 12582912.0f), c16 = pack2(16.0f, 16.0f);
    int columns = -1;                                      // (part, column block) whose scales are in shared memory
    for (int item = first; item < last; ++item) {
        const int part = MANY ? item / per_part_items : 0, in_part = item - part * per_part_items;
        const int cb = in_part / cut.band_steps, band = (in_part - cb * cut.band_steps) * Cfg::kBands + bw;
        const int kbase = cb * Cfg::kCols, array0 = part * cut.per_part, arrays = MANY ? min(cut.per_part, cut.arrays - array0) : 1;
        if (part * cut.col_blocks + cb != columns) {
            columns = part * cut.col_blocks + cb;
            __syncthreads();                               // the scales before have been read
            if (MANY) {
                for (int i = threadIdx.x; i < arrays * Cfg::kCols; i += Cfg::kThreads)
                    s_sm[i] = __ldcg(a + (size_t)(array0 + i / Cfg::kCols) * K + kbase + i % Cfg::kCols);
            } else {
                for (int i = threadIdx.x; i < Cfg::kCols; i += Cfg::kThreads)
                    s_sm[i] = channel_scale_one(mode == kAlphaZero ? 1.0f : __ldcg(a + kbase + i), alpha, mode);
            }
            __syncthreads();
        }
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncwarp();
        const unsigned char* tile = tiles + (item % kQStages) * kQTileBytes + g * kQRowBytes + t * 8;
        // Where this lane's outputs go: packed blocks [band][k-tile][512 bytes], scales [band][stored group][16], zero bytes
        // [band pair][stored group][16], 8 per band; a stored group is the group itself up to 128 columns, else each of its runs of 128.
        const size_t nsg = (size_t)(K / Cfg::kStored), q_step = (size_t)bands * K * 2, d_step = (size_t)bands * nsg * 16;
        const int sg0 = G == 64 ? cb * 2 : cb * kColWarps + cw;
        const int own = t % kSets, own_row = own & 1, own_ti = own >> 1;       // the (row, group) whose parameters this lane forms
        uint32_t* q_out = qweight + (MANY ? array0 * q_step : 0) + ((size_t)band * (K / 64) + (size_t)(kbase / 64 + cw * 2)) * 128 + lane * 4;
        __half* d_out = scales + (MANY ? array0 * d_step : 0) + ((size_t)band * nsg + sg0 + own_ti) * 16 + g + 8 * own_row;
        uint8_t* z_out = zeros + (MANY ? array0 * (d_step / 2) : 0) + ((size_t)(band >> 1) * nsg + sg0) * 16 + (band & 1) * 8 + g;
        for (int ai = 0; ai < arrays; ++ai) {
            // w' = fp32(w) * s  (Eq. 3), once, and the min / max of this lane's columns of each (row, group)
            f32x2 wp[2][2][4][2];                          // [row h][64-column block][word j][columns 4t, 4t+1 | 4t+2, 4t+3]
            float mn[kSets], mx[kSets];
#pragma unroll
            for (int q = 0; q < kSets; ++q) { mn[q] = INFINITY; mx[q] = -INFINITY; }
            const float* sc = s_sm + ai * Cfg::kCols + cw * 128 + 4 * t;
#pragma unroll
            for (int ti = 0; ti < 2; ++ti)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float4 s4 = *reinterpret_cast<const float4*>(sc + ti * 64 + 16 * j);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const uint2 raw = *reinterpret_cast<const uint2*>(tile + h * 8 * kQRowBytes + ti * 128 + j * 32);
                        const float2 f01 = __half22float2(*reinterpret_cast<const __half2*>(&raw.x));
                        const float2 f23 = __half22float2(*reinterpret_cast<const __half2*>(&raw.y));
                        const f32x2 w01 = mul2(pack2(f01.x, f01.y), pack2(s4.x, s4.y)), w23 = mul2(pack2(f23.x, f23.y), pack2(s4.z, s4.w));
                        wp[h][ti][j][0] = w01;
                        wp[h][ti][j][1] = w23;
                        float w0, w1, w2, w3;
                        unpack2(w01, w0, w1);
                        unpack2(w23, w2, w3);
                        const int q = G == 64 ? 2 * ti + h : h;
                        mn[q] = min3(mn[q], w0, w1);
                        mn[q] = min3(mn[q], w2, w3);
                        mx[q] = max3(mx[q], w0, w1);
                        mx[q] = max3(mx[q], w2, w3);
                    }
                }
            if (ai + 1 == arrays) {                        // the tile is in registers: its place takes the one after the next
                __syncwarp();
                fetch(item + 2);
            }
// a row's four lanes meet; lane t ends with set t % kSets: of two (sets of) sets it hands on the one that it does not keep
            auto halve = [&](float keep, float give, int off, bool least) {
                const float v = __shfl_xor_sync(0xFFFFFFFFu, give, off);
                return least ? fminf(keep, v) : fmaxf(keep, v);
            };
            const bool odd = (t & 1) != 0, high = (t & 2) != 0;
            float mn1 = halve(odd ? mn[1] : mn[0], odd ? mn[0] : mn[1], 1, true), mx1 = halve(odd ? mx[1] : mx[0], odd ? mx[0] : mx[1], 1, false);
            if constexpr (kSets == 4) {
                const float mn2 = halve(odd ? mn[3] : mn[2], odd ? mn[2] : mn[3], 1, true), mx2 = halve(odd ? mx[3] : mx[2], odd ? mx[2] : mx[3], 1, false);
                mn1 = halve(high ? mn2 : mn1, high ? mn1 : mn2, 2, true);
                mx1 = halve(high ? mx2 : mx1, high ? mx1 : mx2, 2, false);
            } else {
                mn1 = halve(mn1, mn1, 2, true);
                mx1 = halve(mx1, mx1, 2, false);
            }
            if (kColWarps > 1) {
                // the group spans the block's column warps: the others' min / max through shared memory
                float2(*mm)[Cfg::kBands * 16] = s_mm[kColWarps > 1 ? item & 1 : 0];
                if (t < 2) mm[cw][bw * 16 + g + 8 * t] = make_float2(mn1, mx1);
                __syncthreads();
#pragma unroll
                for (int o = 0; o < kColWarps; ++o) {
                    const float2 v = mm[o][bw * 16 + g + 8 * own_row];
                    mn1 = fminf(mn1, v.x);
                    mx1 = fmaxf(mx1, v.y);
                }
            }
            // Delta, the zero point and 1 / Delta cost three IEEE divisions: once per row and group, then handed on
            const float wabs = fmaxf(fabsf(mn1), fabsf(mx1));      // largest |w'| of the group (before clipping)
            if (CLIP) {
                const int gi = G == 64 ? cb * 2 + own_ti : cb;
                const float r = __ldcg(clip + (size_t)(band * 16 + g + 8 * own_row) * (K / G) + gi);
                mn1 = __fmul_rn(mn1, r);
                mx1 = __fmul_rn(mx1, r);
            }
            __half h16;
            float d1, z1;
            if (SYM) {
                constexpr float half_levels = (float)(1 << (BITS - 1));
                const float d32 = __fdiv_rn(fmaxf(fabsf(mn1), fabsf(mx1)), half_levels);
                h16 = __float2half_rn(d32);
                const unsigned short bits = __half_as_ushort(h16);
                if ((bits & 0x7FFFu) == 0u || (bits & 0x7C00u) == 0x7C00u) h16 = __ushort_as_half(0x3C00u);
                d1 = __half2float(h16);
                z1 = half_levels;
            } else {
                group_params(mn1, mx1, top, h16, d1, z1);
            }
            const float rd1 = __frcp_rn(d1);
            // |w * rd - w / d| <= 1.8e-7 |w / d| (three roundings); the group's largest |w / d|
            // bounds it for every element; quotients beyond 1024 always take the division
            const float tmax = __fmul_rn(wabs, rd1);
            const float thr1 = tmax < 1024.0f ? 0.5f - fmaf(tmax, 4e-7f, 1e-6f) : -1.0f;
            // Clamping to [0, top] can only matter where the group's smallest or largest element leaves the
            // range (the level is monotone in w'): rare without clipping - rne(max / Delta) + rne(-min / Delta)
            // exceeds top only when both quotients sit on a tie - so the warp takes the clamped code only if one
            // of its lanes needs it.
            bool need_clamp = CLIP || SYM;
            if (!need_clamp) {
                const float zc = 12582912.0f - z1;               // exact: z is a small integer
                const float qlo = __fsub_rn(__fmaf_rn(mn1, rd1, 12582912.0f), zc), qhi = __fsub_rn(__fmaf_rn(mx1, rd1, 12582912.0f), zc);
                need_clamp = __any_sync(0xFFFFFFFFu, !(qlo >= 0.0f && qhi <= top));
            }
            if (t < kSets) *d_out = h16;
            float z[2], d[2], rd[2], thr = 0.0f;
#pragma unroll
            for (int ti = 0; ti < 2; ++ti) {
                if (ti == 0 || G == 64) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int from = (lane & ~3) + (G == 64 ? 2 * ti + h : h);
                        d[h] = __shfl_sync(0xFFFFFFFFu, d1, from);
                        z[h] = __shfl_sync(0xFFFFFFFFu, z1, from);
                        rd[h] = __shfl_sync(0xFFFFFFFFu, rd1, from);
                        const float th = __shfl_sync(0xFFFFFFFFu, thr1, from);
                        thr = h == 0 ? th : fminf(thr, th);
                    }
                    if (t == 0)                                  // z + 2^23: z in the low bits
                        z_out[ti * 16] = (uint8_t)((__float_as_uint(z[0] + 8388608.0f) & 15u) | ((__float_as_uint(z[1] + 8388608.0f) & 15u) << 4));
                }
                const f32x2 rdu = pack2(rd[0], rd[0]), rdl = pack2(rd[1], rd[1]);
                uint32_t words[4];
                float dev[4];
                auto quantize_words = [&](auto clamp_tag) {
                    constexpr bool CL = decltype(clamp_tag)::value;
                    // 2^23 + the zero points' own word: the codes are integer + zero point, nibbles (row g, g + 8, g, g + 8)
                    const float zz = fmaf(z[1], 4112.0f, fmaf(z[0], 257.0f, 8388608.0f));
                    const f32x2 zz2 = pack2(zz, zz);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        // minus the integer nearest to the product w' / Delta (ties to even), and the product's distance from it
                        f32x2 nu[2], nl[2], du[2], dl[2];
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            nu[e] = sub2(big2, fma2(wp[0][ti][j][e], rdu, big2));
                            nl[e] = sub2(big2, fma2(wp[1][ti][j][e], rdl, big2));
                            du[e] = fma2(wp[0][ti][j][e], rdu, nu[e]);
                            dl[e] = fma2(wp[1][ti][j][e], rdl, nl[e]);
                        }
                        float x[8];
                        unpack2(du[0], x[0], x[1]);
                        unpack2(du[1], x[2], x[3]);
                        unpack2(dl[0], x[4], x[5]);
                        unpack2(dl[1], x[6], x[7]);
                        dev[j] = max3_nan(max3_nan(max3_nan(fabsf(x[0]), fabsf(x[1]), fabsf(x[2])), fabsf(x[3]), fabsf(x[4])),
                                          max3_nan(fabsf(x[5]), fabsf(x[6]), fabsf(x[7])), 0.0f);
                        // nibbles 0 .. 3 = (g,c) (g+8,c) (g,c+2) (g+8,c+2), nibbles 4 .. 7 the same for c+1, c+3: each half's sum
                        // stays within 2^23 .. 2^23 + 65535, exactly, and is read as bits
                        f32x2 sum;
                        if (CL) {
                            auto clamp2 = [&](f32x2 n, float zp) {
                                float q0, q1;
                                unpack2(sub2(pack2(zp, zp), n), q0, q1);
                                return pack2(fminf(fmaxf(q0, 0.0f), top), fminf(fmaxf(q1, 0.0f), top));
                            };
                            sum = fma2(fma2(clamp2(nl[1], z[1]), c16, clamp2(nu[1], z[0])), c16, clamp2(nl[0], z[1]));
                            sum = add2(fma2(sum, c16, clamp2(nu[0], z[0])), pack2(8388608.0f, 8388608.0f));
                        } else {
                            sum = sub2(zz2, fma2(fma2(fma2(nl[1], c16, nu[1]), c16, nl[0]), c16, nu[0]));
                        }
                        float lo, hi;
                        unpack2(sum, lo, hi);
                        words[j] = __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x5410);
                    }
                };
                if (need_clamp) quantize_words(std::true_type{}); else quantize_words(std::false_type{});
                if (!(max3_nan(dev[0], dev[1], max3_nan(dev[2], dev[3], 0.0f)) < thr)) {       // rare: a word again, element by element
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        if (dev[j] < thr) continue;
                        uint32_t word = 0;
#pragma unroll
                        for (int h = 0; h < 2; ++h)
#pragma unroll
                            for (int e = 0; e < 2; ++e) {
                                float w0, w1;
                                unpack2(wp[h][ti][j][e], w0, w1);
                                word |= (code_of(w0, d[h], rd[h], z[h], top) | (code_of(w1, d[h], rd[h], z[h], top) << 16)) << (4 * h + 8 * e);
                            }
                        words[j] = word;
                    }
                }
                // band-major: block (band, k-tile) is 512 bytes, a band's blocks are contiguous along K
                *reinterpret_cast<uint4*>(q_out + ti * 128) = make_uint4(words[0], words[1], words[2], words[3]);
            }
            if (MANY) { q_out += q_step; d_out += d_step; z_out += d_step / 2; }
        }
    }
}

// Weight clipping (Sec. 3.2).  For every group of w' = w * s and every ratio r of the list, the
// group is quantized on [r * min, r * max] and its squared error summed; the first ratio of least
// error is written to clip[n][group].  The choice decides integer codes downstream, so the error
// is defined operation by operation: dequant = (q - z) * Delta (one fp32 multiply), e = dequant -
// w', err += e * e in fp32 over ascending k (no contraction), a NaN error counts as +inf.
// grid = (K / G, N / 64), block = 256 or 128: one group of columns of 64 rows, its w' in shared memory; a thread takes one (row, J
// ratios) item at a time.
// First an estimate of every (row, ratio)'s error, in steps of Delta and in no particular order: t = w' / Delta by
// w' * (1 / Delta), its nearest integer, clamped, f = t - that, S = sum of f * f, two elements per packed fp32 instruction
// (4 of these, 4 min / max per pair of elements).  The estimate's root is within
//     margin = 1e-5 sqrt(S) Delta + 6e-6 (T + 2) Delta,    T = max|w'| / Delta,
// of the root of the error as it is defined: 1 / Delta is rounded once, f once, and where the product's nearest integer is not the
// quotient's both lie half a step away, so |f| is off by less than 2^-21.6 (T + 1); the defined dequant and difference are each
// rounded once, 2^-22.4 (T + 2) of a step; over 128 elements the norms differ by sqrt(128) times the sum of both, < 5.5e-6 (T + 2); the
// two sums' own roundings are 130 and 70 times 2^-24 of the errors, half of that of the roots.  A ratio whose
// estimate less its margin is above another's plus its margin is not the best.  Where more than one ratio is left (1 % of the rows),
// those are evaluated as defined, in order, the quotient's integer by w' * (1 / Delta) where the largest distance of a product from
// its integer shows that this is safe and by division elsewhere.  Not-a-number and overflow leave a ratio to be evaluated.
// A packed fp32 instruction takes two issue slots, so a pair of elements and a ratio take 12 (12.3 measured on registers alone);
// here they take 15.  4096 -> 4096 with 20 ratios: 94 us, of which 18 are loads, parameters and the choice (every ratio
// evaluated as defined, 9 packed or min / max instructions per pair: 125 us).  128, 192, 320 threads: 103, 101, 96 us; one ratio at a
// time 95, four 99; clamping by the saturation of a scalar multiply-add 91 to 99, at a wider margin.
constexpr int kClipRows = 64;
struct ClipGrid {
    float r[kMaxClipRatios];
    int n;
};

// the error of one (row, ratio) as it is defined; wg = its w'
template <int G>
__device__ __noinline__ float clip_error_by_division(const float* wg, float d, float z, float top) {
    float err = 0.0f;
    for (int k = 0; k < G; ++k) {
        const float w = wg[k];
        const float q = fminf(fmaxf(__fadd_rn(rintf(__fdiv_rn(w, d)), z), 0.0f), top);
        const float e = __fsub_rn(__fmul_rn(__fsub_rn(q, z), d), w);
        err = __fadd_rn(err, __fmul_rn(e, e));
    }
    return err;
}
// the same without a division per element, where that gives the same integers
template <int G>
__device__ __noinline__ float clip_error(const float* wg, float tmax, float d, float rd, float z, float top) {
    // |w rd - fl(w / d)| <= 2^-23 |w / d| (1 / d and the quotient are rounded once each); the distance
    // itself is off by at most 2^-26, the threshold by 2^-25
    const float thr = tmax < 1024.0f ? 0.5f - fmaf(tmax, 1.25e-7f, 6e-8f) : -1.0f;
    float err = 0.0f, dev = 0.0f;
#pragma unroll 8
    for (int k = 0; k < G; ++k) {
        const float w = wg[k];
        const float n = __fsub_rn(12582912.0f, __fmaf_rn(w, rd, 12582912.0f));     // minus the product's integer
        dev = max3_nan(dev, fabsf(__fmaf_rn(w, rd, n)), 0.0f);
        const float e = __fadd_rn(__fmul_rn(fminf(fmaxf(n, z - top), z), d), w);    // minus the difference: its square is the same
        err = __fadd_rn(err, __fmul_rn(e, e));
    }
    return dev < thr ? err : clip_error_by_division<G>(wg, d, z, top);
}

template <int G>
struct ClipSmem {
    static constexpr int kRowFloats = G + 4;                // 16 bytes more, so that rows start on different banks
    float w[kClipRows * kRowFloats];
    float err[kClipRows * (kMaxClipRatios + 1)];
    float2 mm[kClipRows];
    int least[kClipRows];                                   // least estimate plus margin (a float that is not negative)
    int left[kClipRows];                                    // ratios that may be the best
    float s[G];
};

// THREADS per block, items of J ratios of a row
template <int G, int J, int THREADS>
__global__ void __launch_bounds__(THREADS)
clip_search_kernel(const __half* W, const float* a, float alpha, int mode,
                   const __grid_constant__ ClipGrid ratios, float top, float* __restrict__ clip, int N, int K,
                   bool aligned) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ClipSmem<G>& sm = *reinterpret_cast<ClipSmem<G>*>(smem_raw);
    constexpr int kPieces = G / 8, kRowFloats = ClipSmem<G>::kRowFloats;
    const int n0 = blockIdx.y * kClipRows, k0 = blockIdx.x * G;
    const int tid = threadIdx.x;
    start_behind_predecessor();

    for (int i = tid; i < G; i += THREADS) sm.s[i] = channel_scale_one(mode == kAlphaZero ? 1.0f : __ldcg(a + k0 + i), alpha, mode);
    __syncthreads();
    // w' = w * s (Eq. 3), eight columns of a row per thread; the row's min / max over its kPieces lanes
#pragma unroll 4
    for (int i = tid; i < kClipRows * kPieces; i += THREADS) {
        const int row = i / kPieces, p = i % kPieces;
        const __half* src = W + (size_t)(n0 + row) * K + k0 + p * 8;
        __half h[8];
        if (aligned) {
            *reinterpret_cast<uint4*>(h) = __ldcg(reinterpret_cast<const uint4*>(src));
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) h[e] = __ldcg(src + e);
        }
        float mn = INFINITY, mx = -INFINITY;
        float* dst = sm.w + row * kRowFloats + p * 8;
        float wv[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            wv[e] = __fmul_rn(__half2float(h[e]), sm.s[p * 8 + e]);
            mn = fminf(mn, wv[e]);
            mx = fmaxf(mx, wv[e]);
        }
        *reinterpret_cast<float4*>(dst) = make_float4(wv[0], wv[1], wv[2], wv[3]);
        *reinterpret_cast<float4*>(dst + 4) = make_float4(wv[4], wv[5], wv[6], wv[7]);
#pragma unroll
        for (int off = kPieces / 2; off >= 1; off >>= 1) {
            mn = fminf(mn, __shfl_xor_sync(0xFFFFFFFFu, mn, off));
            mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, off));
        }
        if (p == 0) { sm.mm[row] = make_float2(mn, mx); sm.least[row] = 0x7F800000; sm.left[row] = 0; }
    }
    __syncthreads();
    const int nr = ratios.n;
    // Delta, zero point, 1 / Delta and max|w'| / Delta of a (row, ratio)
    auto params = [&](const float2& mm, float r, float& d, float& z, float& rd, float& tmax) {
        __half d16;
        group_params(__fmul_rn(mm.x, r), __fmul_rn(mm.y, r), top, d16, d, z);
        rd = __frcp_rn(d);
        tmax = __fmul_rn(fmaxf(fabsf(mm.x), fabsf(mm.y)), rd);
    };
    const int np = (nr + J - 1) / J;
    for (int item = tid; item < kClipRows * np; item += THREADS) {
        const int row = item / np, i0 = J * (item - row * np);
        const f32x2 big = pack2(12582912.0f, 12582912.0f);
        float d[J], tmax[J], lo[J], hi[J];
        f32x2 rd2[J], sum[J];
#pragma unroll
        for (int j = 0; j < J; ++j) {
            float z, rd;
            params(sm.mm[row], ratios.r[min(i0 + j, nr - 1)], d[j], z, rd, tmax[j]);
            rd2[j] = pack2(rd, rd);
            sum[j] = pack2(0.0f, 0.0f);
            lo[j] = 12582912.0f - z;
            hi[j] = lo[j] + top;
        }
        const float* wg = sm.w + row * kRowFloats;
        constexpr int E = 4;                                     // pairs of elements at a time
#pragma unroll 2
        for (int k = 0; k < G; k += 2 * E) {
            f32x2 w[E], u[J][E];
#pragma unroll
            for (int e = 0; e < E; e += 2) {
                const float4 w4 = *reinterpret_cast<const float4*>(wg + k + 2 * e);
                w[e] = pack2(w4.x, w4.y);
                w[e + 1] = pack2(w4.z, w4.w);
            }
#pragma unroll
            for (int e = 0; e < E; ++e)
#pragma unroll
                for (int j = 0; j < J; ++j) u[j][e] = fma2(w[e], rd2[j], big);       // rounded to an integer in the sum
#pragma unroll
            for (int e = 0; e < E; ++e)
#pragma unroll
                for (int j = 0; j < J; ++j) {
                    float u0, u1;
                    unpack2(u[j][e], u0, u1);
                    u[j][e] = pack2(fminf(fmaxf(u0, lo[j]), hi[j]), fminf(fmaxf(u1, lo[j]), hi[j]));
                }
#pragma unroll
            for (int e = 0; e < E; ++e)
#pragma unroll
                for (int j = 0; j < J; ++j) u[j][e] = fma2(w[e], rd2[j], sub2(big, u[j][e]));
#pragma unroll
            for (int e = 0; e < E; ++e)
#pragma unroll
                for (int j = 0; j < J; ++j) sum[j] = fma2(u[j][e], u[j][e], sum[j]);
        }
#pragma unroll
        for (int j = 0; j < J; ++j) {
            if (i0 + j >= nr) break;
            float s0, s1;
            unpack2(sum[j], s0, s1);
            const float root = sqrtf(s0 + s1) * d[j], margin = fmaf(1e-5f, root, 6e-6f * (tmax[j] + 2.0f) * d[j]);
            const bool sure = tmax[j] < 1024.0f && root + margin < INFINITY;
            sm.err[row * (kMaxClipRatios + 1) + i0 + j] = sure ? root - margin : -INFINITY;
            if (sure) atomicMin(&sm.least[row], __float_as_int(root + margin));
        }
    }
    __syncthreads();
    for (int item = tid; item < kClipRows * nr; item += THREADS) {
        const int row = item / nr, i = item - row * nr;
        if (sm.err[row * (kMaxClipRatios + 1) + i] <= __int_as_float(sm.least[row])) atomicAdd(&sm.left[row], 1);
    }
    __syncthreads();
    for (int item = tid; item < kClipRows * nr; item += THREADS) {
        const int row = item / nr, i = item - row * nr;
        float* e = sm.err + row * (kMaxClipRatios + 1) + i;
        float err = INFINITY;
        if (*e <= __int_as_float(sm.least[row])) {
            err = 0.0f;                                     // the only one left
            if (sm.left[row] > 1) {
                float d, z, rd, tmax;
                params(sm.mm[row], ratios.r[i], d, z, rd, tmax);
                err = clip_error<G>(sm.w + row * kRowFloats, tmax, d, rd, z, top);
                if (err != err) err = INFINITY;
            }
        }
        *e = err;
    }
    __syncthreads();
    if (tid < kClipRows) {
        const float* e = sm.err + tid * (kMaxClipRatios + 1);
        int best = 0;
        for (int i = 1; i < nr; ++i)
            if (e[i] < e[best]) best = i;
        clip[(size_t)(n0 + tid) * (K / G) + blockIdx.x] = ratios.r[best];
    }
}

// One thread per (row, 8 columns): expands the packed arrays (test / debug path).
__global__ void unpack_kernel(const uint32_t* __restrict__ qweight, const __half* __restrict__ scales,
                              const uint8_t* __restrict__ zeros, int N, int K, int group,
                              uint8_t* __restrict__ codes, uint16_t* __restrict__ scales_nk,
                              uint8_t* __restrict__ zeros_nk) {
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t total = (size_t)N * K;
    if (idx >= total) return;
    const int n = (int)(idx / K), k = (int)(idx % K);
    const int band = n / 16, rr = n % 16, g = rr % 8, h = rr / 8;
    const size_t block = (size_t)band * (K / 64) + k / 64;
    const int c = k % 64;
    const int j = c / 16, t = (c % 16) / 4, i = c % 4;
    const uint32_t w = qweight[block * 128 + (g * 4 + t) * 4 + j];
    const int slot = (i / 2) * 4 + h * 2 + (i % 2);
    const int nib = (slot % 2) * 4 + slot / 2;
    codes[idx] = (uint8_t)((w >> (4 * nib)) & 0xFu);
    if (k % group == 0) {
        // the group's first stored entry (groups above 128 columns are stored once per 128 columns)
        const int gi = k / group, ng = K / group;
        const int stored = group < 128 ? group : 128;
        const size_t sgi = k / stored, nsg = K / stored;
        scales_nk[(size_t)n * ng + gi] = __half_as_ushort(scales[((size_t)band * nsg + sgi) * 16 + rr]);
        const uint8_t zb = zeros[((size_t)(band >> 1) * nsg + sgi) * 16 + (band & 1) * 8 + g];
        zeros_nk[(size_t)n * ng + gi] = (uint8_t)((zb >> (4 * h)) & 0xFu);
    }
}

cudaError_t launch_channel_scale(const float* a, float alpha, float* s, int K, cudaStream_t st) {
    channel_scale_kernel<<<(K + 255) / 256, 256, 0, st>>>(a, alpha, (int)alpha_mode(alpha), s, K);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_channel_scales(const float* a, const float* alphas, int n, float* s, int K, cudaStream_t st) {
    Alphas list = {};
    for (int i = 0; i < n; ++i) { list.v[i] = alphas[i]; list.mode[i] = (int)alpha_mode(alphas[i]); }
    const cudaError_t e = launch_behind(channel_scales_kernel, dim3((K + 255) / 256, n), 256, 0, st, a, list, s, K);
    if (e != cudaSuccess) return e;
    count_launch();
    return cudaGetLastError();
}

// Blocks take equal ranges of items.  The scale search's arrays are divided into parts where that evens out the ranges:
// (4096 x 4096: 2048 items of 20 arrays for 592 blocks would be 4 against 3.46 on average).
template <int G, int BITS, bool CLIP, bool SYM, bool MANY = false>
static cudaError_t launch_quantize(const __half* W, const float* a, float alpha, int mode, const float* clip, uint32_t* qweight,
                                   __half* scales, uint8_t* zeros, int N, int K, int arrays, int sms, cudaStream_t st) {
    using Cfg = QCfg<G>;
    static std::mutex mutex;
    static bool done[64] = {};
    auto* kernel = quantize_pack_tile_kernel<G, BITS, CLIP, SYM, MANY>;
    constexpr int tiles = Cfg::kWarps * kQStages * kQTileBytes, most = tiles + (MANY ? kMaxSearchAlphas : 1) * Cfg::kCols * 4;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    {
        std::lock_guard<std::mutex> lock(mutex);
        if (!done[dev & 63]) {
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
            if (e != cudaSuccess) return e;
            done[dev & 63] = true;
        }
    }
    QuantizeCut cut = {};
    cut.N = N;
    cut.K = K;
    cut.col_blocks = K / Cfg::kCols;
    cut.band_steps = N / 16 / Cfg::kBands;             // (N is a multiple of 128)
    cut.arrays = arrays;
    // blocks that can be resident with `per` arrays of scales in shared memory: of 228 KB per SM, a block keeps 1.5 KB beside its dynamic part
    auto resident_with = [&](int per) { return sms * std::min(Cfg::kBlocks, 228 * 1024 / (tiles + per * Cfg::kCols * 4 + 1536)); };
    const long long tiles_all = (long long)cut.col_blocks * cut.band_steps;
    int parts = 1;
    if (MANY) {
        double least = 0.0;
        for (int p = 1; p <= 4 && p <= arrays; ++p) {
            const int per = (arrays + p - 1) / p, real = (arrays + per - 1) / per;
            const int resident = resident_with(per);
            const double rounds = (double)((tiles_all * real + resident - 1) / resident) * (per + 0.5);    // (an item's own start: half an array)
            if (p == 1 || rounds < least) { least = rounds; parts = real; }
        }
    }
    cut.per_part = (arrays + parts - 1) / parts;
    const long long items = tiles_all * parts;
    if (items > 0x7FFFFFFFLL) return cudaErrorInvalidValue;
    cut.items = (int)items;
    const int resident = resident_with(cut.per_part), blocks = items < resident ? (int)items : resident;
    cut.share = cut.items / blocks;
    cut.longer = cut.items % blocks;
    e = launch_behind(kernel, blocks, Cfg::kThreads, (size_t)(tiles + cut.per_part * Cfg::kCols * 4), st, W, a, alpha, mode, clip, qweight, scales, zeros, cut);
    if (e != cudaSuccess) return e;
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_quantize_pack_many(const __half* W, const float* s, int count, int group, uint32_t* qweight, __half* scales,
                                      uint8_t* zeros, int N, int K, int sms, cudaStream_t st) {
    return group == 64 ? launch_quantize<64, 4, false, false, true>(W, s, 1.0f, kAlphaOne, nullptr, qweight, scales, zeros, N, K, count, sms, st)
                       : launch_quantize<128, 4, false, false, true>(W, s, 1.0f, kAlphaOne, nullptr, qweight, scales, zeros, N, K, count, sms, st);
}

cudaError_t launch_quantize_pack(const __half* W, const float* a, float alpha, int group, int bits,
                                 bool symmetric, const float* clip, uint32_t* qweight, __half* scales, uint8_t* zeros,
                                 int N, int K, int sms, cudaStream_t st) {
    const int mode = (int)alpha_mode(alpha);
#define AWQ_QP_LAUNCH(GG, BB, CC, SS) \
    return launch_quantize<GG, BB, CC, SS>(W, a, alpha, mode, clip, qweight, scales, zeros, N, K, 1, sms, st)
#define AWQ_QP_PICK2(GG, SS)                                             \
    do {                                                                 \
        if (bits == 4 && !clip) AWQ_QP_LAUNCH(GG, 4, false, SS);         \
        else if (bits == 4) AWQ_QP_LAUNCH(GG, 4, true, SS);              \
        else if (!clip) AWQ_QP_LAUNCH(GG, 3, false, SS);                 \
        else AWQ_QP_LAUNCH(GG, 3, true, SS);                             \
    } while (0)
#define AWQ_QP_PICK(GG)                                                  \
    do {                                                                 \
        if (symmetric) AWQ_QP_PICK2(GG, true); else AWQ_QP_PICK2(GG, false); \
    } while (0)
    switch (group) {
        case 64: AWQ_QP_PICK(64); break;
        case 128: AWQ_QP_PICK(128); break;
        case 256: AWQ_QP_PICK(256); break;
        case 512: AWQ_QP_PICK(512); break;
        default: AWQ_QP_PICK(1024); break;
    }
#undef AWQ_QP_PICK
#undef AWQ_QP_PICK2
#undef AWQ_QP_LAUNCH
    return cudaErrorInvalidValue;
}

template <int G, int J, int THREADS>
static cudaError_t launch_clip(const __half* W, const float* a, float alpha, int mode, const ClipGrid& ratios, float top,
                               float* clip, int N, int K, bool aligned, cudaStream_t st) {
    static bool done[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (!done[dev & 63]) {
        e = cudaFuncSetAttribute(clip_search_kernel<G, J, THREADS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ClipSmem<G>));
        if (e != cudaSuccess) return e;
        done[dev & 63] = true;
    }
    e = launch_behind(clip_search_kernel<G, J, THREADS>, dim3(K / G, N / kClipRows), THREADS, sizeof(ClipSmem<G>), st, W, a, alpha, mode, ratios, top, clip, N, K, aligned);
    if (e != cudaSuccess) return e;
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_clip_search(const __half* W, const float* a, float alpha, int group, int bits,
                               const float* ratios, int n_ratios, float* clip, int N, int K,
                               cudaStream_t st) {
    ClipGrid grid_r;
    grid_r.n = n_ratios;
    for (int i = 0; i < kMaxClipRatios; ++i) grid_r.r[i] = i < n_ratios ? ratios[i] : 1.0f;
    const int mode = (int)alpha_mode(alpha);
    const float top = (float)((1 << bits) - 1);
    const bool aligned = (reinterpret_cast<uintptr_t>(W) & 15u) == 0;   // rows are multiples of 256 bytes
    // Groups of 64 and up to four ratios: smaller blocks, which the items of one or two ratios fill (11008 x 4096, us, against 256 threads and two
    // ratios an item: 1 ratio 72.1 -> 59.9, 2: 76.1 -> 64.5, 3: 83.4 -> 73.9, 4: 85.7 -> 76.0; groups of 128, whose rows keep a thread busy for
    // twice as long: 63.0 -> 75.3, 65.9 -> 80.3, 71.1 -> 86.8, 72.6 -> 87.7).
    if (group == 64 && n_ratios <= 2) return launch_clip<64, 1, 128>(W, a, alpha, mode, grid_r, top, clip, N, K, aligned, st);
    if (group == 64 && n_ratios <= 4) return launch_clip<64, 2, 128>(W, a, alpha, mode, grid_r, top, clip, N, K, aligned, st);
    return group == 128 ? launch_clip<128, 2, 256>(W, a, alpha, mode, grid_r, top, clip, N, K, aligned, st)
                        : launch_clip<64, 2, 256>(W, a, alpha, mode, grid_r, top, clip, N, K, aligned, st);
}

cudaError_t launch_unpack(const uint32_t* qweight, const __half* scales, const uint8_t* zeros,
                          int N, int K, int group, uint8_t* codes, uint16_t* scales_nk,
                          uint8_t* zeros_nk, cudaStream_t st) {
    const size_t total = (size_t)N * K;
    unpack_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(qweight, scales, zeros, N, K, group,
                                                                    codes, scales_nk, zeros_nk);
    count_launch();
    return cudaGetLastError();
}

// ---- 3-bit storage: four nibble words of a piece (codes < 8) <-> three words.  One thread per piece.
__global__ void pack_int3_kernel(const uint4* __restrict__ q4, uint32_t* __restrict__ q3, size_t pieces) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= pieces) return;
    const uint4 w = q4[i];
    q3[3 * i + 0] = (w.x & 0x77777777u) | ((w.w & 0x11111111u) << 3);
    q3[3 * i + 1] = (w.y & 0x77777777u) | (((w.w >> 1) & 0x11111111u) << 3);
    q3[3 * i + 2] = (w.z & 0x77777777u) | (((w.w >> 2) & 0x11111111u) << 3);
}
__global__ void unpack_int3_kernel(const uint32_t* __restrict__ q3, uint4* __restrict__ q4, size_t pieces) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= pieces) return;
    const uint32_t u0 = q3[3 * i], u1 = q3[3 * i + 1], u2 = q3[3 * i + 2];
    uint4 w;
    w.x = u0 & 0x77777777u;
    w.y = u1 & 0x77777777u;
    w.z = u2 & 0x77777777u;
    w.w = ((u0 >> 3) & 0x11111111u) | ((u1 >> 2) & 0x22222222u) | ((u2 >> 1) & 0x44444444u);
    q4[i] = w;
}

cudaError_t launch_pack_int3(const void* q4, void* q3, int N, int K, cudaStream_t st) {
    const size_t pieces = (size_t)N * K / 32;
    pack_int3_kernel<<<(unsigned)((pieces + 255) / 256), 256, 0, st>>>(
        reinterpret_cast<const uint4*>(q4), reinterpret_cast<uint32_t*>(q3), pieces);
    count_launch();
    return cudaGetLastError();
}
cudaError_t launch_unpack_int3(const void* q3, void* q4, int N, int K, cudaStream_t st) {
    const size_t pieces = (size_t)N * K / 32;
    unpack_int3_kernel<<<(unsigned)((pieces + 255) / 256), 256, 0, st>>>(
        reinterpret_cast<const uint32_t*>(q3), reinterpret_cast<uint4*>(q4), pieces);
    count_launch();
    return cudaGetLastError();
}

}  // namespace awq
