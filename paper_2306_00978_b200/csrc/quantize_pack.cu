// Offline step of the layer: channel scale (Eq. 5), fold into W (Eq. 3), group-wise
// asymmetric 4-bit round-to-nearest (Eq. 2) and the packed tile layout (Sec. 4.2).
//
// HBM-bound: 2 bytes read and ~0.52 bytes written per weight.  One warp owns a band of 16
// rows x 128 columns; lane (g, t) loads rows g and g+8, columns 16j+4t..+3 (j = 0..3) of both
// 64-column tiles (sixteen 8-byte loads in flight per thread; the four lanes of a row read 32
// contiguous bytes), which is exactly the data of the two 16-byte packed pieces it writes, so
// no shared-memory transpose is needed.  Every
// rounding point is an explicit IEEE operation (no contraction); the per-weight division is
// replaced by a multiplication only where that provably rounds to the same integer.
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
__global__ void channel_scales_kernel(const float* __restrict__ a, const __grid_constant__ Alphas alphas, float* __restrict__ s, int K) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x, i = blockIdx.y, mode = alphas.mode[i];
    if (k < K) s[(size_t)i * K + k] = channel_scale_one(mode == kAlphaZero ? 1.0f : a[k], alphas.v[i], mode);
}

__device__ __forceinline__ uint2 ldg_stream(const uint2* p) {
    uint2 v;
    asm volatile("ld.global.nc.L1::no_allocate.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
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
// four codes (exact small integers held in floats) as four nibbles: q0 + 16 q1 + 256 q2 + 4096 q3 is
// exact in fp32, so three FFMAs and one conversion replace four conversions and the shifts and ORs
__device__ __forceinline__ uint32_t pack4(float q0, float q1, float q2, float q3) {
    return (uint32_t)fmaf(q3, 4096.0f, fmaf(q2, 256.0f, fmaf(q1, 16.0f, q0)));
}

// grid = (K/128, N/32), block = 128: warp w takes band w % 2 of the block's 32 rows and block w / 2 of
// the 128 columns, a lane 2 rows x 16 columns - exactly the data of the 16-byte packed piece it writes.
// The products w' = w * s stay in registers (32), formed once (64 registers, 32 warps per SM).  For
// G = 128 the two warps that share a group exchange their min / max through shared memory.  The
// division w' / Delta is done only where it can matter: w' * (1 / Delta) rounds to the same integer
// unless it lies within the group's own error bound of a half-integer; that test is taken per
// packed word and row (the largest distance of the word's products from their rounded values), so
// there is no branch per element, and a word that fails is redone element by element with the
// division (code_of).  Rounding is by adding 1.5 * 2^23 (the zero point rides in the subtraction
// that follows), group min / max take three-input min / max instructions, clamping to [0, top] is
// compiled in only for the warps one of whose groups can leave the range, the nibbles of four codes
// are assembled by FFMA and converted once.
// What bounds it (measured on 4096 -> 11008, 113.6 MB): a block loads, computes and stores in
// phases, and the blocks of an SM run in step, so the loads overlap the arithmetic only as far as
// the blocks drift apart.  With 512-thread blocks (two per SM) 45.4 us, whatever the instruction
// count (a form with a third more instructions and half the warps: 45 us; a third fewer
// integer-pipe instructions: 44.3 us); 256-thread blocks 41.6 us, 128-thread blocks 37.9 us, 64-thread
// blocks 41.0 us (the 128 channel scales are then formed per 64 threads).  A persistent form whose
// producer warp keeps six 32 KB tiles in flight by tensor-map copies for sixteen quantizing warps
// measured 58 us: the arithmetic needs the 32 warps.  The same 128-thread blocks made persistent
// (eight per SM, each walking the tiles): 44.0 us - blocks that never leave stay in step.
__device__ __forceinline__ float min3(float a, float b, float c) {
    float d; asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c)); return d;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
    float d; asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c)); return d;
}
// code (still a float) = clamp(rne(w * rd) + z): zc = 1.5 * 2^23 - z, so that (w * rd + 1.5 * 2^23) - zc
// is the rounded product plus the zero point, exactly (the product enters the sum unrounded, by a
// fused multiply-add: 4 instead of 5 instructions per weight, 38.0 -> 35.7 us on 4096 -> 11008)
// `dev` receives |t - rne(t)|, the distance that decides whether the product may stand for the
// quotient; CLAMP = false where the group's smallest and largest element are known to stay in range.
template <bool CLAMP>
__device__ __forceinline__ float level_fast2(float w, float rd, float zc, float top, float& dev) {
    // one rounding to the integer grid (the product is not rounded first), and the distance of the
    // exact product from that integer, by one fused multiply-add each
    const float u = __fmaf_rn(w, rd, 12582912.0f);
    const float r = __fsub_rn(u, 12582912.0f);
    dev = fabsf(__fmaf_rn(w, rd, -r));
    const float q = __fsub_rn(u, zc);
    return CLAMP ? fminf(fmaxf(q, 0.0f), top) : q;
}

// One warp per band (16 rows) and 64-column block.  A thread block covers one group of columns (two
// groups for G = 64) so that the group's min / max meet in shared memory: 2 bands x 2 blocks up to
// G = 128, 1 band x G / 64 blocks above.  Scales and zero points are stored per 128 columns for
// G > 128 (each group's entry G / 128 times), so that the layer kernels need no variant for them.
template <int G> struct QCfg {
    static constexpr int kBlocks = G < 128 ? 2 : G / 64;            // 64-column blocks per thread block
    static constexpr int kBands = kBlocks <= 4 ? 4 / kBlocks : 1;   // bands per thread block
    static constexpr int kThreads = kBlocks * kBands * 32;
    static constexpr int kStored = G < 128 ? G : 128;               // columns per stored scale / zero point
};

// MANY (the scale search): `a` is `many` arrays of K scales; W is quantized with each, its 32 values per lane loaded once,
// and the packed arrays follow one another (4096 x 4096 with 20 arrays: 12.3 us each in launches of their own, ~9 us here; with
// four blocks per SM, which nothing spills in, the whole search takes 538 us, with five 545, with six 556).
template <int G, int BITS, bool CLIP, bool SYM, bool MANY = false>
__global__ void __launch_bounds__(QCfg<G>::kThreads, (MANY ? 512 : 1024) / QCfg<G>::kThreads)
quantize_pack_tile_kernel(const __half* __restrict__ W, const float* __restrict__ a, float alpha,
                          int mode, const float* __restrict__ clip,
                          uint32_t* __restrict__ qweight, __half* __restrict__ scales,
                          uint8_t* __restrict__ zeros, int N, int K, int many) {
    constexpr float top = (float)((1 << BITS) - 1);       // largest code
    constexpr int kQBands = QCfg<G>::kBands, kQBlocks = QCfg<G>::kBlocks, kQThreads = QCfg<G>::kThreads;
    __shared__ __align__(16) float s_sm[kQBlocks * 64];
    __shared__ float2 s_mm[kQBlocks][kQBands * 16];        // G >= 128: [64-column block][row] (min, max)
    const int kblk = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int bw = warp % kQBands, ti = warp / kQBands;
    const int g = lane >> 2, t = lane & 3;
    const int n0 = (blockIdx.y * kQBands + bw) * 16 + g;   // this lane's upper row; lower = n0 + 8
    const int kbase = kblk * (kQBlocks * 64);

    uint2 raw[2][4];                                       // [row h][word j] = columns 16j + 4t .. +3 of the block
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            raw[h][j] = ldg_stream(reinterpret_cast<const uint2*>(
                W + (size_t)(n0 + 8 * h) * K + kbase + ti * 64 + 16 * j + 4 * t));
    static_assert(!MANY || kQBlocks * 64 == kQThreads, "one scale per thread");
    float s_next = 0.0f;
    if (MANY) s_next = a[kbase + (int)threadIdx.x];
    for (int rest = MANY ? many : 1; rest > 0; --rest) {
    if (MANY) {
        s_sm[threadIdx.x] = s_next;
        a += K;
        if (rest > 1) s_next = a[kbase + (int)threadIdx.x];
    } else {
        for (int i = threadIdx.x; i < kQBlocks * 64; i += kQThreads) {
            const int k = kbase + i;
            s_sm[i] = channel_scale_one(mode == kAlphaZero ? 1.0f : a[k], alpha, mode);
        }
    }
    __syncthreads();

    // w' = fp32(w) * s  (Eq. 3), once, and the min / max of this lane's 16 columns of each row
    float wp[2][4][4];
    float mn[2], mx[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) { mn[h] = INFINITY; mx[h] = -INFINITY; }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float4 s4 = *reinterpret_cast<const float4*>(&s_sm[ti * 64 + 16 * j + 4 * t]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float2 f01 = __half22float2(*reinterpret_cast<const __half2*>(&raw[h][j].x));
            const float2 f23 = __half22float2(*reinterpret_cast<const __half2*>(&raw[h][j].y));
            wp[h][j][0] = __fmul_rn(f01.x, s4.x);
            wp[h][j][1] = __fmul_rn(f01.y, s4.y);
            wp[h][j][2] = __fmul_rn(f23.x, s4.z);
            wp[h][j][3] = __fmul_rn(f23.y, s4.w);
            mn[h] = min3(mn[h], wp[h][j][0], wp[h][j][1]);
            mn[h] = min3(mn[h], wp[h][j][2], wp[h][j][3]);
            mx[h] = max3(mx[h], wp[h][j][0], wp[h][j][1]);
            mx[h] = max3(mx[h], wp[h][j][2], wp[h][j][3]);
        }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int off = 1; off <= 2; off <<= 1) {
            mn[h] = fminf(mn[h], __shfl_xor_sync(0xFFFFFFFFu, mn[h], off));
            mx[h] = fmaxf(mx[h], __shfl_xor_sync(0xFFFFFFFFu, mx[h], off));
        }
    if (G >= 128) {
        // the group spans all 64-column blocks of the thread block: the others' min / max through shared memory
        if (t == 0) {
            s_mm[ti][bw * 16 + g] = make_float2(mn[0], mx[0]);
            s_mm[ti][bw * 16 + g + 8] = make_float2(mn[1], mx[1]);
        }
        __syncthreads();
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int o = 1; o < kQBlocks; ++o) {
                const float2 v = s_mm[(ti + o) % kQBlocks][bw * 16 + g + 8 * h];
                mn[h] = fminf(mn[h], v.x);
                mx[h] = fmaxf(mx[h], v.y);
            }
    }
    float wabs[2];                                          // largest |w'| of each group (before clipping)
#pragma unroll
    for (int h = 0; h < 2; ++h) wabs[h] = fmaxf(fabsf(mn[h]), fabsf(mx[h]));
    const int gi = (G == 64) ? kblk * 2 + ti : kblk;
    const int ng = K / G;
    if (CLIP) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float r = __ldg(clip + (size_t)(n0 + 8 * h) * ng + gi);
            mn[h] = __fmul_rn(mn[h], r);
            mx[h] = __fmul_rn(mx[h], r);
        }
    }
    // Delta, the zero point and 1 / Delta cost three IEEE divisions: each of a row's four lanes needs both rows', so even lanes
    // form the upper row's and odd ones the lower row's, and they exchange them (4096 -> 11008: 32.9 -> 31.2 us).
    const bool low = (t & 1) != 0;
    float d[2], z[2], rd[2], thr[2], zc[2];
    {
        const float mn1 = low ? mn[1] : mn[0], mx1 = low ? mx[1] : mx[0], wabs1 = low ? wabs[1] : wabs[0];
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
        const float tmax = __fmul_rn(wabs1, rd1);
        const float thr1 = tmax < 1024.0f ? 0.5f - fmaf(tmax, 4e-7f, 1e-6f) : -1.0f;
        const float d2 = __shfl_xor_sync(0xFFFFFFFFu, d1, 1), z2 = __shfl_xor_sync(0xFFFFFFFFu, z1, 1);
        const float rd2 = __shfl_xor_sync(0xFFFFFFFFu, rd1, 1), thr2 = __shfl_xor_sync(0xFFFFFFFFu, thr1, 1);
        d[0] = low ? d2 : d1; d[1] = low ? d1 : d2;
        z[0] = low ? z2 : z1; z[1] = low ? z1 : z2;
        rd[0] = low ? rd2 : rd1; rd[1] = low ? rd1 : rd2;
        thr[0] = low ? thr2 : thr1; thr[1] = low ? thr1 : thr2;
#pragma unroll
        for (int h = 0; h < 2; ++h) zc[h] = 12582912.0f - z[h];      // exact: z is a small integer
    }
    // Clamping to [0, top] can only matter where the group's smallest or largest element leaves the
    // range (the level is monotone in w'): rare without clipping - rne(max / Delta) + rne(-min / Delta)
    // exceeds top only when both quotients sit on a tie - so the warp takes the clamped code only if one
    // of its lanes needs it.
    bool need_clamp = CLIP || SYM;
    if (!need_clamp) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float dummy;
            const float qlo = level_fast2<false>(mn[h], rd[h], zc[h], top, dummy);
            const float qhi = level_fast2<false>(mx[h], rd[h], zc[h], top, dummy);
            need_clamp = need_clamp || !(qlo >= 0.0f && qhi <= top);
        }
        need_clamp = __any_sync(0xFFFFFFFFu, need_clamp);
    }
    uint32_t words[4];
    auto quantize_words = [&](auto clamp_tag) {
        constexpr bool CL = decltype(clamp_tag)::value;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float qu[4], ql[4], du[4], dl[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                qu[e] = level_fast2<CL>(wp[0][j][e], rd[0], zc[0], top, du[e]);
                ql[e] = level_fast2<CL>(wp[1][j][e], rd[1], zc[1], top, dl[e]);
            }
            // the word's largest distance from the rounded value, per row, decides
            const float dmu = max3(max3(du[0], du[1], du[2]), du[3], 0.0f);
            const float dml = max3(max3(dl[0], dl[1], dl[2]), dl[3], 0.0f);
            const bool bad = !(dmu < thr[0]) || !(dml < thr[1]);
            // nibbles 0 .. 3 = (g,c) (g+8,c) (g,c+2) (g+8,c+2), nibbles 4 .. 7 the same for c+1, c+3
            words[j] = pack4(qu[0], ql[0], qu[2], ql[2]) | (pack4(qu[1], ql[1], qu[3], ql[3]) << 16);
            if (bad)                                               // rare: the word again, element by element
                words[j] = (code_of(wp[0][j][0], d[0], rd[0], z[0], top) << 0) | (code_of(wp[0][j][1], d[0], rd[0], z[0], top) << 16) |
                           (code_of(wp[1][j][0], d[1], rd[1], z[1], top) << 4) | (code_of(wp[1][j][1], d[1], rd[1], z[1], top) << 20) |
                           (code_of(wp[0][j][2], d[0], rd[0], z[0], top) << 8) | (code_of(wp[0][j][3], d[0], rd[0], z[0], top) << 24) |
                           (code_of(wp[1][j][2], d[1], rd[1], z[1], top) << 12) | (code_of(wp[1][j][3], d[1], rd[1], z[1], top) << 28);
        }
    };
    if (need_clamp) quantize_words(std::true_type{}); else quantize_words(std::false_type{});
    // band-major: block (band, k-tile) is 512 bytes, a band's blocks are contiguous along K
    const size_t band = (size_t)blockIdx.y * kQBands + bw;
    const size_t block = band * (K / 64) + (size_t)kblk * kQBlocks + ti;
    uint4* dst = reinterpret_cast<uint4*>(qweight) + block * 32 + lane;
    *dst = make_uint4(words[0], words[1], words[2], words[3]);
    if (t == 0 && (G == 64 || (ti & 1) == 0)) {
        // scales: [band][stored group][16]; zero bytes: [band pair][stored group][16], 8 per band; a
        // stored group is the group itself up to 128 columns, else each of its runs of 128 columns
        const size_t nsg = K / QCfg<G>::kStored;
        const size_t sgi = (G == 64) ? (size_t)gi : (size_t)kblk * (kQBlocks / 2) + ti / 2;
        scales[(band * nsg + sgi) * 16 + g] = __float2half_rn(d[0]);         // exact: Delta is an fp16 value
        scales[(band * nsg + sgi) * 16 + g + 8] = __float2half_rn(d[1]);
        zeros[((band >> 1) * nsg + sgi) * 16 + (band & 1) * 8 + g] =
            (uint8_t)((uint32_t)z[0] | ((uint32_t)z[1] << 4));
    }
    if (MANY) {
        qweight += (size_t)N * K / 8;
        scales += (size_t)N * (K / QCfg<G>::kStored);
        zeros += (size_t)N * (K / QCfg<G>::kStored) / 2;
        __syncthreads();                                     // s_sm and s_mm have been read
    }
    }
}

// Weight clipping (Sec. 3.2).  For every group of w' = w * s and every ratio r of the list, the
// group is quantized on [r * min, r * max] and its squared error summed; the first ratio of least
// error is written to clip[n][group].  The choice decides integer codes downstream, so the error
// is defined operation by operation: dequant = (q - z) * Delta (one fp32 multiply), e = dequant -
// w', err += e * e in fp32 over ascending k (no contraction), a NaN error counts as +inf.
// grid = (K / G, N / 64), block = 128: one group of columns of 64 rows.  Its w' stay in shared memory, and
// a thread takes one (row, two ratios) item at a time and walks the group's elements
// in order, both ratios in one packed fp32 instruction each (multiply, add and fused multiply-add on two
// floats round each half as the scalar ones do).  As in the quantizer the quotient's rounded value comes
// from w' * (1 / Delta) by one fused multiply-add, and the largest distance of a product from its integer
// decides per (row, ratio) whether that was safe; if not (about 0.05 % of them) the item is redone with
// the division.  Arithmetic bounds it: 6 packed instructions, two moves and 5 min / max per element and
// ratio pair, ~5.6 us per ratio on 4096 -> 4096 and ~15 us for the rest.  4096 -> 4096 with 20 ratios 306 us
// with a scalar division per element and ratio (a row's 2048 columns per 256 threads); packed with the
// pairs (w', w') kept in shared memory, 11 warps per SM, 153 us; w' kept once, 20 warps, 117 us; with four
// times four elements unrolled 112 us (192 or 256 threads: 119, 113 us); with the products kept from
// contraction (mul2) 126 us.
constexpr int kClipRows = 64, kClipThreads = 128;
struct ClipGrid {
    float r[kMaxClipRatios];
    int n;
    float minus_zero;                                       // -0.0f, see mul2
};

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
// The rounded product, as a * b + (-0.0) with the zero in a kernel argument: with mul.rn.f32x2 and an
// add.rn.f32x2 behind it about one group in 10^5 came out with another ratio than the definition, as if the
// two had been fused (the scalar forms with explicit rounding did not); like this all agree.
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b, f32x2 minus_zero) { return fma2(a, b, minus_zero); }
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b)); return d;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
    f32x2 d; asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b)); return d;
}

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

template <int G>
struct ClipSmem {
    static constexpr int kRowFloats = G + 4;                // 16 bytes more, so that rows start on different banks
    float w[kClipRows * kRowFloats];
    float err[kClipRows * (kMaxClipRatios + 1)];
    float2 mm[kClipRows];
    float s[G];
};

template <int G>
__global__ void __launch_bounds__(kClipThreads)
clip_search_kernel(const __half* __restrict__ W, const float* __restrict__ a, float alpha, int mode,
                   const __grid_constant__ ClipGrid ratios, float top, float* __restrict__ clip, int N, int K,
                   bool aligned) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ClipSmem<G>& sm = *reinterpret_cast<ClipSmem<G>*>(smem_raw);
    constexpr int kPieces = G / 8, kRowFloats = ClipSmem<G>::kRowFloats;
    const int n0 = blockIdx.y * kClipRows, k0 = blockIdx.x * G;
    const int tid = threadIdx.x;

    for (int i = tid; i < G; i += kClipThreads) sm.s[i] = channel_scale_one(mode == kAlphaZero ? 1.0f : a[k0 + i], alpha, mode);
    __syncthreads();
    // w' = w * s (Eq. 3), eight columns of a row per thread; the row's min / max over its kPieces lanes
#pragma unroll 4
    for (int i = tid; i < kClipRows * kPieces; i += kClipThreads) {
        const int row = i / kPieces, p = i % kPieces;
        const __half* src = W + (size_t)(n0 + row) * K + k0 + p * 8;
        __half h[8];
        if (aligned) {
            *reinterpret_cast<uint4*>(h) = __ldg(reinterpret_cast<const uint4*>(src));
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) h[e] = src[e];
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
        if (p == 0) sm.mm[row] = make_float2(mn, mx);
    }
    __syncthreads();
    const int nr = ratios.n, np = (nr + 1) / 2;
    for (int item = tid; item < kClipRows * np; item += kClipThreads) {
        const int row = item / np, i0 = 2 * (item - row * np), i1 = min(i0 + 1, nr - 1);
        const float2 mm = sm.mm[row];
        float d[2], z[2], rd[2], thr[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const float r = ratios.r[j ? i1 : i0];
            __half d16;
            group_params(__fmul_rn(mm.x, r), __fmul_rn(mm.y, r), top, d16, d[j], z[j]);
            rd[j] = __frcp_rn(d[j]);
            // |w rd - fl(w / d)| <= 2^-23 |w / d| (1 / d and the quotient are rounded once each); the distance
            // itself is off by at most 2^-26, the threshold by 2^-25
            const float tmax = __fmul_rn(fmaxf(fabsf(mm.x), fabsf(mm.y)), rd[j]);
            thr[j] = tmax < 1024.0f ? 0.5f - fmaf(tmax, 1.25e-7f, 6e-8f) : -1.0f;
        }
        const f32x2 rd2 = pack2(rd[0], rd[1]), d2 = pack2(d[0], d[1]), big = pack2(12582912.0f, 12582912.0f);
        const f32x2 mz = pack2(ratios.minus_zero, ratios.minus_zero);
        const float lo0 = z[0] - top, lo1 = z[1] - top, hi0 = z[0], hi1 = z[1];
        const float* wg = sm.w + row * kRowFloats;
        f32x2 err = pack2(0.0f, 0.0f);
        float dm0 = 0.0f, dm1 = 0.0f;
#pragma unroll 4
        for (int k = 0; k < G; k += 4) {
            const float4 w4 = *reinterpret_cast<const float4*>(wg + k);
            const float we[4] = {w4.x, w4.y, w4.z, w4.w};
            float da[4], db[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const f32x2 w = pack2(we[e], we[e]);
                const f32x2 u = fma2(w, rd2, big);               // rounded to an integer in the sum
                const f32x2 nr2 = sub2(big, u);                  // minus that integer
                unpack2(fma2(w, rd2, nr2), da[e], db[e]);        // its distance from the product
                float q0, q1;
                unpack2(nr2, q0, q1);
                q0 = fminf(fmaxf(q0, lo0), hi0);                 // z - q
                q1 = fminf(fmaxf(q1, lo1), hi1);
                const f32x2 dif = add2(mul2(pack2(q0, q1), d2, mz), w);  // minus the difference: its square is the same
                err = add2(err, mul2(dif, dif, mz));
            }
            dm0 = max3(max3(dm0, fabsf(da[0]), fabsf(da[1])), fabsf(da[2]), fabsf(da[3]));
            dm1 = max3(max3(dm1, fabsf(db[0]), fabsf(db[1])), fabsf(db[2]), fabsf(db[3]));
        }
        float e0, e1;
        unpack2(err, e0, e1);
        if (!(dm0 < thr[0])) e0 = clip_error_by_division<G>(wg, d[0], z[0], top);
        if (!(dm1 < thr[1])) e1 = clip_error_by_division<G>(wg, d[1], z[1], top);
        float* out = sm.err + row * (kMaxClipRatios + 1);
        out[i0] = (e0 != e0) ? INFINITY : e0;
        if (i1 > i0) out[i1] = (e1 != e1) ? INFINITY : e1;
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
    channel_scales_kernel<<<dim3((K + 255) / 256, n), 256, 0, st>>>(a, list, s, K);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_quantize_pack_many(const __half* W, const float* s, int count, int group, uint32_t* qweight, __half* scales,
                                      uint8_t* zeros, int N, int K, cudaStream_t st) {
    if (group == 64)
        quantize_pack_tile_kernel<64, 4, false, false, true><<<dim3(K / 128, N / (16 * QCfg<64>::kBands)), QCfg<64>::kThreads, 0, st>>>(
            W, s, 1.0f, kAlphaOne, nullptr, qweight, scales, zeros, N, K, count);
    else
        quantize_pack_tile_kernel<128, 4, false, false, true><<<dim3(K / 128, N / (16 * QCfg<128>::kBands)), QCfg<128>::kThreads, 0, st>>>(
            W, s, 1.0f, kAlphaOne, nullptr, qweight, scales, zeros, N, K, count);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_quantize_pack(const __half* W, const float* a, float alpha, int group, int bits,
                                 bool symmetric, const float* clip, uint32_t* qweight, __half* scales, uint8_t* zeros,
                                 int N, int K, cudaStream_t st) {
    const int mode = (int)alpha_mode(alpha);
#define AWQ_QP_LAUNCH(GG, BB, CC, SS)                                                                           \
    quantize_pack_tile_kernel<GG, BB, CC, SS><<<dim3(K / (QCfg<GG>::kBlocks * 64), N / (16 * QCfg<GG>::kBands)), \
                                                QCfg<GG>::kThreads, 0, st>>>(W, a, alpha, mode, clip, qweight, scales, zeros, N, K, 1)
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
    count_launch();
    return cudaGetLastError();
}

template <int G>
static cudaError_t launch_clip(const __half* W, const float* a, float alpha, int mode, const ClipGrid& ratios, float top,
                               float* clip, int N, int K, bool aligned, cudaStream_t st) {
    static bool done[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (!done[dev & 63]) {
        e = cudaFuncSetAttribute(clip_search_kernel<G>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ClipSmem<G>));
        if (e != cudaSuccess) return e;
        done[dev & 63] = true;
    }
    clip_search_kernel<G><<<dim3(K / G, N / kClipRows), kClipThreads, sizeof(ClipSmem<G>), st>>>(
        W, a, alpha, mode, ratios, top, clip, N, K, aligned);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_clip_search(const __half* W, const float* a, float alpha, int group, int bits,
                               const float* ratios, int n_ratios, float* clip, int N, int K,
                               cudaStream_t st) {
    ClipGrid grid_r;
    grid_r.n = n_ratios;
    grid_r.minus_zero = -0.0f;
    for (int i = 0; i < kMaxClipRatios; ++i) grid_r.r[i] = i < n_ratios ? ratios[i] : 1.0f;
    const int mode = (int)alpha_mode(alpha);
    const float top = (float)((1 << bits) - 1);
    const bool aligned = (reinterpret_cast<uintptr_t>(W) & 15u) == 0;   // rows are multiples of 256 bytes
    return group == 128 ? launch_clip<128>(W, a, alpha, mode, grid_r, top, clip, N, K, aligned, st)
                        : launch_clip<64>(W, a, alpha, mode, grid_r, top, clip, N, K, aligned, st);
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
