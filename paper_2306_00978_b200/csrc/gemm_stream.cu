// The layer for 9 .. 256 tokens (and fewer on long rows or few output rows; Sec. 4.2: fused dequantize + product) on the
// tensor cores, where the weights or the start of a launch set the time rather than the products.
//
// Pairs of thread blocks (a cluster of two SMs) issue tcgen05.mma.cta_group::2 of 256 output channels x bn <= 128
// tokens: weights -> q - z (exactly), straight into tensor memory as the A operand, tokens on the N side, each block
// staging half of them.  The tiles' K loops (256 input channels a stage), of up to four matrices that read the same x, are
// laid end to end and cut into one range per pair, so that all pairs end together whatever the sizes.  A tile
// that a cut divides leaves its parts' fp32 sums in the workspace, and a second, small kernel adds them in a fixed order:
// deterministic, no counters, nobody waits for another pair.
//   * a stage is 8 bands x 256 input channels of packed weights (16 KB), its scales and zero points, and the block's half
//     of x (128-byte swizzle), one tensor-map copy each, up to six stages ahead;
//   * sixteen dequantizer warps, each owning a band and every second stage; a slot of A in tensor memory is a stage;
//   * one warp issues the products, four (16 tokens) or eight epilogue warps drain them.
// A is stored in the 16x128b form (17 cycles per 16 x 32 columns; 16x256b, which is the packed piece as it is, takes 33, and
// up to 48 while products run).  In that form lane t of a row holds the 32-bit columns 4i + t, while its words hold
// pairs 2t and 2t + 1 of each 16 channels: so A's channels come permuted inside each 16, pair 2t + p at place
// 4p + t, and the dequantizers bring the stage's x into the same order in shared memory (the products' sum over 16
// channels does not depend on the order).  The product with 1 / s of awq_linear_scaled rides on that pass.
//
// Up to 32 tokens (EXACT) A is the integer q - z, every group has an accumulator of its own and the epilogue adds Delta times it
// in fp32: nothing is rounded before the output (a 2-norm error of 2.1e-4); above A is fp16 (q - z) * Delta (2.8e-4).
//
// What bounds it: a stage takes 970 / 1130 / 1410 cycles at 16 / 32 / 64 tokens (18944 channels, one tile per pair, the slope of chained
// calls with cold weights between 4096 and 12288 input channels; 1010 / 1140 / 1410 while a stage was freed by the epilogue behind its
// products; 700 at the HBM rate), of which the products' and the dequantizers' own cycles, counted in a copy of the kernel at 16
// tokens, are about 880 each.  Above 64 tokens x through L2 (32 KB a stage and SM at 128 tokens, half of a tile's, beside 16 KB of
// weights) comes on top, on short launches their start (~3 us until the first products are drained) and the second kernel (~1.5 us).
// What it took, 28672 -> 8192 / 4096 -> 4096 at 16 tokens, us (one machine, cold weights; 30.5 to 33.2 and 6 to 6.4 by now on others):
//   one SM per 128 channels, chunks of K with x resident, whole units per block       37.6 / 7.9
//   pairs, even ranges; parts added by the last pair to arrive                         45 / 10
//   scales and zero points with the stage instead of loads ahead                       42 / 10
//   copies issued before tensor memory and the cluster are ready, host-made divisors   37.5 / 8.6
//   warp number through a shuffle and tensor memory at column 0, so that a product's operands are formed in uniform
//     registers (46 -> 32 cycles a product)                                            31 / 8
//   64 registers, so that a block of the second kernel fits beside the first's         30 / 6.4
//   (another machine: 30.5 / 5.85) a stage freed by its products, the scales read before, not by the epilogue behind them   29.2 / 5.72
//   three stages of weights ahead at the start (kStAhead), six in all                  28.7 / 5.67
// Adding the parts inside this kernel cost more: by the last pair to arrive 9.5 us, by all of a tile's pairs 9.6 us,
// through distributed shared memory of clusters of 4 or 8 blocks (whole tiles only; 33 and 15 clusters fit) 7.0 us.
#include "tcgen05.cuh"

namespace awq {

namespace {

// warps: 0 weight copies, 1 products (leader), 2 x copies, 4-7 and 24-27 epilogue, 8-23 dequantizers
constexpr int kStTiles = 4;                              // k-blocks per stage
constexpr int kStStageK = kStTiles * kBK;                // 256 input channels
constexpr int kStBlockBytes = 512;                       // 16 rows x 64 columns (384 in the 3-bit storage)
constexpr int kStWBytes = 8 * kStTiles * kStBlockBytes;  // 8 bands x 4 k-blocks
constexpr int kStInvBytes = kStStageK * 4;               // the stage's 1 / s
constexpr int kStZeroBytes = 256, kStScaleBytes = 1024;  // zero points [4 band pairs][groups][16], scales [8 bands][groups][16]
constexpr int kStMaxSmem = 226 * 1024 - 64;              // dynamic part: a few static bytes, and a block of the second kernel, come on top
// Stages of weights that may be under way before the first has landed.  With the whole ring asked for at once x, which may be asked for
// only after the launch in front, arrives behind it: 11008 -> 4096 at 16 / 32 tokens 10.2 / 11.6 us against 9.2 / 10.5, 4096 -> 12288 at 16
// 10.7 against 9.6 (two: 9.5, but 4096 -> 22016 15.7 against 15.0; six stages in all instead of eight are as fast in the long run and faster here).
constexpr int kStAhead = 3;
constexpr int kStMaxThreads = 1024;                      // what registers are kept free for: the second kernel's block

// BN: tokens per tile at most (N of the products is a multiple of 16 up to that)
template <int BN, bool XS> struct StCfg {
    static constexpr bool kExact = BN <= 32;             // q - z as an integer, Delta applied in fp32 (see the kernel)
    static constexpr int kHalf = BN / 2;                 // tokens staged by each block of the pair
    static constexpr int kXBytes = kStTiles * kHalf * 128;
    static constexpr int kParOff = kXBytes + kStWBytes;  // [scales | 1 / s | zero points]
    static constexpr int kInvOff = kParOff + kStScaleBytes, kZeroOff = kInvOff + (XS ? kStInvBytes : 0);
    static constexpr int kStageBytes = (kZeroOff + kStZeroBytes + 1023) / 1024 * 1024;
    static constexpr int kOutBytes = kExact ? 0 : 8 * 2048;
    static constexpr int kFixed = 1024 /*align*/ + 512 /*barriers*/ + kOutBytes;
    static constexpr int kFit = (kStMaxSmem - kFixed) / kStageBytes;
    static constexpr int kStages = kFit < 6 ? kFit : 6;
    // tensor memory: accumulators (EXACT: of pairs of groups), then 128 columns of A per slot
    static constexpr uint32_t kAccCols = kExact ? 2 * BN : BN;
    static constexpr uint32_t kNumAcc = BN == 16 ? 4 : BN <= 64 ? 2 : 1;
    static constexpr int kEpilogue = BN == 16 ? 1 : 2;   // warps per 32 channels, which divide the tokens
    static constexpr int kEpTokens = BN / kEpilogue;
    static constexpr int kThreads = (24 + (kEpilogue - 1) * 4) * 32;
    static constexpr int kA0 = 128;
    static constexpr int kSlots = (512 - kA0) / 128;
    static constexpr int kSmemBytes = kFixed + kStages * kStageBytes;
    static_assert(kNumAcc * kAccCols <= (uint32_t)kA0, "accumulators and A slots overlap");
    static_assert(kStages > kSlots, "a slot's previous use is found by its stage's barrier");
};

// up to kMaxMulti matrices that read the same x
struct StMats {
    CUtensorMap w[kMaxMulti], sc[kMaxMulti], z[kMaxMulti];
};
// Tiles (256 channels x bn tokens, all matrices' end to end), their K loops cut into one range of stages per pair.
struct StCut {
    int M, K;
    int nks, total, pairs;                               // stages per tile, of all tiles, ranges
    int share, longer;                                   // total / pairs, total % pairs
    int tiles;
    float inv_nks;                                       // 1 / nks
    int bn, rows, m_tiles;                               // tokens per tile, rows of a partial tile, token tiles
    int slab_end[kMaxMulti];                             // first 256-channel slab of the next matrix
    int n[kMaxMulti];
    __half* y[kMaxMulti];
};

__device__ __forceinline__ int st_range_start(const StCut& c, int p) { return p * c.share + min(p, c.longer); }
// s / nks (s below 2^22: the quotient in fp32 is at most one off)
__device__ __forceinline__ int st_tile_of(const StCut& c, int s) {
    const int q = (int)((float)s * c.inv_nks), r = s - q * c.nks;
    return r < 0 ? q - 1 : r >= c.nks ? q + 1 : q;
}
__device__ __forceinline__ int st_pair_of(const StCut& c, int s) {
    const int in_longer = c.longer * (c.share + 1);
    return s < in_longer ? s / (c.share + 1) : c.longer + (s - in_longer) / c.share;
}
// A pair's stages: `count` of them, the first one stage ks of `tile`.
struct StRange { int count, tile, ks; };
__device__ __forceinline__ StRange st_range(const StCut& c, int pair) {
    StRange r;
    const int s0 = st_range_start(c, pair);
    r.count = st_range_start(c, pair + 1) - s0;
    r.tile = st_tile_of(c, s0);
    r.ks = s0 - r.tile * c.nks;
    return r;
}
// where a tile lies: matrix, 256-channel slab of it, token tile
struct StTile { int mi, slab, mt; };
__device__ __forceinline__ StTile st_tile(const StCut& c, int tile) {
    StTile t = {0, c.m_tiles == 1 ? tile : tile / c.m_tiles, 0};
    t.mt = tile - t.slab * c.m_tiles;
    int base = 0;
#pragma unroll
    for (int i = 0; i + 1 < kMaxMulti; ++i)
        if (t.slab >= c.slab_end[i]) { t.mi = i + 1; base = c.slab_end[i]; }
    t.slab -= base;
    return t;
}
// the fp32 sums of a pair's part of a tile: slot 2p + 1 for the part that starts its tile, 2p for the other
// one; [rank][row][128 channels]
__device__ __forceinline__ size_t st_slot(const StCut& c, int slot, int rank) {
    return (size_t)(slot * 2 + rank) * (size_t)(c.rows * 128);
}
// arrives on the barrier at this offset in both blocks of the pair when the products issued so far are done
__device__ __forceinline__ void st_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(bar), "h"((unsigned short)3) : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld_8cols(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld_16cols(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr) : "memory");
}
template <int C> __device__ __forceinline__ void tmem_ld_cols(uint32_t taddr, uint32_t (&r)[C]) {
    static_assert(C == 8 || C == 16, "columns per load");
    if constexpr (C == 8) tmem_ld_8cols(taddr, r); else tmem_ld_16cols(taddr, r);
}
// 16 lanes x 32 columns in the 16x128b register layout: lane (g, t) holds, for i = 0 .. 7, rows g and
// g + 8 of column 4i + t in registers 2i and 2i + 1.
__device__ __forceinline__ void tmem_st_16x32cols_128b(uint32_t taddr, const uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.16x128b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
        "%14, %15, %16};"
        ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
          "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
        : "memory");
}
// two fp16 activations times their 1 / s: fp16_rne(fp32(x) * inv_s) each
__device__ __forceinline__ uint32_t scale_pair(uint32_t h, float2 s) {
    const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&h));
    const __half2 r = __floats2half2_rn(__fmul_rn(f.x, s.x), __fmul_rn(f.y, s.y));
    return *reinterpret_cast<const uint32_t*>(&r);
}
// a += d * x, b += d * y in one instruction (each rounded like fmaf)
__device__ __forceinline__ void fma_pair(float& a, float& b, float d, uint32_t x, uint32_t y) {
    asm("{\n\t.reg .b64 s, t, u;\n\t"
        "mov.b64 s, {%0, %1};\n\tmov.b64 t, {%2, %2};\n\tmov.b64 u, {%3, %4};\n\t"
        "fma.rn.f32x2 s, t, u, s;\n\tmov.b64 {%0, %1}, s;\n\t}"
        : "+f"(a), "+f"(b) : "f"(d), "r"(x), "r"(y));
}
// a time-out bounded end of copies in flight: the block may exit only when they have landed
__device__ __forceinline__ void drain(uint32_t bar, uint32_t parity, const WaitCtl& ctl) {
    const unsigned long long t0 = global_ns();
    while (!mbar_try_wait(bar, parity) && global_ns() - t0 < drain_limit_ns(ctl)) {}
}

// A lane's piece of one block.  3-bit storage: three words, whose nibbles' top bits are the fourth's (the readers mask them out).
template <int TB> __device__ __forceinline__ uint4 st_piece(const unsigned char* p) {
    if constexpr (TB == kStBlockBytes) return *reinterpret_cast<const uint4*>(p);
    const uint32_t* u = reinterpret_cast<const uint32_t*>(p);
    return make_uint4(u[0], u[1], u[2], ((u[0] >> 3) & 0x11111111u) | ((u[1] >> 2) & 0x22222222u) | ((u[2] >> 1) & 0x44444444u));
}

// TB: bytes of a packed block (16 rows x 64 columns): 512 for 4-bit codes, 384 for the 3-bit storage, whose fourth word costs five
// instructions per piece and the others none (their masks leave out a nibble's top bit): 8192 -> 28672 at 16 / 32 / 64 tokens 32.1 / 36.7 /
// 44.2 us plainly ordered, 4-bit codes in chained launches 30.6 / 35.7 / 45.5.
template <int G, int BN, bool XS, int TB = kStBlockBytes>
__global__ void __launch_bounds__(kStMaxThreads, 1)
gemm_stream_kernel(const __grid_constant__ StCut cut, const float* __restrict__ inv_s, float* partial, unsigned int* status_word, const __grid_constant__ CUtensorMap x_map,
                   const __grid_constant__ StMats mats) {
    using Cfg = StCfg<BN, XS>;
    constexpr bool EXACT = Cfg::kExact;
    constexpr int S = Cfg::kStages, SL = Cfg::kSlots;
    constexpr int KPG = G / kBK;                         // k-blocks per group
    constexpr int GPS = kStTiles / KPG;                  // groups per stage
    constexpr int kBlockK = TB / 8, kWBytes = 8 * kStTiles * TB;  // a block's 64-bit elements per band, a stage's weights
    constexpr uint32_t NACC = Cfg::kNumAcc;
    static_assert(8 * (3 * S + 2 * SL + 2 * (int)NACC) <= 512, "barriers");
    extern __shared__ unsigned char smem_dyn[];
    __shared__ unsigned int s_abort;
    __shared__ uint32_t s_tmem_base;

    const uint32_t dyn = smem_u32(smem_dyn);
    const uint32_t base = (dyn + 1023u) & ~1023u;
    unsigned char* base_ptr = smem_dyn + (base - dyn);
    // stage: [x: 4 k-blocks of BN / 2 rows x 128 bytes, 128-byte swizzle | packed weights | 1 / s]
    auto x_off = [&](uint32_t s) { return s * (uint32_t)Cfg::kStageBytes; };
    auto w_off = [&](uint32_t s) { return s * (uint32_t)Cfg::kStageBytes + (uint32_t)Cfg::kXBytes; };
    constexpr uint32_t kOutOff = (uint32_t)(S * Cfg::kStageBytes);
    const uint32_t bars = base + kOutOff + (uint32_t)Cfg::kOutBytes;
    auto w_full = [&](uint32_t s) { return bars + 8u * s; };                       // weights landed
    auto x_full = [&](uint32_t s) { return bars + 8u * (uint32_t)(S + s); };       // own half of x landed
    auto empty = [&](uint32_t s) { return bars + 8u * (uint32_t)(2 * S + s); };    // the stage may be filled again
    auto a_full = [&](uint32_t s) { return bars + 8u * (uint32_t)(3 * S + s); };   // leader: both blocks' A and x are ready
    auto acc_full = [&](uint32_t b) { return bars + 8u * ((uint32_t)(3 * S + SL) + b); };
    auto acc_empty = [&](uint32_t b) { return bars + 8u * ((uint32_t)(3 * S + SL) + NACC + b); };    // leader
    auto a_empty = [&](uint32_t s) { return bars + 8u * ((uint32_t)(3 * S + SL) + 2u * NACC + s); }; // the slot's products are done

    // (the shuffle tells the compiler that all lanes of a warp take the same role: addresses stay in uniform registers)
    const int warp = __shfl_sync(0xFFFFFFFFu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const int pair = (int)cluster_id_x();
    const int nks = cut.nks, half_rows = cut.bn >> 1;
    const StRange range = st_range(cut, pair);

    // The copies need nothing but their barriers: they start before tensor memory is there and before the other block
    // of the pair is (the first weights land 2600 instead of 4000 cycles after the start).
    if (warp == 0) {
        if (lane == 0) {
            s_abort = 0u;
            for (uint32_t s = 0; s < (uint32_t)S; ++s) {
                mbar_init(w_full(s), 1); mbar_init(x_full(s), 1);
                mbar_init(empty(s), EXACT ? 1 + 4 * Cfg::kEpilogue : 1);  // the products, and (EXACT) the epilogue has read the scales
            }
            for (uint32_t s = 0; s < (uint32_t)SL; ++s) { mbar_init(a_full(s), 16); mbar_init(a_empty(s), 1); }
            for (uint32_t b = 0; b < NACC; ++b) { mbar_init(acc_full(b), 1); mbar_init(acc_empty(b), 8 * Cfg::kEpilogue); }
            mbar_fence_init();
        }
        __syncwarp();
        named_barrier_sync(1, 64);
    } else if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&s_tmem_base)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        tc_fence_before();
    } else if (warp == 2) {
        named_barrier_sync(1, 64);
    }
    if (warp == 0 || warp == 2) {
        asm volatile("bar.arrive 2, %0;" ::"r"(Cfg::kThreads) : "memory");
        cluster_arrive_start();
    } else {
        named_barrier_sync(2, Cfg::kThreads);
        cluster_arrive_start();
        cluster_wait();                   // both blocks' barriers exist before anyone arrives remotely
        tc_fence_after();
    }
    constexpr uint32_t tmem_base = 0;        // all 512 columns are this block's
    const WaitCtl ctl{status_word, &s_abort};
    // programmatic dependent launch: the packed arrays are constants of the layer and are copied before
    // the work in front of this launch has completed; x and the workspace are touched after it
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (warp == 0) {
        // ------------------------------------------------------------ weight copies
        const bool lead = elect_one();
        uint32_t stage = 0, phase = 0;
        int issued = 0, tile = range.tile, ks = range.ks;
        StTile at = st_tile(cut, tile);
        bool ok = true;
        for (int n = 0; n < range.count; ++n) {
            if (n >= kStAhead && n < S && !mbar_wait_warp(w_full((uint32_t)(n - kStAhead)), 0u, ctl)) { ok = false; break; }
            if (!mbar_wait_warp(empty(stage), phase ^ 1u, ctl)) { ok = false; break; }
            if (lead) {
                mbar_arrive_expect_tx(w_full(stage), kWBytes + GPS * (64 + 256));
                // 8 bands x 4 k-blocks (256 or 192 64-bit elements); past the last band or k-block zeros are filled in
                tma_load_2d(base + w_off(stage), &mats.w[at.mi], ks * kStTiles * kBlockK, at.slab * 16 + (int)rank * 8, w_full(stage));
                tma_load_2d(base + x_off(stage) + Cfg::kZeroOff, &mats.z[at.mi], ks * GPS * 16, at.slab * 8 + (int)rank * 4, w_full(stage));
                tma_load_2d(base + x_off(stage) + Cfg::kParOff, &mats.sc[at.mi], ks * GPS * 16, at.slab * 16 + (int)rank * 8, w_full(stage));
            }
            __syncwarp();
            ++issued;
            if (++stage == (uint32_t)S) { stage = 0; phase ^= 1u; }
            if (++ks == nks) { ks = 0; at = st_tile(cut, ++tile); }
        }
        if (!ok) {
            for (int i = 0; i < S && i < issued; ++i) {
                if (stage == 0) { stage = S - 1; phase ^= 1u; } else { --stage; }
                drain(w_full(stage), phase, ctl);
            }
        }
    } else if (warp == 2) {
        // ------------------------------------------------------------ x copies
        const bool lead = elect_one();
        uint32_t stage = 0, phase = 0;
        int issued = 0, tile = range.tile, ks = range.ks;
        StTile at = st_tile(cut, tile);
        bool ok = true;
        asm volatile("griddepcontrol.wait;" ::: "memory");
        for (int n = 0; n < range.count; ++n) {
            const int inv_bytes = min(kStStageK, cut.K - ks * kStStageK) * 4;
            if (!mbar_wait_warp(empty(stage), phase ^ 1u, ctl)) { ok = false; break; }
            if (lead) {
                mbar_arrive_expect_tx(x_full(stage), (uint32_t)(Cfg::kXBytes + (XS ? inv_bytes : 0)));
                // this block's half of the tile's tokens x 4 k-blocks; past the last token or k-block zeros
                tma_load_3d(base + x_off(stage), &x_map, 0, at.mt * cut.bn + (int)rank * half_rows, ks * kStTiles, x_full(stage));
                if (XS) bulk_load(base + x_off(stage) + Cfg::kInvOff, inv_s + (size_t)ks * kStStageK, (uint32_t)inv_bytes, x_full(stage));
            }
            __syncwarp();
            ++issued;
            if (++stage == (uint32_t)S) { stage = 0; phase ^= 1u; }
            if (++ks == nks) { ks = 0; at = st_tile(cut, ++tile); }
        }
        if (!ok) {
            for (int i = 0; i < S && i < issued; ++i) {
                if (stage == 0) { stage = S - 1; phase ^= 1u; } else { --stage; }
                drain(x_full(stage), phase, ctl);
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ products (leader block only)
        if (rank == 0) {
            const bool lead = elect_one();
            const uint32_t idesc = (1u << 4) | ((uint32_t)(cut.bn >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
            constexpr int kb_step = (Cfg::kHalf * 128) >> 4;     // a k-block of x, in descriptor units
            uint32_t stage = 0, slot = 0, slot_phase = 0, acc = 0, acc_phase = 0;
            int ks = range.ks;
            bool ok = true;
            for (int n = 0; n < range.count; ++n) {
                const bool first = n == 0 || ks == 0, last = n + 1 == range.count || ks + 1 == nks;
                // both barriers are normally complete already: they are polled together
                const bool ar = mbar_try_wait(a_full(slot), slot_phase), er = mbar_try_wait(acc_empty(acc), acc_phase ^ 1u);
                if (!__all_sync(0xFFFFFFFFu, ar) && !mbar_wait_warp(a_full(slot), slot_phase, ctl)) break;
                if ((EXACT || first) && !__all_sync(0xFFFFFFFFu, er) && !mbar_wait_warp(acc_empty(acc), acc_phase ^ 1u, ctl)) break;
                tc_fence_after();
                const uint32_t a_tmem = tmem_base + (uint32_t)(Cfg::kA0 + slot * 128);
                const uint64_t bdesc = smem_desc_sw128(base + x_off(stage));
                // k-blocks h0 .. h1-1 of the stage into an accumulator
                auto products = [&](uint32_t d_tmem, int h0, int h1, bool start) {
#pragma unroll
                    for (int h = h0; h < h1; ++h)
#pragma unroll
                        for (int k = 0; k < kBK / 16; ++k)       // A: +8 columns, B: +32 bytes per K = 16 step
                            umma_pair_f16_a_tmem(d_tmem, a_tmem + (uint32_t)(32 * h + 8 * k), bdesc + (uint64_t)(h * kb_step) + (uint64_t)(2 * k),
                                    idesc, (!start || h != h0 || k != 0) ? 1u : 0u);
                };
                if (EXACT) {
#pragma unroll
                    for (int q = 0; q < GPS; q += 2) {           // pairs of groups
                        if (q > 0) {
                            if (!mbar_wait_warp(acc_empty(acc), acc_phase ^ 1u, ctl)) { ok = false; break; }
                            tc_fence_after();
                        }
                        if (lead) {
                            const uint32_t d_tmem = tmem_base + acc * Cfg::kAccCols;
                            products(d_tmem, q * KPG, (q + 1) * KPG, true);
                            products(d_tmem + (uint32_t)BN, (q + 1) * KPG, (q + 2) * KPG, true);
                            // The slot before the last pair's sums: what the epilogue waits for comes last,
                            // so that no arrival is outstanding when the block exits.
                            if (q + 2 >= GPS) { st_commit(a_empty(slot)); st_commit(empty(stage)); }
                            st_commit(acc_full(acc));
                        }
                        __syncwarp();
                        if (++acc == NACC) { acc = 0; acc_phase ^= 1u; }
                    }
                    if (!ok) break;
                } else {
                    if (lead) {
                        products(tmem_base + acc * Cfg::kAccCols, 0, kStTiles, first);
                        st_commit(empty(stage));
                        if (last) st_commit(acc_full(acc));
                    }
                    __syncwarp();
                    if (last && ++acc == NACC) { acc = 0; acc_phase ^= 1u; }
                }
                if (++stage == (uint32_t)S) stage = 0;
                if (++slot == (uint32_t)SL) { slot = 0; slot_phase ^= 1u; }
                if (++ks == nks) ks = 0;
            }
            // the epilogues' last arrivals, the other block's among them, are waited for here (see cluster_sync_end)
            for (uint32_t b = 0; b < NACC && mbar_wait_warp(acc_empty(acc), acc_phase ^ 1u, ctl); ++b)
                if (++acc == NACC) { acc = 0; acc_phase ^= 1u; }
        }
    } else if (warp >= 8 && warp < 24) {
        // ------------------------------------------------------------ dequantizers
        // warp (band, parity): the band's 16 rows, all four k-blocks of every second stage.  Lane (g, t)
        // holds, per k-block, the piece (rows g and g+8, columns 16j + 4t .. +3 for j = 0..3).
        const int wi = warp - 8, quad = wi & 3, hsel = (wi >> 2) & 1, par2 = wi >> 3;
        const int band = 2 * quad + hsel;                // bands 0..7 <-> TMEM lanes 16 * band .. +15
        const int g = lane >> 2;
        const uint32_t taddr_band = tmem_base + ((uint32_t)(quad * 32 + hsel * 16) << 16) + (uint32_t)Cfg::kA0;
        const uint32_t leader_a_full0 = map_to_rank(a_full(0), 0);
        const unsigned char* w_lane = base_ptr + Cfg::kXBytes + band * (kStTiles * TB) + lane * (TB / 32);
        // x's channels are brought into A's order in shared memory, 16 of a token (32 bytes) per thread and pass
        constexpr int kThreadsPerKb = 4 * Cfg::kHalf, kKbPerPass = 256 / kThreadsPerKb < kStTiles ? 256 / kThreadsPerKb : kStTiles;
        const int t256 = (wi & 7) * 32 + lane, xkb = t256 / kThreadsPerKb, xm = (t256 >> 2) % Cfg::kHalf, xj = t256 & 3;
        const bool x_active = xkb < kKbPerPass && xm < half_rows;

        // this lane's rows' parameters of a stage
        const unsigned char* z_lane = base_ptr + Cfg::kZeroOff + (band >> 1) * (GPS * 16) + (band & 1) * 8 + g;
        const unsigned char* d_lane = base_ptr + Cfg::kParOff + band * (GPS * 32) + g * 2;
        uint32_t stage = (uint32_t)par2, phase = 0, slot = (uint32_t)par2;
        // the slot's previous use was SL stages ago: its products are done when that stage is empty (EXACT: a barrier of its own)
        uint32_t old = (uint32_t)(EXACT ? par2 : par2 + S - SL), old_phase = 1u;
        constexpr uint32_t kOldRing = EXACT ? SL : S;
        const uint32_t old_bar0 = EXACT ? a_empty(0) : empty(0);
        int to_last = nks - 1 - range.ks - par2;         // stages up to its tile's last one
        if (to_last < 0) to_last += nks;
        const int last_kb = cut.K / kBK - (nks - 1) * kStTiles;  // k-blocks of that stage
        for (int n = par2; n < range.count; n += 2) {
            const uint32_t so = x_off(stage);
            bool ok = mbar_wait(w_full(stage), phase, ctl);
            uint4 pk[kStTiles];
#pragma unroll
            for (int h = 0; h < kStTiles; ++h) pk[h] = st_piece<TB>(w_lane + so + h * TB);
            ok = mbar_wait(old_bar0 + 8u * old, old_phase, ctl) && ok;
            tc_fence_after();
            uint32_t zc[GPS], du[GPS], dl[GPS];
#pragma unroll
            for (int q = 0; q < GPS; ++q) {
                zc[q] = z_lane[so + q * 16];
                if (EXACT) { du[q] = dl[q] = 0u; continue; }
                du[q] = *reinterpret_cast<const unsigned short*>(d_lane + so + q * 32);
                dl[q] = *reinterpret_cast<const unsigned short*>(d_lane + so + q * 32 + 16);
            }
#pragma unroll
            for (int h = 0; h < kStTiles; ++h) {
                const int q = h / KPG;
                // 1024 + z for the low nibble; -(64 + z) for the high one (bits 4-7 of the byte are z << 4)
                const uint32_t zlo = __byte_perm((zc[q] & 0xFu) | 0x6400u, 0u, 0x1010), zhi = __byte_perm((zc[q] & 0xF0u) | 0xD400u, 0u, 0x1010);
                const uint32_t d_up = __byte_perm(du[q], 0u, 0x1010), d_lo = __byte_perm(dl[q], 0u, 0x1010);
                const uint32_t wds[4] = {pk[h].x, pk[h].y, pk[h].z, pk[h].w};
                // word j: (row g | g+8: c, c+1) in its low bytes, (c+2, c+3) in the bytes above
                uint32_t v[16];
#pragma unroll
                for (int jw = 0; jw < 4; ++jw) {
                    constexpr uint32_t kSixteenth = 0x2C002C00u;
                    const uint32_t w = wds[jw], w8 = w >> 8;
                    constexpr uint32_t kLow = TB == kStBlockBytes ? kLowCodes : kLowCodes & 0x77777777u, kHigh = TB == kStBlockBytes ? kHighCodes : kHighCodes & 0x77777777u;
                    v[4 * jw + 0] = hsub2_u32(code_pair(w, kLow), zlo);                  // q - z, exactly
                    v[4 * jw + 1] = hfma2_u32(code_pair(w, kHigh), kSixteenth, zhi);
                    v[4 * jw + 2] = hsub2_u32(code_pair(w8, kLow), zlo);
                    v[4 * jw + 3] = hfma2_u32(code_pair(w8, kHigh), kSixteenth, zhi);
                    if (EXACT) continue;
                    v[4 * jw + 0] = hmul2_u32(v[4 * jw + 0], d_up);
                    v[4 * jw + 1] = hmul2_u32(v[4 * jw + 1], d_lo);
                    v[4 * jw + 2] = hmul2_u32(v[4 * jw + 2], d_up);
                    v[4 * jw + 3] = hmul2_u32(v[4 * jw + 3], d_lo);
                }
                tmem_st_16x32cols_128b(taddr_band + slot * 128u + (uint32_t)(32 * h), v);
            }
            // the stage's x, in place, times 1 / s where that is folded in
            ok = mbar_wait(x_full(stage), phase, ctl) && ok;
            if (!__all_sync(0xFFFFFFFFu, ok)) break;
            if (x_active) {
                unsigned char* st = base_ptr + so;
                const int kb_valid = to_last == 0 ? last_kb : kStTiles;
#pragma unroll
                for (int p = 0; p < kStTiles / kKbPerPass; ++p) {
                    const int kb = p * kKbPerPass + xkb;
                    if (kb >= kb_valid) break;                   // zeros stay zeros
                    unsigned char* row = st + kb * (Cfg::kHalf * 128) + xm * 128;
                    uint4* c0 = reinterpret_cast<uint4*>(row + (((2 * xj) ^ (xm & 7)) << 4));
                    uint4* c1 = reinterpret_cast<uint4*>(row + (((2 * xj + 1) ^ (xm & 7)) << 4));
                    uint4 a = *c0, b = *c1;
                    if (XS) {
                        const float4* is = reinterpret_cast<const float4*>(st + Cfg::kInvOff) + (kb * kBK + xj * 16) / 4;
                        const float4 i0 = is[0], i1 = is[1], i2 = is[2], i3 = is[3];
                        a.x = scale_pair(a.x, make_float2(i0.x, i0.y)); a.y = scale_pair(a.y, make_float2(i0.z, i0.w));
                        a.z = scale_pair(a.z, make_float2(i1.x, i1.y)); a.w = scale_pair(a.w, make_float2(i1.z, i1.w));
                        b.x = scale_pair(b.x, make_float2(i2.x, i2.y)); b.y = scale_pair(b.y, make_float2(i2.z, i2.w));
                        b.z = scale_pair(b.z, make_float2(i3.x, i3.y)); b.w = scale_pair(b.w, make_float2(i3.z, i3.w));
                    }
                    *c0 = make_uint4(a.x, a.z, b.x, b.z);        // pairs 0 2 4 6
                    *c1 = make_uint4(a.y, a.w, b.y, b.w);        // pairs 1 3 5 7
                }
                fence_proxy_async_smem();                        // the products read x through the asynchronous proxy
            }
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(leader_a_full0 + 8u * slot);
            stage += 2;
            if (stage >= (uint32_t)S) { stage -= S; phase ^= 1u; }
            old += 2;
            if (old >= kOldRing) { old -= kOldRing; old_phase ^= 1u; }
            slot += 2;
            if (slot >= (uint32_t)SL) slot -= SL;
            to_last -= 2;
            while (to_last < 0) to_last += nks;
        }
    } else if (warp >= 4) {
        // ------------------------------------------------------------ epilogue
        // warp (quad, half): 32 of the block's channels x half of the tile's tokens
        asm volatile("griddepcontrol.wait;" ::: "memory");
        const int quad = warp & 3, thalf = warp >= 24 ? 1 : 0;
        const uint32_t taddr0 = tmem_base + ((uint32_t)(quad * 32) << 16);
        const uint32_t leader_acc_empty0 = map_to_rank(acc_empty(0), 0);
        const unsigned char* sc_lane = base_ptr + Cfg::kParOff + (2 * quad + (lane >> 4)) * (GPS * 32) + (lane & 15) * 2;
        uint32_t acc = 0, acc_phase = 0, stage = 0, phase = 0;
        bool ok = true;
        const int tok0 = thalf * (EXACT ? Cfg::kEpTokens : half_rows);               // this warp's first token of a tile
        int tile = range.tile, k0 = range.ks;
        for (int left = range.count; left > 0 && ok; ++tile, k0 = 0) {
            const int k1 = min(nks, k0 + left);
            left -= k1 - k0;
            const bool whole = k0 == 0 && k1 == nks;
            const StTile at = st_tile(cut, tile);
            const int N = cut.n[at.mi], ch0 = at.slab * 256 + (int)rank * 128;      // this block's first channel
            const int rows = min(cut.bn, cut.M - at.mt * cut.bn);                   // tokens of the tile that are there
            __half* y = cut.y[at.mi] + (size_t)(at.mt * cut.bn) * N + ch0;
            float* mine = partial + st_slot(cut, 2 * pair + (k0 == 0 ? 1 : 0), (int)rank) + (size_t)tok0 * 128 + quad * 32 + lane;
            if constexpr (EXACT) {
                constexpr int TH = Cfg::kEpTokens;
                float v[TH];
#pragma unroll
                for (int i = 0; i < TH; ++i) v[i] = 0.0f;
                for (int ks = k0; ks < k1 && ok; ++ks) {
                    // Delta of this lane's channel: row lane % 16 of band 2 quad + lane / 16
                    ok = __all_sync(0xFFFFFFFFu, mbar_wait(w_full(stage), phase, ctl));
                    if (!ok) break;
                    float d[GPS];
#pragma unroll
                    for (int q = 0; q < GPS; ++q)
                        d[q] = __half2float(*reinterpret_cast<const __half*>(sc_lane + x_off(stage) + q * 32));
                    __syncwarp();
                    if (lane == 0) mbar_arrive(empty(stage));    // (with the products' commit it frees the stage)
#pragma unroll
                    for (int q = 0; q < GPS; q += 2) {
                        ok = __all_sync(0xFFFFFFFFu, mbar_wait(acc_full(acc), acc_phase, ctl));
                        if (!ok) break;
                        tc_fence_after();
                        uint32_t r0[TH], r1[TH];
                        const uint32_t t0 = taddr0 + acc * Cfg::kAccCols + (uint32_t)tok0;
                        tmem_ld_cols<TH>(t0, r0);
                        tmem_ld_cols<TH>(t0 + (uint32_t)BN, r1);
                        tmem_ld_wait(r0, r1);
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive_cluster(leader_acc_empty0 + 8u * acc);
#pragma unroll
                        for (int i = 0; i < TH; i += 2) fma_pair(v[i], v[i + 1], d[q], r0[i], r0[i + 1]);
#pragma unroll
                        for (int i = 0; i < TH; i += 2) fma_pair(v[i], v[i + 1], d[q + 1], r1[i], r1[i + 1]);
                        if (++acc == NACC) { acc = 0; acc_phase ^= 1u; }
                    }
                    if (++stage == (uint32_t)S) { stage = 0; phase ^= 1u; }
                }
                if (!ok) break;
                if (!whole) {
#pragma unroll
                    for (int i = 0; i < TH; ++i)
                        if (tok0 + i < rows) __stcg(mine + (size_t)i * 128, v[i]);
                } else if (ch0 < N) {
#pragma unroll
                    for (int i = 0; i < TH; ++i)
                        if (tok0 + i < rows) y[(size_t)(tok0 + i) * N + quad * 32 + lane] = __float2half_rn(v[i]);
                }
            } else {
                const int th = half_rows, my_rows = min(th, rows - tok0);       // (may be none)
                unsigned char* out = base_ptr + kOutOff + (thalf * 4 + quad) * 2048;
                // 32 tokens x 32 channels through shared memory: 16 bytes of a token per lane and store
                auto store = [&](int c, const float (&v)[32]) {
                    if (ch0 >= N) return;
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < 32; ++i)
                        *reinterpret_cast<__half*>(out + i * 64 + lane * 2) = __float2half_rn(v[i]);
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int t = i * 8 + (lane >> 2);
                        if (c + t < my_rows)
                            *reinterpret_cast<uint4*>(y + (size_t)(tok0 + c + t) * N + quad * 32 + (lane & 3) * 8) =
                                *reinterpret_cast<const uint4*>(out + t * 64 + (lane & 3) * 16);
                    }
                };
                ok = __all_sync(0xFFFFFFFFu, mbar_wait(acc_full(acc), acc_phase, ctl));
                if (!ok) break;
                tc_fence_after();
#pragma unroll 1
                for (int c = 0; c < th; c += 32) {
                    uint32_t r[32];
                    tmem_ld_32cols(taddr0 + acc * Cfg::kAccCols + (uint32_t)(tok0 + c), r);
                    tmem_ld_wait(r);
                    if (c + 32 >= th) {
                        // the accumulator is in registers: the next part's products may overwrite it
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive_cluster(leader_acc_empty0 + 8u * acc);
                    }
                    if (whole) {
                        float v[32];
#pragma unroll
                        for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
                        store(c, v);
                    } else {
#pragma unroll
                        for (int i = 0; i < 32; ++i)
                            if (c + i < my_rows) __stcg(mine + (size_t)(c + i) * 128, __uint_as_float(r[i]));
                    }
                }
                if (++acc == NACC) { acc = 0; acc_phase ^= 1u; }
            }
        }
    }

    __syncwarp();
    if (warp == 0 || warp == 2) cluster_wait();
    tc_fence_before();
    __syncthreads();
    cluster_sync_end(*ctl.abort != 0u);      // nothing of the pair still refers to this block
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    }
}

__device__ __forceinline__ void add4(float4& a, const float4& b) { a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w; }
// The parts of a cut tile, added in a fixed order: block x = (tile, rank), 4 R tokens per block y, four channels of R tokens a thread.
template <int R>
__global__ void __launch_bounds__(128, 8)
stream_reduce_kernel(const __grid_constant__ StCut cut, const float* partial) {
    // launched with programmatic stream serialization behind the kernel above: it may be resident before that
    // kernel has finished (so the sums are read through L2), and lets the launch behind it start its own copies
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int tile = blockIdx.x >> 1, rank = blockIdx.x & 1;
    const int owner = st_pair_of(cut, tile * cut.nks), parts = st_pair_of(cut, tile * cut.nks + cut.nks - 1) - owner + 1;
    const StTile at = st_tile(cut, tile);
    const int row0 = blockIdx.y * (4 * R) + (threadIdx.x >> 5), c4 = (threadIdx.x & 31) * 4;
    const int N = cut.n[at.mi], ch = at.slab * 256 + rank * 128 + c4;
    const int rows = min(cut.bn, cut.M - at.mt * cut.bn);
    const size_t step = 2 * st_slot(cut, 1, 0);                  // from a pair's slot to the next pair's
    const float* first = partial + c4 + st_slot(cut, 2 * owner + 1, rank);
    const float* others = partial + c4 + st_slot(cut, 2 * (owner + 1), rank);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (parts == 1 || ch >= N) return;
    float4 sum[R];
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (row0 + 4 * r < rows) sum[r] = __ldcg(reinterpret_cast<const float4*>(first + (row0 + 4 * r) * 128));
    constexpr int B = 8 / R;
    for (int p = 1; p < parts; p += B) {
        float4 v[B][R];
#pragma unroll
        for (int i = 0; i < B; ++i)
#pragma unroll
            for (int r = 0; r < R; ++r)
                v[i][r] = p + i < parts && row0 + 4 * r < rows
                              ? __ldcg(reinterpret_cast<const float4*>(others + (size_t)(p - 1 + i) * step + (row0 + 4 * r) * 128))
                              : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        // neighbours first, then neighbouring sums: fewer roundings act on each part than one after the other
#pragma unroll
        for (int w = 1; w < B; w *= 2)
#pragma unroll
            for (int i = 0; i + w < B; i += 2 * w)
#pragma unroll
                for (int r = 0; r < R; ++r) add4(v[i][r], v[i + w][r]);
#pragma unroll
        for (int r = 0; r < R; ++r) add4(sum[r], v[0][r]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (row0 + 4 * r >= rows) break;
        const __half2 lo = __floats2half2_rn(sum[r].x, sum[r].y), hi = __floats2half2_rn(sum[r].z, sum[r].w);
        uint2 o;
        o.x = *reinterpret_cast<const uint32_t*>(&lo);
        o.y = *reinterpret_cast<const uint32_t*>(&hi);
        *reinterpret_cast<uint2*>(cut.y[at.mi] + (size_t)(at.mt * cut.bn + row0 + 4 * r) * N + ch) = o;
    }
}

// ------------------------------------------------------------------------------ host
int st_tile_tokens(int M) {                              // tokens per tile: a multiple of 16 up to 128
    if (M <= 32) return M <= 16 ? 16 : 32;
    const int tiles = (M + 127) / 128;
    return ((M + tiles - 1) / tiles + 15) / 16 * 16;
}

// pairs that can be resident at once on the current device (0 if the query fails); cached once there is one
template <int G, int BN, bool XS, int TB>
cudaError_t st_resident_pairs(int sms, int* out) {
    static std::mutex mutex;
    static bool done[64] = {};
    static int pairs[64] = {};
    using Cfg = StCfg<BN, XS>;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    dev &= 63;
    std::lock_guard<std::mutex> lock(mutex);
    if (!done[dev]) {
        e = cudaFuncSetAttribute(gemm_stream_kernel<G, BN, XS, TB>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::kSmemBytes);
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3((unsigned)(sms & ~1));
        cfg.blockDim = dim3(Cfg::kThreads);
        cfg.dynamicSmemBytes = Cfg::kSmemBytes;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, gemm_stream_kernel<G, BN, XS, TB>, &cfg) != cudaSuccess) {
            (void)cudaGetLastError();
            n = 0;
        }
        pairs[dev] = n < sms / 2 ? n : sms / 2;          // (what the workspace is sized for)
        done[dev] = n > 0;
    }
    *out = pairs[dev];
    return cudaSuccess;
}

template <int G, int BN, bool XS, int TB = kStBlockBytes>
cudaError_t st_launch(const CUtensorMap& xmap, const StMats& mats, const float* inv_s, StCut cut,
                      void* workspace, unsigned int* status_word, int sms, bool serialize, cudaStream_t st) {
    int resident = 0;
    cudaError_t e = st_resident_pairs<G, BN, XS, TB>(sms, &resident);
    if (e != cudaSuccess) return e;
    if (resident < 1) return cudaErrorNotSupported;          // the caller's cue to take another kernel
    cut.pairs = cut.total < resident ? cut.total : resident;
    cut.share = cut.total / cut.pairs;
    cut.longer = cut.total % cut.pairs;
    // no tile is cut where every range starts at a tile, as all do where a tile is one stage
    const bool second = cut.nks > 1 && (cut.longer != 0 || cut.share % cut.nks != 0);
    float* partial = reinterpret_cast<float*>(static_cast<unsigned char*>(workspace) + kCounterBytes);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3((unsigned)(2 * cut.pairs));
    cfg.blockDim = dim3(StCfg<BN, XS>::kThreads);
    cfg.dynamicSmemBytes = StCfg<BN, XS>::kSmemBytes;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = serialize ? 1 : 2;
    e = cudaLaunchKernelEx(&cfg, gemm_stream_kernel<G, BN, XS, TB>, cut, inv_s, partial, status_word, xmap, mats);
    if (e != cudaSuccess) return e;
    count_launch();
    if (!second) return cudaGetLastError();
    // Its blocks run beside the kernel's as soon as there are (one fits per SM), so where they can they all do.
    int per = 1;
    while (per < 4 && 2 * cut.tiles * ((cut.rows + 4 * per - 1) / (4 * per)) > sms) per *= 2;
    if (2 * cut.tiles * ((cut.rows + 4 * per - 1) / (4 * per)) > sms) per = 1;
    cfg.gridDim = dim3((unsigned)(2 * cut.tiles), (unsigned)((cut.rows + 4 * per - 1) / (4 * per)));
    cfg.blockDim = dim3(128);
    cfg.dynamicSmemBytes = 0;
    cfg.attrs = attr + 1;
    cfg.numAttrs = 1;
    auto* reduce = per == 1 ? stream_reduce_kernel<1> : per == 2 ? stream_reduce_kernel<2> : stream_reduce_kernel<4>;
    e = cudaLaunchKernelEx(&cfg, reduce, cut, (const float*)partial);
    if (e != cudaSuccess) return e;
    count_launch();
    return cudaGetLastError();
}

}  // namespace

bool gemm_stream_applies(int M, int N, int K, int group) {
    return M >= 1 && N % 128 == 0 && K % 128 == 0 && (group == 64 || group == 128) && encode_fn() != nullptr;
}

size_t gemm_stream_workspace_bytes(int M, int sms) {
    const int bn = st_tile_tokens(M);
    return kCounterBytes + (size_t)(sms / 2) * 2 * 256 * (bn < M ? bn : M) * sizeof(float);
}

// Estimated time above 64 tokens, us: start, stages of the longest range, the parts that a pair leaves, and how many of them
// make up a tile.  A fit to 70 / 100 / 128 / 192 / 256 tokens on 7 shapes (2048 -> 2048 .. 28672 -> 8192); on 36 other problems
// (N 1024 .. 28672, K 1024 .. 28672, 65 .. 224 tokens) it is 5 % off on average.
double gemm_stream_estimate(int M, int slabs, int K, int sms) {
    const int bn = st_tile_tokens(M), nks = (K + kStStageK - 1) / kStStageK;
    const long long total = (long long)slabs * ((M + bn - 1) / bn) * nks, pairs = sms / 2;
    const double share = total < pairs ? 1.0 : (double)total / (double)pairs;
    const double parts = 1.0 + (share < nks ? share / nks : 1.0), per_tile = (double)nks / share;
    return 1.6 + (double)((long long)(share + 0.999)) * (0.45 + 0.0048 * bn) + (2.63 + 0.0208 * bn) * parts + 0.1 * per_tile;
}

cudaError_t launch_gemm_stream(const void* x, const GemvMatrix* mats, int count, int M, int K, int group,
                               const float* inv_s, void* workspace, unsigned int* status_word, int sms,
                               bool serialize, cudaStream_t st, int bits) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return cudaErrorNotSupported;
    StCut cut = {};
    cut.bn = st_tile_tokens(M);
    cut.rows = cut.bn < M ? cut.bn : M;
    cut.m_tiles = (M + cut.bn - 1) / cut.bn;
    cut.M = M;
    cut.K = K;
    cut.nks = (K + kStStageK - 1) / kStStageK;
    cut.inv_nks = 1.0f / (float)cut.nks;
    const int cls = cut.bn <= 16 ? 16 : cut.bn <= 32 ? 32 : cut.bn <= 64 ? 64 : 128;
    CUtensorMap xmap;
    StMats sm;
    {
        // x as [k-block][token][64] fp16 in boxes of four k-blocks x half of the most tokens of a tile (its own may be fewer), 128-byte swizzle; rows past M
        // and k-blocks past K read as zeros
        const cuuint64_t dims[3] = {(cuuint64_t)kBK, (cuuint64_t)M, (cuuint64_t)(K / kBK)};
        const cuuint64_t strides[2] = {(cuuint64_t)K * 2, (cuuint64_t)kBK * 2};
        const cuuint32_t box[3] = {(cuuint32_t)kBK, (cuuint32_t)(cls / 2), (cuuint32_t)kStTiles}, estr[3] = {1, 1, 1};
        if (enc(&xmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<void*>(x), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    int slabs = 0;
    for (int i = 0; i < kMaxMulti; ++i) {
        const GemvMatrix& m = mats[i < count ? i : 0];
        if (i < count) {
            slabs += (m.n + 255) / 256;
            // packed weights: one row of K * 8 (3-bit storage: K * 6) bytes per band, as 64-bit elements; boxes of 8 bands x 4 k-blocks
            const int per_block = bits * 16;             // 64-bit elements of a band's k-block
            const cuuint64_t wdims[2] = {(cuuint64_t)(K / kBK) * per_block, (cuuint64_t)(m.n / 16)}, wstr[1] = {wdims[0] * 8};
            const cuuint32_t wbox[2] = {(cuuint32_t)(kStTiles * per_block), 8}, estr[2] = {1, 1};
            if (enc(&sm.w[i], CU_TENSOR_MAP_DATA_TYPE_UINT64, 2, const_cast<void*>(m.qweight), wdims, wstr, wbox, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
                return cudaErrorInvalidValue;
            // scales: fp16 [band][group][16], zero points: bytes [band pair][group][16]; boxes of a stage's groups
            const int ng = K / group, gps = kStStageK / group;
            const cuuint64_t sdims[2] = {(cuuint64_t)ng * 16, (cuuint64_t)(m.n / 16)}, sstr[1] = {(cuuint64_t)ng * 32};
            const cuuint64_t zdims[2] = {(cuuint64_t)ng * 16, (cuuint64_t)(m.n / 32)}, zstr[1] = {(cuuint64_t)ng * 16};
            const cuuint32_t sbox[2] = {(cuuint32_t)(gps * 16), 8}, zbox[2] = {(cuuint32_t)(gps * 16), 4};
            if (enc(&sm.sc[i], CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void*>(m.scales), sdims, sstr, sbox, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS ||
                enc(&sm.z[i], CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(m.zeros), zdims, zstr, zbox, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
                return cudaErrorInvalidValue;
        } else {
            sm.w[i] = sm.w[0]; sm.sc[i] = sm.sc[0]; sm.z[i] = sm.z[0];      // never used
        }
        cut.y[i] = static_cast<__half*>(m.y);
        cut.n[i] = m.n;
        cut.slab_end[i] = slabs;
    }
    if ((long long)slabs * cut.m_tiles * cut.nks > (1LL << 22)) return cudaErrorInvalidValue;
    cut.tiles = slabs * cut.m_tiles;
    cut.total = cut.tiles * cut.nks;
    if (bits == 3) {                                     // (up to 64 tokens, nothing folded in)
        if (inv_s || cls > 64) return cudaErrorInvalidValue;
#define AWQ_ST_LAUNCH3(GG, BNN) return st_launch<GG, BNN, false, 384>(xmap, sm, inv_s, cut, workspace, status_word, sms, serialize, st)
        if (group == 128) { if (cls == 16) AWQ_ST_LAUNCH3(128, 16); if (cls == 32) AWQ_ST_LAUNCH3(128, 32); AWQ_ST_LAUNCH3(128, 64); }
        if (cls == 16) AWQ_ST_LAUNCH3(64, 16); if (cls == 32) AWQ_ST_LAUNCH3(64, 32); AWQ_ST_LAUNCH3(64, 64);
#undef AWQ_ST_LAUNCH3
    }
#define AWQ_ST_LAUNCH(GG, BNN)                                                                                             \
    return inv_s ? st_launch<GG, BNN, true>(xmap, sm, inv_s, cut, workspace, status_word, sms, serialize, st)       \
                 : st_launch<GG, BNN, false>(xmap, sm, inv_s, cut, workspace, status_word, sms, serialize, st)
    if (group == 128) {
        switch (cls) { case 16: AWQ_ST_LAUNCH(128, 16); case 32: AWQ_ST_LAUNCH(128, 32);
                       case 64: AWQ_ST_LAUNCH(128, 64); default: AWQ_ST_LAUNCH(128, 128); }
    }
    switch (cls) { case 16: AWQ_ST_LAUNCH(64, 16); case 32: AWQ_ST_LAUNCH(64, 32);
                   case 64: AWQ_ST_LAUNCH(64, 64); default: AWQ_ST_LAUNCH(64, 128); }
#undef AWQ_ST_LAUNCH
}

}  // namespace awq
