// Prefill path of the layer for large token counts (Sec. 4.2: fused dequantize + matrix-matrix
// product): the dataflow of gemm_tcgen05.cu, run by PAIRS of thread blocks (a cluster of two SMs)
// that issue one tcgen05.mma.cta_group::2 of M = 256 output channels x N = 64 .. 256 tokens.
//
// Why pairs, and why 128-channel stages.  With one block per 128 x 256 tile every 64-wide k-block
// moves 72 KB through shared memory and costs the MMA-issuing warp two barrier polls, four MMAs and a
// commit: it, not the tensor pipe (one 128 x 256 x 16 MMA per 128 cycles), set the pace.  In a pair
// each block stages only its half of the tokens (the tensor cores of both SMs read both halves), and
// a stage covers K = 128, so the polls and commits are paid once per eight MMAs.
// Tiles are 64, 128, 192 or 256 tokens wide (choose_tile).  At 256 a stage takes ~1070 cycles against the
// pipe's 1024.  Narrower tiles are bound by the dequantizers (~620 cycles a stage, whatever the
// width up to 128: the conversion's instructions and the tensor-memory stores) once nothing waits: sixteen
// dequantizer warps, and a ring of up to eight stages in shared memory behind the four whose A is in tensor
// memory (128 tokens, one tile per pair, 108 stages: 55 us with four stages, 42 us with eight; 256 tokens gain
// nothing from a fifth).
//
// The start of a launch: chained to the one in front by programmatic dependent launch, weight copies (a warp of their own, x's are
// another's) issued before tensor memory and the cluster are ready.  Chained calls, before and after: 333 tokens on
// 4096 -> 4096 19.3 -> 15.7 us, 700 on 2048 -> 2048 13.5 -> 10.7, 100 on 5120 -> 13824 22.7 -> 19.2.
//
// Block r of a pair (r = rank in the cluster) owns
//   - A: output channels 128 r .. 128 r + 127 of the 256-channel slab, dequantized by its own
//        warps into its own tensor memory (64 columns per stage),
//   - B: its half of the tile's tokens in its own shared memory (two 64-wide 128-byte-swizzled
//        halves per stage),
//   - D: the fp32 accumulator rows of its 128 channels x all tokens in its own tensor memory (two of them
//        up to 128 tokens), drained by its own epilogue warps (half of the tokens each four).
// Only the leader (rank 0) issues MMAs.  Barriers that the leader's MMA thread waits on live in the
// leader's shared memory: x_full (both blocks' x copies complete their bytes there), a_full (16
// dequantizer warps, 8 of each block), acc_empty (16 epilogue warps).  The MMA
// thread's tcgen05.commit arrives on "empty" and "acc_full" of BOTH blocks.
//
// Tile balance: with a workspace, and when whole tiles would leave pairs idle for long, the tiles'
// K loops are cut into equal ranges over the pairs (stream-K, see PieceIter and the epilogue).
//
// Every wait is bounded (about two seconds): a wait that runs out writes a code to the status word
// and every role of that block leaves its loop; the other block of the pair then runs into its
// own limits.  Both blocks meet at a cluster barrier before they free tensor memory and exit, so
// that no remote arrival can land in the shared memory of a block that has already gone.
#include "tcgen05.cuh"

namespace awq {

namespace {

constexpr int kStageK = 128;                     // input channels per pipeline stage (two k-tiles)

// BN = tokens per tile (N of the MMA); each block stages half of them
template <int BN> struct PairCfg {
    // 256 tokens: a stage's products take 1024 cycles, eight dequantizer warps (one per band) keep up; with
    // fewer tokens sixteen, every second stage each, so that a warp's chain of latencies spans two stages
    static constexpr int kDequantWarps = BN >= 256 ? 8 : 16;
    static constexpr int kEpilogueWarp1 = 8 + kDequantWarps;                 // first warp of the second epilogue half
    static constexpr int kThreads = (kEpilogueWarp1 + 4) * 32;               // warps: 0 copy, 1 MMA, 4-7 epilogue, 8.. dequant, 4 epilogue
    static constexpr int kHalf = BN / 2;                                     // tokens staged by each block, and per epilogue half
    static constexpr int kXHalfBytes = kHalf * kBK * 2;                      // one 64-wide swizzled half
    static constexpr int kXTileBytes = 2 * kXHalfBytes;                      // BN / 2 tokens x 128 channels
    static constexpr int kWBytes = 2 * kTileBytes;                           // 8 bands x 2 k-tiles x 512 bytes
    static constexpr int kStageBytes = kXTileBytes + kWBytes;                // 40 KB at 256 tokens
    static constexpr int kOutBytes = 8 * 2 * 2048;                           // 8 epilogue warps x 2 staging blocks
    static constexpr int kStages = BN >= 256 ? 4 : BN >= 192 ? 6 : 8;        // what shared memory holds
    static constexpr int kSlots = 4;                                         // stages whose A is in tensor memory
    static constexpr uint32_t kNumAcc = BN <= 128 ? 2 : 1;                   // accumulators in tensor memory
    static constexpr int kAColumn0 = 256;                                    // tensor memory: accumulators, then A
    static constexpr int kAColsPerStage = 64;                                // 8 columns per K = 16
    static constexpr int kTmemCols = 512;                                    // 256 + kSlots x 64
    static constexpr int kSmemBytes = kStages * kStageBytes + kOutBytes + 1024 /*align*/ + 512 /*barriers*/;
    static constexpr int kPartialFloats = 256 * BN;                          // one pair's fp32 accumulator
};

// ---------------------------------------------------------------- cluster-scope PTX wrappers
// x tile copy whose bytes are counted on a barrier of the pair's leader
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int c0, int c1,
                                                 uint32_t leader_bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(leader_bar) : "memory");
}
// arrives on ONE barrier (a shared::cluster address) when the pair's MMAs issued so far are done
__device__ __forceinline__ void umma_pair_commit(uint32_t cluster_bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                 ::"r"(cluster_bar) : "memory");
}
__host__ __device__ constexpr uint32_t instr_desc_pair(int bn) {     // D fp32, A/B fp16 K-major, M = 256, N = bn
    return (1u << 4) | ((uint32_t)(bn >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
}

// Work of one pair: a sequence of pieces (tile, stages k0 .. k1-1 of the tile's K / 128).
// Without a workspace every piece is a whole tile and tiles go round-robin over the pairs.
// With one ("stream-K"), the tiles' stages are laid end to end and cut into equal contiguous
// ranges, one per pair, so that all pairs finish together whatever the tile count; a tile that
// a cut splits is summed up by the pair that holds its first stages (see the epilogue).
struct PieceIter {
    long long s, s_end;              // stream-K: global stage range still to do
    int tile, tile_step, total_tiles, nks;
    bool streamk;
    __device__ bool next(int& t, int& k0, int& k1) {
        if (streamk) {
            if (s >= s_end) return false;
            t = (int)(s / nks);
            k0 = (int)(s - (long long)t * nks);
            const long long left = s_end - s;
            k1 = left < (long long)(nks - k0) ? k0 + (int)left : nks;
            s += k1 - k0;
            return true;
        }
        if (tile >= total_tiles) return false;
        t = tile; k0 = 0; k1 = nks;
        tile += tile_step;
        return true;
    }
};
// first global stage of pair c when `total` stages are cut into `C` ranges that differ by at most one
__device__ __forceinline__ long long range_start(long long total, int C, int c) {
    const long long q = total / C, r = total % C;
    return (long long)c * q + (c < r ? c : r);
}
__device__ __forceinline__ unsigned int ld_acquire_u32(const unsigned int* p) {
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Several products of the same shape end to end (the scale search): their channels stacked in the packed arrays, each with
// `rows` rows of x and y of its own.  One product: all slabs, rows 0.
struct PairBlocks {
    int slabs;                       // 256-channel slabs of a product
    int n;                           // its channels
    int rows;                        // rows from a product's x (and y) to the next one's
};

// ------------------------------------------------------------------------- the kernel
template <int G, int BN>
__global__ void __launch_bounds__(PairCfg<BN>::kThreads, 1)
gemm_pair_kernel(const __grid_constant__ CUtensorMap x_map, const __grid_constant__ CUtensorMap w_map,
                 const __grid_constant__ CUtensorMap y_map,
                 const __half* __restrict__ scales, const unsigned char* __restrict__ zeros,
                 int M, int N, int K, unsigned int* status_word,
                 float* partials, unsigned int* flags, const PairBlocks blocks) {
    using Cfg = PairCfg<BN>;
    constexpr int S = Cfg::kStages, SL = Cfg::kSlots;
    constexpr uint32_t NACC = Cfg::kNumAcc;
    constexpr int GPS = kStageK / G;                 // quantization groups per stage: 1 or 2
    extern __shared__ unsigned char smem_dyn[];
    __shared__ unsigned int s_abort;
    __shared__ uint32_t s_tmem_base;

    const uint32_t dyn = smem_u32(smem_dyn);
    const uint32_t base = (dyn + 1023u) & ~1023u;                    // 1024-byte aligned stage ring
    unsigned char* base_ptr = smem_dyn + (base - dyn);
    // stage layout: [x, k-half 0 (BN / 2 tokens x 64) | x, k-half 1 | packed weights (8 bands x 1 KB)]
    auto x_addr = [&](int s) { return base + (uint32_t)s * Cfg::kStageBytes; };
    auto w_ptr = [&](int s) { return base_ptr + (size_t)s * Cfg::kStageBytes + Cfg::kXTileBytes; };
    const uint32_t out_base = base + (uint32_t)S * Cfg::kStageBytes;
    const uint32_t bars = out_base + (uint32_t)Cfg::kOutBytes;
    auto w_full = [&](int s) { return bars + 8u * (uint32_t)s; };               // own weights landed
    auto x_full = [&](int s) { return bars + 8u * (uint32_t)(S + s); };         // leader: both blocks' x landed
    auto empty = [&](int s) { return bars + 8u * (uint32_t)(2 * S + s); };      // stage free again: its products are done
    auto a_full = [&](int s) { return bars + 8u * (uint32_t)(3 * S + s); };     // leader: both blocks' A stored (per slot)
    auto acc_full = [&](uint32_t b) { return bars + 8u * ((uint32_t)(3 * S + SL) + b); };        // accumulator complete
    auto acc_empty = [&](uint32_t b) { return bars + 8u * ((uint32_t)(3 * S + SL + 2) + b); };   // leader: accumulator drained

    // (the shuffle tells the compiler that all lanes of a warp take the same role: addresses stay in uniform registers)
    const int warp = __shfl_sync(0xFFFFFFFFu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const int m_tiles = (M + BN - 1) / BN;
    const int total_tiles = ((N + 255) / 256) * m_tiles;     // an odd last slab of 128 channels pairs with an absent one
    const int cluster = (int)cluster_id_x(), num_clusters = (int)num_clusters_x();
    const int nks = K / kStageK;                     // stages per tile
    const long long total_stages = (long long)total_tiles * nks;
    PieceIter pieces;
    pieces.streamk = partials != nullptr;
    pieces.s = range_start(total_stages, num_clusters, cluster);
    pieces.s_end = range_start(total_stages, num_clusters, cluster + 1);
    pieces.tile = cluster; pieces.tile_step = num_clusters; pieces.total_tiles = total_tiles; pieces.nks = nks;
    int tile, k0, k1;

    // the weight copies need nothing but their own block's barriers: they start before tensor memory and the cluster are ready
    if (warp == 0) {
        if (lane == 0) {
            s_abort = 0u;
            for (int s = 0; s < S; ++s) {
                mbar_init(w_full(s), 1); mbar_init(x_full(s), 1); mbar_init(empty(s), 1);
            }
            for (int s = 0; s < SL; ++s) mbar_init(a_full(s), 16);
            for (uint32_t b = 0; b < NACC; ++b) { mbar_init(acc_full(b), 1); mbar_init(acc_empty(b), 16); }
            mbar_fence_init();
        }
        __syncwarp();
        asm volatile("bar.arrive 1, %0;" ::"r"(Cfg::kThreads) : "memory");
        cluster_arrive_start();
    } else {
        if (warp == 1) {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                         ::"r"(smem_u32(&s_tmem_base)), "r"((uint32_t)Cfg::kTmemCols) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
            tc_fence_before();
        }
        named_barrier_sync(1, Cfg::kThreads);
        cluster_arrive_start();
        cluster_wait();                      // both blocks' barriers exist before anyone arrives remotely
        tc_fence_after();
    }
    constexpr uint32_t tmem_base = 0;        // all 512 columns are this block's
    const WaitCtl ctl{status_word, &s_abort};
    // programmatic dependent launch: the packed arrays are constants of the layer and are read before the work in front of
    // this launch has completed; x is read and y and the workspace are written after it
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (warp == 0) {
        // ------------------------------------------------------------------ weight copies
        const bool lead = elect_one();
        uint32_t stage = 0, phase = 0;
        unsigned int issued = 0;
        bool ok = true;
        while (ok && pieces.next(tile, k0, k1)) {
            const int slab = (tile / m_tiles) * 2 + (int)rank;              // 128-channel slab of this block
            for (int ks = k0; ks < k1; ++ks) {
                if (!mbar_wait_warp(empty(stage), phase ^ 1u, ctl)) { ok = false; break; }
                if (lead) {
                    const uint32_t bar = w_full(stage);
                    mbar_arrive_expect_tx(bar, (uint32_t)Cfg::kWBytes);
                    // weights: box of 8 bands x 1 KB (256 words: two k-tiles) at (stage, first band)
                    tma_load_2d(x_addr(stage) + Cfg::kXTileBytes, &w_map, ks * 256, slab * 8, bar);
                }
                __syncwarp();
                ++issued;
                if (++stage == S) { stage = 0; phase ^= 1u; }
            }
        }
        if (!ok) {
            // giving up: let the copies already issued land before the block exits
            const unsigned int pending = issued < (unsigned)S ? issued : (unsigned)S;
            uint32_t st = stage, ph = phase;
            for (unsigned int i = 0; i < pending; ++i) {
                if (st == 0) { st = S - 1; ph ^= 1u; } else { --st; }
                const unsigned long long t0 = global_ns();
                while (!mbar_try_wait(w_full(st), ph) && global_ns() - t0 < 100000000ull) {}
            }
        }
    } else if (warp == 2) {
        // ------------------------------------------------------------------ x copies
        const bool lead = elect_one();
        const uint32_t leader_x_full0 = map_to_rank(x_full(0), 0);
        uint32_t stage = 0, phase = 0;
        bool ok = true;
        asm volatile("griddepcontrol.wait;" ::: "memory");
        while (ok && pieces.next(tile, k0, k1)) {
            const int tok0 = (tile / m_tiles / blocks.slabs) * blocks.rows + (tile % m_tiles) * BN + (int)rank * Cfg::kHalf;
            for (int ks = k0; ks < k1; ++ks) {
                if (!mbar_wait_warp(empty(stage), phase ^ 1u, ctl)) { ok = false; break; }
                if (lead) {
                    if (rank == 0) mbar_arrive_expect_tx(x_full(stage), 2u * Cfg::kXTileBytes);
                    const uint32_t xbar = leader_x_full0 + 8u * stage;
                    tma_load_2d_pair(x_addr(stage), &x_map, ks * kStageK, tok0, xbar);
                    tma_load_2d_pair(x_addr(stage) + Cfg::kXHalfBytes, &x_map, ks * kStageK + kBK, tok0, xbar);
                }
                __syncwarp();
                if (++stage == S) { stage = 0; phase ^= 1u; }
            }
        }
        if (!ok) {                                                  // giving up: the x halves are counted on the leader
            const unsigned long long t1 = global_ns();
            while (global_ns() - t1 < 1000000ull) __nanosleep(1000);
        }
    } else if (warp == 1) {
        // ------------------------------------------------- MMA issuer (leader block only)
        if (rank == 0) {
            const bool lead = elect_one();
            constexpr uint32_t idesc = instr_desc_pair(BN);
            const uint32_t peer_acc_full0 = map_to_rank(acc_full(0), 1);
            const uint32_t peer_empty0 = map_to_rank(empty(0), 1);
            uint32_t stage = 0, phase = 0, slot = 0, slot_phase = 0, acc = 0, acc_phase = 0;
            bool ok = true;
            while (ok && pieces.next(tile, k0, k1)) {
                if (!mbar_wait_warp(acc_empty(acc), acc_phase ^ 1u, ctl)) { ok = false; break; }
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + acc * (uint32_t)BN;
                for (int ks = k0; ks < k1; ++ks) {
                    // both barriers are normally complete already: poll them together
                    const bool xr = mbar_try_wait(x_full(stage), phase), ar = mbar_try_wait(a_full(slot), slot_phase);
                    if (!__all_sync(0xFFFFFFFFu, xr && ar) &&
                        (!mbar_wait_warp(x_full(stage), phase, ctl) || !mbar_wait_warp(a_full(slot), slot_phase, ctl))) {
                        ok = false; break;
                    }
                    tc_fence_after();
                    const uint32_t a_tmem = tmem_base + (uint32_t)(Cfg::kAColumn0 + slot * Cfg::kAColsPerStage);
                    const uint64_t bdesc = smem_desc_sw128(x_addr(stage));
                    if (lead) {
#pragma unroll
                        for (int k = 0; k < kStageK / 16; ++k) {
                            // A: 8 columns per K = 16; B: 32 bytes per K = 16 inside a 64-wide half
                            const uint64_t boff = (uint64_t)(((k >> 2) * Cfg::kXHalfBytes + (k & 3) * 32) >> 4);
                            umma_pair_f16_a_tmem(d_tmem, a_tmem + (uint32_t)(8 * k), bdesc + boff, idesc,
                                                 (ks > k0 || k > 0) ? 1u : 0u);
                        }
                        umma_pair_commit(empty(stage));
                        umma_pair_commit(peer_empty0 + 8u * stage);
                    }
                    __syncwarp();
                    if (++stage == S) { stage = 0; phase ^= 1u; }
                    if (++slot == SL) { slot = 0; slot_phase ^= 1u; }
                }
                if (ok && lead) { umma_pair_commit(acc_full(acc)); umma_pair_commit(peer_acc_full0 + 8u * acc); }
                __syncwarp();
                if (++acc == NACC) { acc = 0; acc_phase ^= 1u; }
            }
            // the epilogues' last arrivals, the other block's among them, are waited for here (see cluster_sync_end)
            for (uint32_t b = 0; b < NACC && mbar_wait_warp(acc_empty(acc), acc_phase ^ 1u, ctl); ++b)
                if (++acc == NACC) { acc = 0; acc_phase ^= 1u; }
        }
    } else if (warp >= 8 && warp < Cfg::kEpilogueWarp1) {
        // -------------------------------------------------------------- dequantizers
        // a warp takes a 16-row band of this block's 128 channels, two k-tiles per stage - every stage, or
        // every STEPth of those of all its pieces end to end; see gemm_tcgen05.cu for the piece <-> register layout
        constexpr int STEP = Cfg::kDequantWarps / 8;
        const int wi = warp - 8, quad = wi & 3, hsel = (wi >> 2) & 1;
        const int band = 2 * quad + hsel;
        const int g = lane >> 2;
        const int ng = K / G, bands = N / 16;
        const uint32_t taddr_band = tmem_base + ((uint32_t)(quad * 32 + hsel * 16) << 16) + (uint32_t)Cfg::kAColumn0;
        const uint32_t leader_a_full0 = map_to_rank(a_full(0), 0);
        int first = wi >> 3;                             // this warp's first stage inside the next piece
        uint32_t stage = (uint32_t)first, phase = 0, slot = (uint32_t)first;
        // the slot's previous use was kSlots stages ago: its products are done when that stage is empty
        uint32_t old = (uint32_t)(first + S - SL), old_phase = 1u;     // (both below S: first <= 1, and 0 where S = SL)
        static_assert(S > SL || STEP == 1, "stage index of the slot's previous use");
        bool ok = true;
        while (ok && pieces.next(tile, k0, k1)) {
            // (an absent slab's warps read the last band's parameters for rows that nobody keeps)
            const int gband = min(((tile / m_tiles) * 2 + (int)rank) * 8 + band, bands - 1);
            // this lane's rows' parameters: scales [band][group][16], zero bytes [band pair][group][16]
            const unsigned short* sc_g = reinterpret_cast<const unsigned short*>(scales) + (size_t)gband * ng * 16 + g;
            const unsigned char* z_g = zeros + (size_t)(gband >> 1) * ng * 16 + (gband & 1) * 8 + g;
            // parameters of the current stage's groups and of this warp's next stage's (fetched one ahead)
            uint32_t du[GPS], dl[GPS], zb[GPS], du1[GPS], dl1[GPS], zb1[GPS];
#pragma unroll
            for (int q = 0; q < GPS; ++q) {
                const int g0 = min((k0 + first) * GPS + q, ng - 1);
                du1[q] = __ldg(sc_g + g0 * 16); dl1[q] = __ldg(sc_g + g0 * 16 + 8); zb1[q] = __ldg(z_g + g0 * 16);
            }
            int ks = k0 + first;
            for (; ks < k1; ks += STEP) {
#pragma unroll
                for (int q = 0; q < GPS; ++q) {
                    du[q] = du1[q]; dl[q] = dl1[q]; zb[q] = zb1[q];
                    const int gn = min((ks + STEP) * GPS + q, ng - 1);
                    du1[q] = __ldg(sc_g + gn * 16); dl1[q] = __ldg(sc_g + gn * 16 + 8); zb1[q] = __ldg(z_g + gn * 16);
                }
                ok = mbar_wait(w_full(stage), phase, ctl) && mbar_wait(empty(old), old_phase, ctl);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                tc_fence_after();
#pragma unroll
                for (int h = 0; h < 2; ++h) {                     // the stage's two 64-wide k-tiles
                    const int q = GPS == 2 ? h : 0;
                    const uint4 pk = *reinterpret_cast<const uint4*>(w_ptr(stage) + band * 1024 + h * 512 + lane * 16);
                    const uint32_t d_up = du[q] | (du[q] << 16), d_lo = dl[q] | (dl[q] << 16);
                    const uint32_t zu = 0x6400u + (zb[q] & 0xFu), zl = 0xD400u + ((zb[q] >> 4) << 4);
                    const uint32_t zlo = zu | (zu << 16), zhi = zl | (zl << 16);
                    const uint32_t wds[4] = {pk.x, pk.y, pk.z, pk.w};
                    // per word j: (row g: c, c+1) (row g: c+2, c+3) (row g+8: c, c+1) (row g+8: c+2, c+3)
                    uint32_t v[16];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        constexpr uint32_t kSixteenth = 0x2C002C00u;
                        const uint32_t w = wds[j], w8 = w >> 8;
                        v[4 * j + 0] = hmul2_u32(hsub2_u32(code_pair(w, kLowCodes), zlo), d_up);
                        v[4 * j + 1] = hmul2_u32(hsub2_u32(code_pair(w8, kLowCodes), zlo), d_up);
                        v[4 * j + 2] = hmul2_u32(hfma2_u32(code_pair(w, kHighCodes), kSixteenth, zhi), d_lo);
                        v[4 * j + 3] = hmul2_u32(hfma2_u32(code_pair(w8, kHighCodes), kSixteenth, zhi), d_lo);
                    }
                    tmem_st_16x32cols(taddr_band + slot * (uint32_t)Cfg::kAColsPerStage + 32u * h, v);
                }
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(leader_a_full0 + 8u * slot);
                stage += STEP;
                if (stage >= (uint32_t)S) { stage -= S; phase ^= 1u; }
                old += STEP;
                if (old >= (uint32_t)S) { old -= S; old_phase ^= 1u; }
                slot = (slot + STEP) % SL;
            }
            first = ks - k1;                             // where this warp's stages resume
        }
    } else if (warp >= 4) {
        // ------------------------------------------------------------------ epilogue
        // warps 4-7 drain the first half of the accumulator's token columns, the last four warps the second
        asm volatile("griddepcontrol.wait;" ::: "memory");
        const int quad = warp & 3;                     // TMEM lanes 32*quad .. +31
        const int half = warp >= Cfg::kEpilogueWarp1 ? 1 : 0;
        const uint32_t leader_acc_empty0 = map_to_rank(acc_empty(0), 0);
        // this warp's part of a pair's fp32 partial tile: [rank][warp][chunk][register][lane]
        const size_t part_off = (size_t)((((int)rank * 8 + half * 4 + quad) * (Cfg::kHalf / 32)) * 1024 + lane);
        uint32_t acc = 0, acc_phase = 0;
        int obuf = 0;
        bool ok = true;
        while (ok && pieces.next(tile, k0, k1)) {
            // A piece that does not start the tile is a contribution: its fp32 sums go to this pair's
            // slot of the workspace.  A piece that starts the tile but does not end it waits for the
            // contributions of the pairs after this one (they were produced at the start of those
            // pairs' ranges, long before) and adds them in pair order: the sum is reproducible.
            const bool contributes = k0 > 0;
            int n_contrib = 0;
            if (k0 == 0 && k1 < nks) {
                const long long tile_end = (long long)(tile + 1) * nks;
                while (cluster + 1 + n_contrib < num_clusters &&
                       range_start(total_stages, num_clusters, cluster + 1 + n_contrib) < tile_end)
                    ++n_contrib;
            }
            // while this piece's MMAs run: wait for the contributions (normally there long ago) and
            // fetch the first one's first chunk, so that the drain below does not wait for memory
            for (int j = 0; j < n_contrib && ok; ++j) {
                const unsigned int* f = flags + cluster + 1 + j;
                const unsigned long long t0 = global_ns();
                while (ld_acquire_u32(f) < 16u) {                   // 16 epilogue warps of that pair
                    if (*ctl.abort) { ok = false; break; }
                    if (global_ns() - t0 > wait_limit_ns(ctl)) {
                        *ctl.abort = 1u;
                        atomicExch(ctl.status, kTimeoutCode);
                        ok = false;
                        break;
                    }
                    __nanosleep(64);
                }
            }
            constexpr bool kPrefetch = Cfg::kDequantWarps == 8;     // (with sixteen there are too few registers)
            float p[32];
            const float* src0 = partials + (size_t)(cluster + 1) * Cfg::kPartialFloats + part_off;
            if (kPrefetch && n_contrib > 0 && ok) {
#pragma unroll
                for (int i = 0; i < 32; ++i) p[i] = __ldcg(src0 + i * 32);
            }
            ok = ok && mbar_wait(acc_full(acc), acc_phase, ctl);
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            tc_fence_after();
            int row = (tile % m_tiles) * BN + half * Cfg::kHalf;        // this warp's first token, then its row of y
            const int block = tile / m_tiles / blocks.slabs, n0 = ((tile / m_tiles - block * blocks.slabs) * 2 + (int)rank) * 128 + quad * 32;
            const int rows = n0 < blocks.n ? M - row : 0;               // what there is to store
            row += block * blocks.rows;
            const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + acc * (uint32_t)BN + (uint32_t)(half * Cfg::kHalf);
#pragma unroll 1
            for (int c = 0; c < Cfg::kHalf; c += 32) {
                uint32_t r[32];
                tmem_ld_32cols(taddr + (uint32_t)c, r);
                tmem_ld_wait(r);
                if (c + 32 >= Cfg::kHalf) {
                    // the accumulator is in registers: the MMA thread may start the next piece
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(leader_acc_empty0 + 8u * acc);
                }
                if (contributes) {
                    float* dst = partials + (size_t)cluster * Cfg::kPartialFloats + part_off + (size_t)c * 32;
#pragma unroll
                    for (int i = 0; i < 32; ++i) __stcg(dst + i * 32, __uint_as_float(r[i]));
                    continue;
                }
                if (n_contrib > 0) {
                    if (kPrefetch) {
#pragma unroll
                        for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) + p[i]);
                    }
                    for (int j = kPrefetch ? 1 : 0; j < n_contrib; ++j) {
                        const float* src = src0 + (size_t)j * Cfg::kPartialFloats + (size_t)c * 32;
#pragma unroll
                        for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) + __ldcg(src + i * 32));
                    }
                    if (kPrefetch && c + 32 < Cfg::kHalf) {         // the next chunk of the first contribution
#pragma unroll
                        for (int i = 0; i < 32; ++i) p[i] = __ldcg(src0 + (size_t)(c + 32) * 32 + i * 32);
                    }
                }
                // stage the 32 x 32 block as [token][channel] fp16 and hand it to the copy engine
                // (rows past M are clipped by the tensor map; blocks that lie outside y are left out)
                if (c >= rows) continue;
                if (lane == 0) bulk_wait_read_1();                  // the store that last used this buffer
                __syncwarp();
                const uint32_t tb = out_base + (uint32_t)(((half * 4 + quad) * 2 + obuf) * 2048);
                unsigned char* tp = base_ptr + (tb - base);
#pragma unroll
                for (int i = 0; i < 32; ++i)
                    *reinterpret_cast<__half*>(tp + i * 64 + lane * 2) = __float2half_rn(__uint_as_float(r[i]));
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    tma_store_2d(&y_map, n0, row + c, tb);
                    bulk_commit_group();
                }
                obuf ^= 1;
            }
            if (contributes) {
                __threadfence();                                    // the sums before the flag
                __syncwarp();
                if (lane == 0) atomicAdd(flags + cluster, 1u);
            }
            if (lane == 0) {
                // the 16 readers of a slot count themselves in after the 16 writers; the last one
                // clears the flag, so the workspace is ready for the next launch
                for (int j = 0; j < n_contrib; ++j)
                    if (atomicAdd(flags + cluster + 1 + j, 1u) == 31u) atomicExch(flags + cluster + 1 + j, 0u);
            }
            if (++acc == NACC) { acc = 0; acc_phase ^= 1u; }
        }
        if (lane == 0) bulk_wait_all();                             // all of y written before exit
    }

    __syncwarp();
    if (warp == 0) cluster_wait();
    tc_fence_before();
    __syncthreads();
    cluster_sync_end(*ctl.abort != 0u);      // nothing of the pair still refers to this block
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;"
                     ::"r"(tmem_base), "r"((uint32_t)Cfg::kTmemCols) : "memory");
    }
}

// ------------------------------------------------------------------------------ host
// stream-K's part of the workspace: a flag per pair in its head, one fp32 tile per pair behind that
size_t streamk_bytes(int bn, int pairs) { return kCounterBytes + (size_t)pairs * 256 * bn * sizeof(float); }

// pairs that can be resident at once on the current device (0 if the query fails); cached once there is one
template <int G, int BN>
int resident_pairs(int sms, cudaError_t* err) {
    static bool done[64] = {};
    static int pairs[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    *err = cudaSuccess;
    if (!done[dev & 63]) {
        *err = cudaFuncSetAttribute(gemm_pair_kernel<G, BN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    PairCfg<BN>::kSmemBytes);
        if (*err != cudaSuccess) return 0;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3((unsigned)(sms & ~1));
        cfg.blockDim = dim3(PairCfg<BN>::kThreads);
        cfg.dynamicSmemBytes = PairCfg<BN>::kSmemBytes;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, gemm_pair_kernel<G, BN>, &cfg) != cudaSuccess) {
            (void)cudaGetLastError();
            n = 0;
        }
        pairs[dev & 63] = n;
        done[dev & 63] = n > 0;
    }
    return pairs[dev & 63];
}

template <int G, int BN>
cudaError_t launch_pair(const CUtensorMap& xmap, const CUtensorMap& wmap, const CUtensorMap& ymap,
                        const void* scales, const void* zeros, int M, int N, int K, bool streamk,
                        void* workspace, size_t workspace_bytes, const PairBlocks& blocks,
                        unsigned int* status_word, int sms, bool serialize, cudaStream_t st, bool* launched) {
    using Cfg = PairCfg<BN>;
    cudaError_t e;
    const int resident = resident_pairs<G, BN>(sms, &e);
    if (e != cudaSuccess) return e;
    // pairs that cannot all be resident at once would leave SMs idle (and a tile's owner waiting)
    if (resident * 2 < sms - 4) { *launched = false; return cudaSuccess; }
    const long long tiles = (long long)((N + 255) / 256) * ((M + BN - 1) / BN);
    const long long stages = tiles * (K / kStageK);
    // (choose_tile asked for room for sms / 2 pairs; resident ones are never more)
    streamk = streamk && workspace_bytes >= streamk_bytes(BN, resident) && (size_t)resident * sizeof(unsigned int) <= kCounterBytes;
    long long want = tiles;
    if (streamk && stages / 4 > want) want = stages / 4;          // at least four stages per pair
    const int clusters = (int)(want < resident ? want : resident);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3((unsigned)(2 * clusters));
    cfg.blockDim = dim3(Cfg::kThreads);
    cfg.dynamicSmemBytes = Cfg::kSmemBytes;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = serialize ? 1 : 2;
    float* partials = streamk ? reinterpret_cast<float*>(static_cast<unsigned char*>(workspace) + kCounterBytes)
                              : nullptr;
    unsigned int* flags = static_cast<unsigned int*>(workspace);
    e = cudaLaunchKernelEx(&cfg, gemm_pair_kernel<G, BN>, xmap, wmap, ymap, reinterpret_cast<const __half*>(scales),
                           reinterpret_cast<const unsigned char*>(zeros), M, N, K, status_word, partials, flags, blocks);
    if (e != cudaSuccess) return e;
    count_launch();
    *launched = true;
    return cudaGetLastError();
}

// Tokens per tile, and whether to cut the tiles' K loops into equal ranges (stream-K).  A launch takes `start`
// us plus `stage` us per 128 input channels of each wave of tiles (both measured with one tile per pair, on
// 4096 -> 4096 and 13824 -> 5120: 17.4 / 17.2 / 21.9 / 26.8 and 42.8 / 42.2 / 54.8 / 69.2 us with 64 / 128 /
// 192 / 256 tokens, a launch by itself; chained ones start 3 us sooner, which is in `start`); stream-K replaces the last wave by an even share but costs its pairs two more
// drains and a pass over a partial tile (8.5 us at 64 tokens, 10 us at 256; at 128 and 192, with
// sixteen dequantizer warps too few registers are left to fetch those sums in one go, 16 us and more: not
// offered) and, where a tile is cut among many pairs, the addition of their sums one after the other by
// the pair that finishes it (1.5 us each at 64 tokens, 4.4 us at 256).  With all pairs busy a stage of any size
// takes up to 1.3 times as long, so the estimates
// rank, they do not predict.  256 tokens are kept unless another tile promises 4 % (they move the
// fewest bytes per product), and launches beyond about 0.3 ms, which run into the power limit, keep
// whole tiles: idle pairs let the busy ones clock higher (an even split measured 5 % slower there).
// 4096 -> 4096 at 333 tokens: 26.6 us with 256 tokens per tile (32 tiles for 74 pairs), 18.7 us with 128;
// 5120 -> 13824 at 100 tokens 34 -> 24.6 us; 13824 -> 5120 at 2048 tokens 205 us (256, stream-K), 202 us (192).
// Over 120 problems (N 256 .. 8192, K 4096 .. 28672, 70 .. 1000 tokens, every tile timed) the choice is 0.9 % off
// the best on average and 19 % at worst (27 % and a factor of 5 without the term for the additions:
// 28672 -> 1152 at 130 tokens 88.8 us with 256 tokens and stream-K, 35.3 us with 64).
// Stream-K is offered only for tiles whose partial sums fit the workspace at hand, so that what was chosen
// is what runs (28672 -> 1152 at 130 tokens with a workspace too small for any: 77.1 us, as without one).
struct PairChoice { int bn; bool streamk; double us; };
PairChoice choose_tile(int M, int N, int K, int pairs, size_t workspace_bytes) {
    static const struct { int bn; double start, stage, streamk, addition; } kTiles[] = {
        {256, 6.0, 0.557, 10.0, 4.4}, {192, 5.5, 0.425, 0.0, 0.0}, {128, 4.0, 0.325, 0.0, 0.0}, {64, 3.6, 0.330, 8.5, 1.5}};
    PairChoice best = {256, false, 1e30};
    double least = 1e30;                             // with the bias
    const long long nks = K / kStageK;
    for (const auto& t : kTiles) {
        const long long tiles = (long long)((N + 255) / 256) * ((M + t.bn - 1) / t.bn);
        const long long waves = (tiles + pairs - 1) / pairs;
        const double bias = t.bn == 256 ? 1.0 : 1.04;
        const double plain = t.start + (double)(waves * nks) * t.stage;
        if (bias * plain < least) { least = bias * plain; best = {t.bn, false, plain}; }
        if (t.streamk == 0.0 || workspace_bytes < streamk_bytes(t.bn, pairs)) continue;
        const long long share = (tiles * nks + pairs - 1) / pairs, range = share > 4 ? share : 4;     // (at least four stages per pair)
        const double additions = nks > range ? (double)nks / (double)range - 1.0 : 0.0;
        const double even = t.start + (double)share * t.stage + t.streamk + additions * t.addition;
        if ((double)share * t.stage < 225.0 && bias * even < least) { least = bias * even; best = {t.bn, true, even}; }
    }
    return best;
}

}  // namespace

// Above 64 tokens always; below, on wide matrices when the stream kernel does not serve the call.
bool gemm_pair_applies(int M, int N) { return M > 64 || (M >= 32 && N >= 16384); }

// workspace with which the pair kernel balances its tiles over all SM pairs (stream-K)
size_t gemm_pair_workspace_bytes(int sms) {
    return streamk_bytes(256, sms / 2);
}

// its estimated time, us
double gemm_pair_estimate(int M, int N, int K, int sms, size_t workspace_bytes) {
    return choose_tile(M, N, K, sms / 2, workspace_bytes).us;
}

// Launches the pair kernel if this device can keep (nearly) all its SMs busy with pairs;
// otherwise *launched is false and the caller uses the single-block kernel.
cudaError_t launch_gemm_pair(const void* x, const CUtensorMap& wmap, const CUtensorMap& ymap,
                             const void* scales, const void* zeros, int M, int N, int K, int group,
                             void* workspace, size_t workspace_bytes,
                             unsigned int* status_word, int sms, bool serialize, cudaStream_t st, bool* launched, int count, int rows) {
    const PairBlocks blocks = {(N / count + 255) / 256, N / count, rows};
    const PairChoice c = choose_tile(M, N, K, sms / 2, workspace ? workspace_bytes : 0);
    // Long launches are not chained.  They run at the power limit, where an early start buys nothing and sometimes costs: back to back,
    // chained / unchained, us: 700 and 2048 tokens on 4096 -> 4096 24.4 / 25.4 and 59.0 / 60.0, 1024 on 13824 -> 5120 118 / 121 (estimates
    // below 85); 2048 on 4096 -> 11008, 8192 -> 8192 and 13824 -> 5120 152 / 153, 224 / 224 and 249 / 249 (95 to 146); 3000 on 8192 -> 8192
    // 341 / 338, 4096 on 11008 -> 4096 358 / 352, 1024 on 28672 -> 8192 429 / 412, 1500 on 8192 -> 28672 560 / 570, 4096 on 13824 -> 5120
    // 501 / 496 (182 to 362).  Over 12 problems whose estimate is above 150 chaining loses 0.5 %, over 11 below it gains 1.2 %.
    serialize = serialize || c.us > 150.0;
    CUtensorMap xmap;
    {
        // x as [M][K] fp16 in boxes of half a tile's tokens x one k-block, 128-byte swizzle
        const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)(count > 1 ? (long long)count * rows : M)};
        const cuuint64_t strides[1] = {(cuuint64_t)K * 2};
        const cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)(c.bn / 2)}, estr[2] = {1, 1};
        if (encode_fn()(&xmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void*>(x), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
#define AWQ_PAIR_CASE(GG, BNN)                                                                                     \
    return launch_pair<GG, BNN>(xmap, wmap, ymap, scales, zeros, M, N, K, c.streamk, workspace, workspace_bytes, blocks, \
                                status_word, sms, serialize, st, launched)
    if (group == 128) {
        switch (c.bn) { case 64: AWQ_PAIR_CASE(128, 64); case 128: AWQ_PAIR_CASE(128, 128);
                        case 192: AWQ_PAIR_CASE(128, 192); default: AWQ_PAIR_CASE(128, 256); }
    }
    switch (c.bn) { case 64: AWQ_PAIR_CASE(64, 64); case 128: AWQ_PAIR_CASE(64, 128);
                    case 192: AWQ_PAIR_CASE(64, 192); default: AWQ_PAIR_CASE(64, 256); }
#undef AWQ_PAIR_CASE
}

}  // namespace awq
