// The layer for 9 .. 64 tokens (and fewer where the output rows are too few for the band kernel; Sec. 4.2:
// fused dequantize + product) on the tensor cores, where the weights still set the time: every packed byte should cross HBM once and nothing else should
// be slower than that.
//
// The prefill kernels (gemm_tcgen05*.cu) are built for many tokens: per 64-wide k-block a tile
// fetches its x tile again, and split-K meets through counters and a fix-up pass.  This kernel keeps
// their arithmetic (weights -> exact fp16 (q - z), times Delta in fp16, straight into tensor memory as
// the A operand of tcgen05.mma; tokens on the N side, fp32 accumulator in tensor memory) and
// changes the decomposition, like the chunked matrix-vector kernel:
//   * a work unit is one 128-channel slab x one chunk of K; a block takes a contiguous range of
//     units that stay in one chunk as long as possible, so the chunk's slice of x (BN tokens, 128-byte
//     swizzle) is fetched once per chunk and stays in shared memory as the B operand of every slab;
//     up to four matrices that read the same x lay their slabs end to end in one launch;
//   * a stage of the weight ring is 8 bands x 256 input channels = 16 KB (one tensor-map copy),
//     released when its words have been converted; a slot of A in tensor memory is 128 columns
//     (the same 256 input channels), released by the completion of its products;
//   * sixteen dequantizer warps, each owning a band and every second stage, so that a warp pays its
//     barrier polls, parameter reads and arrivals once per 16 packed words;
//   * one warp issues the products, four epilogue warps write the unit's fp32 sums to
//     [chunk][token][channel] in the workspace, and a second, small kernel adds the chunks in ascending
//     order: deterministic, no counters, no waiting between blocks.
//
// What bounds it.  Steady state: the dequantizers' instruction stream - per scheduler 21 cycles a packed word of
// 32 lanes with the product by Delta, ~15 without, against 22 at the HBM rate - and L2: the slices of x
// and the partial sums together are as many bytes as the weights at 64 tokens (~4.5 TB/s).  Short launches: ~4 us
// of hand-overs (the launch in front, x, the second kernel).  What it took, 8192 -> 28672 at 32 tokens:
//   * 8 KB stages, products issued inside `if (lane == 0)` 64 us; issued by an elected lane of a converged warp
//     (tcgen05.cuh) 49 us;
//   * 16 KB stages, 16x128b stores of A (17 cycles per 16 x 32 columns; the 16x256b form, which is the packed piece as
//     it is, takes 33, and up to 48 while products run) 46 us.  In that form lane t of a row holds the 32-bit
//     columns 4i + t, while its words hold pairs 2t and 2t + 1 of each 16 channels: so A's channels come
//     permuted inside each 16, pair 2t + p at place 4p + t, and the slice of x is brought into the same order
//     in shared memory by the dequantizers (a part of it after each of their first stages; the products'
//     sum over 16 channels does not depend on the order).  The product with 1 / s of awq_linear_scaled
//     rides on that pass;
//   * mask and magic number in one three-input instruction (code_pair) 42 us; chunk lengths by the estimate
//     at make_plan;
//   * Delta in the epilogue up to 32 tokens (EXACT): as fast (45 us; 4096 -> 4096 9.3 instead of 9.7 us,
//     4096 -> 11008 15.5 instead of 15.6 us) and without the rounding.
// At 16 tokens 37.9 us (3.3 TB/s of weights); a 7B layer's seven linears at 32 tokens, as four calls: 71 us
// (111 us with a launch per matrix, 8 KB stages and a separate scaling kernel).
#include <cstring>

#include "tcgen05.cuh"

namespace awq {

namespace {

// warp 0 weight copies, 1 products, 2 x copies, 4-7 epilogue, 8-23 dequantizers (EXACT: 24-27 epilogue too)
constexpr int kSkThreads = 768, kSkExactThreads = 896;
constexpr int kSkStageTiles = 4;                 // k-blocks per stage
constexpr int kSkStageBytes = kSkStageTiles * kTileBytes;    // 8 bands x 4 k-blocks x 512 bytes
constexpr int kSkMaxRing = 8;                    // stages of packed weights in shared memory
constexpr int kSkXBytes = 128 * 1024;            // most that the chunk's slice of x may take
constexpr int kSkPartTiles = 8;                  // k-blocks of x per part (two stages: one per dequantizer parity)
constexpr int kSkMaxParts = 4;
// tensor memory: two accumulators of BN <= 64 columns (two units in flight), then 128 columns of
// dequantized weights per stage
constexpr int kSkA0 = 128, kSkSlotCols = 128, kSkSlots = (512 - kSkA0) / kSkSlotCols;
constexpr int kSkTmemCols = 512;
constexpr int kSkMaxAcc = 2;                     // accumulators: two units' (BN columns), or two pairs of groups' (EXACT, 2 BN columns)
constexpr int kSkMaxGroups = 16;                 // groups per chunk (one tensor-map box of scales / zero points)
constexpr int kSkParBytes = kSkMaxGroups * (8 * 32 + 4 * 16);   // a unit's scales [8 bands][groups][16] fp16 + zero bytes [4][groups][16]
constexpr int kSkMaxSmem = 227 * 1024 - 64;          // dynamic part: a few static bytes come on top
constexpr int kSkFixed = 1024 /*align*/ + 512 /*barriers*/ + 2 * kSkParBytes;
// A stage may pass from the warps of one parity to the others' (an odd ring): what tells them apart is that a warp
// has seen the products of five stages ago complete, so a ring is even or has at least five stages.
static_assert((kSkMaxSmem - kSkFixed - kSkXBytes - kSkMaxParts * kSkPartTiles * kBK * 4) / kSkStageBytes >= 4, "ring");

struct SkMaps {                                  // up to kMaxMulti matrices, slabs laid end to end
    CUtensorMap w[kMaxMulti], sc[kMaxMulti], z[kMaxMulti];
    int slab_end[kMaxMulti];                     // first slab of the next matrix
};

struct SkPlan {
    int ck = 0, blocks = 0;                      // k-blocks per chunk, thread blocks
    UnitStarts starts;
};

__device__ __forceinline__ void tmem_ld_16cols(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld_8cols(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
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

// EXACT = false: A is fp16 (q - z) * Delta, rounded once, one accumulator per unit.  EXACT = true (up to 32
// tokens): A is the integer q - z, every group has an accumulator of its own (handed over in pairs), and
// the epilogue adds Delta times it in fp32 registers: no rounding before the output, like the
// matrix-vector kernels (a 2-norm error of 2.1e-4 instead of 2.8e-4, the output's own rounding).
template <int G, int BN, bool XS, bool EXACT>
__global__ void __launch_bounds__(EXACT ? kSkExactThreads : kSkThreads, 1)
gemm_skinny_kernel(const __grid_constant__ CUtensorMap x_map, const __grid_constant__ SkMaps maps,
                   const float* __restrict__ inv_s, float* __restrict__ partial, int M, int nslabs, int K, int CK,
                   int R, const __grid_constant__ UnitStarts starts, unsigned int* status_word) {
    constexpr int S = kSkSlots;
    constexpr int KPG = G / kBK;                     // k-blocks per group
    constexpr int GPS = kSkStageTiles / KPG;         // groups per stage
    constexpr uint32_t NACC = kSkMaxAcc;
    constexpr uint32_t kAccCols = EXACT ? 2 * BN : BN;
    static_assert(NACC * kAccCols <= kSkA0, "accumulators and A slots overlap");
    extern __shared__ unsigned char smem_dyn[];
    __shared__ unsigned int s_abort;
    __shared__ uint32_t s_tmem_base;

    const uint32_t dyn = smem_u32(smem_dyn);
    const uint32_t base = (dyn + 1023u) & ~1023u;
    unsigned char* base_ptr = smem_dyn + (base - dyn);
    // [x slice: CK tiles of BN rows x 128 bytes | ring of weight stages | two parameter buffers | 1 / s | barriers]
    const uint32_t x_base = base;
    const uint32_t w_base = base + (uint32_t)(CK * BN * 128);
    const uint32_t par_base = w_base + (uint32_t)(R * kSkStageBytes);
    const uint32_t inv_base = par_base + 2u * (uint32_t)kSkParBytes;
    const uint32_t bars = inv_base + (XS ? (uint32_t)(CK * kBK * 4) : 0u);
    // the packed weights' ring (raw_*: filled by the copy engine, released by the dequantizers when they
    // have used the words) and the ring of A slots in tensor memory (a_*: filled by the
    // dequantizers, released by the products' completion)
    auto raw_full = [&](uint32_t r) { return bars + 8u * r; };
    auto raw_empty = [&](uint32_t r) { return bars + 8u * (uint32_t)(kSkMaxRing + r); };
    auto a_full = [&](uint32_t s) { return bars + 8u * (uint32_t)(2 * kSkMaxRing + s); };
    auto a_empty = [&](uint32_t s) { return bars + 8u * (uint32_t)(2 * kSkMaxRing + S + s); };
    constexpr int B1 = 2 * kSkMaxRing + 2 * S;
    auto acc_full = [&](uint32_t b) { return bars + 8u * (uint32_t)(B1 + b); };
    auto acc_empty = [&](uint32_t b) { return bars + 8u * (uint32_t)(B1 + kSkMaxAcc + b); };
    constexpr int B2 = B1 + 2 * kSkMaxAcc;
    auto par_full = [&](uint32_t b) { return bars + 8u * (uint32_t)(B2 + b); };
    auto par_empty = [&](uint32_t b) { return bars + 8u * (uint32_t)(B2 + 2 + b); };
    // the slice of x, in parts: landed, in the products' order, no longer needed
    auto x_raw = [&](uint32_t p) { return bars + 8u * (uint32_t)(B2 + 4 + p); };
    auto x_full = [&](uint32_t p) { return bars + 8u * (uint32_t)(B2 + 4 + kSkMaxParts + p); };
    const uint32_t x_empty = bars + 8u * (uint32_t)(B2 + 4 + 2 * kSkMaxParts);
    const int gpc = CK / KPG;                        // groups per chunk (<= kSkMaxGroups)
    const uint32_t z_in_par = (uint32_t)(gpc * 8 * 32), par_bytes = (uint32_t)(gpc * (8 * 32 + 4 * 16));

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nkb = K / kBK;
    const int u0 = starts.v[blockIdx.x], u1 = starts.v[blockIdx.x + 1];
    // unit u = chunk * nslabs + slab; a chunk has nt k-blocks, ceil(nt / 4) stages (CK is a multiple of
    // 4, the last chunk's nt a multiple of 2: the copies past K fill zeros that no product reads)
    auto chunk_of = [&](int u) { return u / nslabs; };
    auto tiles_of = [&](int c) { return min(CK, nkb - c * CK); };

    if (threadIdx.x == 0) {
        s_abort = 0u;
        for (int r = 0; r < R; ++r) { mbar_init(raw_full(r), 1); mbar_init(raw_empty(r), 8); }
        for (int s = 0; s < S; ++s) { mbar_init(a_full(s), 8); mbar_init(a_empty(s), 1); }
        for (uint32_t b = 0; b < NACC; ++b) { mbar_init(acc_full(b), 1); mbar_init(acc_empty(b), EXACT ? 8 : 4); }
        // the parameters are read by the dequantizers and (EXACT) by the epilogue
        for (uint32_t b = 0; b < 2; ++b) { mbar_init(par_full(b), 1); mbar_init(par_empty(b), EXACT ? 24 : 16); }
        for (int p = 0; p < kSkMaxParts; ++p) { mbar_init(x_raw(p), 1); mbar_init(x_full(p), 16); }
        mbar_init(x_empty, 1);
        mbar_fence_init();
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&s_tmem_base)), "r"((uint32_t)kSkTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = s_tmem_base;
    const WaitCtl ctl{status_word, &s_abort};
    // programmatic dependent launch: the packed arrays are constants of the layer and are copied before
    // the work in front of this launch has completed; x, 1 / s and the workspace are touched after it
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (warp == 0) {
        // ------------------------------------------------------------ weight copies
        const bool lead = elect_one();
        uint32_t stage = 0, phase = 0;
        int issued = 0, par_issued = 0;
        bool ok = true;
        for (int u = u0; u < u1 && ok; ++u) {
            const int c = chunk_of(u);
            int slab = u - c * nslabs, mi = 0;
#pragma unroll
            for (int i = 0; i + 1 < kMaxMulti; ++i) mi += slab >= maps.slab_end[i] ? 1 : 0;
            if (mi > 0) slab -= maps.slab_end[mi - 1];
            const int kb0 = c * CK, nt = tiles_of(c);
            // the unit's scales and zero points: boxes of 8 bands (4 band pairs) x the chunk's groups
            const uint32_t pb = (uint32_t)(u - u0) & 1u, puse = ((uint32_t)(u - u0) >> 1) & 1u;
            if (!mbar_wait_warp(par_empty(pb), puse ^ 1u, ctl)) { ok = false; break; }
            if (lead) {
                mbar_arrive_expect_tx(par_full(pb), par_bytes);
                tma_load_2d(par_base + pb * (uint32_t)kSkParBytes, &maps.sc[mi], (kb0 / KPG) * 16, slab * 8, par_full(pb));
                tma_load_2d(par_base + pb * (uint32_t)kSkParBytes + z_in_par, &maps.z[mi], (kb0 / KPG) * 16, slab * 4, par_full(pb));
            }
            __syncwarp();
            ++par_issued;
            for (int j = 0; j < nt; j += kSkStageTiles) {
                if (!mbar_wait_warp(raw_empty(stage), phase ^ 1u, ctl)) { ok = false; break; }
                if (lead) {
                    mbar_arrive_expect_tx(raw_full(stage), kSkStageBytes);
                    // 8 bands x 4 k-blocks (256 64-bit elements) at (element kb * 64 of the band's run, first band)
                    tma_load_2d(w_base + stage * kSkStageBytes, &maps.w[mi], (kb0 + j) * 64, slab * 8, raw_full(stage));
                }
                __syncwarp();
                ++issued;
                if (++stage == (uint32_t)R) { stage = 0; phase ^= 1u; }
            }
        }
        if (!ok) {
            // giving up: let the copies already issued land before the block exits
            const int pending = issued < R ? issued : R;
            uint32_t st = stage, ph = phase;
            for (int i = 0; i < pending; ++i) {
                if (st == 0) { st = R - 1; ph ^= 1u; } else { --st; }
                const unsigned long long t0 = global_ns();
                while (!mbar_try_wait(raw_full(st), ph) && global_ns() - t0 < drain_limit_ns(ctl)) {}
            }
            for (int i = 0; i < 2 && i < par_issued; ++i) {
                const unsigned int k = par_issued - 1 - i;               // the k-th parameter copy: buffer k & 1, use k >> 1
                const unsigned long long t0 = global_ns();
                while (!mbar_try_wait(par_full(k & 1u), (k >> 1) & 1u) && global_ns() - t0 < drain_limit_ns(ctl)) {}
            }
        }
    } else if (warp == 2) {
        // ------------------------------------------------------------ x copies, one slice per chunk
        const bool lead = elect_one();
        int cur = -1;
        uint32_t n = 0;
        for (int u = u0; u < u1; ++u) {
            const int c = chunk_of(u);
            if (c == cur) continue;
            // the products that read the previous slice have completed
            if (n > 0 && !__all_sync(0xFFFFFFFFu, mbar_wait_relaxed(x_empty, (n - 1u) & 1u, ctl))) break;
            const int nt = tiles_of(c);
            if (n == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
            if (lead) {
                for (int kb = 0, p = 0; kb < nt; kb += kSkPartTiles, ++p) {
                    const int ke = min(kb + kSkPartTiles, nt);
                    mbar_arrive_expect_tx(x_raw(p), (uint32_t)((ke - kb) * BN * 128 + (XS && p == 0 ? nt * kBK * 4 : 0)));
                    if (XS && p == 0) bulk_load(inv_base, inv_s + (size_t)c * CK * kBK, (uint32_t)(nt * kBK * 4), x_raw(0));
                    for (int k = kb; k < ke; ++k)
                        tma_load_2d(x_base + (uint32_t)(k * BN * 128), &x_map, (c * CK + k) * kBK, 0, x_raw(p));
                }
            }
            __syncwarp();
            cur = c;
            ++n;
        }
        if (s_abort && n > 0) {
            // giving up: the last slice's copies must have landed before the block exits
            const int parts = (tiles_of(cur) + kSkPartTiles - 1) / kSkPartTiles;
            for (int p = 0; p < parts; ++p) {
                // a part that earlier, shorter slices lacked has seen fewer phases: its own count decides
                uint32_t uses = 0;
                for (int c = chunk_of(u0); c <= cur; ++c) uses += tiles_of(c) > p * kSkPartTiles ? 1u : 0u;
                const unsigned long long t0 = global_ns();
                while (!mbar_try_wait(x_raw(p), (uses - 1u) & 1u) && global_ns() - t0 < drain_limit_ns(ctl)) {}
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ products
        const bool lead = elect_one();
        constexpr uint32_t idesc = instr_desc(BN);
        uint32_t stage = 0, phase = 0, xn = 0, acc = 0, acc_phase = 0;
        int cur = -1;
        bool ok = true;
        for (int u = u0; u < u1 && ok; ++u) {
            const int c = chunk_of(u);
            const int nt = tiles_of(c);
            const bool fresh = c != cur;                         // first unit on this slice of x: wait for its parts
            if (fresh) { ++xn; cur = c; }
            if (!EXACT) {
                if (!mbar_wait_warp(acc_empty(acc), acc_phase ^ 1u, ctl)) break;
                tc_fence_after();
            }
            uint64_t bdesc = smem_desc_sw128(x_base);
            for (int j = 0; j < nt; j += kSkStageTiles) {
                // slices that are not the last have all parts: a part's phase is the slice's number
                if (fresh && j % kSkPartTiles == 0 && !mbar_wait_warp(x_full(j / kSkPartTiles), (xn - 1u) & 1u, ctl)) { ok = false; break; }
                if (!mbar_wait_warp(a_full(stage), phase, ctl)) { ok = false; break; }
                tc_fence_after();
                const uint32_t a_tmem = tmem_base + (uint32_t)(kSkA0 + stage * kSkSlotCols);
                // k-blocks h0 .. h1-1 of the stage into an accumulator
                auto products = [&](uint32_t d_tmem, int h0, int h1, bool start) {
#pragma unroll
                    for (int h = h0; h < h1; ++h) {
                        if (h >= 2 && j + h >= nt) break;        // nt is even
#pragma unroll
                        for (int k = 0; k < kBK / 16; ++k)       // A: +8 columns, B: +32 bytes per K = 16 step
                            umma_f16_a_tmem(d_tmem, a_tmem + (uint32_t)(32 * h + 8 * k),
                                            bdesc + (uint64_t)((h * BN * 128) >> 4) + (uint64_t)(2 * k), idesc,
                                            (!start || h != h0 || k != 0) ? 1u : 0u);
                    }
                };
                if (EXACT) {
#pragma unroll
                    for (int q = 0; q < GPS; q += 2) {           // pairs of groups (G = 128: a chunk may end on half a pair)
                        if (j + q * KPG >= nt) break;
                        if (!mbar_wait_warp(acc_empty(acc), acc_phase ^ 1u, ctl)) { ok = false; break; }
                        tc_fence_after();
                        if (lead) {
                            const uint32_t d_tmem = tmem_base + acc * kAccCols;
                            products(d_tmem, q * KPG, (q + 1) * KPG, true);
                            if (j + (q + 1) * KPG < nt) products(d_tmem + (uint32_t)BN, (q + 1) * KPG, (q + 2) * KPG, true);
                            // The slot of A before the last pair's sums: what the epilogue waits for comes last,
                            // so that no arrival is outstanding when the block exits.
                            if (q + 2 >= GPS || j + (q + 2) * KPG >= nt) umma_commit(a_empty(stage));
                            umma_commit(acc_full(acc));
                        }
                        __syncwarp();
                        if (++acc == NACC) { acc = 0; acc_phase ^= 1u; }
                    }
                    if (!ok) break;
                } else if (lead) {
                    products(tmem_base + acc * kAccCols, 0, kSkStageTiles, j == 0);
                    umma_commit(a_empty(stage));
                }
                __syncwarp();
                bdesc += (uint64_t)((kSkStageTiles * BN * 128) >> 4);
                if (++stage == (uint32_t)S) { stage = 0; phase ^= 1u; }
            }
            if (!ok) break;
            if (lead) {
                if (!EXACT) umma_commit(acc_full(acc));
                // the slice of x may be replaced once the products of its last unit have completed
                if (u + 1 < u1 && chunk_of(u + 1) != c) umma_commit(x_empty);
            }
            __syncwarp();
            if (!EXACT && ++acc == NACC) { acc = 0; acc_phase ^= 1u; }
        }
    } else if (warp >= 8 && warp < 24) {
        // ------------------------------------------------------------ dequantizers
        // warp (band, parity): the band's 16 rows, all four k-blocks of every second stage (stages are
        // counted through the whole range of units).  Lane (g, t) holds, per k-block, the piece (rows g
        // and g+8, columns 16j + 4t .. +3 for j = 0..3).
        const int wi = warp - 8, quad = wi & 3, hsel = (wi >> 2) & 1, par2 = wi >> 3;
        const int band = 2 * quad + hsel;               // bands 0..7 <-> TMEM lanes 16 * band .. +15
        const int g = lane >> 2;
        const uint32_t taddr_band = tmem_base + ((uint32_t)(quad * 32 + hsel * 16) << 16) + (uint32_t)kSkA0;
        const unsigned char* w_lane = base_ptr + (w_base - base) + band * (kSkStageTiles * 512) + lane * 16;

        // one part of the slice of x, brought into A's order in place (a thread takes 32 bytes = 16
        // channels of a token at a time), times 1 / s where that is folded in
        auto order_x = [&](int part, int nt, uint32_t parity) -> bool {
            if (!__all_sync(0xFFFFFFFFu, mbar_wait(x_raw(part), parity, ctl))) return false;
            if (XS && part != 0 && !__all_sync(0xFFFFFFFFu, mbar_wait(x_raw(0), parity, ctl))) return false;
            const int kb0 = part * kSkPartTiles;
#pragma unroll
            for (int i = 0; i < BN / 16; ++i) {
                const int item = i * 512 + wi * 32 + lane;       // [k-block of the part][token][16 channels]
                const int kb = kb0 + item / (BN * 4), m = (item / 4) % BN, j = item % 4;
                if (kb < nt) {
                    unsigned char* row = base_ptr + kb * (BN * 128) + m * 128;
                    uint4* c0 = reinterpret_cast<uint4*>(row + (((2 * j) ^ (m & 7)) << 4));
                    uint4* c1 = reinterpret_cast<uint4*>(row + (((2 * j + 1) ^ (m & 7)) << 4));
                    uint4 a = *c0, b = *c1;
                    if (XS) {
                        const float4* is = reinterpret_cast<const float4*>(base_ptr + (inv_base - base)) + (kb * kBK + j * 16) / 4;
                        const float4 s0 = is[0], s1 = is[1], s2 = is[2], s3 = is[3];
                        a.x = scale_pair(a.x, make_float2(s0.x, s0.y)); a.y = scale_pair(a.y, make_float2(s0.z, s0.w));
                        a.z = scale_pair(a.z, make_float2(s1.x, s1.y)); a.w = scale_pair(a.w, make_float2(s1.z, s1.w));
                        b.x = scale_pair(b.x, make_float2(s2.x, s2.y)); b.y = scale_pair(b.y, make_float2(s2.z, s2.w));
                        b.z = scale_pair(b.z, make_float2(s3.x, s3.y)); b.w = scale_pair(b.w, make_float2(s3.z, s3.w));
                    }
                    *c0 = make_uint4(a.x, a.z, b.x, b.z);        // pairs 0 2 4 6
                    *c1 = make_uint4(a.y, a.w, b.y, b.w);        // pairs 1 3 5 7
                }
            }
            fence_proxy_async_smem();                            // the products read it through the asynchronous proxy
            __syncwarp();
            if (lane == 0) mbar_arrive(x_full(part));
            return true;
        };

        uint32_t stage = (uint32_t)par2, phase = 0;     // slot of A in tensor memory (this warp's next)
        uint32_t rstage = (uint32_t)par2, rphase = 0;   // stage of the packed weights' ring
        int first = par2;                               // this warp's first stage inside the next unit
        int cur = -1, xpart = 0, xparts = 0;            // parts of the current slice of x already brought into order
        uint32_t xn = 0;
        bool ok = true;
        for (int u = u0; u < u1 && ok; ++u) {
            const int c = chunk_of(u);
            const int nt = tiles_of(c), nst = (nt + kSkStageTiles - 1) / kSkStageTiles;
            if (c != cur) { cur = c; xpart = 0; xparts = (nt + kSkPartTiles - 1) / kSkPartTiles; ++xn; }
            const uint32_t pb = (uint32_t)(u - u0) & 1u, puse = ((uint32_t)(u - u0) >> 1) & 1u;
            ok = __all_sync(0xFFFFFFFFu, mbar_wait(par_full(pb), puse, ctl));
            if (!ok) break;
            // this lane's rows' parameters: scales [band][group][16], zero bytes [band pair][group][16]
            const unsigned char* par = base_ptr + (par_base - base) + pb * kSkParBytes;
            const unsigned char* psc = par + band * (gpc * 32) + g * 2;
            const unsigned char* pz = par + z_in_par + (band >> 1) * (gpc * 16) + (band & 1) * 8 + g;
            int j = first;
            for (; j < nst; j += 2) {
                ok = mbar_wait(raw_full(rstage), rphase, ctl);
                uint4 pk[kSkStageTiles];
#pragma unroll
                for (int h = 0; h < kSkStageTiles; ++h)
                    pk[h] = *reinterpret_cast<const uint4*>(w_lane + rstage * kSkStageBytes + h * 512);
                ok = __all_sync(0xFFFFFFFFu, ok && mbar_wait(a_empty(stage), phase ^ 1u, ctl));
                if (!ok) break;
                tc_fence_after();
                // parameters of the stage's groups
                uint32_t d_up[GPS], d_lo[GPS], zlo[GPS], zhi[GPS];
#pragma unroll
                for (int q = 0; q < GPS; ++q) {
                    const int gi = GPS * j + q;                       // group inside the chunk
                    d_up[q] = __byte_perm(*reinterpret_cast<const unsigned short*>(psc + gi * 32), 0u, 0x1010);
                    d_lo[q] = __byte_perm(*reinterpret_cast<const unsigned short*>(psc + gi * 32 + 16), 0u, 0x1010);
                    const uint32_t zb = pz[gi * 16];
                    // 1024 + z for the low nibble; -(64 + z) for the high one (bits 4-7 of the byte are z << 4)
                    zlo[q] = __byte_perm((zb & 0xFu) | 0x6400u, 0u, 0x1010);
                    zhi[q] = __byte_perm((zb & 0xF0u) | 0xD400u, 0u, 0x1010);
                }
#pragma unroll
                for (int h = 0; h < kSkStageTiles; ++h) {
                    constexpr int q_of[4] = {0, 1 / KPG, 2 / KPG, 3 / KPG};
                    const int q = q_of[h];
                    const uint32_t wds[4] = {pk[h].x, pk[h].y, pk[h].z, pk[h].w};
                    // word j: (row g | g+8: c, c+1) in its low bytes, (c+2, c+3) in the bytes above
                    uint32_t v[16];
#pragma unroll
                    for (int jw = 0; jw < 4; ++jw) {
                        constexpr uint32_t kSixteenth = 0x2C002C00u;
                        const uint32_t w = wds[jw], w8 = w >> 8;
                        v[4 * jw + 0] = hsub2_u32(code_pair(w, kLowCodes), zlo[q]);                  // q - z, exactly
                        v[4 * jw + 1] = hfma2_u32(code_pair(w, kHighCodes), kSixteenth, zhi[q]);
                        v[4 * jw + 2] = hsub2_u32(code_pair(w8, kLowCodes), zlo[q]);
                        v[4 * jw + 3] = hfma2_u32(code_pair(w8, kHighCodes), kSixteenth, zhi[q]);
                        if (EXACT) continue;
                        v[4 * jw + 0] = hmul2_u32(v[4 * jw + 0], d_up[q]);
                        v[4 * jw + 1] = hmul2_u32(v[4 * jw + 1], d_lo[q]);
                        v[4 * jw + 2] = hmul2_u32(v[4 * jw + 2], d_up[q]);
                        v[4 * jw + 3] = hmul2_u32(v[4 * jw + 3], d_lo[q]);
                    }
                    tmem_st_16x32cols_128b(taddr_band + stage * (uint32_t)kSkSlotCols + (uint32_t)(32 * h), v);
                }
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                // The stage is given back with the slot: only the use of a word shows that its load is done.
                // Given back in front of the wait for the slot, a stage was refilled while late warps still
                // read it (4096 -> 8192 at 24 tokens, whose ring of five stages wraps during its first
                // conversions: 96 of 36000 calls had wrong channels in one or more bands; now none of 72000).
                if (lane == 0) {
                    mbar_arrive(raw_empty(rstage));
                    mbar_arrive(a_full(stage));
                }
                stage += 2;
                if (stage >= (uint32_t)S) { stage -= S; phase ^= 1u; }
                rstage += 2;
                if (rstage >= (uint32_t)R) { rstage -= R; rphase ^= 1u; }
                if (xpart < xparts) {
                    ok = order_x(xpart, nt, (xn - 1u) & 1u);
                    ++xpart;
                    if (!ok) break;
                }
            }
            if (!ok) break;
            for (; xpart < xparts && ok; ++xpart) ok = order_x(xpart, nt, (xn - 1u) & 1u);
            first = j - nst;                             // 0 or 1: where this warp's stages resume
            __syncwarp();
            if (lane == 0) mbar_arrive(par_empty(pb));               // the unit's parameters may be replaced
        }
    } else if (warp >= 4) {
        // ------------------------------------------------------------ epilogue
        asm volatile("griddepcontrol.wait;" ::: "memory");
        const int quad = warp & 3;                     // TMEM lanes 32 * quad .. +31
        const size_t N = (size_t)nslabs * 128;         // all matrices' channels
        const uint32_t taddr0 = tmem_base + ((uint32_t)(quad * 32) << 16);
        uint32_t acc = 0, acc_phase = 0;
        bool ok = true;
        for (int u = u0; u < u1 && ok; ++u) {
            const int c = chunk_of(u), slab = u - c * nslabs;
            float* out = partial + (size_t)c * M * N + slab * 128 + quad * 32 + lane;
            if (!EXACT) {
                if (!__all_sync(0xFFFFFFFFu, mbar_wait(acc_full(acc), acc_phase, ctl))) break;
                tc_fence_after();
#pragma unroll 1
                for (int c0 = 0; c0 < BN; c0 += 16) {
                    uint32_t r[16];
                    tmem_ld_16cols(taddr0 + acc * kAccCols + (uint32_t)c0, r);
                    tmem_ld_wait(r);
                    if (c0 + 16 >= BN) {
                        // the accumulator is in registers: the next unit's products may overwrite it
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(acc_empty(acc));
                    }
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        if (c0 + i < M) out[(size_t)(c0 + i) * N] = __uint_as_float(r[i]);
                }
                if (++acc == NACC) { acc = 0; acc_phase ^= 1u; }
                continue;
            }
            // EXACT: this lane's channel of the slab is row lane % 16 of band 2 quad + lane / 16; this warp's
            // tokens are one half of BN
            constexpr int TH = EXACT ? BN / 2 : 8;
            const int tok0 = warp >= 24 ? TH : 0;
            const int ngr = tiles_of(c) / KPG;
            const uint32_t pb = (uint32_t)(u - u0) & 1u, puse = ((uint32_t)(u - u0) >> 1) & 1u;
            ok = __all_sync(0xFFFFFFFFu, mbar_wait(par_full(pb), puse, ctl));
            if (!ok) break;
            const unsigned char* psc = base_ptr + (par_base - base) + pb * kSkParBytes +
                                       (2 * quad + (lane >> 4)) * (gpc * 32) + (lane & 15) * 2;
            float y[TH];
#pragma unroll
            for (int i = 0; i < TH; ++i) y[i] = 0.0f;
            for (int gi = 0; gi < ngr; gi += 2) {
                const bool two = gi + 1 < ngr;
                const float d0 = __half2float(*reinterpret_cast<const __half*>(psc + gi * 32));
                const float d1 = __half2float(*reinterpret_cast<const __half*>(psc + (two ? gi + 1 : gi) * 32));
                ok = __all_sync(0xFFFFFFFFu, mbar_wait(acc_full(acc), acc_phase, ctl));
                if (!ok) break;
                tc_fence_after();
                uint32_t r0[TH], r1[TH];
                const uint32_t t0 = taddr0 + acc * kAccCols + (uint32_t)tok0;
                tmem_ld_cols<TH>(t0, r0);
                tmem_ld_cols<TH>(t0 + (two ? (uint32_t)BN : 0u), r1);
                tmem_ld_wait(r0, r1);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(acc_empty(acc));
#pragma unroll
                for (int i = 0; i < TH; ++i) y[i] = fmaf(d0, __uint_as_float(r0[i]), y[i]);
                if (two) {
#pragma unroll
                    for (int i = 0; i < TH; ++i) y[i] = fmaf(d1, __uint_as_float(r1[i]), y[i]);
                }
                if (++acc == NACC) { acc = 0; acc_phase ^= 1u; }
            }
            if (!ok) break;
#pragma unroll
            for (int i = 0; i < TH; ++i)
                if (tok0 + i < M) out[(size_t)(tok0 + i) * N] = y[i];
            __syncwarp();
            if (lane == 0) mbar_arrive(par_empty(pb));           // the unit's parameters may be replaced
        }
    }

    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;"
                     ::"r"(tmem_base), "r"((uint32_t)kSkTmemCols) : "memory");
    }
}

// y_i[m][n] = fp16(sum over the chunks, ascending, of partial[c][m][offset_i + n]): four outputs per
// thread, one token per block row.
struct SkOutputs {
    __half* y[kMaxMulti];
    int end[kMaxMulti];                              // first channel of the next matrix
};
template <int B>
__global__ void __launch_bounds__(256)
skinny_reduce_kernel(const float* partial, const __grid_constant__ SkOutputs out, int chunks, int M, int N) {
    // launched with programmatic stream serialization behind the kernel above: it may be resident
    // before that kernel has finished (so the sums, written during its lifetime, are no read-only data: they
    // are read through L2), and lets the launch behind it start its own weight copies
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int n = (int)(blockIdx.x * blockDim.x + threadIdx.x) * 4, m = blockIdx.y;
    if (n >= N) return;
    const size_t mn = (size_t)M * N;
    const float4 s = add_chunks<B>(partial + (size_t)m * N + n, chunks, mn);
    const __half2 lo = __floats2half2_rn(s.x, s.y), hi = __floats2half2_rn(s.z, s.w);
    uint2 o;
    o.x = *reinterpret_cast<const uint32_t*>(&lo);
    o.y = *reinterpret_cast<const uint32_t*>(&hi);
    int mi = 0;
#pragma unroll
    for (int i = 0; i + 1 < kMaxMulti; ++i) mi += n >= out.end[i] ? 1 : 0;
    const int n0 = mi > 0 ? out.end[mi - 1] : 0, width = out.end[mi] - n0;
    *reinterpret_cast<uint2*>(out.y[mi] + (size_t)m * width + (n - n0)) = o;
}

int skinny_bn(int M) { return M <= 16 ? 16 : M <= 32 ? 32 : 64; }

int skinny_max_ck(int bn, int group) {
    const int by_x = kSkXBytes / (bn * 128), by_groups = kSkMaxGroups * (group / kBK), by_parts = kSkMaxParts * kSkPartTiles;
    const int ck = by_x < by_groups ? by_x : by_groups;
    return ck < by_parts ? ck : by_parts;
}

// Blocks and chunk length for a problem.  Units of the last chunk are shorter; blocks take contiguous
// ranges.  For a given chunk length the ranges are cut greedily at the smallest limit with which the
// blocks suffice; of the chunk lengths (multiples of a stage) the one with the least estimate is taken.
// The estimate is a fit to 27 problems (1536 x 2048 to 8192 x 28672, 16 / 32 / 64 tokens), every chunk length
// timed: 4 us + 0.12 us per k-block of the longest block (4 KB of weights; a unit counts four more for
// its hand-overs and epilogue, a change of chunk the next slice of x) + the slice of x and the partial
// sums, both of which go through L2 at ~4.5 TB/s and pull in opposite directions.  What it picks is within
// 1.3 % of the best chunk length on average, 13 % at worst.  All in k-blocks.
constexpr double kUnitCost = 4.0, kSliceCost = 0.009, kChangeCost = 0.04, kPartialCost = 10.3e-6;
SkPlan make_plan(int M, int N, int K, int group, int sms) {
    const int bn = skinny_bn(M), nkb = K / kBK, nslabs = N / 128;
    const int max_blocks = sms < kUnitMaxBlocks ? sms : kUnitMaxBlocks;
    SkPlan best;
    double best_cost = 1e30;
    for (int ck = kSkStageTiles; ck <= skinny_max_ck(bn, group); ck += kSkStageTiles) {
        const int chunks = (nkb + ck - 1) / ck;
        const double change = kChangeCost * bn * ck;
        auto cut = [&](double limit, UnitStarts* st) {           // blocks needed
            int blocks = 0;
            double load = 1e30;
            for (int c = 0; c < chunks; ++c) {
                const int nt = nkb - c * ck < ck ? nkb - c * ck : ck;
                const double unit = nt + kUnitCost;
                for (int left = nslabs; left > 0;) {
                    const double extra = (left == nslabs && blocks > 0) ? change : 0.0;   // a block that goes on into this chunk
                    int fit = (int)((limit - load - extra) / unit);
                    if (load > 1e29 || fit < 1) {
                        if (blocks >= kUnitMaxBlocks) return kUnitMaxBlocks + 1;
                        if (st) st->v[blocks] = c * nslabs + (nslabs - left);
                        ++blocks;
                        load = 0.0;
                        fit = (int)(limit / unit);
                        if (fit < 1) return kUnitMaxBlocks + 1;
                    } else {
                        load += extra;
                    }
                    const int take = fit < left ? fit : left;
                    load += take * unit;
                    left -= take;
                }
            }
            if (st) for (int b = blocks; b <= kUnitMaxBlocks; ++b) st->v[b] = chunks * nslabs;
            return blocks;
        };
        double lo = ((double)nkb * nslabs) / max_blocks, hi = lo + 2.0 * (ck + kUnitCost) + change + chunks;
        while (cut(hi, nullptr) > max_blocks) hi *= 1.25;
        for (int i = 0; i < 12; ++i) {
            const double mid = 0.5 * (lo + hi);
            if (cut(mid, nullptr) <= max_blocks) hi = mid; else lo = mid;
        }
        const double cost = hi + kSliceCost * bn * (ck < nkb ? ck : nkb) + kPartialCost * chunks * M * N;
        if (cost < best_cost) {
            best_cost = cost;
            best.ck = ck;
            best.blocks = cut(hi, &best.starts);
        }
        if (ck >= nkb) break;
    }
    return best;
}

// Plans are pure functions of the problem; the last few are kept (some 20 us each to make).  Fills
// *out if it is given and returns the chunk length.
int plan_for(int M, int N, int K, int group, int sms, SkPlan* out) {
    struct Entry { int key[5]; SkPlan plan; };
    constexpr int kEntries = 64;
    static Entry table[kEntries];
    static int used = 0, next = 0;
    static std::mutex mutex;
    const int key[5] = {M, N, K, group, sms};
    {
        std::lock_guard<std::mutex> lock(mutex);
        for (int i = 0; i < used; ++i)
            if (!std::memcmp(table[i].key, key, sizeof(key))) {
                if (out) *out = table[i].plan;
                return table[i].plan.ck;
            }
    }
    const SkPlan p = make_plan(M, N, K, group, sms);
    if (out) *out = p;
    std::lock_guard<std::mutex> lock(mutex);
    std::memcpy(table[next].key, key, sizeof(key));
    table[next].plan = p;
    if (used < kEntries) ++used;
    next = (next + 1) % kEntries;
    return p.ck;
}

template <int G, int BN, bool XS, bool EXACT>
cudaError_t launch_one_skinny(cudaLaunchConfig_t& cfg, const CUtensorMap& xmap, const SkMaps& maps, const float* inv_s,
                              float* partial, int M, int nslabs, int K, int R, const SkPlan& plan,
                              unsigned int* status_word) {
    static bool done[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (!done[dev & 63]) {
        e = cudaFuncSetAttribute(gemm_skinny_kernel<G, BN, XS, EXACT>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSkMaxSmem);
        if (e != cudaSuccess) return e;
        done[dev & 63] = true;
    }
    return cudaLaunchKernelEx(&cfg, gemm_skinny_kernel<G, BN, XS, EXACT>, xmap, maps, inv_s, partial, M, nslabs, K, plan.ck, R,
                              plan.starts, status_word);
}

}  // namespace

bool gemm_skinny_applies(int M, int N, int K, int group) {
    return M >= 1 && M <= 64 && N % 128 == 0 && K % 128 == 0 && (group == 64 || group == 128) &&
           encode_fn() != nullptr;
}

size_t gemm_skinny_workspace_bytes(int M, int N, int K, int group, int sms) {
    const int ck = plan_for(M, N, K, group, sms, nullptr);
    return kCounterBytes + (size_t)((K / kBK + ck - 1) / ck) * M * N * sizeof(float);
}

cudaError_t launch_gemm_skinny(const void* x, const GemvMatrix* mats, int count, int M, int K, int group,
                               const float* inv_s, void* workspace, unsigned int* status_word, int sms,
                               bool serialize, cudaStream_t st) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return cudaErrorNotSupported;
    const bool exact = M <= 32;
    int N = 0;
    for (int i = 0; i < count; ++i) N += mats[i].n;
    SkPlan plan;
    plan_for(M, N, K, group, sms, &plan);
    const int bn = skinny_bn(M), ck = plan.ck;
    const int ng = K / group, gpc = ck / (group / kBK);
    const cuuint32_t estr[2] = {1, 1};
    CUtensorMap xmap;
    SkMaps maps;
    SkOutputs out;
    {
        // x as [M][K] fp16 in boxes of BN tokens x one k-block, 128-byte swizzle; rows past M read as zeros
        const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)M};
        const cuuint64_t strides[1] = {(cuuint64_t)K * 2};
        const cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)bn};
        if (enc(&xmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void*>(x), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    int slabs = 0;
    for (int i = 0; i < kMaxMulti; ++i) {
        if (i < count) {
            const GemvMatrix& m = mats[i];
            slabs += m.n / 128;
            out.y[i] = static_cast<__half*>(m.y);
            // packed weights: one row of K * 8 bytes per band, as 64-bit elements; boxes of 8 bands x 4 k-blocks
            const cuuint64_t wdims[2] = {(cuuint64_t)K, (cuuint64_t)(m.n / 16)}, wstr[1] = {(cuuint64_t)K * 8};
            const cuuint32_t wbox[2] = {(cuuint32_t)(kSkStageTiles * 64), 8};
            // scales: fp16 [band][group][16]; boxes of 8 bands x a chunk's groups
            const cuuint64_t sdims[2] = {(cuuint64_t)ng * 16, (cuuint64_t)(m.n / 16)}, sstr[1] = {(cuuint64_t)ng * 32};
            const cuuint32_t sbox[2] = {(cuuint32_t)(gpc * 16), 8};
            // zero points: bytes [band pair][group][16]; boxes of 4 pairs x a chunk's groups
            const cuuint64_t zdims[2] = {(cuuint64_t)ng * 16, (cuuint64_t)(m.n / 32)}, zstr[1] = {(cuuint64_t)ng * 16};
            const cuuint32_t zbox[2] = {(cuuint32_t)(gpc * 16), 4};
            if (enc(&maps.w[i], CU_TENSOR_MAP_DATA_TYPE_UINT64, 2, const_cast<void*>(m.qweight), wdims, wstr, wbox, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS ||
                enc(&maps.sc[i], CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void*>(m.scales), sdims, sstr, sbox, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS ||
                enc(&maps.z[i], CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(m.zeros), zdims, zstr, zbox, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
                return cudaErrorInvalidValue;
        } else {
            maps.w[i] = maps.w[0]; maps.sc[i] = maps.sc[0]; maps.z[i] = maps.z[0];      // never used
            out.y[i] = out.y[0];
        }
        maps.slab_end[i] = slabs;
        out.end[i] = slabs * 128;
    }
    float* partial = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(workspace) + kCounterBytes);
    const int chunks = (K / kBK + ck - 1) / ck;
    const int xbytes = ck * bn * 128, ibytes = inv_s ? ck * kBK * 4 : 0;
    int R = (kSkMaxSmem - kSkFixed - xbytes - ibytes) / kSkStageBytes;
    if (R > kSkMaxRing) R = kSkMaxRing;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3((unsigned)plan.blocks);
    cfg.blockDim = dim3(exact ? kSkExactThreads : kSkThreads);
    cfg.dynamicSmemBytes = (size_t)(kSkFixed + xbytes + ibytes + R * kSkStageBytes);
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = serialize ? 0 : 1;
    cudaError_t e;
#define AWQ_SK_LAUNCH(GG, BNN, EX)                                                                                        \
    e = inv_s ? launch_one_skinny<GG, BNN, true, EX>(cfg, xmap, maps, inv_s, partial, M, slabs, K, R, plan, status_word)  \
              : launch_one_skinny<GG, BNN, false, EX>(cfg, xmap, maps, inv_s, partial, M, slabs, K, R, plan, status_word)
#define AWQ_SK_PICK(GG)                                                                             \
    do {                                                                                            \
        if (bn == 16) AWQ_SK_LAUNCH(GG, 16, true);                                           \
        else if (bn == 32) AWQ_SK_LAUNCH(GG, 32, true);                                               \
        else AWQ_SK_LAUNCH(GG, 64, false);                                                          \
    } while (0)
    if (group == 128) AWQ_SK_PICK(128); else AWQ_SK_PICK(64);
#undef AWQ_SK_PICK
#undef AWQ_SK_LAUNCH
    if (e != cudaSuccess) return e;
    count_launch();
    cfg.gridDim = dim3((unsigned)((N / 4 + 255) / 256), (unsigned)M);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = 0;
    cfg.numAttrs = 1;
    // loads in flight: eight only where that many chunks are there (28672 -> 8192 at 16 tokens, 16 chunks: 40.2 -> 36.6 us;
    // 8192 -> 28672, 5 chunks: 38.5 us with eight, 37.6 us with four; 4096 -> 4096, 4 chunks: 7.9 and 6.9 us)
    e = chunks > 8 ? cudaLaunchKernelEx(&cfg, skinny_reduce_kernel<8>, (const float*)partial, out, chunks, M, N)
                   : cudaLaunchKernelEx(&cfg, skinny_reduce_kernel<4>, (const float*)partial, out, chunks, M, N);
    if (e != cudaSuccess) return e;
    count_launch();
    return cudaGetLastError();
}

}  // namespace awq
