// tcgen05 / TMA wrappers (inline PTX) and tensor-map helpers shared by the prefill kernels.
#pragma once
#include <cuda.h>

#include <mutex>

#include "async_copy.cuh"
#include "common.cuh"

namespace awq {

constexpr int kBK = 64;   // k-block: 64 input channels = one 128-byte swizzle row of fp16

// ------------------------------------------------------------------ small PTX wrappers
// One lane of a converged warp, chosen the same way every time.  The warps that issue copies and products
// run their whole loop converged - every lane polls the barriers and forms the operands - and only the
// instruction itself is predicated on this lane.  With the loop inside `if (lane == 0)` a thread issued a
// product per ~80 - 105 cycles; converged, 8192 -> 28672 at 32 tokens went from 64 to 49 us.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p) :: "memory");
    return p != 0;
}
// the bounded wait of a converged warp: true only if no lane gave up
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, const WaitCtl& ctl) {
    return __all_sync(0xFFFFFFFFu, mbar_wait(bar, parity, ctl));
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(bar) : "memory");
}
// shared -> global tensor store of one box (bulk async-group completion)
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, int c0, int c1, uint32_t src) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];"
                 ::"l"(map), "r"(c0), "r"(c1), "r"(src) : "memory");
}
__device__ __forceinline__ void bulk_commit_group() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// wait until at most one / none of this thread's store groups still reads shared memory
__device__ __forceinline__ void bulk_wait_read_1() { asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// D (tensor memory) += A (tensor memory: 128 lanes x 8 columns of fp16 pairs per K = 16) * B (smem)
__device__ __forceinline__ void umma_f16_a_tmem(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                                uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// A warp stores 16 lanes x 32 columns: four blocks of 8 columns, each in the 16x256b register
// layout (lane-group g = lane / 4 holds rows g and g+8; t = lane % 4 holds columns 2t, 2t+1 of
// the block; registers 4i .. 4i+3 of block i = (g, 2t) (g, 2t+1) (g+8, 2t) (g+8, 2t+1)).
__device__ __forceinline__ void tmem_st_16x32cols(uint32_t taddr, const uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.16x256b.x4.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
        "%14, %15, %16};"
        ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
          "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
        : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// ------------------------------------------------------------------ pairs of blocks (clusters of two)
__device__ __forceinline__ uint32_t cluster_ctarank() {
    uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r;
}
__device__ __forceinline__ uint32_t cluster_id_x() {
    uint32_t r; asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r)); return r;
}
__device__ __forceinline__ uint32_t num_clusters_x() {
    uint32_t r; asm volatile("mov.u32 %0, %%nclusterid.x;" : "=r"(r)); return r;
}
// address of the same shared-memory location in block `rank` of the cluster
__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank) {
    uint32_t r; asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank)); return r;
}
// Arrival on a barrier of another block of the cluster.  What is handed over lives in tensor memory or was written by the copy
// engine, and tcgen05.fence::before_thread_sync orders it; or (x in the stream kernel) it lies in the arriving block's own shared
// memory, fenced to the asynchronous proxy, and only that block's half of the products reads it.  So the default release at
// block scope is used; a cluster-scope release costs about a thousand cycles per arrival here.
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// Between the blocks of a cluster.  At the start of a kernel nothing is handed over but the barriers' initialisation, which has a
// fence of its own, so the arrival may be relaxed.
__device__ __forceinline__ void cluster_arrive_start() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// In front of a block's end, which gives its shared memory away: no arrival of the other block may still be on the way there.
// Either every remote arrival has been waited for by then (the warp that issues the products waits for the last ones too), or the
// block is giving up and the barrier releases what is under way.  (Releasing always made the launches 0.4 us longer: the
// epilogue's stores to global memory are under way as well.)
__device__ __forceinline__ void cluster_sync_end(bool gave_up) {
    if (gave_up) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    else asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    cluster_wait();
}
// D (both blocks' tensor memory) += A (tensor memory, 128 lanes per block) * B (both blocks' smem)
__device__ __forceinline__ void umma_pair_f16_a_tmem(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc,
                                                     uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, rows of 128 bytes,
// 8-row atoms 1024 bytes apart.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);          // start address, 16-byte units
    d |= (uint64_t)1 << 16;                           // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(1024 >> 4) << 32;                 // stride byte offset between 8-row atoms
    d |= (uint64_t)1 << 46;                           // descriptor version (sm_100)
    d |= (uint64_t)2 << 61;                           // layout: 128-byte swizzle
    return d;
}

// Instruction descriptor: D fp32, A and B fp16, both K-major, M = 128, N = BN.
__host__ __device__ constexpr uint32_t instr_desc(int bn) {
    return (1u << 4) | (0u << 7) | (0u << 10) | ((uint32_t)(bn >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

__device__ __forceinline__ uint32_t hsub2_u32(uint32_t a, uint32_t b) {
    uint32_t d; asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b)); return d;
}
__device__ __forceinline__ uint32_t hfma2_u32(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t d; asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c)); return d;
}
__device__ __forceinline__ uint32_t hmul2_u32(uint32_t a, uint32_t b) {
    uint32_t d; asm("mul.rn.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b)); return d;
}

// Two codes of a packed word as fp16: (w & mask) | 0x6400 in both halves, i.e. 1024 + q (low nibbles) or
// 1024 + 16 q (high ones).  Asked for as one three-input instruction with both constants in registers: written
// as C, 16 packed words with four tensor-memory stores of four warps per scheduler took 420 cycles a warp, like
// this they take 340.
__device__ __forceinline__ uint32_t code_pair(uint32_t w, uint32_t mask) {
    uint32_t d; asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(d) : "r"(w), "r"(mask), "r"(0x64006400u)); return d;
}
constexpr uint32_t kLowCodes = 0x000F000Fu, kHighCodes = 0x00F000F0u;

__device__ __forceinline__ void tmem_ld_32cols(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr) : "memory");
}
// Waits for this thread's loads from tensor memory.  The loaded registers pass through it: a load's outputs
// are ordinary values to the compiler from the load on, and nothing else would keep arithmetic on
// them behind the wait.
template <int C>
__device__ __forceinline__ void tmem_loaded(uint32_t (&r)[C]) {
#pragma unroll
    for (int i = 0; i < C; ++i) asm volatile("" : "+r"(r[i]));
}
template <int... C>
__device__ __forceinline__ void tmem_ld_wait(uint32_t (&... r)[C]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    (tmem_loaded(r), ...);
}

// ------------------------------------------------------------------------------ host
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}


// the pair (two-SM) kernel: weight map with a box of 256 words; an optional workspace enables stream-K
// tile balancing
bool gemm_pair_applies(int M, int N);
size_t gemm_pair_workspace_bytes(int sms);
double gemm_pair_estimate(int M, int N, int K, int sms, size_t workspace_bytes);
cudaError_t launch_gemm_pair(const void* x, const CUtensorMap& wmap, const CUtensorMap& ymap,
                             const void* scales, const void* zeros, int M, int N, int K, int group,
                             void* workspace, size_t workspace_bytes,
                             unsigned int* status_word, int sms, bool serialize, cudaStream_t st, bool* launched,
                             int count = 1, int rows = 0);     // count products of N / count channels, rows of x and y apart

}  // namespace awq
