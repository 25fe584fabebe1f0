// Thin inline-PTX wrappers for the asynchronous machinery of sm_100a: mbarriers, bulk (TMA) copies,
// proxy fences and the tcgen05 tensor-core / tensor-memory instructions.  Every wait is bounded.
#pragma once
#include <stdint.h>

namespace tf {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// The next 1024-byte boundary of dynamic shared memory.  An offset from the array, not a rounded address: the compiler then
// still knows that it points into shared memory and uses shared-memory instructions (32-bit addresses, shorter latency)
// for everything that is reached through it.  With a rounded address it fell back to generic ones: a GEMV of 20 MB took
// 6.7 / 8.4 / 10.6 us at 1 / 4 / 16 tokens, with this 6.4 / 7.8 / 9.5.
__device__ __forceinline__ uint8_t* align_shared(uint8_t* p) { return p + ((0u - smem_u32(p)) & 1023u); }

// True in one lane of a converged warp, the same one every time.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.b32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}

// ---- mbarrier ----------------------------------------------------------------------------------
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_init_fence() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    return done != 0;
}
// The same without the moment for which a thread may be held up.
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    return done != 0;
}

// Bounded waits.  A wait gives up after about a second of polling, or as soon as another thread of the CTA has given up
// (`abort_flag[0]` != 0).  On giving up it records `site` in the flag and returns false; the caller must then leave its role loop
// and go to the common teardown.
// Of the threads of a warp that poll for themselves one may see the data arrive and the next the limit run out; the first would go
// on to a shuffle, a vote or an MMA of the whole warp and wait there, without a limit, for threads that have left.  So a
// role of one thread waits with mbar_wait, a role of a whole warp with mbar_wait_warp (or a loop of its own around
// wait_given_up), which decides by a vote.
// `abort_flag` points at two words of shared memory: [0] the flag, [1] the limit of a wait in units of 1024
// cycles, written once by the CTA's first thread from the kernel's `debug` argument (see wait_limit_kcycles).
constexpr long long kWaitLimitCycles = 2000000000ll;
// Kernel argument `debug` (0 in normal operation; set through tf_debug_inject for tests of the failure path):
// bit 0 = the packed-weight producer issues no copies, so every wait for weights runs out; bits 8..31 = limit of a
// wait in units of 1024 cycles (0 = the default of about a second).
constexpr uint32_t kDebugDropWeights = 1u;
__device__ __forceinline__ uint32_t wait_limit_kcycles(uint32_t debug) {
    return (debug >> 8) != 0 ? (debug >> 8) : (uint32_t)(kWaitLimitCycles >> 10);
}
__device__ __forceinline__ bool wait_expired(long long t_begin, volatile uint32_t* abort_flag) {
    return clock64() - t_begin > ((long long)abort_flag[1] << 10);
}
// One turn of a converged warp's wait that has not been met yet: whether the warp, all of it, gives up.
__device__ __forceinline__ bool wait_given_up(long long t_begin, volatile uint32_t* abort_flag, uint32_t site) {
    const bool expired = wait_expired(t_begin, abort_flag);
    if (expired && *abort_flag == 0) *abort_flag = site;
    return __any_sync(0xFFFFFFFFu, expired || *abort_flag != 0);
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag,
                                          uint32_t site) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    for (uint32_t it = 1;; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 0xFFu) == 0) {
            if (*abort_flag != 0) return false;
            if (wait_expired(t0, abort_flag)) {
                *abort_flag = site;
                return false;
            }
        }
    }
}

// The same by a whole converged warp, which leaves it by a vote.  (The compiler then also knows that what the loop around it
// carries is uniform in the warp and keeps it in uniform registers, where tcgen05.mma wants its operands.
// The limit is looked at on every turn: looked at on every 256th, with a counter, the GEMM's dequant warps spilled, 2048x4096x14336
// 187.9 us against 185.9.)
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag, uint32_t site) {
    if (__all_sync(0xFFFFFFFFu, mbar_try_wait(bar, parity))) return true;
    const long long t0 = clock64();
    while (!__all_sync(0xFFFFFFFFu, mbar_try_wait(bar, parity)))
        if (wait_given_up(t0, abort_flag, site)) return false;
    return true;
}

// ---- programmatic dependent launch -------------------------------------------------------------------
// Let the next kernel of the stream start launching now; it still has to call grid_dependency_wait()
// before it touches anything this kernel writes.
__device__ __forceinline__ void grid_launch_dependents() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// Block until every kernel this one depends on has completed and its writes are visible.
__device__ __forceinline__ void grid_dependency_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
// Loads of what earlier kernels of the stream have written, for a kernel that may have started before they ended: volatile, which
// keeps them behind the wait, and coherent.  (__ldg and const __restrict__ promise data that nobody writes while the grid exists.
// __ldcg and __ldcs promise nothing, but the compiler takes them for functions of the address and may move them ahead of a wait or out of a
// loop.)
__device__ __forceinline__ uint32_t load_behind_wait(const uint16_t* p) {
    uint16_t v;
    asm volatile("ld.global.u16 %0, [%1];" : "=h"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ uint32_t load_behind_wait(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ uint2 load_behind_wait(const uint2* p) {
    uint2 v;
    asm volatile("ld.global.cg.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ float4 load_behind_wait(const float4* p) {
    float4 v;
    asm volatile("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ uint2 load_once_behind_wait(const uint2* p) {       // not wanted again: first to leave the L2
    uint2 v;
    asm volatile("ld.global.cs.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}

// ---- thread-block clusters ---------------------------------------------------------------------------
// Address of the same shared-memory location in CTA `rank` of this cluster (shared::cluster window).
__device__ __forceinline__ uint32_t map_to_cta(uint32_t smem_addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr), "r"(rank));
    return r;
}
__device__ __forceinline__ uint32_t cta_rank_in_cluster() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// Arrival on an mbarrier of any CTA of the cluster, and the wait for such arrivals.  For what lies in tensor memory: tcgen05.wait has it done,
// tcgen05.fence::before_thread_sync puts it ahead of the arrival and ::after_thread_sync behind the wait, and for that order the arrival itself may be
// relaxed, but its scope has to hold the waiting thread, which the default (the arriving CTA) does not.  It orders nothing else.  (As a release for the
// cluster it waits for everything that the thread has on its way: 2700 cycles in the GEMM's dequantization warps, where this takes 50 to 100.)
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_bar) {
    asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait_cluster(uint32_t bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    return done != 0;
}
__device__ __forceinline__ bool mbar_wait_warp_cluster(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag, uint32_t site) {
    if (__all_sync(0xFFFFFFFFu, mbar_try_wait_cluster(bar, parity))) return true;
    const long long t0 = clock64();
    while (!__all_sync(0xFFFFFFFFu, mbar_try_wait_cluster(bar, parity)))
        if (wait_given_up(t0, abort_flag, site)) return false;
    return true;
}
// Hardware barrier over all threads of the cluster.
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// ---- stmatrix: four 8 x 8 matrices of 16-bit elements, transposed; lanes 8i .. 8i + 7 give the row addresses of matrix i ----
__device__ __forceinline__ void stmatrix_x4_trans(uint32_t smem_addr, const uint32_t m[4]) {
    asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1,%2,%3,%4};" ::"r"(smem_addr), "r"(m[0]), "r"(m[1]), "r"(m[2]), "r"(m[3]) : "memory");
}

// ---- bulk (TMA) copies ----------------------------------------------------------------------------
// 1-D bulk copy global -> shared; both addresses 16-byte aligned, bytes % 16 == 0.
__device__ __forceinline__ void bulk_copy_g2s(uint32_t dst_smem, const void* src_gmem, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst_smem),
                 "l"(src_gmem), "r"(bytes), "r"(bar)
                 : "memory");
}
// 3-D tiled tensor copy global -> shared memory of this CTA only; x = innermost coordinate (x * elem size % 16 == 0).
__device__ __forceinline__ void tma_load_3d(uint32_t dst_smem, const void* tensor_map, int x, int y, int z, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cta.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst_smem),
        "l"(tensor_map), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void mbar_arrive_n(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void prefetch_tensormap(const void* tensor_map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(tensor_map) : "memory");
}

// ---- tcgen05: tensor memory and MMA ------------------------------------------------------------------
__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols) {   // whole warp
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {                               // whole warp
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {    // whole warp
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// D[tmem] (+)= A[tmem] . B[smem desc], kind::f16 (bf16 inputs, fp32 accumulate); one thread issues.  The 128-row
// operand A is read from tensor memory: 128 lanes x 8 columns of bf16 pairs per 16 k.
__device__ __forceinline__ void tc_mma_f16_tmem_a(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                                  uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// Arrive on an mbarrier once every tcgen05.mma issued so far by this thread has completed.
__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// ---- the same for a pair of CTAs (a cluster of two): one MMA of 256 rows, 128 in the tensor memory of either CTA (operand and sums, at the same
// address in both), whose other operand lies half in the shared memory of either (at the same address).  One thread of the CTA of
// even rank issues; tensor memory is allocated and freed by a warp of both.
__device__ __forceinline__ void tmem_alloc_pair(uint32_t dst_smem, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_mma_f16_tmem_a_pair(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// ... on the mbarrier at this address in both CTAs
__device__ __forceinline__ void tc_commit_pair(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar), "h"((uint16_t)3) : "memory");
}
// To this CTA's shared memory; `bar` (a cluster address) may be the other CTA's.
__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst_smem, const void* tensor_map, int x, int y, int z, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst_smem),
        "l"(tensor_map), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}
// Store 16 lanes x 16 columns (8 registers per thread): thread (g = lane/4, t = lane%4), register 4i+j holds
// TMEM lane (g + 8*(j>>1)), column 8i + 2t + (j&1) relative to `taddr` (whose lane must be a multiple of 16).
__device__ __forceinline__ void tmem_st_16x256b_x2(uint32_t taddr, const uint32_t r[8]) {
    asm volatile("tcgen05.st.sync.aligned.16x256b.x2.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]),
                 "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                 : "memory");
}
__device__ __forceinline__ void tmem_st_wait() {
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
// 32 lanes x 8 or 16 columns as 8 x 8 matrices: thread (g, t) gets of lane 16h + 8j + g, columns 8c + 2t and 8c + 2t + 1, the values
// v[4 C h + 4c + 2j] and the next (C = 1 or 2 matrices side by side).  They are there after the wait.
__device__ __forceinline__ void tmem_ld_16x256b(uint32_t taddr, float (&v)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%4];" : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "r"(taddr) : "memory");
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%4];"
                 : "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]) : "r"(taddr + (16u << 16)) : "memory");
}
__device__ __forceinline__ void tmem_ld_16x256b(uint32_t taddr, float (&v)[16]) {
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]) : "r"(taddr) : "memory");
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=f"(v[8]), "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15]) : "r"(taddr + (16u << 16)) : "memory");
}
// The wait makes the values, as the compiler sees it: it cannot use them before.
__device__ __forceinline__ void tmem_ld_wait_for(float (&v)[8]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7])::"memory");
}
__device__ __forceinline__ void tmem_ld_wait_for(float (&v)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7]), "+f"(v[8]), "+f"(v[9]), "+f"(v[10]),
                   "+f"(v[11]), "+f"(v[12]), "+f"(v[13]), "+f"(v[14]), "+f"(v[15])::"memory");
}

// Shared-memory matrix descriptor for a K-major bf16 operand stored as rows of 128 bytes (64 k)
// with the 128-byte swizzle (16-byte chunk index XOR (row & 7)); 8-row groups are 1024 bytes apart.
__device__ __forceinline__ uint64_t umma_desc_k_sw128(uint32_t smem_addr) {
    uint64_t d = 0;
    d |= static_cast<uint64_t>((smem_addr & 0x3FFFFu) >> 4);          // start address        bits  0..13
    d |= static_cast<uint64_t>(1) << 16;                              // leading byte offset   (unused here)
    d |= static_cast<uint64_t>(1024 >> 4) << 32;                      // stride byte offset    bits 32..45
    d |= static_cast<uint64_t>(1) << 46;                              // descriptor version (sm_100)
    d |= static_cast<uint64_t>(2) << 61;                              // layout: 128-byte swizzle
    return d;
}
// Instruction descriptor: bf16 x bf16 -> fp32, both operands K-major, D is m x n.
__host__ __device__ constexpr uint32_t umma_idesc_bf16(int m, int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(n >> 3) << 17) |
           (static_cast<uint32_t>(m >> 4) << 24);
}

}  // namespace tf
