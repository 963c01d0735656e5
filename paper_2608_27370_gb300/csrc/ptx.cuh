// ptx.cuh -- thin inline-PTX wrappers for sm_103a (Blackwell) used by the
// quantise and GEMM kernels: mbarriers, TMA (cp.async.bulk.tensor), bulk
// copies, and the tcgen05 tensor-core / tensor-memory instructions.
// Every wrapper is one documented PTX instruction (PTX ISA 8.7+) or a few.
#pragma once

#include <cuda.h>
#include <cstdint>

#define PURO_DEV __device__ __forceinline__

namespace puro {

PURO_DEV uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// 1 in one lane of the warp (always the same one), 0 in the others.  The forms
// below with a suffix _e are run by a whole warp and take effect in that lane,
// so that their operands can stay in uniform registers.
PURO_DEV uint32_t elect_one() {
    uint32_t r;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(r));
    return r;
}

PURO_DEV uint64_t global_timer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// --------------------------------------------- programmatic dependent launch
// Kernels are launched with programmatic stream serialisation: a kernel may
// start (and run its prologue: barrier set-up, tensor-memory allocation,
// descriptor prefetch) while the previous kernel on the stream finishes.
// pdl_wait() blocks until the previous kernels have completed and their
// memory is visible; every kernel calls it before it writes global memory and
// before it reads any that the kernel just before may write, and only then
// pdl_launch_dependents(), which lets the next kernel start launching.  So what
// the kernel before the previous one wrote is complete when a kernel starts.
// Two accesses come before the wait: the RMSNorm quantiser's first tile of h
// (see launch_quantize_rmsnorm) and the GEMM's prefetch of B into L2, which
// delivers nothing.
PURO_DEV void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
PURO_DEV void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ------------------------------------------------------ named barriers
// Barrier `id` (1..15) among `threads` threads (a multiple of 32); with the
// AND of every participant's predicate.
PURO_DEV void named_bar_sync(uint32_t id, uint32_t threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
// Arrive without waiting (others wait with named_bar_sync).
PURO_DEV void named_bar_arrive(uint32_t id, uint32_t threads) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
PURO_DEV bool named_bar_and(uint32_t id, uint32_t threads, bool pred) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.and.pred q, %2, %3, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"(pred ? 1u : 0u), "r"(id), "r"(threads)
        : "memory");
    return r != 0;
}

// ---------------------------------------------------------------- mbarrier
PURO_DEV void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

PURO_DEV void fence_mbarrier_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Order this thread's generic-proxy shared-memory writes before later
// async-proxy operations (TMA stores, tcgen05.cp / tcgen05.mma reads).
PURO_DEV void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

PURO_DEV void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

PURO_DEV bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Non-blocking test of the phase with the given parity (never suspends).
PURO_DEV bool mbar_test_wait(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wait for the phase with the given parity to complete, giving up after
// `timeout_ns` of wall time (%globaltimer).  Returns false on time-out.
PURO_DEV bool mbar_wait_bounded(uint64_t *bar, uint32_t parity, uint64_t timeout_ns) {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = global_timer_ns();
    while (true) {
        if (mbar_try_wait(bar, parity)) return true;
        if (global_timer_ns() - t0 > timeout_ns) return false;
    }
}

// ------------------------------------------------------------------- TMA
PURO_DEV void tma_prefetch_desc(const CUtensorMap *map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

// 2-D tiled load global -> shared, completion counted on `bar` (bytes).
PURO_DEV void tma_load_2d(void *dst, const CUtensorMap *map, uint64_t *bar, int32_t x, int32_t y) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4}], [%2];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y)
        : "memory");
}

// 2-D tiled store shared -> global (bulk-group completion).
PURO_DEV void tma_store_2d(const CUtensorMap *map, const void *src, int32_t x, int32_t y) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(smem_u32(src)), "r"(x), "r"(y)
                 : "memory");
}

// (with its commit)
PURO_DEV void tma_store_2d_e(uint32_t e, const CUtensorMap *map, const void *src, int32_t x, int32_t y) {
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %4, 0;\n\t"
        "@q cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];\n\t"
        "@q cp.async.bulk.commit_group;\n\t}" ::"l"(reinterpret_cast<uint64_t>(map)),
        "r"(smem_u32(src)), "r"(x), "r"(y), "r"(e)
        : "memory");
}

// 2-D tiled element-wise add shared -> global (bulk-group completion): each
// element of the box is added to the global tensor's element (the tensor
// map's type; f32 adds round to nearest).
PURO_DEV void tma_reduce_add_2d(const CUtensorMap *map, const void *src, int32_t x, int32_t y) {
    asm volatile("cp.reduce.async.bulk.tensor.2d.global.shared::cta.add.tile.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(smem_u32(src)), "r"(x), "r"(y)
                 : "memory");
}

// Contiguous bulk copy global -> shared; both addresses 16-byte aligned,
// bytes a multiple of 16.
PURO_DEV void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

PURO_DEV void bulk_commit_group() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// Wait until all committed bulk stores have finished reading shared memory.
PURO_DEV void bulk_wait_group_read0() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
// Wait until at most N committed bulk stores still read shared memory.
template <int N>
PURO_DEV void bulk_wait_group_read() { asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory"); }
// Wait until all committed bulk stores are complete.
PURO_DEV void bulk_wait_group0() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// ------------------------------------------------------------- tcgen05
// Tensor memory: 128 lanes x 512 columns of 32-bit cells per SM.  An
// address is (lane << 16) | column.

// The GEMM runs every tcgen05 operation as a CTA pair (cta_group::2): the
// two CTAs of a 2-CTA cluster allocate the same tensor-memory columns
// collectively (one warp in each), a pair MMA issued by one thread of the
// even CTA reads A and B from both CTAs' shared memory (each holds its own
// 128 rows of A and half of the N rows of B) and writes each CTA's 128 rows
// of D into that CTA's tensor memory, and a pair tcgen05.cp copies each
// CTA's shared memory into its own tensor memory.  All tcgen05 instructions
// of a kernel use the same cta_group.

PURO_DEV uint32_t cluster_ctarank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// Store to shared memory of a cluster CTA (16-byte aligned address from mapa_shared).
PURO_DEV void st_cluster_v4(uint32_t addr, const uint4 &v) {
    asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
                 : "memory");
}

// Barrier of all threads of all CTAs of the cluster (release / acquire), in two
// halves for work in between.
PURO_DEV void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
PURO_DEV void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// Address of the same shared-memory variable in cluster CTA `rank`.
PURO_DEV uint32_t mapa_shared(uint32_t saddr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
    return r;
}

// Arrive on an mbarrier given by its shared::cluster address (this CTA's or
// a peer's), releasing this thread's prior writes at cluster scope.
PURO_DEV void mbar_arrive_cluster(uint32_t bar_cluster) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar_cluster) : "memory");
}

// The same arrive with release semantics at CTA scope only (the default of
// mbarrier.arrive).  For a signal that publishes no generic memory -- an
// epilogue telling the MMA thread that its tcgen05.ld reads of an
// accumulator are done, ordered by tcgen05.wait::ld and the tcgen05 fences
// around the barrier -- this is enough, and it does not wait, as the
// cluster-scope release does, for the thread's earlier memory operations
// (measured: about 1,500 cycles per arrive behind the epilogue's stores).
PURO_DEV void mbar_arrive_cluster_cta_scope(uint32_t bar_cluster) {
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar_cluster) : "memory");
}

// 2-D tiled load into this CTA's shared memory whose completion is counted
// on an mbarrier that may live in the peer CTA of the pair.
PURO_DEV void tma_load_2d_pair_e(uint32_t e, void *dst, const CUtensorMap *map, uint32_t bar_cluster, int32_t x,
                                 int32_t y) {
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %5, 0;\n\t"
        "@q cp.async.bulk.tensor.2d.shared::cta.global.tile.mbarrier::complete_tx::bytes.cta_group::2"
        " [%0], [%1, {%2, %3}], [%4];\n\t}" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar_cluster), "r"(e)
        : "memory");
}

// The 128-byte line at p into L2 (a hint: nothing waits for it).
PURO_DEV void prefetch_l2(const void *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

PURO_DEV void tmem_alloc_pair(uint32_t *dst_smem, uint32_t ncols) {  // one warp in each CTA of the pair
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
                 "r"(ncols)
                 : "memory");
}
PURO_DEV void tmem_relinquish_alloc_permit_pair() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
PURO_DEV void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {  // one warp in each CTA of the pair
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
PURO_DEV void tc_fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
PURO_DEV void tc_fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Arrive (once) on `bar` of this CTA when every pair MMA / copy previously
// issued by this thread has completed.
PURO_DEV void tc_commit_pair(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     smem_u32(bar))
                 : "memory");
}

// Each thread of the warp reads 32 consecutive 32-bit columns of its own
// lane (warp w may address lanes 32*(w%4) .. 32*(w%4)+31 only).
PURO_DEV void tmem_ld_32x32b_x32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
          "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
          "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
          "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
PURO_DEV void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Pair MMA D(tmem) (+)= A(smem) * B(smem)^T, kind::f16 (bf16/fp16 inputs,
// f32 accumulate).
PURO_DEV void mma_pair_f16_e(uint32_t e, uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                             uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %5, 0;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(e)
        : "memory");
}
// kind::f8f6f4 (e4m3/e5m2 inputs, f32 accumulate), no block scaling.
PURO_DEV void mma_pair_f8_e(uint32_t e, uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                            uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %5, 0;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(e)
        : "memory");
}
// kind::mxf8f6f4 with one UE8M0 scale per 32 elements of K for each row of
// A and of B (scale_vec::1X); the scales are read from tensor memory (each
// CTA's own: its 128 rows of A, all N rows of B).
PURO_DEV void mma_pair_mxf8_e(uint32_t e, uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                              uint32_t sfa_tmem, uint32_t sfb_tmem, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %7, 0;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::mxf8f6f4.block_scale.scale_vec::1X [%0], %1, %2, %3, [%5], [%6], p;\n\t}\n" ::"r"(
            d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(sfa_tmem), "r"(sfb_tmem), "r"(e)
        : "memory");
}
// Copy 32 rows x 128 bits from shared memory into tensor memory, replicated
// into each of the four 32-lane quarters (warpx4): row r lands in lane r of
// every quarter, its four 32-bit words in columns taddr .. taddr+3.  The
// pair form copies each CTA's shared memory into its own tensor memory.
PURO_DEV void tmem_cp_pair_32x128b_warpx4_e(uint32_t e, uint32_t taddr, uint64_t sdesc) {
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %2, 0;\n\t@q tcgen05.cp.cta_group::2.32x128b.warpx4 [%0], %1;\n\t}" ::"r"(
            taddr),
        "l"(sdesc), "r"(e)
        : "memory");
}
// tc_commit_pair arriving on `bar` in every cluster CTA of `cta_mask`.
PURO_DEV void tc_commit_pair_multicast_e(uint32_t e, uint64_t *bar, uint16_t cta_mask) {
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %2, 0;\n\t"
        "@q tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n\t}" ::"r"(
            smem_u32(bar)),
        "h"(cta_mask), "r"(e)
        : "memory");
}

// ------------------------------------------------- matrix descriptors
// Shared-memory matrix descriptor (tcgen05 form):
//   [0,14)  start address >> 4       [16,30) leading byte offset >> 4
//   [32,46) stride byte offset >> 4  [46,49) fixed 0b001
//   [49,52) base offset (0: atoms 1024-byte aligned)
//   [61,64) swizzle: 0 none, 2 = 128-byte swizzle
// K-major operand tile with 128-byte rows and the 128-byte swizzle (the
// layout TMA writes with CU_TENSOR_MAP_SWIZZLE_128B): 8-row atoms of 1024
// bytes, so SBO = 1024; LBO is not used for this layout (encoded 1).
PURO_DEV uint64_t smem_desc_k_sw128(uint32_t saddr) {
    uint64_t d = 0;
    d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
    d |= static_cast<uint64_t>(1) << 16;
    d |= static_cast<uint64_t>(1024 >> 4) << 32;
    d |= static_cast<uint64_t>(1) << 46;
    d |= static_cast<uint64_t>(2) << 61;
    return d;
}

// Un-swizzled K-major layout of 8-row x 16-byte core matrices stored
// contiguously (128 bytes each): SBO = 128 between 8-row groups; a single
// core matrix along K, so LBO is unused (0).  Source form of tcgen05.cp.
PURO_DEV uint64_t smem_desc_plain_16B_rows(uint32_t saddr) {
    uint64_t d = 0;
    d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
    d |= static_cast<uint64_t>(128 >> 4) << 32;
    d |= static_cast<uint64_t>(1) << 46;
    return d;
}

}  // namespace puro
