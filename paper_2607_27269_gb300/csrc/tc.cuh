// Thin inline-PTX wrappers for the sm_100-family tensor-core path:
// tcgen05 (TMEM allocation, MMA, commit, TMEM loads/stores), TMA tensor
// loads and mbarrier transaction counts.
#pragma once

#include <cuda.h>  // CUtensorMap (type only)

#include "common.cuh"

namespace gbmla {
namespace tc {

// ---------------------------------------------------------------- descriptors

// Shared-memory layout (swizzle) codes of the tcgen05 matrix descriptor.
enum : uint32_t { kSwizzleNone = 0, kSwizzle128B = 2, kSwizzle64B = 4, kSwizzle32B = 6 };

// 64-bit shared-memory matrix descriptor: start address, leading- and
// stride-dimension byte offsets (all in 16-byte units), descriptor version 1
// (bits 46-47), swizzle layout in bits 61-63.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes,
                                              uint32_t layout)
{
    uint64_t d = 0;
    d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
    d |= static_cast<uint64_t>((lbo_bytes >> 4) & 0x3FFFu) << 16;
    d |= static_cast<uint64_t>((sbo_bytes >> 4) & 0x3FFFu) << 32;
    d |= static_cast<uint64_t>(1) << 46;
    d |= static_cast<uint64_t>(layout & 7u) << 61;
    return d;
}

// Instruction descriptor of kind::f16 with bf16 A and B and an fp32
// accumulator: D format bits 4-5, A/B format bits 7-9 / 10-12, A/B major
// bits 15/16 (1 = MN-major), N>>3 in bits 17-22, M>>4 in bits 24-28.
__host__ __device__ constexpr uint32_t idesc_bf16_f32(int M, int N, bool a_mn_major, bool b_mn_major)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn_major ? 1u : 0u) << 15) | ((b_mn_major ? 1u : 0u) << 16) |
           (static_cast<uint32_t>(N >> 3) << 17) | (static_cast<uint32_t>(M >> 4) << 24);
}

// ---------------------------------------------------------------- TMEM

__device__ __forceinline__ void tmem_alloc(uint32_t smem_result_addr, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_result_addr),
                 "r"(ncols)
                 : "memory");
}

__device__ __forceinline__ void tmem_relinquish()
{
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

__device__ __forceinline__ void fence_before_sync()
{
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void fence_after_sync()
{
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Warp-collective forms: the whole warp executes them converged and one
// elected lane issues.  A lone lane running the issue loop pays a large
// per-iteration cost for every branch; a converged warp does not.
__device__ __forceinline__ void mma_bf16_elect(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                               uint32_t accumulate)
{
    asm volatile(
        "{\n .reg .pred p, e;\n elect.sync _|e, 0xffffffff;\n setp.ne.b32 p, %4, 0;\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// Four steps of a product whose operands advance by `da` and `db` (16-byte
// units) per step, then a commit to `mbar`: one election for all of it.
__device__ __forceinline__ void mma4_bf16_commit_elect(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                                       uint32_t accumulate, uint32_t da, uint32_t db, uint32_t mbar)
{
    const uint64_t a1 = a_desc + da, a2 = a1 + da, a3 = a2 + da, b1 = b_desc + db, b2 = b1 + db, b3 = b2 + db;
    asm volatile(
        "{\n .reg .pred p, t, e;\n elect.sync _|e, 0xffffffff;\n setp.ne.b32 p, %4, 0;\n setp.eq.b32 t, 0, 0;\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], %5, %6, %3, t;\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], %7, %8, %3, t;\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], %9, %10, %3, t;\n"
        " @e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%11];\n}\n" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "l"(a1), "l"(b1), "l"(a2), "l"(b2), "l"(a3), "l"(b3),
        "r"(mbar)
        : "memory");
}

// Eight steps, likewise.
__device__ __forceinline__ void mma8_bf16_commit_elect(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                                       uint32_t accumulate, uint32_t da, uint32_t db, uint32_t mbar)
{
    const uint64_t a1 = a_desc + da, a2 = a1 + da, a3 = a2 + da, b1 = b_desc + db, b2 = b1 + db, b3 = b2 + db;
    asm volatile(
        "{\n .reg .pred p, t, e;\n .reg .b64 x, y;\n elect.sync _|e, 0xffffffff;\n setp.ne.b32 p, %4, 0;\n"
        " setp.eq.b32 t, 0, 0;\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], %5, %6, %3, t;\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], %7, %8, %3, t;\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], %9, %10, %3, t;\n"
        " add.s64 x, %1, %12;\n add.s64 y, %2, %13;\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], x, y, %3, t;\n"
        " add.s64 x, %5, %12;\n add.s64 y, %6, %13;\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], x, y, %3, t;\n"
        " add.s64 x, %7, %12;\n add.s64 y, %8, %13;\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], x, y, %3, t;\n"
        " add.s64 x, %9, %12;\n add.s64 y, %10, %13;\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], x, y, %3, t;\n"
        " @e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%11];\n}\n" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "l"(a1), "l"(b1), "l"(a2), "l"(b2), "l"(a3), "l"(b3),
        "r"(mbar), "l"(static_cast<uint64_t>(4 * da)), "l"(static_cast<uint64_t>(4 * db))
        : "memory");
}

__device__ __forceinline__ void commit_elect(uint32_t mbar)
{
    asm volatile(
        "{\n .reg .pred e;\n elect.sync _|e, 0xffffffff;\n"
        " @e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(mbar)
        : "memory");
}

__device__ __forceinline__ void wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// 32 lanes x 32-bit: thread t of the warp reads lane (taddr.lane + t),
// columns taddr.col .. + 15.
__device__ __forceinline__ void ld_32x32b_x16(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}

__device__ __forceinline__ void st_32x32b_x16(uint32_t taddr, const uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
            taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}

// ---------------------------------------------------------------- mbarrier / TMA

__device__ __forceinline__ void mbar_arrive(uint32_t mbar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t mbar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(bytes) : "memory");
}

__device__ __forceinline__ void tma_store_4d(const CUtensorMap *map, uint32_t src, int32_t c0, int32_t c1, int32_t c2,
                                             int32_t c3)
{
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%1, %2, %3, %4}], [%5];" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(src)
                 : "memory");
}

__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// every committed store has finished reading shared memory / has completed
__device__ __forceinline__ void bulk_wait_read0() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait0() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// The address in CTA `rank` of this cluster that `addr` is here.
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}

// bytes (a multiple of 16) from this CTA's shared memory to a peer's, completing
// on the peer's barrier (which expects them).
__device__ __forceinline__ void bulk_copy_cluster(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "r"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

__device__ __forceinline__ void fence_barrier_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Order this thread's generic-proxy shared-memory writes before later
// async-proxy (tensor core / TMA) accesses.
__device__ __forceinline__ void fence_proxy_async_smem()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// L2 eviction policies for cache-hinted loads.
__device__ __forceinline__ uint64_t policy_evict_last()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}

__device__ __forceinline__ uint64_t policy_evict_first()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}

__device__ __forceinline__ void tma_load_3d_hint(uint32_t dst, const CUtensorMap *map, int32_t c0, int32_t c1,
                                                 int32_t c2, uint32_t mbar, uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, "
        "%3, %4}], [%5], %6;" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(mbar), "l"(policy)
        : "memory");
}

// Warp-collective forms (the whole warp converged, one elected lane issues).
__device__ __forceinline__ void mbar_arrive_expect_tx_elect(uint32_t mbar, uint32_t bytes)
{
    asm volatile(
        "{\n .reg .pred e;\n elect.sync _|e, 0xffffffff;\n"
        " @e mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n}\n" ::"r"(mbar),
        "r"(bytes)
        : "memory");
}

__device__ __forceinline__ void tma_load_2d_hint_elect(uint32_t dst, const CUtensorMap *map, int32_t c0, int32_t c1,
                                                       uint32_t mbar, uint64_t policy)
{
    asm volatile(
        "{\n .reg .pred e;\n elect.sync _|e, 0xffffffff;\n"
        " @e cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, "
        "{%2, %3}], [%4], %5;\n}\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(mbar), "l"(policy)
        : "memory");
}

__device__ __forceinline__ void tma_load_3d_hint_elect(uint32_t dst, const CUtensorMap *map, int32_t c0, int32_t c1,
                                                       int32_t c2, uint32_t mbar, uint64_t policy)
{
    asm volatile(
        "{\n .reg .pred e;\n elect.sync _|e, 0xffffffff;\n"
        " @e cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, "
        "{%2, %3, %4}], [%5], %6;\n}\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(mbar), "l"(policy)
        : "memory");
}

// The same with a 2-d box (of another map) as the last load.
__device__ __forceinline__ void tma_refill_q_elect(uint32_t mbar, uint32_t bytes, const CUtensorMap *map, int32_t c0,
                                                   int32_t c1, uint32_t dst, int32_t blk, uint32_t dst2, int32_t blk2,
                                                   uint32_t two, uint64_t policy, const CUtensorMap *map_q, int32_t q0,
                                                   int32_t q1, uint32_t dst_q, uint64_t policy_q)
{
    asm volatile(
        "{\n .reg .pred e, f, t;\n elect.sync _|e, 0xffffffff;\n setp.ne.b32 t, %9, 0;\n and.pred f, e, t;\n"
        " @e mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n"
        " @e cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%5], [%2, {%3, "
        "%4, %6}], [%0], %10;\n"
        " @f cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%7], [%2, {%3, "
        "%4, %8}], [%0], %10;\n"
        " @e cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%14], [%11, "
        "{%12, %13}], [%0], %15;\n}\n" ::"r"(mbar),
        "r"(bytes), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(dst), "r"(blk), "r"(dst2), "r"(blk2),
        "r"(two), "l"(policy), "l"(reinterpret_cast<uint64_t>(map_q)), "r"(q0), "r"(q1), "r"(dst_q), "l"(policy_q)
        : "memory");
}

// A ring entry of two column chunks `step` bytes apart (columns c0 and c0 + 64)
// in one election: one box per chunk, or two (the second `half` bytes further on).
__device__ __forceinline__ void tma_refill_pair_elect(uint32_t mbar, uint32_t bytes, const CUtensorMap *map, int32_t c0,
                                                      int32_t c1, uint32_t dst, uint32_t step, int32_t blk, uint32_t half,
                                                      int32_t blk2, uint32_t two, uint64_t policy)
{
    asm volatile(
        "{\n .reg .pred e, f, t;\n elect.sync _|e, 0xffffffff;\n setp.ne.b32 t, %9, 0;\n and.pred f, e, t;\n"
        " @e mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n"
        " @e cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%5], [%2, {%3, "
        "%4, %6}], [%0], %10;\n"
        " @f cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%7], [%2, {%3, "
        "%4, %8}], [%0], %10;\n"
        " @e cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%11], [%2, {%13, "
        "%4, %6}], [%0], %10;\n"
        " @f cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%12], [%2, {%13, "
        "%4, %8}], [%0], %10;\n}\n" ::"r"(mbar),
        "r"(bytes), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(dst), "r"(blk), "r"(dst + half), "r"(blk2),
        "r"(two), "l"(policy), "r"(dst + step), "r"(dst + step + half), "r"(c0 + 64)
        : "memory");
}

__device__ __forceinline__ void tma_load_2d_elect(uint32_t dst, const CUtensorMap *map, int32_t c0, int32_t c1,
                                                  uint32_t mbar)
{
    asm volatile(
        "{\n .reg .pred e;\n elect.sync _|e, 0xffffffff;\n"
        " @e cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n}\n" ::"r"(
            dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(mbar)
        : "memory");
}

__device__ __forceinline__ void tma_load_3d_elect(uint32_t dst, const CUtensorMap *map, int32_t c0, int32_t c1,
                                                  int32_t c2, uint32_t mbar)
{
    asm volatile(
        "{\n .reg .pred e;\n elect.sync _|e, 0xffffffff;\n"
        " @e cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];\n}\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(mbar)
        : "memory");
}

__device__ __forceinline__ void tma_load_4d_elect(uint32_t dst, const CUtensorMap *map, int32_t c0, int32_t c1,
                                                  int32_t c2, int32_t c3, uint32_t mbar)
{
    asm volatile(
        "{\n .reg .pred e;\n elect.sync _|e, 0xffffffff;\n"
        " @e cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];\n}\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(mbar)
        : "memory");
}

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ void prefetch_tensormap(const CUtensorMap *map)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

}  // namespace tc
}  // namespace gbmla
