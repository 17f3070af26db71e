// Inline-PTX helpers shared by the fifth-generation tensor-core kernels
// (tcgen05 MMAs with operands in shared memory and accumulators in tensor
// memory) and their mbarrier / bulk-copy plumbing.  Every wait is bounded:
// after kTcWaitLimit polls it returns false and the caller reports a status
// word instead of hanging the GPU.
#pragma once

#include <cuda.h>
#include <stdint.h>

namespace flosic {

constexpr long long kTcWaitLimit = 1LL << 24;

__device__ __forceinline__ uint32_t tc_smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void tc_mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(tc_smem_addr(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void tc_mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tc_smem_addr(bar)), "r"(bytes)
                 : "memory");
}

// true once the phase with the given parity has completed; false after the limit
__device__ __forceinline__ bool tc_mbar_wait(uint64_t* bar, uint32_t parity) {
    for (long long i = 0; i < kTcWaitLimit; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(tc_smem_addr(bar)), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

// 2-D tiled bulk copy global -> shared, completion counted in bytes on bar
__device__ __forceinline__ void tc_tma_load_2d(void* dst, const CUtensorMap* map, int c0, int c1, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            tc_smem_addr(dst)),
        "l"((unsigned long long)map), "r"(c0), "r"(c1), "r"(tc_smem_addr(bar))
        : "memory");
}

// 4-D tiled bulk copy global -> shared (x, y, z, orbital), completion counted in bytes on bar
__device__ __forceinline__ void tc_tma_load_4d(void* dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                               uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(
            tc_smem_addr(dst)),
        "l"((unsigned long long)map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(tc_smem_addr(bar))
        : "memory");
}

// Shared-memory matrix descriptor: K-major, 128-byte swizzle, consecutive
// 8-row groups 1024 bytes apart (stride byte offset), descriptor version 1.
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t saddr) {
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;                  // leading byte offset (unused by swizzled K-major)
    d |= (uint64_t)(1024 >> 4) << 32;        // stride byte offset
    d |= (uint64_t)1 << 46;                  // version
    d |= (uint64_t)2 << 61;                  // 128-byte swizzle
    return d;
}

// The same with a 64-byte swizzle: rows of 64 bytes (32 bf16), 8-row groups
// 512 bytes apart, 16-byte piece c of row m at c ^ ((m >> 1) & 3).
__device__ __forceinline__ uint64_t umma_desc_sw64(uint32_t saddr) {
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(512 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)4 << 61;                  // 64-byte swizzle
    return d;
}

// Instruction descriptor of kind::f16: bf16 A and B (K-major), float32 D.
__host__ __device__ constexpr uint32_t umma_idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// D (tensor memory) (+)= A B^T, both operands bf16 in shared memory
__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, int acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(da), "l"(db), "r"(idesc), "r"(acc)
        : "memory");
}

// the mbarrier arrives once every tcgen05 operation this thread issued before it has completed
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(tc_smem_addr(bar))
                 : "memory");
}

// One lane of a converged warp (1 there, 0 in the others).  The MMAs below are
// issued by a whole warp whose control flow and operands are warp-uniform,
// predicated on this lane: the descriptors then live in uniform registers and
// an M = 128, K = 16 MMA issues in N / 2 cycles (the tensor pipe's own rate:
// 32 at N = 64, 64 at N = 128, measured).  Issued from a lane-0 branch, each
// MMA moves its operands to uniform registers first and takes 86 cycles
// whatever its N.
__device__ __forceinline__ uint32_t tc_elect() {
    uint32_t r;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(r));
    return r;
}
// A warp-uniform value v in a form that the compiler knows to be uniform (the
// reduction's result is a uniform register; a shuffle's is not).
__device__ __forceinline__ uint32_t tc_uniform(uint32_t v) { return __reduce_or_sync(0xffffffffu, v); }

// The last of `count` commits made in turn to the mbarriers of a ring of `ring`
// slots (one commit per phase): its slot (-1: none) and the parity of its phase.
struct TcLastCommit {
    int slot;
    uint32_t parity;
};
__host__ __device__ constexpr TcLastCommit tc_last_commit(int count, int ring) {
    return count > 0 ? TcLastCommit{(count - 1) % ring, (uint32_t)(((count - 1) / ring) & 1)} : TcLastCommit{-1, 0u};
}
static_assert(tc_last_commit(0, 4).slot == -1 && tc_last_commit(1, 4).slot == 0 && tc_last_commit(1, 4).parity == 0 &&
                  tc_last_commit(4, 4).slot == 3 && tc_last_commit(4, 4).parity == 0 &&
                  tc_last_commit(5, 4).slot == 0 && tc_last_commit(5, 4).parity == 1 &&
                  tc_last_commit(9, 3).slot == 2 && tc_last_commit(9, 3).parity == 0,
              "slot and phase of the last commit");

// D (tensor memory) (+)= A B^T issued by the elected lane of a converged warp:
// both operands in shared memory, or A in tensor memory (row i in lane i, two
// bf16 K-values per 32-bit column)
__device__ __forceinline__ void umma_bf16_el(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, int acc,
                                             uint32_t el) {
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(da), "l"(db), "r"(idesc), "r"(acc), "r"(el)
        : "memory");
}
__device__ __forceinline__ void umma_bf16_ts_el(uint32_t tmem_d, uint32_t tmem_a, uint64_t db, uint32_t idesc, int acc,
                                                uint32_t el) {
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(tmem_d),
        "r"(tmem_a), "l"(db), "r"(idesc), "r"(acc), "r"(el)
        : "memory");
}

// 4 consecutive 32-bit columns of this warp's 32 tensor-memory lanes (one register each)
__device__ __forceinline__ void tmem_st4(uint32_t taddr, uint32_t v0, uint32_t v1, uint32_t v2, uint32_t v3) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr), "r"(v0), "r"(v1),
                 "r"(v2), "r"(v3)
                 : "memory");
}
// this thread's tensor-memory stores have completed
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// 32 consecutive columns of this warp's 32 tensor-memory lanes (one column per register)
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* out) {
    uint32_t v[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
        "%14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]),
          "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]),
          "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]),
          "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int j = 0; j < 32; ++j) out[j] = __uint_as_float(v[j]);
}

// 16 consecutive columns of this warp's 32 tensor-memory lanes
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* out) {
    uint32_t v[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
        "%14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int j = 0; j < 16; ++j) out[j] = __uint_as_float(v[j]);
}

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// plain arrival (no transaction count) on an mbarrier
__device__ __forceinline__ void tc_mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc_smem_addr(bar)) : "memory");
}

// Bounded wait that also gives up as soon as *abort (shared) becomes nonzero.
// Each poll may suspend the thread for up to about a microsecond (it resumes as
// soon as the phase completes), so a waiting warp takes almost no issue slots;
// gives up after about two seconds.
__device__ __forceinline__ bool tc_mbar_sleep_or_abort(uint64_t* bar, uint32_t parity, const volatile int* abort) {
    for (int i = 0; i < (1 << 21); ++i) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(tc_smem_addr(bar)), "r"(parity), "r"(1000u)
            : "memory");
        if (ok) return true;
        if (*abort) return false;
    }
    return false;
}

// The same for a converged warp: true if every lane saw the phase complete.  The
// lanes poll on their own and may disagree near the limit or when *abort changes;
// a warp whose code has collective operations ahead must branch on the vote, or
// some lanes would wait for the others at the next one, outside any limit.
__device__ __forceinline__ bool tc_mbar_warp_wait(uint64_t* bar, uint32_t parity, const volatile int* abort) {
    return __all_sync(0xffffffffu, tc_mbar_sleep_or_abort(bar, parity, abort));
}

// The vote of a converged warp on a flag that another warp may set at any time
__device__ __forceinline__ bool tc_warp_any(int flag) { return __any_sync(0xffffffffu, flag) != 0; }

// named barrier over `count` threads (a multiple of 32) of the CTA
__device__ __forceinline__ void tc_named_sync(int id, int count) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// generic-proxy shared-memory writes become visible to the async proxy (MMA operand reads)
__device__ __forceinline__ void tc_fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// warp-collective tensor-memory allocation; the base address lands in *dst (shared)
__device__ __forceinline__ void tmem_alloc(uint32_t* dst, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_smem_addr(dst)), "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t base, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(cols) : "memory");
}

}  // namespace flosic
