// The few instructions that the row kernels write as inline PTX.
#pragma once
#include <stdint.h>

namespace bcs {

// Position of the highest set bit, -1 for 0 (one instruction).
__device__ __forceinline__ int top_bit(uint32_t v)
{
    int d;
    asm("bfind.u32 %0, %1;" : "=r"(d) : "r"(v));
    return d;
}

// Byte permutation: nibble i of `pick` says which byte of (b, a) becomes byte i; with its top bit set, that byte's
// sign bit eight times (0 for a byte below 128).
__device__ __forceinline__ uint32_t pick_bytes(uint32_t a, uint32_t b, uint32_t pick)
{
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(pick));
    return d;
}

// Loads that are not taken from the L1 cache or from an earlier load of the same place.
__device__ __forceinline__ uint32_t load_relaxed(const uint32_t *at)
{
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(at) : "memory");
    return v;
}

__device__ __forceinline__ uint64_t load_relaxed(const uint64_t *at)
{
    uint64_t v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(at) : "memory");
    return v;
}

// Makes this thread's shared-memory writes visible to the copies that bulk_store() starts.
__device__ __forceinline__ void fence_before_bulk() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// `bytes` (a multiple of 16) from shared memory to global memory, both 16-byte aligned, by the TMA unit.
__device__ __forceinline__ void bulk_store(void *dst, const void *from_shared, uint32_t bytes)
{
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                 :: "l"(reinterpret_cast<uint64_t>(dst)), "r"((uint32_t)__cvta_generic_to_shared(from_shared)), "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// True for one lane of a full warp, the same one each time (the compiler then knows that what follows is done by one thread).
__device__ __forceinline__ bool elect_one()
{
    uint32_t one;
    asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}" : "=r"(one) :: "memory");
    return one != 0u;
}

// The copies that this thread has started have read their shared memory.
__device__ __forceinline__ void bulk_stores_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }

// ---------------------------------------------------------------- work that CTAs take from one another
// A CTA that asks for the work of one that has not started yet gets its index, and that one is not launched (cluster launch control).  The answer
// (16 bytes) arrives in shared memory and completes a phase of the barrier.
__device__ __forceinline__ void barrier_init(uint64_t *bar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"((uint32_t)__cvta_generic_to_shared(bar)) : "memory");
}

__device__ __forceinline__ void ask_for_work(uint4 *answer, uint64_t *bar)
{
    const uint32_t b = (uint32_t)__cvta_generic_to_shared(bar);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], 16;" :: "r"(b) : "memory");
    asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];"
                 :: "r"((uint32_t)__cvta_generic_to_shared(answer)), "r"(b) : "memory");
}

// Waits for the phase of the given parity, two seconds at most; false: it has not come.
__device__ __forceinline__ bool barrier_wait(uint64_t *bar, uint32_t parity)
{
    const uint32_t b = (uint32_t)__cvta_generic_to_shared(bar);
    uint64_t begin = 0, now = 0;
    for (;;) {
        uint32_t done;
        asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
                     : "=r"(done) : "r"(b), "r"(parity) : "memory");
        if (done) return true;
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(now) :: "memory");
        if (begin == 0) begin = now;
        if (now - begin > 2000000000ull) return false;
    }
}

// Whether an answer names a CTA, and which.
__device__ __forceinline__ bool work_given(const uint4 *answer, uint32_t *cta)
{
    const uint4 a = *answer;
    uint32_t given, x;
    asm volatile("{\n.reg .b128 r;\n.reg .pred p;\n.reg .b64 lo, hi;\nmov.b64 lo, {%2, %3};\nmov.b64 hi, {%4, %5};\nmov.b128 r, {lo, hi};\n"
                 "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, r;\nselp.u32 %0, 1, 0, p;\nmov.u32 %1, 0;\n"
                 "@p clusterlaunchcontrol.query_cancel.get_first_ctaid.v4.b32.b128 {%1, _, _, _}, r;\n}"
                 : "=r"(given), "=r"(x) : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w) : "memory");
    *cta = x;
    return given != 0u;
}

}  // namespace bcs
