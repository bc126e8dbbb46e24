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

// The copies that this thread has started have read their shared memory.
__device__ __forceinline__ void bulk_stores_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }

}  // namespace bcs
