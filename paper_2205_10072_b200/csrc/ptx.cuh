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

// Bytes of a (0..3) and b (4..7) by the nibbles of kPick, one for each byte of the result; with 8 added the sign of that byte eight times.
template <uint32_t kPick>
__device__ __forceinline__ uint32_t sign_bytes(uint32_t a, uint32_t b)
{
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "n"(kPick));
    return r;
}

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

// Polls came() until it is true or until the time spent waiting, by clock() in nanoseconds, reaches `limit`.  What passes between two looks at the clock
// counts as a millisecond at most, and the last thing before giving up is a poll: a context that was switched out for seconds (a debugger, a suspended
// process) finds what has come meanwhile, and goes on waiting for what has not.
template <class Came, class Clock>
__host__ __device__ __forceinline__ bool wait_with_limit(Came came, Clock clock, uint64_t limit)
{
    constexpr uint64_t most = 1000000;
    uint64_t waited = 0, last = 0;
    for (bool timed = false; !came(); timed = true) {
        if (waited >= limit) return false;
        const uint64_t now = clock(), passed = timed ? now - last : 0;
        waited += passed < most ? passed : most;
        last = now;
    }
    return true;
}

struct NanosecondClock {
    __device__ __forceinline__ uint64_t operator()() const
    {
        uint64_t now;
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(now) :: "memory");
        return now;
    }
};

// Whether the phase of the given parity has come (a poll: it may suspend the thread for a while).
struct PhaseCame {
    uint32_t bar, parity;
    __device__ __forceinline__ PhaseCame(uint64_t *at, uint32_t of) : bar((uint32_t)__cvta_generic_to_shared(at)), parity(of) {}
    __device__ __forceinline__ bool operator()() const
    {
        uint32_t done;
        asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
                     : "=r"(done) : "r"(bar), "r"(parity) : "memory");
        return done != 0u;
    }
};

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

// What a CTA learns from the answer to ask_for_work().
enum class Work { given, none, expired };

// For some thread of the CTA the time was up: whether the phase has come for any of them by now.  (Out of line: the kernels have few registers left.)
static __device__ __noinline__ bool came_for_any(uint64_t *bar, uint32_t parity, bool came)
{
    if (!came) came = PhaseCame(bar, parity)();
    return __syncthreads_or(came);
}

// Waits for the answer, `limit` nanoseconds at most; by all threads of the CTA, behind a barrier behind which nobody else reads an answer.  Ends with a barrier:
// the next one may be asked for.  All threads return the same.
__device__ __forceinline__ Work await_work(uint4 *answer, uint64_t *bar, uint32_t parity, uint64_t limit, uint32_t *cta)
{
    bool came = wait_with_limit(PhaseCame(bar, parity), NanosecondClock(), limit);
    bool given = came && work_given(answer, cta);
    fence_before_bulk();                                         // (the answer is written by the asynchronous proxy: it has been read)
    if (!__syncthreads_and(came)) {
        // If it has come for any, the answer is there for all; a turn that it names is nobody else's.
        if (!came_for_any(bar, parity, came)) return Work::expired;
        given = work_given(answer, cta);
        fence_before_bulk();
        __syncthreads();
    }
    return given ? Work::given : Work::none;
}

}  // namespace bcs
