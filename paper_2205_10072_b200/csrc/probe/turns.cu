// Turns that CTAs take from one another, on their own (see bcs_probe.h): what the row kernels do with them, with nothing else around it.
#include "bcs_common.cuh"
#include "bcs_probe.h"

namespace bcs {
namespace {

constexpr int kTurnThreads = 96;

__global__ void __launch_bounds__(kTurnThreads)
turns_kernel(uint32_t *taken)
{
    __shared__ __align__(16) uint4 answer;
    __shared__ uint64_t answered;
    if (threadIdx.x == 0) barrier_init(&answered);
    __syncthreads();
    uint32_t turn = blockIdx.x, parity = 0;
    for (;;) {
        if (threadIdx.x == 0) ask_for_work(&answer, &answered);
        atomicAdd(taken + turn, 1u);
        if (await_work(&answer, &answered, parity, 2000000000, &turn) != Work::given) break;
        parity ^= 1u;
    }
}

__global__ void __launch_bounds__(kTurnThreads)
unanswered_kernel(uint64_t limit, uint32_t *results)
{
    __shared__ __align__(16) uint4 answer;
    __shared__ uint64_t answered;
    if (threadIdx.x == 0) {
        answer = make_uint4(0u, 0u, 0u, 0u);
        barrier_init(&answered);
    }
    __syncthreads();
    uint32_t turn = 12345u;
    const Work work = await_work(&answer, &answered, 0u, limit, &turn);      // (nothing has been asked for)
    results[threadIdx.x] = work == Work::expired && turn == 12345u ? 1u : 2u;
}

}  // namespace
}  // namespace bcs

using namespace bcs;

extern "C" {

bcs_status bcs_probe_turns(uint32_t ctas, uint32_t *taken_dev, void *cuda_stream)
{
    if (ctas == 0 || taken_dev == nullptr) return BCS_ERR_ARG;
    turns_kernel<<<ctas, kTurnThreads, 0, static_cast<cudaStream_t>(cuda_stream)>>>(taken_dev);
    return launch_status();
}

bcs_status bcs_probe_unanswered(uint64_t limit_ns, uint32_t *results_dev, void *cuda_stream)
{
    if (limit_ns > 1000000000ull || results_dev == nullptr) return BCS_ERR_ARG;
    unanswered_kernel<<<1, kTurnThreads, 0, static_cast<cudaStream_t>(cuda_stream)>>>(limit_ns, results_dev);
    return launch_status();
}

}  // extern "C"
