// Receive and send rows of a stretch of ranks of one p: the kernel behind bcs_build and its relatives.
//
// One launch, nothing read from memory, no table of all ranks (rows.cuh).  Before it: skip codes of all ranks, a
// search on them per round, a round-major copy and its transposition, three launches.  All ranks of
// 100 003: 23.2 -> 10.2 us, of about 2^20: 38.4 -> 22.7 us, 65 553 ranks of it 104 -> 10.3 us (send rows whose
// to-processor lies outside the range were searched for one by one), 32 ranks without a workspace 572 -> 8.2 us (a
// descent of the homeranges per window), 8 chunks of about 2^28 ranks 9.35 -> 3.94 ms.  Small calls
// last as long as launch, table and one item; large ones are bound by instruction issue (seven eighths of the slots).
#include <atomic>

#include "rows.cuh"

namespace bcs {
namespace {

constexpr unsigned kSms = 148;
constexpr unsigned kRowThreads = 1024;

// One CTA per SM at most; every warp takes items of `item` (32, 64 or 128) consecutive ranks, neighbouring warps
// neighbouring items.  first: rank of the first row (< p); the count <= p ranks go on at 0 behind p - 1.
template <int kWords>
__global__ void __launch_bounds__(kRowThreads, 1)
rows_kernel(const __grid_constant__ RowConsts rc, uint32_t first, uint32_t count, uint32_t item, int8_t *recv,
            int8_t *send)
{
    extern __shared__ __align__(128) uint8_t sm[];
    const RowLayout at(rc.q);
    const RowTable t(sm, at);
    if (threadIdx.x < kRow + kLow + 1) t.s[threadIdx.x] = rc.s[threadIdx.x];
    __syncthreads();
    build_row_table(t, rc.q, rc.odd);
    const uint32_t n_warps = blockDim.x >> 5, warp = threadIdx.x >> 5;
    uint8_t *mine = sm + at.warps + warp * at.warp_bytes;
    const uint64_t stride = (uint64_t)gridDim.x * n_warps * item;
    for (uint64_t b = ((uint64_t)blockIdx.x * n_warps + warp) * item; b < count; b += stride) {
        const uint32_t n = count - (uint32_t)b < item ? count - (uint32_t)b : item;
        uint32_t x0 = first + (uint32_t)b;
        if (x0 >= rc.p) x0 -= rc.p;
        const uint64_t byte = b * (uint64_t)rc.q;
        warp_rows<kWords, true>(t, mine, rc.q, rc.odd, rc.inv, x0, n, recv ? recv + byte : nullptr,
                                send ? send + byte : nullptr);
    }
    stage_free();
}

// Opts a kernel in to large dynamic shared memory, once per device.
template <auto kKernel>
bool allow_shared()
{
    static std::atomic<uint64_t> done{0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    const uint64_t bit = dev < 64 ? 1ull << dev : 0;
    if (done.load(std::memory_order_relaxed) & bit) return true;
    if (cudaFuncSetAttribute(kKernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) != cudaSuccess)
        return false;
    done.fetch_or(bit, std::memory_order_relaxed);
    return true;
}

template <int kWords>
bcs_status launch(const RowConsts &rc, uint32_t first, uint32_t count, int8_t *recv, int8_t *send, cudaStream_t stream)
{
    if ((rc.q + 3) / 4 != kWords) {
        if constexpr (kWords < (BCS_MAX_Q + 3) / 4) return launch<kWords + 1>(rc, first, count, recv, send, stream);
        return BCS_ERR_UNSUPPORTED;
    }
    if (!allow_shared<rows_kernel<kWords>>()) return BCS_ERR_CUDA;
    // Items of 128 ranks where they fill the card, smaller ones before that: the latency of an item is
    // what counts then, although the ranks behind it that it looks up (up to 64) are more for a small one (all
    // ranks of 100 003: 16.0 us with items of 128 ranks only, 10.2 us like this).
    uint32_t item = kItemRanks;
    while (item > 32u && count < kSms * (kRowThreads / 32) * item) item /= 2;
    const unsigned items = (count + item - 1) / item;
    rows_kernel<kWords><<<items < kSms ? items : kSms, kRowThreads, RowLayout(rc.q).total(kRowThreads / 32), stream>>>(
        rc, first, count, item, recv, send);
    return launch_status();
}

}  // namespace

bcs_status launch_rows(uint32_t p, uint64_t first, uint64_t count, int8_t *recv, int8_t *send, cudaStream_t stream)
{
    RowConsts rc = {};
    rc.p = p;
    rc.q = ceil_log2_u32(p);
    uint32_t v = p;
    for (int k = rc.q; k >= 0; --k) {                            // Algorithm 1
        rc.s[k] = v;
        v = (v + 1u) / 2u;
    }
    for (int k = 1; k <= rc.q; ++k) rc.odd |= (2u * rc.s[k - 1] - rc.s[k]) << k;
    rc.inv = (uint32_t)((1ull << (rc.q - low_levels(rc.q) + 32)) / p);
    return launch<1>(rc, (uint32_t)first, (uint32_t)count, recv, send, stream);
}

}  // namespace bcs
