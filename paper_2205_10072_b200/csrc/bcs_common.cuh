// Shared pieces of the schedule, round-table and checksum translation units: per-p tables,
// the Section 2 primitives of arXiv 2205.10072 as device functions, lists of p, launches.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "bcs.h"
#include "ptx.cuh"

namespace bcs {

constexpr int kTile = 256;                    // ranks (= threads) per CTA of the checks (validate.cu)
constexpr uint32_t kFusedMaxP = 1024;         // batch: a p up to here is built by one CTA
constexpr int kRow = BCS_SKIPS_STRIDE;        // words per table row

// Per-p constants (kernel parameter of the single-p kernels).
//   s[k] = skips[k] of Algorithm 1, k = 0..q (q <= 31), then 0
struct PTable {
    uint32_t s[kRow];
    uint32_t p;
    int q;
};

struct BatchArgs {
    const uint32_t *p_list;
    const uint64_t *rank_off;
    const uint64_t *entry_off;
    uint32_t num_p;
    uint64_t total_ranks;
};

__host__ __device__ inline int ceil_log2_u32(uint32_t p)
{
    int q = 0;
    while (q < 32 && (uint64_t(1) << q) < p) ++q;
    return q;
}

__device__ __forceinline__ int ceil_log2_fast(uint32_t p) { return p > 1u ? 32 - __clz(p - 1u) : 0; }

// ---------------------------------------------------------------- Section 2 primitives
// Largest k with skips[k] <= x (the homerange of x), 1 <= x < p.  Algorithm 1 gives
// 2^(k-1) < skips[k] <= 2^k, so k is floor(log2 x) or one more.
__device__ __forceinline__ int home_of(const uint32_t *s, uint32_t x)
{
    int m = 31 - __clz(x);
    return m + (s[m + 1] <= x ? 1 : 0);
}

// Skip code of rank x (0 <= x < p): bit k set iff skips[k] is a term of the greedy
// decomposition x = skips[k1] + skips[k2] + ... that Algorithm 2 walks down (largest skip
// not above the remainder first; the remainder after taking skips[k] is below skips[k], so a
// downward scan over the levels finds the same terms).  The baseblock of x is the lowest set
// bit, its homerange the highest.  Codes order like ranks.
__host__ __device__ inline uint32_t skip_code(const uint32_t *s, int q, uint32_t x)
{
    uint32_t code = 0;
    for (int k = q - 1; k >= 0; --k) {
        if (x >= s[k]) {
            x -= s[k];
            code |= 1u << k;
        }
    }
    return code;
}

// ---------------------------------------------------------------- spans of rows, lists of p
// Copies in[byte0, byte0+len) to stage[shift, shift+len), (byte0 & 15) == shift, `in` 16-byte
// aligned: 16-byte loads but for the ragged ends.
__device__ __forceinline__ void load_span(uint8_t *stage, uint32_t shift, uint32_t len,
                                          const int8_t *in, uint64_t byte0)
{
    const uint8_t *src = reinterpret_cast<const uint8_t *>(in) + (byte0 - shift);
    const uint32_t end = shift + len;
    const uint32_t nvec = (end + 15u) >> 4;
    for (uint32_t v = threadIdx.x; v < nvec; v += blockDim.x) {
        const uint32_t lo = v << 4, hi = lo + 16u;
        if (lo >= shift && hi <= end) {
            *reinterpret_cast<uint4 *>(stage + lo) = *reinterpret_cast<const uint4 *>(src + lo);
        } else {
            const uint32_t from = lo < shift ? shift : lo, to = hi > end ? end : hi;
            for (uint32_t e = from; e < to; ++e) stage[e] = src[e];
        }
    }
}

// Largest j with off[j] <= g (off[0] <= g), by a whole warp: 32 probes per step, so a table of a few thousand offsets takes
// three dependent loads.  Whatever off holds, it ends, with some j < num.  All 32 lanes must call.
__device__ __forceinline__ uint32_t find_segment_warp(const uint64_t *off, uint32_t num, uint64_t g)
{
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t lo = 0, hi = num;                       // answer in [lo, hi)
    while (hi - lo > 1u) {
        const uint32_t step = (hi - lo + 31u) / 32u;
        const uint32_t idx = lo + lane * step;
        const bool le = lane == 0u || (idx < hi && load_relaxed(off + idx) <= g);
        const uint32_t hits = __popc(__ballot_sync(0xffffffffu, le));
        lo += (hits - 1u) * step;
        hi = lo + step < hi ? lo + step : hi;
    }
    return lo;
}

// ---------------------------------------------------------------- dependent launches
// Calls follow one another on a stream, many of them a few microseconds long, so the time in which one grid drains and
// the next is brought onto the SMs counts.  A kernel launched with launch_dependent() may be made resident as soon as every CTA
// of the kernel before it on the stream has called grid_launch_dependents() (or has exited); it
// runs its set-up, which relies on nothing that another kernel may have written, and then blocks in grid_dependency_wait() until
// that kernel has completed and its writes are visible.  Both calls do nothing in a kernel that was launched the ordinary way.
__device__ __forceinline__ void grid_dependency_wait()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

__device__ __forceinline__ void grid_launch_dependents()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// ---------------------------------------------------------------- host helpers
bcs_status make_table(uint32_t p, PTable *tab);

// Rows of the count <= p ranks first, first+1, ... (mod p; first < p, p > 1): rows.cu.  Either output may be null.
bcs_status launch_rows(uint32_t p, uint64_t first, uint64_t count, int8_t *recv, int8_t *send, cudaStream_t stream);

// Waits with a limit that ran out in the row kernels of the current device: rows.cu.
bool expired_wait_count(unsigned long long *count);

// Launch with programmatic stream serialisation (see above); `dependent` false: ordinary launch.
template <class... Params, class... Args>
inline void launch_dependent(bool dependent, void (*kernel)(Params...), dim3 grid, unsigned block, size_t shared,
                             cudaStream_t stream, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = shared;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = dependent ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, Params(args)...);
}

// Opts a kernel in to large dynamic shared memory (what a little static use leaves of 227 KB), once per device.  If the
// runtime refuses, its error is not left for launch_status() of a later call.
template <auto kKernel>
bool allow_shared()
{
    static std::atomic<uint64_t> done{0};
    int dev = 0;
    const bool known = cudaGetDevice(&dev) == cudaSuccess;
    const uint64_t bit = dev < 64 ? 1ull << dev : 0;
    if (known && (done.load(std::memory_order_relaxed) & bit)) return true;
    if (!known || cudaFuncSetAttribute(kKernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    done.fetch_or(bit, std::memory_order_relaxed);
    return true;
}

inline bool aligned16(const void *ptr) { return (reinterpret_cast<uintptr_t>(ptr) & 15u) == 0; }

inline bcs_status launch_status()
{
    return cudaGetLastError() == cudaSuccess ? BCS_OK : BCS_ERR_CUDA;
}

inline bcs_status check_range(uint32_t p, uint64_t r_begin, uint64_t r_end)
{
    if (p == 0) return BCS_ERR_RANGE;
    if (p > 0x7fffffffu) return BCS_ERR_UNSUPPORTED;
    if (r_begin > r_end || r_end > p) return BCS_ERR_RANGE;
    return BCS_OK;
}

__host__ __device__ inline uint64_t align_up(uint64_t v, uint64_t a) { return (v + a - 1) / a * a; }

}  // namespace bcs
