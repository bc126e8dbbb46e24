// Receive and send rows of a stretch of ranks of one p: the kernels behind bcs_build and its relatives.
//
// One launch, nothing read from memory but constants, no table of all ranks (rows.cuh).  Two forms, by size (launch_rows):
//   * rows_kernel, a rank per lane.  Bound by latency: launch, table, one or two items per warp.  From Python 32 ranks 3.2 to 3.5 us back to
//     back, all ranks of 1152 3.3 to 3.7, 65 553 ranks 3.5 (2.7 on the device).  The table holds what the
//     CTA's segments need where these are few, and a CTA has no more warps than items.
//   * wide_kernel, 16 output bytes per lane (wide.cuh).  Up to some 2^23 ranks bound by instruction issue and latency: a segment of 65 ranks
//     takes a warp 1250 cycles, most of them in the step in which it ends.  Up to 2^20 ranks two CTAs fit an SM, so that the next call's table is
//     built beside the rows, above it the 61 440 registers of a CTA leave no room and the table's time (some 4800 cycles, half of
//     them for the send table) is in series.
//     From about 2^25 ranks on bound by memory writes.  All ranks of 100 003 4.6 to 5.1 us by the card, of 1.06 million 13.7, 8 chunks of about
//     2^28 2.34 to 2.46 ms (6.4 to 6.1 TB/s; the power cap shows in long runs).
// Both are launched as dependents of whatever runs before them on the stream and wait for it before their first store.
#include <type_traits>

#include "batch.cuh"     // (in this unit, too: the constants of rows.cuh are in the module once)
#include "rows.cuh"
#include "wide.cuh"

namespace bcs {
namespace {

constexpr unsigned kRowThreads = 1024;
constexpr uint32_t kShortRun = 192;               // see wide_kernel

// One CTA per SM at most; every warp takes items of `item` (32, 64 or 128) consecutive ranks, in turn over the CTAs.
// first: rank of the first row (< p); the count <= p ranks go on at 0 behind p - 1.
template <int kWords>
__global__ void __launch_bounds__(kRowThreads, 1)
rows_kernel(const __grid_constant__ RowConsts rc, uint32_t first, uint32_t count, uint32_t item, int8_t *recv,
            int8_t *send)
{
    extern __shared__ __align__(128) uint8_t sm[];
    grid_launch_dependents();
    const RowLayout at(rc.q);
    const RowTable t(sm, at);
    const uint32_t n_warps = blockDim.x >> 5, warp = threadIdx.x >> 5;
    const uint64_t stride = (uint64_t)gridDim.x * n_warps * item;
    const uint64_t begin = ((uint64_t)warp * gridDim.x + blockIdx.x) * item;
    auto rank = [&](uint64_t b) {
        const uint32_t x = first + (uint32_t)b;
        return x >= rc.p ? x - rc.p : x;
    };
    if (threadIdx.x < kRow + kLow + 1) t.s[threadIdx.x] = rc.s[threadIdx.x];
    if (rc.q > kLow) {
        // Where every warp has one item at most, the CTA's segments are few: rows for those only (all ranks of
        // 1152 and 32 ranks of any p need two or three of up to 25 groups of rows).
        const bool few = count <= stride;
        if (threadIdx.x == 0) *t.wanted = few ? 0u : (2u << (rc.q - kLow)) - 1u;
        if (few) {
            __syncthreads();
            if (begin < count) {
                const uint32_t mask = wanted_rows(rc.q, rc.inv, rank(begin), item + kHalo);
                if ((threadIdx.x & 31u) == 0u) atomicOr(t.wanted, mask);
            }
        }
    }
    __syncthreads();
    build_row_table(t, rc.q, rc.odd);
    uint8_t *mine = sm + at.warps + warp * at.warp_bytes;
    for (uint64_t b = begin; b < count; b += stride) {
        const uint32_t n = count - (uint32_t)b < item ? count - (uint32_t)b : item;
        const uint64_t byte = b * (uint64_t)rc.q;
        warp_rows<kWords, true>(t, mine, rc.q, rc.odd, rc.inv, rank(b), n, recv ? recv + byte : nullptr,
                                send ? send + byte : nullptr);
    }
    stage_free();
}

// The same for larger tables, q >= 16 (wide.cuh), one CTA per SM; `item` is a multiple of 16.  halves: every warp has one item of
// one table, half of the warps write the receive rows and half the send rows; otherwise all warps the ones before the others.
// (No more than 640 threads: at the speed of the memory the write streams of 1024 cost 20 % and more.)
template <unsigned kThreads, int kCtas, bool kAnyStep>
__global__ void __launch_bounds__(kThreads, kCtas)
wide_kernel(const __grid_constant__ RowConsts rc, uint32_t first, uint32_t count, uint32_t item, bool halves,
            int8_t *recv, int8_t *send)
{
    extern __shared__ __align__(128) uint8_t sm[];
    grid_launch_dependents();
    const WideLayout at(rc.q);
    const RowTable t(sm, at.base);
    if (threadIdx.x < kRow + kLow + 1) t.s[threadIdx.x] = rc.s[threadIdx.x];
    if (halves) {
        // One run per warp, those of the CTA side by side: rows for their segments only (all ranks of 100 003: five of 11
        // groups of rows, of about 2^20 nine of 15; 6.13 -> 5.97 and 16.8 -> 15.7 us, 1.3 million ranks 17.6 -> 16.5).
        const uint32_t warps = (blockDim.x >> 5) / (recv != nullptr && send != nullptr ? 2u : 1u);
        // A CTA that has no ranks stays until the kernel before is done, too.  If it left at once, CTAs of the call after next would
        // take its place, two of one call on some SMs, and the whole call would wait for those: in a row of calls 700 001 ranks 12.5 us
        // and not 9.65, 1 000 003 16.7 and not 12.0, receive rows of 1 000 003 9.8 and not 7.5 (none is without ranks at 1 048 576: 12.4 both
        // ways).  Runs of both tables of kShortRun ranks and less take no longer than what comes before them, and the call after next is
        // welcome: 98 304 ranks 5.0 us, 5.15 with the wait, 140 000 ranks of q = 20 5.05, 5.5; but 180 000 6.0, 5.95, 300 001 7.0, 6.7.
        if (blockIdx.x * warps * item >= count) {
            if (item > kShortRun || recv == nullptr || send == nullptr) grid_dependency_wait();
            return;
        }
        const uint32_t x0 = first + blockIdx.x * warps * item;
        want_rows(t, rc.q, rc.inv, x0 >= rc.p ? x0 - rc.p : x0, warps * item + 1u);      // (the last vectors look at the rank behind)
    } else {
        if (threadIdx.x == 0) *t.wanted = (2u << (rc.q - kLow)) - 1u;
        __syncthreads();
    }
    build_row_table(t, rc.q, rc.odd);
    if (send != nullptr) build_send_table(t, reinterpret_cast<uint2 *>(sm + at.send), rc.q, rc.odd);
    const uint32_t warp = threadIdx.x >> 5;
    uint32_t n_warps = blockDim.x >> 5, index = warp;
    auto all = [&](auto is_send, int8_t *out) {
        WideLane mine;
        mine.template init<kAnyStep>(rc.q, 0u);
        const uint64_t stride = (uint64_t)gridDim.x * n_warps * item;
        for (uint64_t b = ((uint64_t)blockIdx.x * n_warps + index) * item; b < count; b += stride) {
            const uint32_t n = count - (uint32_t)b < item ? count - (uint32_t)b : item;
            uint32_t x0 = first + (uint32_t)b;
            if (x0 >= rc.p) x0 -= rc.p;
            wide_rows<decltype(is_send)::value, kAnyStep, true>(t, sm, at.send, sm + at.ends + warp * 32u, rc.p, rc.q, rc.odd, rc.inv,
                                                mine, x0, n, b == 0, b + n == count, out + b * (uint64_t)rc.q);
        }
    };
    bool receives = recv != nullptr, sends = send != nullptr;
    if (halves && receives && sends) {
        n_warps /= 2;
        sends = warp >= n_warps;
        receives = !sends;
        if (sends) index -= n_warps;
    }
    if (receives) all(std::false_type(), recv);
    if (sends) all(std::true_type(), send);
}

template <unsigned kThreads, int kCtas, bool kAnyStep = false>
bcs_status launch_wide(const RowConsts &rc, uint32_t first, uint32_t count, uint32_t item, bool halves, int8_t *recv, int8_t *send,
                       cudaStream_t stream)
{
    if constexpr (!kAnyStep) {
        if (step_ranks(rc.q) != 16u) return launch_wide<kThreads, kCtas, true>(rc, first, count, item, halves, recv, send, stream);
    }
    if (!allow_shared<wide_kernel<kThreads, kCtas, kAnyStep>>()) return BCS_ERR_CUDA;
    const unsigned items = (count + item - 1) / item;
    launch_dependent(true, wide_kernel<kThreads, kCtas, kAnyStep>, items < kSms ? items : kSms, kThreads,
                     WideLayout(rc.q).bytes, stream, rc, first, count, item, halves, recv, send);
    return launch_status();
}

// Warps of a CTA of the per-rank form of which two fit an SM, 16 to 18: 56 registers a thread, 228 KB (1 KB of each CTA the system's).
uint32_t paired_warps(int q)
{
    const RowLayout at(q);
    const uint32_t warps = (228u * 512u - 1024u - at.warps) / at.warp_bytes;
    return warps > 18u ? 18u : (warps < 16u ? 16u : warps);
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
    const unsigned grid = items < kSms ? items : kSms;
    // as many warps as there are items for, at least 8 (for the table): small CTAs let the next call's start beside them
    unsigned warps = (items + grid - 1) / grid;
    warps = warps < 8u ? 8u : (warps > kRowThreads / 32 ? kRowThreads / 32 : warps);
    launch_dependent(true, rows_kernel<kWords>, grid, 32u * warps, RowLayout(rc.q).total(warps), stream, rc, first, count,
                     item, recv, send);
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
    const uint32_t ranks = (uint32_t)count, x0 = (uint32_t)first;
    // The wide kernel for larger tables.  The per-rank form gets slower in steps: where the next call's CTA no longer fits beside one
    // (paired_warps) and above 148 x 32 x 32 ranks (151 552), where items have more than 32.  Both tables, us, per rank / wide, back to back:
    //     ranks     q = 18, 20   q = 19, 21, 22    q = 24     q = 26     q = 30
    //     65 536     2.8/4.5        2.7/4.3       2.8/4.2    2.8/4.4    2.9/4.4
    //     90 112     4.7/5.3        4.8/5.1       4.8/5.4    4.9/5.1    5.0/5.2
    //     98 304     4.7/5.3        4.8/5.0       4.9/5.5    4.9/5.1    5.0/5.0
    //    120 000     5.4/5.4        5.5/5.4       5.6/5.7    5.6/5.4    5.7/5.4
    //    140 000     5.8/5.2        5.9/5.3       6.0/5.4    6.1/5.3    6.2/5.4
    //    151 552     5.8/5.6        5.9/5.5       6.1/5.7    6.3/5.5    6.4/5.6
    // A call that is waited for takes 15.7 us per rank and 17.6 wide at 98 304 ranks, 15.9 and 17.7 at 131 072.  The lines, 98 304 up to
    // q = 22 and 151 552 above, are a compromise of the two: back to back the forms cross at some 105 000 (q = 18, 20, 24: 125 000) ranks.
    // One table alone: the wide form where the per-rank form's CTAs no longer fit an SM in pairs, above 85 248 ranks up to q = 24, 80 512 up
    // to 26, 75 776 for larger q.  Receive (send) rows, us, per rank / wide:
    //     ranks             q = 18               q = 24               q = 26               q = 30
    //     75 777    2.3/3.5 (2.7/3.4)    2.3/3.6 (2.7/3.6)    2.3/3.5 (2.8/3.4)    3.8/3.5 (4.5/3.4)
    //     83 000    2.5/3.5 (2.8/3.5)    2.5/3.7 (2.9/3.6)    4.1/3.6 (4.5/3.4)    4.0/3.6 (4.6/3.4)
    //     90 112    3.8/3.7 (4.3/3.5)    3.8/3.7 (4.4/3.6)    3.8/3.5 (4.4/3.4)    3.8/3.5 (4.5/3.4)
    //    131 072    4.3/3.6 (4.8/3.7)    4.3/3.6 (5.0/3.7)    4.4/3.6 (5.1/3.5)    4.4/3.6 (5.3/3.5)
    // Up to 2^23 ranks every warp has one run of one table; up to 2^20 the CTA is half an SM, so that the next call's tables
    // are built beside it.  (Above, 640 threads in one CTA: 1.06 million 13.5 us, with 768 13.7, with two CTAs of 448 15.1, of 384 15.3.)
    // Beyond, all receive rows before the send rows, item by item: an item's start costs as
    // much as some 50 ranks, but from 2^25 ranks on the memory bounds it, and items close together are written
    // faster (12.3 million ranks 54 us a table with items of 800, 61 with 400; 2^25: 151 and 146 us).
    const bool one = recv == nullptr || send == nullptr;
    if (rc.q >= kWideMinQ && count >= (one ? kSms * paired_warps(rc.q) * 32u + 1u : (rc.q <= 22 ? 98304u : kSms * 32u * 32u + 1u))) {
        const bool halves = count < (1u << 23);
        auto run = [&](uint32_t warps) {
            if (recv != nullptr && send != nullptr) warps /= 2;
            return (ranks + kSms * warps * kStep - 1u) / (kSms * warps * kStep) * kStep;
        };
        if (count <= (1u << 20)) return launch_wide<384, 2>(rc, x0, ranks, run(12), halves, recv, send, stream);
        if (halves) return launch_wide<640, 1>(rc, x0, ranks, run(20), halves, recv, send, stream);
        const uint32_t item = count >= (1u << 25) ? 384u : 768u;            // (whole steps: 400 and 800 where these have 20 ranks)
        return launch_wide<640, 1>(rc, x0, ranks, step_ranks(rc.q) == 20u ? item / 24u * 25u : item, halves, recv, send, stream);
    }
    return launch<1>(rc, x0, ranks, recv, send, stream);
}

}  // namespace bcs
