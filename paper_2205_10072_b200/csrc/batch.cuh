// All ranks of many p at once: bcs_build_batch.
//
// A CTA builds the row table of a p (rows.cuh) and computes rows from it; where several CTAs share an SM, one builds a
// table while the others compute.  Three kernels take a p by its size:
//   * up to 1024 ranks: a CTA of 128 or 256 threads per p, a rank per lane or four (rule at the end of this file);
//   * up to 2^21 ranks: CTAs of 256 threads take equal shares of the flattened ranks of the list, p by p;
//   * more: CTAs of 640 threads, one per SM, work on one p after another (launched only when the list is long enough to hold one).
// Each is launched as a dependent of the kernel before it on the stream and may run beside it until it waits for it.
// The plan is the caller's memory: the kernel before may still be writing it, or what it has written may not be visible yet.
// So what the plan shows before the wait is a guess, good for one thing: a table of row entries is a function of p
// alone, and the one that the guess asks for is built while the wait lasts.  Any p in a kernel's range gives a table
// within bounds, the search stays inside the plan's arrays whatever they hold, and nothing else is done.  Behind the wait all is
// read again (past the L1 cache, which may hold what the guess has read), and the table is built again if p is another.
// (With row tables computed in place, back to back, every p up to 1024, in any order: 17.7 us with the guess taken as it is, 18.3 like
// this, 25.4 with the first load behind the wait, 22.5 with an ordinary launch; one p of 2000: 6.7, 7.2, 10.5, 10.3; 16 p of 2^10..2^13: 16.8,
// 18.7.)
//
// Up to 1024 ranks: instruction issue, and a CTA's chain from its p to its last row.  Every p up to 1024, four ranks per lane, 10.2 us in any order
// (a rank per lane 13.9).
// Above, instruction issue and the integer pipe: 1024 p of 2^10..2^20 1250 us (both tables 4.7 TB/s).  That kernel holds two narrow and two wide
// forms in 80 registers and spills a few bytes at its three CTAs per SM; two per SM take 1368 us, four 1490.
#pragma once
#include <type_traits>

#include "quad.cuh"
#include "rows.cuh"
#include "wide.cuh"

namespace bcs {
namespace {

constexpr uint32_t kSmallP = 1024;
constexpr int kSmallQ = 10;
constexpr int kMiddleQ = 21;
constexpr uint32_t kLargeThreads = 640, kBatchThreads = 256, kBatchWarps = kBatchThreads / 32;
constexpr unsigned kMiddleCtas = 3;               // per SM

// What a CTA works on.
struct BatchJob {
    uint64_t rank0, rank1, entry0;   // flattened ranks and first byte of the p
    uint32_t p, odd, inv;
};

// One warp: constants of a p (any from 1 to 2^31 - 1) into t and job.  They depend on p only: skips[k] is p / 2^(q-k),
// rounded up (Algorithm 1).
__device__ __forceinline__ void load_p(uint32_t p, const RowTable &t, BatchJob &job)
{
    const int lane = (int)(threadIdx.x & 31u);
    const int q = ceil_log2_fast(p);
    const uint32_t skip = lane <= q ? (p + ((1u << (q - lane)) - 1u)) >> (q - lane) : 0u;
    const uint32_t before = __shfl_up_sync(0xffffffffu, skip, 1);
    const uint32_t odd = __ballot_sync(0xffffffffu, lane >= 1 && lane <= q && 2u * before != skip);
    t.s[lane] = skip;
    if (lane < kLow + 1) t.s[kRow + lane] = 0u;
    if (lane == 0) {
        job.p = p;
        job.odd = odd;
        job.inv = p > 1u ? (uint32_t)((1ull << (q - low_levels(q) + 32)) / p) : 0u;
        *t.wanted = q > kLow ? (2u << (q - kLow)) - 1u : 1u;
    }
}

// Ranks r0 .. r1-1 of a p by the warps of the CTA, the per-rank form, `item` (<= 128) ranks at a time.
template <int kWords>
__device__ __forceinline__ void narrow_piece(const RowTable &t, uint8_t *mine, const BatchJob &job, uint64_t entry0, int q,
                                             uint32_t r0, uint32_t r1, uint32_t item, int8_t *recv, int8_t *send)
{
    for (uint32_t r = r0 + (threadIdx.x >> 5) * item; r < r1; r += (blockDim.x >> 5) * item) {
        const uint32_t n = r1 - r < item ? r1 - r : item;
        const uint64_t byte = entry0 + (uint64_t)r * (uint64_t)q;
        warp_rows<kWords, false>(t, mine, q, job.odd, job.inv, r, n, recv + byte, send ? send + byte : nullptr);
    }
}

// Ranks r0 .. r1-1 of a p (multiples of 16, or r1 = p), wide form: every warp takes one run, receive rows then send rows.
__device__ __forceinline__ void wide_piece(const RowTable &t, const uint8_t *sm, const WideLayout &at, uint8_t *ends,
                                           const BatchJob &job, int q, uint32_t r0, uint32_t r1, int8_t *recv, int8_t *send)
{
    const uint32_t item = ((r1 - r0 + kBatchWarps - 1u) / kBatchWarps + kStep - 1u) / kStep * kStep;
    const uint32_t r = r0 + (threadIdx.x >> 5) * item;
    if (r >= r1) return;
    const uint32_t n = r1 - r < item ? r1 - r : item;
    const bool head = r == 0u, tail = r + n == job.p;
    const uint64_t byte = job.entry0 + (uint64_t)r * (uint64_t)q;
    WideLane lane;
    lane.init<true>(q, (uint32_t)(byte & 15u));                        // (the outputs start on 16-byte boundaries)
    wide_rows<false, true, false>(t, sm, at.send, ends, job.p, q, job.odd, job.inv, lane, r, n, head, tail, recv + byte);
    if (send != nullptr) {
        lane.home = -1;
        wide_rows<true, true, false>(t, sm, at.send, ends, job.p, q, job.odd, job.inv, lane, r, n, head, tail, send + byte);
    }
}

constexpr uint32_t kSmallRun = 256;               // ranks of a warp's run
// With room for more segments than it can have, an eighth CTA of 128 threads did not fit an SM: 5000 p of 777 42.0 us and not 40.5, 1100 of 300..1024 12.3, 11.8.
// (CTAs of 256 threads fit; one p of 500 3.48 us, with less room 3.56.)
__host__ __device__ constexpr uint32_t small_segments(uint32_t threads) { return threads == 128u ? run_segments(kSmallRun) : roomy_segments(kSmallRun); }

// All ranks of a p of 129..1024 by the warps of the CTA, four ranks per lane.  Runs begin where rows begin (nearly) on a 16-byte boundary.
// kSegments: how many the warps have room for.
template <int Q, uint32_t kSegments>
__device__ __forceinline__ void quad_small(const RowTable &t, uint8_t *sm, const BatchJob &job, uint64_t entry0, int8_t *recv, int8_t *send)
{
    const QuadLayout<false> at(Q, kSegments);
    const uint32_t warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    uint8_t *mine = sm + at.warps + warp * at.warp_bytes;
    const uint32_t best = quad_shift(entry0, Q), up = best & 15u, shift = best >> 4;
    const int begin = up ? (int)up - 16 : 0, p = (int)job.p;
    const int share = (int)(((uint32_t)(p - begin) + warps * kQuads - 1u) / (warps * kQuads) * kQuads);
    const int stop = begin + ((int)warp + 1) * share < p ? begin + ((int)warp + 1) * share : p;
    for (int a = begin + (int)warp * share; a < stop; a += (int)kSmallRun) {
        const uint32_t n = stop - a < (int)kSmallRun ? (uint32_t)(stop - a) : kSmallRun;
        const uint32_t lead = a < 0 ? (uint32_t)-a : 0u;
        const int64_t byte = (int64_t)entry0 + (int64_t)a * Q;
        quad_run<Q, false, false>(t, sm + at.table, mine, at, t.s, job.odd, job.inv, a < 0 ? job.p - lead : (uint32_t)a, n, lead, shift, recv + byte,
                                  send ? send + byte : nullptr);
    }
}

// p <= 1024: a CTA per p.  kQuad: four ranks per lane for p > 128.
template <unsigned kThreads, int kCtas, bool kQuad>
__global__ void __launch_bounds__(kThreads, kCtas)
batch_small_kernel(const __grid_constant__ BatchArgs ba, int8_t *recv, int8_t *send)
{
    extern __shared__ __align__(128) uint8_t sm[];
    __shared__ BatchJob job;
    __shared__ uint32_t guess;
    grid_launch_dependents();
    const uint32_t j = ba.num_p - 1u - blockIdx.x;               // (lists often ascend: the longest first)
    // The table is built for the p that the plan shows before the wait, see the top of this file.
    auto build = [&](uint32_t p) {
        const int q = ceil_log2_fast(p);
        const RowTable t(sm, RowLayout(q));
        if (threadIdx.x < 32u) load_p(p, t, job);
        __syncthreads();
        if (kQuad && q > kLow) build_row_table<true>(t, q, job.odd);
        else build_row_table<false, 1>(t, q, job.odd);
    };
    auto fits = [](uint32_t p) { return p > 1u && p <= kSmallP; };
    if (threadIdx.x == 0) guess = load_relaxed(ba.p_list + j);
    __syncthreads();
    const uint32_t built = guess;                                // (not written again)
    if (fits(built)) build(built);
    grid_dependency_wait();
    const uint32_t p = load_relaxed(ba.p_list + j);
    const uint64_t entry0 = load_relaxed(ba.entry_off + j);
    if (!fits(p)) return;
    if (p != built) build(p);
    const int q = ceil_log2_fast(p);
    const RowLayout at(q);
    const RowTable t(sm, at);
    if (kQuad && q > kLow) {
        constexpr uint32_t segments = small_segments(kThreads);
        if (q == 8) quad_small<8, segments>(t, sm, job, entry0, recv, send);
        else if (q == 9) quad_small<9, segments>(t, sm, job, entry0, recv, send);
        else quad_small<10, segments>(t, sm, job, entry0, recv, send);
        stage_free<true>();
    } else {
        uint8_t *mine = sm + at.warps + (threadIdx.x >> 5) * at.warp_bytes;
        constexpr uint32_t warps = kThreads / 32;
        const uint32_t turns = (p + warps * kItemRanks - 1u) / (warps * kItemRanks) * warps;
        const uint32_t item = ((p + turns - 1u) / turns + 31u) & ~31u;
        if (q <= 4) narrow_piece<1>(t, mine, job, entry0, q, 0u, p, item, recv, send);
        else if (q <= 8) narrow_piece<2>(t, mine, job, entry0, q, 0u, p, item, recv, send);
        else if constexpr (!kQuad) narrow_piece<3>(t, mine, job, entry0, q, 0u, p, item, recv, send);
        stage_free<false>();
    }
}

// 1024 < p <= 2^21: the CTA's share is `share` (a multiple of 16) flattened ranks.
__global__ void __launch_bounds__(kBatchThreads, kMiddleCtas)
batch_middle_kernel(const __grid_constant__ BatchArgs ba, uint32_t share, int8_t *recv, int8_t *send)
{
    extern __shared__ __align__(128) uint8_t sm[];
    __shared__ BatchJob job;
    __shared__ uint32_t found;
    __shared__ uint32_t home, from;                              // first warp only: what a guess has found to hold rank g0, where to look on
    grid_launch_dependents();
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t g0 = (uint64_t)blockIdx.x * share;
    const uint64_t g1 = g0 + share < ba.total_ranks ? g0 + share : ba.total_ranks;
    // (CTAs beyond those that fit at once start when others of the grid have ended: nothing is left to wait for)
    bool sure = blockIdx.x >= kSms * kMiddleCtas;                // the wait is behind us
    if (sure) grid_dependency_wait();
    uint32_t built = 0;                                          // the p whose tables are in shared memory
    if (threadIdx.x < 32u) {
        const uint32_t j = find_segment_warp(ba.rank_off, ba.num_p, g0);
        if (lane == 0u) home = from = j;
    }
    for (;;) {
        __syncthreads();                                         // the p before is done with
        if (threadIdx.x < 32u) {
            uint32_t hits = 0, p = 0;
            uint64_t rank0 = 0, rank1 = 0, entry0 = 0;
            uint32_t base = from;
            bool again = base == home;
            for (;; base += 32u) {
                const uint32_t j = base + lane;
                const bool listed = j < ba.num_p;
                rank0 = listed ? load_relaxed(ba.rank_off + j) : 0u;
                rank1 = listed ? load_relaxed(ba.rank_off + j + 1) : 0u;
                entry0 = listed ? load_relaxed(ba.entry_off + j) : 0u;
                p = listed ? load_relaxed(ba.p_list + j) : 0u;
                if (again && __any_sync(0xffffffffu, lane == 0u && (rank0 > g0 || rank1 <= g0))) {
                    again = false;
                    base = find_segment_warp(ba.rank_off, ba.num_p, g0) - 32u;
                    continue;
                }
                again = false;
                const bool inside = listed && rank0 < g1;
                hits = __ballot_sync(0xffffffffu, inside && p > kSmallP && p <= (1u << kMiddleQ));
                if (hits != 0u || __any_sync(0xffffffffu, !inside) || !sure) break;
            }
            if (hits != 0u) {
                const uint32_t nth = (uint32_t)__ffs(hits) - 1u;
                if (lane == nth) {
                    job.rank0 = rank0;
                    job.rank1 = rank1;
                    job.entry0 = entry0;
                }
                p = __shfl_sync(0xffffffffu, p, nth);
                if (p != built) load_p(p, RowTable(sm, RowLayout(ceil_log2_fast(p))), job);
                base += nth + 1u;
            }
            if (lane == 0u) {
                found = hits != 0u ? p : 0u;
                if (sure) {                                      // (a guess is looked at again)
                    from = base;
                    home = 0xffffffffu;
                }
            }
        }
        __syncthreads();
        const uint32_t p = found;
        if (p == 0u && sure) break;
        const int q = ceil_log2_fast(p);
        const bool narrow = q < kWideMinQ;
        const RowLayout at_narrow(q);
        const WideLayout at(q);
        const RowTable t(sm, at_narrow);
        const uint32_t r0 = g0 > job.rank0 ? ((uint32_t)(g0 - job.rank0) + 15u) & ~15u : 0u;
        const uint32_t end = g1 < job.rank1 ? ((uint32_t)(g1 - job.rank0) + 15u) & ~15u : p;
        const uint32_t r1 = end < p ? end : p;
        if (p != built) {
            built = 0u;
            if (p != 0u && r0 < r1) {
                build_row_table<false, 2>(t, q, job.odd);
                if (!narrow && send != nullptr) build_send_table_wide(t, reinterpret_cast<uint2 *>(sm + at.send), q, job.odd);
                built = p;
            }
        }
        if (!sure) {                                             // that was a guess: look again
            grid_dependency_wait();
            sure = true;
            continue;
        }
        if (r0 >= r1) continue;
        if (narrow) {
            uint8_t *mine = sm + at_narrow.warps + (threadIdx.x >> 5) * at_narrow.warp_bytes;
            if (q <= 12) narrow_piece<3>(t, mine, job, job.entry0, q, r0, r1, kItemRanks, recv, send);
            else narrow_piece<4>(t, mine, job, job.entry0, q, r0, r1, kItemRanks, recv, send);
            stage_free<false>();
        } else {
            wide_piece(t, sm, at, sm + at.ends + (threadIdx.x >> 5) * 32u, job, q, r0, r1, recv, send);
        }
    }
}

// p > 2^21: all CTAs on every such p of the list.
__global__ void __launch_bounds__(kLargeThreads, 1)
batch_large_kernel(const __grid_constant__ BatchArgs ba, int8_t *recv, int8_t *send)
{
    extern __shared__ __align__(128) uint8_t sm[];
    __shared__ BatchJob job;
    grid_launch_dependents();
    grid_dependency_wait();
    constexpr uint32_t item = 768;
    uint32_t j = 0;
    for (;;) {
        for (; j < ba.num_p; ++j) {                              // the next one, kLargeThreads at a glance
            if (j % kLargeThreads == 0u) {
                const uint32_t k = j + threadIdx.x;
                if (!__syncthreads_or(k < ba.num_p && ba.p_list[k] > (1u << kMiddleQ))) {
                    j += kLargeThreads - 1u;
                    continue;
                }
            }
            if (ba.p_list[j] > (1u << kMiddleQ)) break;
        }
        if (j >= ba.num_p) break;
        const uint32_t p = ba.p_list[j];
        const int q = ceil_log2_fast(p);
        const WideLayout at(q);
        const RowTable t(sm, at.base);
        __syncthreads();                                         // the p before is done with
        if (threadIdx.x < 32u) load_p(p, t, job);
        const uint64_t entry0 = ba.entry_off[j];
        __syncthreads();
        build_row_table<false, 1>(t, q, job.odd);
        if (send != nullptr) build_send_table_wide(t, reinterpret_cast<uint2 *>(sm + at.send), q, job.odd);
        const uint32_t warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
        auto all = [&](auto is_send, int8_t *out) {
            WideLane lane;
            lane.init<true>(q, (uint32_t)(entry0 & 15u));
            for (uint64_t r = ((uint64_t)blockIdx.x * n_warps + warp) * item; r < p; r += (uint64_t)gridDim.x * n_warps * item) {
                const uint32_t n = p - (uint32_t)r < item ? p - (uint32_t)r : item;
                wide_rows<decltype(is_send)::value, true, false>(t, sm, at.send, sm + at.ends + warp * 32u, p, q, job.odd, job.inv, lane,
                                                    (uint32_t)r, n, r == 0, r + n == p, out + entry0 + r * (uint64_t)q);
            }
        };
        all(std::false_type(), recv);
        if (send != nullptr) all(std::true_type(), send);
        ++j;
    }
}

// A CTA per p of the list, up to kCtas of them per SM.  alone: no larger p, nothing runs beside them.  Where the list is then
// too short to fill the card, they ask for so much shared memory that they spread over all SMs (else some held five and
// others one: 300 p of 3..900 11.9 -> 8.4 us).
template <unsigned kThreads, int kCtas, bool kQuad>
bcs_status launch_small(const BatchArgs &ba, bool alone, int8_t *recv, int8_t *send, cudaStream_t stream)
{
    constexpr uint32_t fits = 228u * 1024u / kCtas - 1024u - (uint32_t)sizeof(BatchJob) - 16u;       // (1 KB of each CTA is the system's)
    uint32_t shared = RowLayout(kSmallQ).total(kThreads / 32);
    if constexpr (kQuad) {
        constexpr QuadLayout<false> at(kSmallQ, small_segments(kThreads));
        static_assert(at.total(kThreads / 32) <= fits, "shared memory for kCtas CTAs per SM");
        shared = at.total(kThreads / 32);
    }
    const uint32_t per_sm = (ba.num_p + kSms - 1) / kSms;
    if (alone && per_sm < (uint32_t)kCtas) {
        const uint32_t spread = (226u * 1024u / per_sm - 1280u) & ~127u;
        if (shared < spread) shared = spread;
    }
    if (!allow_shared<batch_small_kernel<kThreads, kCtas, kQuad>>()) return BCS_ERR_CUDA;
    launch_dependent(true, batch_small_kernel<kThreads, kCtas, kQuad>, ba.num_p, kThreads, shared, stream, ba, recv, send);
    return launch_status();
}

}  // namespace
}  // namespace bcs

using namespace bcs;

extern "C" {

size_t bcs_build_batch_workspace_bytes(uint64_t total_ranks, uint64_t total_copy)
{
    if (total_ranks == 0) return 0;
    if (total_copy == 0) return 256;
    return (size_t)(align_up(4ull * total_ranks, 256) + total_copy);
}

bcs_status bcs_build_batch(const uint32_t *p_list_dev, const uint64_t *rank_off_dev,
                           const uint64_t *entry_off_dev, const uint64_t *tile_off_dev,
                           const uint64_t *copy_off_dev, const uint32_t *skips_tab_dev,
                           const uint32_t *full_tab_dev, uint32_t num_p, uint64_t total_ranks,
                           uint64_t total_entries, uint64_t total_tiles, uint64_t total_copy,
                           int8_t *recv_out, int8_t *send_out, void *workspace, size_t workspace_bytes,
                           void *cuda_stream)
{
    if (num_p == 0 || total_ranks == 0) return BCS_OK;
    if (p_list_dev == nullptr || rank_off_dev == nullptr || entry_off_dev == nullptr ||
        skips_tab_dev == nullptr || full_tab_dev == nullptr)
        return BCS_ERR_ARG;
    if (total_entries == 0) return BCS_OK;   // only p == 1 in the list
    if (recv_out == nullptr) return BCS_ERR_ARG;
    if (!aligned16(recv_out) || !aligned16(send_out) || !aligned16(workspace)) return BCS_ERR_ALIGN;
    if ((total_ranks + kTile - 1) / kTile > 0x7fffffffull || total_tiles > 0x3fffffffull) return BCS_ERR_UNSUPPORTED;
    (void)copy_off_dev;                      // the rows need no scratch memory, see rows.cuh
    (void)total_copy;
    (void)workspace_bytes;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    const BatchArgs ba = {p_list_dev, rank_off_dev, entry_off_dev, num_p, total_ranks};
    static_assert(kSmallP == kFusedMaxP, "the plan counts tiles for the p above kSmallP");
    // (without the plan's tiles the host cannot tell what sizes the list holds)
    const bool small_only = tile_off_dev != nullptr && total_tiles == 0;
    if (!small_only) {
        const WideLayout wide(kMiddleQ);
        const RowLayout narrow(kWideMinQ - 1);
        const uint32_t shared = wide.bytes > narrow.total(kBatchWarps) ? wide.bytes : narrow.total(kBatchWarps);
        if (!allow_shared<batch_middle_kernel>()) return BCS_ERR_CUDA;
        // Up to 2^23 ranks a share per resident CTA: every share costs a search and a table or two (16 p
        // of 2^10..2^20 83 us with three, 76 with one; 3000 of 2^10..2^11 115, 106).  Beyond, three, so that none
        // ends last by much (150 p of 2^12..2^18 146 us, with one 152; 300 of 2^14..2^18 286, 296; 3000 of 2^12..2^13 277, 341;
        // but 64 of 2^17..2^18, few tables, 140, 137).  At most 32768 ranks, at least 1024 (a table costs as much as some
        // hundred ranks of each warp).
        const uint64_t ctas = kSms * kMiddleCtas * (total_ranks <= (1u << 23) ? 1u : 3u);
        uint64_t share = align_up(total_ranks / ctas, 128);
        share = share < 1024 ? 1024 : (share > 32768 ? 32768 : share);
        const uint64_t shares = (total_ranks + share - 1) / share;
        launch_dependent(true, batch_middle_kernel, (unsigned)shares, kBatchThreads, shared, stream, ba, (uint32_t)share,
                         recv_out, send_out);
        if (total_ranks > (1u << kMiddleQ)) {
            if (!allow_shared<batch_large_kernel>()) return BCS_ERR_CUDA;
            launch_dependent(true, batch_large_kernel, kSms, kLargeThreads, WideLayout(BCS_MAX_Q).bytes, stream, ba, recv_out,
                             send_out);
        }
    }
    // Four ranks per lane for lists without a larger p whose p are 400 on average or more; us with it / the per-rank form: every p up to 1024 in any order
    // 10.2/13.9, and with seven CTAs per SM 11.7, ascending 10.8/15.4, 5000 of 777 43.6/60.8, 800 of 1000 8.1/12.9, 740 of 280..1019 8.8/9.8.  A CTA takes one p, and CTAs whose p
    // have other q run other code, which counts where there is little to do for each: 900 of 64..256 6.3/5.9, 300 of 64..1000 7.5/6.7, 700 of 2^6..2^12
    // (beside the kernel for larger p) 33.3/29.8.  CTAs of 256 threads while three of them per SM take the list (140 of 900 4.6, with 128 threads 5.1).
    if (small_only && total_ranks >= 400ull * num_p) {
        if (num_p <= kSms * 3u) return launch_small<256, 3, true>(ba, true, recv_out, send_out, stream);
        return launch_small<128, 8, true>(ba, true, recv_out, send_out, stream);
    }
    // Per rank: CTAs of 256 threads while all are resident at once (the shorter chain counts), else of 128 (less waiting at
    // barriers, longer items): us with 256 / 128, 300 p of 3..900 7.0/8.8, 700 of 3..702 9.4/10.2;
    // 900 of 64..256 8.4/6.0, 1000 of 33 6.4/3.7, 2000 of 2..1024 20.7/20.7.
    if (num_p <= kSms * 5u) return launch_small<256, 5, false>(ba, small_only, recv_out, send_out, stream);
    return launch_small<128, 8, false>(ba, small_only, recv_out, send_out, stream);
}

}  // extern "C"
