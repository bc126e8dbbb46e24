// Receive and send rows of a stretch of ranks of one p: the kernels behind bcs_build and its relatives.
//
// One launch, nothing read from memory but constants, no table of all ranks (rows.cuh).  By size (launch_rows):
//   * rows_kernel, a rank per lane.  Bound by latency: launch, table, one or two items per warp.  From Python 32 ranks 3.2 us back to
//     back, all ranks of 1152 3.3, 65 553 ranks 3.2 (2.7 on the device).  The table holds what the
//     CTA's segments need where these are few, and a CTA has no more warps than items.
//   * quad_kernel, four ranks per lane (quad.cuh).  Up to some 2^21 ranks bound by instruction issue, the integer pipe with it, above by
//     memory writes.  All ranks of 100 003 2.4 us, of 1.06 million 9.6, 2^24 ranks of q = 28 133, 2^25 receive rows 140 (6.7 TB/s).  With vectors
//     of 16 output bytes per lane in its place, some 40 warp instructions for every 32 of them where a segment ends: 4.9, 13.3, 148 and 148.
//   * wide_send_kernel, 16 output bytes per lane (wide.cuh): send rows alone of some million ranks.
// All are launched as dependents of whatever runs before them on the stream and wait for it before their first store.
#include "batch.cuh"     // (in this unit, too: the constants of rows.cuh are in the module once)
#include "rows.cuh"
#include "quad.cuh"
#include "wide.cuh"

namespace bcs {
namespace {

constexpr unsigned kRowThreads = 1024;

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
    stage_free<true>();
}

// Send rows alone of 1.9 to 6 million ranks, or from where quad_kernel takes turns (q >= 27), 16 output bytes per lane (wide.cuh): a run per warp, one CTA per SM.  Its table of send rows holds those of all the
// CTA's segments, and nothing is looked up twice.  us, this / quad_kernel: 2 million ranks of q = 21 11.3/11.4, of q = 28 12.1/12.8, 3.1 million of q = 23
// 16.0/18.9, 4.8 million 22.4/23.5, 1.7 million of q = 31 12.0/12.9, 1.86 million of q = 28 11.2/12.8; 1.5 million of q = 21 10.2/9.1, 6.5 million of q = 24 31.7/29.9, of q = 28 34.7/30.9.
constexpr unsigned kWideThreads = 640;
constexpr uint32_t kWideFrom = 1900000, kWideTo = 6000000;

template <bool kAnyStep>
__global__ void __launch_bounds__(kWideThreads, 1)
wide_send_kernel(const __grid_constant__ RowConsts rc, uint32_t first, uint32_t count, uint32_t run, int8_t *send)
{
    extern __shared__ __align__(128) uint8_t sm[];
    grid_launch_dependents();
    const WideLayout at(rc.q);
    const RowTable t(sm, at.base);
    if (threadIdx.x < kRow + kLow + 1) t.s[threadIdx.x] = rc.s[threadIdx.x];
    const uint32_t warps = kWideThreads / 32u, warp = threadIdx.x >> 5, begin = blockIdx.x * warps * run;
    if (begin >= count) {                                        // (stays until the kernel before is done, or CTAs of the next calls pile up here)
        grid_dependency_wait();
        return;
    }
    auto rank = [&](uint32_t b) {
        const uint32_t x = first + b;
        return x >= rc.p ? x - rc.p : x;
    };
    want_rows(t, rc.q, rc.inv, rank(begin), warps * run + 1u);   // (the last vectors look at the rank behind)
    build_row_table(t, rc.q, rc.odd);
    build_send_table_wide(t, reinterpret_cast<uint2 *>(sm + at.send), rc.q, rc.odd);
    const uint32_t b = begin + warp * run;
    if (b >= count) return;
    const uint32_t n = count - b < run ? count - b : run;
    WideLane mine;
    mine.template init<kAnyStep>(rc.q, 0u);
    wide_rows<true, kAnyStep, true>(t, sm, at.send, sm + at.ends + warp * 32u, rc.p, rc.q, rc.odd, rc.inv, mine, rank(b), n, b == 0u, b + n == count,
                                    send + (uint64_t)b * (uint64_t)rc.q);
}

template <bool kAnyStep>
bcs_status launch_wide_send(const RowConsts &rc, uint32_t first, uint32_t count, int8_t *send, cudaStream_t stream)
{
    if (!allow_shared<wide_send_kernel<kAnyStep>>()) return BCS_ERR_CUDA;
    const uint32_t all = kSms * kWideThreads / 32u * kStep, run = (count + all - 1u) / all * kStep;
    launch_dependent(true, wide_send_kernel<kAnyStep>, kSms, kWideThreads, WideLayout(rc.q).bytes, stream, rc, first, count, run, send);
    return launch_status();
}

// Half an SM's shared memory, and the warps of a CTA that have room in it for runs of `run` ranks.
constexpr uint32_t kQuadHalf = (228u * 512u - 1024u - 128u) & ~127u;
template <int Q, bool kTable>
constexpr uint32_t quad_bytes(uint32_t warps, uint32_t run) { return QuadLayout<kTable>(Q, roomy_segments(run)).total(warps); }
template <int Q, bool kTable>
constexpr uint32_t quad_warps(uint32_t run)
{
    uint32_t warps = 10;
    while (warps > 4u && quad_bytes<Q, kTable>(warps, run) > kQuadHalf) --warps;
    return warps;
}
// Threads that registers are shared among: ten warps; for q = 28, whose rows need the most, as many as a CTA ever has (with ten it spills: one million ranks 11.1 -> 10.7 us,
// 400 000 send rows 4.4 -> 3.9; q = 25 to 27 spill a word; for larger q more registers are no better, 300 000 receive rows of q = 30 2.84 -> 3.03).
template <int Q, bool kTable>
constexpr uint32_t kQuadThreads = 32u * (Q == 28 ? quad_warps<Q, kTable>(kTable ? 4u * kQuads : kQuads) : 10u);

__device__ unsigned long long expired_waits;      // waits with a limit that ran out
constexpr uint64_t kWaitLimit = 2000000000;       // two seconds (an answer takes a microsecond)

// Two CTAs per SM.  A turn of a CTA is a run per warp.  once: a CTA for each turn, all of them run at once.  Otherwise the CTAs that run take the turns of
// those that have not started yet: SMs do not write equally fast (a fill by CTAs of equal shares reaches 6.3 TB/s, by CTAs of 16 KB in
// any order 7.5), and one table serves all turns of a CTA.
template <int Q, bool kTable>
__global__ void __launch_bounds__((kQuadThreads<Q, kTable>), 2)
quad_kernel(const __grid_constant__ RowConsts rc, uint32_t first, uint32_t count, uint32_t run, bool once, int8_t *recv, int8_t *send)
{
    extern __shared__ __align__(128) uint8_t sm[];
    __shared__ __align__(16) uint4 answer;
    grid_launch_dependents();
    __shared__ uint64_t answered;
    const QuadLayout<kTable> at(Q, roomy_segments(run));
    const uint32_t warps = blockDim.x >> 5, warp = threadIdx.x >> 5;
    const RowTable t(sm, at.base);
    if (threadIdx.x < kRow + kLow + 1) t.s[threadIdx.x] = rc.s[threadIdx.x];
    if (once) {
        const uint32_t x0 = first + blockIdx.x * warps * run;
        want_rows(t, Q, rc.inv, x0 >= rc.p ? x0 - rc.p : x0, warps * run + kHalo);
    } else {
        if (threadIdx.x == 0) {
            *t.wanted = (2u << (Q - kLow)) - 1u;
            barrier_init(&answered);
        }
        __syncthreads();
    }
    build_row_table<true>(t, Q, rc.odd);
    if constexpr (kTable) build_send_table(t, reinterpret_cast<uint2 *>(sm + at.table), Q, rc.odd);
    uint8_t *mine = sm + at.warps + warp * at.warp_bytes;
    uint32_t turn = blockIdx.x, parity = 0;
    for (;;) {
        if (!once && threadIdx.x == 0) ask_for_work(&answer, &answered);
        const uint64_t b = ((uint64_t)turn * warps + warp) * run;
        if (b < count) {
            const uint32_t n = count - (uint32_t)b < run ? count - (uint32_t)b : run;
            uint32_t x0 = first + (uint32_t)b;
            if (x0 >= rc.p) x0 -= rc.p;
            const uint64_t byte = b * Q;
            quad_run<Q, kTable, true>(t, sm + at.table, mine, at, rc.s, rc.odd, rc.inv, x0, n, 0u, 0u, recv ? recv + byte : nullptr, send ? send + byte : nullptr);
        }
        if (once) break;
        const Work more = await_work(&answer, &answered, parity, kWaitLimit, &turn);
        if (more == Work::expired && threadIdx.x == 0) atomicAdd(&expired_waits, 1ull);          // (bcs_wait_expired)
        if (more != Work::given) break;
        parity ^= 1u;
    }
    stage_free<true>();
}

// Turns and CTAs.  Runs are whole look-ups (128 ranks): partly filled ones cost as much.  The shortest run with which at most 296 CTAs of up to ten warps
// (as many as two CTAs per SM have shared memory for) have all ranks at once; and no more warps than make 148 CTAs, which leave room for the
// next call's (back to back, us, the kernel as it was when this was chosen: all ranks of 100 003 2.4, with the ranks spread over 296 CTAs 4.5; 200 000 ranks of q = 21 4.2 and 4.9, 524 288 6.6
// and 6.5, 1.06 million 10.2 and 10.3).  One table: two look-ups as soon as 148 CTAs do not do with one (200 000 receive rows 2.6 us, with runs of 128 3.0).
// The shared memory is filled up to half an SM, lest three CTAs of one call meet on an SM while another one has one.
// Longer ranges: turns of 512 ranks per warp, of 768 for one table from 3.5 million on (2^24 send rows of q = 28 71 us, with 512 74; receive rows of 3
// million 15.6, with 512 14.9).
template <int Q, bool kTable>
bcs_status launch_quad(const RowConsts &rc, uint32_t first, uint32_t count, int8_t *recv, int8_t *send, cudaStream_t stream)
{
    if (!allow_shared<quad_kernel<Q, kTable>>()) return BCS_ERR_CUDA;
    const uint32_t quads = (count + kQuads - 1u) / kQuads;
    const bool one = recv == nullptr || send == nullptr;
    uint32_t k = 1;
    while (k * kQuads <= kMostRun && quad_warps<Q, kTable>(k * kQuads) * k * kSms * (one && k == 1u ? 1u : 2u) < quads) ++k;
    const bool once = k * kQuads <= kMostRun;
    if (!once) k = one && count >= 3500000u ? 6u : 4u;
    const uint32_t run = k * kQuads;
    uint32_t warps = quad_warps<Q, kTable>(run);
    if (once) {
        const uint32_t enough = (quads + k * kSms - 1u) / (k * kSms);
        warps = warps < enough ? warps : (enough < 4u ? 4u : enough);
    }
    const uint32_t need = quad_bytes<Q, kTable>(warps, run), turn = warps * run;
    launch_dependent(true, quad_kernel<Q, kTable>, (unsigned)(((uint64_t)count + turn - 1u) / turn), 32u * warps, need < kQuadHalf ? kQuadHalf : need, stream, rc, first,
                     count, run, once, recv, send);
    return launch_status();
}

// kTable from 2^22 ranks on: building the table of send rows pays (send rows of q = 28, us, without / with it: 1 million 7.1/8.0, 3 million 17.6/17.4, 8 million
// 43/37, 2^25 164/137; both tables 4 million 33.9/35.0, 8 million 66.6/65.7).
template <int Q>
bcs_status launch_quads(const RowConsts &rc, uint32_t first, uint32_t count, int8_t *recv, int8_t *send, cudaStream_t stream)
{
    if constexpr (Q > BCS_MAX_Q) return BCS_ERR_UNSUPPORTED;
    else {
        if (rc.q != Q) return launch_quads<Q + 1>(rc, first, count, recv, send, stream);
        constexpr uint32_t at_once = quad_warps<Q, false>(kMostRun) * (kMostRun / kQuads) * 2u * kSms * kQuads;
        if (recv == nullptr && (count >= kWideFrom || count > at_once) && count < kWideTo)
            return step_ranks(Q) == 16u ? launch_wide_send<false>(rc, first, count, send, stream) : launch_wide_send<true>(rc, first, count, send, stream);
        if constexpr (Q >= 22)                                   // (2^22 ranks are more than a smaller p has)
            if (send != nullptr && count >= (1u << 22)) return launch_quad<Q, true>(rc, first, count, recv, send, stream);
        return launch_quad<Q, false>(rc, first, count, recv, send, stream);
    }
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

bool expired_wait_count(unsigned long long *count)
{
    return cudaMemcpyFromSymbol(count, expired_waits, sizeof *count) == cudaSuccess;
}

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
    // Four ranks per lane where two of the per-rank form's CTAs no longer fit an SM (148 x 16 x 32 ranks).  Both tables, us back to back, per rank / four
    // per lane (a call that is waited for):
    //     ranks          q = 20                 q = 24                 q = 28                 q = 31
    //     32 768    2.0/2.2 (14.3/16.0)    2.1/2.5 (14.3/15.0)    2.1/2.6 (14.3/15.2)    2.1/2.9 (14.6/15.5)
    //     65 553    2.7/2.4 (14.6/15.4)    2.7/2.6 (14.6/15.1)    2.8/2.7 (14.6/15.0)    2.8/2.9 (14.9/15.5)
    //     75 777    2.7/2.2 (15.5/15.1)    2.8/2.3 (15.7/15.5)    4.4/2.3 (15.9/15.7)    4.5/2.6 (16.0/15.9)
    //     98 304    4.9/2.4 (17.5/15.0)    4.6/2.7 (16.1/15.4)    4.5/2.7 (16.3/15.6)    4.7/3.0 (16.4/15.7)
    // (The first two lines with the kernel as it was before low ranks were put together by their entries' zero bytes, on another box.)
    if (rc.q >= kQuadMinQ && count > kSms * 16u * 32u) return launch_quads<kQuadMinQ>(rc, x0, ranks, recv, send, stream);
    return launch<1>(rc, x0, ranks, recv, send, stream);
}

}  // namespace bcs
