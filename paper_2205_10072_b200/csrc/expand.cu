// Round tables of the n-block broadcast (arXiv 2205.10072, Algorithm 6 without the
// Send||Recv): a pure store stream, one 16-byte record per (rank, round).
#include "bcs_common.cuh"
#include "paper_path.cuh"

namespace bcs {
namespace {

// ---------------------------------------------------------------- Algorithm 6: round tables
// Records and threads of a CTA.  Memory writes bound it, and small CTAs in the order of the records write fastest (SMs do not write equally fast, so the
// hardware's handing out of CTAs balances them): p = 100 003, n = 1000 219 us with 1024 records (7.4 TB/s), 222 with 2048, 227 with 4096, 234 with 8192.
// By the number of records, us with 512 records and 256 threads / 512, 128 / 1024, 128: 1.0 million (p = 40 000, n = 10) 7.6/8.0/12.3, 0.9 million (3000, 300)
// 4.2/4.3/6.1; 1.9 million (30 000, 50) 8.5/7.3/8.7, 2.0 million (1000, 2000) 7.2/6.3/6.8; 5.4 million (200 000, 10) 32.5/27.8/27.6, 11.6 million
// (100 003, 100) 40.6/32.2/28.0.
// More than one CTA per SM, but fewer than run at once (eight per SM of 256 threads): as few records each as let them, a record or two per thread.
// us with 512 / 256 or 384: 0.19 million (6000, 20) 4.0/2.4, 0.15 million (300, 500) 2.6/2.1, 0.32 million (20 000, 2) 5.7/4.6, 0.33 million (3000, 100) 3.2/2.7,
// 0.36 million (1152, 300) 2.9/2.6, 0.40 million (12 000, 20) 4.3/3.5; but rows of more than 512 rounds, 0.30 million (300, 1000) 2.3/2.7, (100, 3000) 2.3/2.6.
constexpr uint32_t kExpandRecords = 1024, kExpandFewer = 512, kExpandStep = 128, kExpandFewest = 256;
constexpr uint32_t kExpandSms = 148, kExpandAtOnce = 148 * 8;
constexpr uint64_t kExpandMany = 4000000, kExpandFew = 1200000;
constexpr int kExpandThreads = 128, kExpandThreadsFew = 256;
constexpr uint32_t kExpandBuilt = 8192;        // where the CTA builds the rows of its ranks, whole ranks then
constexpr uint32_t kExpandCtas = 148 * 4;      // and every SM four CTAs
constexpr uint32_t kExpandSharedBytes = 48 * 1024;

// What is the same for all threads, and took them divisions.
struct Walk {
    uint64_t by_rounds;                        // 2^64 / rounds, rounded up (not for 1)
    uint32_t by_rounds_32, by_q;               // 2^32 / rounds, 2^32 / q, rounded up
    uint32_t rounds, x;                        // n - 1 + q; rounds before the first one: i = j + x
    int step_k, step_add, row_k, row_add;      // what the CTA's threads' records, and a whole row, add to the entry k = i mod q and to q floor(i / q)
};

// The records of all ranks are one flat stream, and a CTA takes `records` of them wherever ranks begin and end.  The threads walk them, thread t at the
// records t - shift, t - shift + 128 (256), ...: `shift` (0..7) is chosen so that a warp's 32 x 16 bytes are four whole
// 128-byte lines of memory wherever the stretch starts (stores that cut lines or 32-byte sectors
// cost up to a fifth of the write bandwidth), and short rows (few rounds) fill the threads as
// well as long ones.  Rank, round, entry and phase of a thread's record are kept incrementally; where a CTA and a thread
// begin is found with multiplications (divisions took longer than the four records of a thread: 20 000 ranks, n = 300 14.9 us with them).
// kBuildRows: the caller gave no schedule tables, so the CTA computes the rows of its ranks as
// Algorithm 6 itself does: the receive entry of round k by running Algorithm 4 up to round k,
// the send entry as the receive entry of the to-processor (Algorithm 5) -- one (rank, round)
// pair per thread, the paper's own per-rank construction, no table and no scratch memory.
template <bool kBuildRows, int kThreads>
__global__ void __launch_bounds__(kThreads)
expand_kernel(const __grid_constant__ PTable tab, const __grid_constant__ Walk walk, uint32_t n, uint64_t r_begin, uint64_t total, uint32_t records,
              const int8_t *__restrict__ recv, const int8_t *__restrict__ send, int4 *__restrict__ table_out)
{
    // per rank of the CTA and per round k of a phase: {send entry - x, recv entry - x, to, from}.
    // Algorithm 6 adds q to an entry after each use and starts entries k < x at +q because
    // their first use is in the second phase; both are covered by adding q * floor(i / q).
    grid_launch_dependents();
    extern __shared__ int4 entries[];          // [ranks][q], then (kBuildRows) the skips: in front of the entries all took 4 % longer
    uint32_t *skips_sh = reinterpret_cast<uint32_t *>(entries + (kBuildRows ? (size_t)(records / walk.rounds) * tab.q : 0));
    if (kBuildRows) {
        if (threadIdx.x < kRow) skips_sh[threadIdx.x] = tab.s[threadIdx.x];
        __syncthreads();
    }
    const uint32_t q = (uint32_t)tab.q;
    const uint32_t p = tab.p;
    const uint32_t rounds = walk.rounds, x = walk.x;
    const uint64_t first = (uint64_t)blockIdx.x * records;           // the CTA's first record: round e0 of rank j0
    const uint32_t len = (uint32_t)(total - first < (uint64_t)records ? total - first : (uint64_t)records);
    uint64_t j0 = rounds > 1u ? __umul64hi(first, walk.by_rounds) : first;
    if ((int64_t)(first - j0 * rounds) < 0) --j0;                    // (one too many, at most)
    const uint32_t e0 = (uint32_t)(first - j0 * rounds);
    // rank of the record f rounds behind the start of j0 (f rounds < 2^32 where that is multiplied)
    auto rank_of = [&](uint32_t f) { return rounds >= records ? (f >= rounds ? 1u : 0u) : (rounds > 1u ? __umulhi(f, walk.by_rounds_32) : f); };
    auto phase_of = [&](uint32_t i) { return q > 1u ? __umulhi(i, walk.by_q) : i; };
    const uint32_t ranks = rank_of(e0 + len - 1u) + 1u;
    grid_dependency_wait();                    // (the rows may be the work of the kernel before this one)
    {
        const int8_t *srow = kBuildRows ? nullptr : send + j0 * q;   // the CTA's rows are contiguous
        const int8_t *rrow = kBuildRows ? nullptr : recv + j0 * q;
        for (uint32_t e = threadIdx.x; e < ranks * q; e += kThreads) {
            const uint32_t g = phase_of(e), k = e - g * q;
            const uint32_t r = (uint32_t)(r_begin + j0 + g);
            const uint32_t sk = tab.s[k];
            uint32_t to = r + sk;
            if (to >= p) to -= p;
            const uint32_t from = r >= sk ? r - sk : r + p - sk;
            int sent, received;
            if (kBuildRows) {
                received = (int8_t)recv_rounds(skips_sh, p, (int)q, r, (int)k, nullptr);
                sent = (int8_t)recv_rounds(skips_sh, p, (int)q, to, (int)k, nullptr);
            } else {
                sent = srow[e];
                received = rrow[e];
            }
            entries[e] = make_int4(sent - (int)x, received - (int)x, (int)to, (int)from);
        }
    }
    __syncthreads();
    int4 *out = table_out + first;
    const uint32_t shift = (uint32_t)((reinterpret_cast<uintptr_t>(table_out) >> 4) + first) & 7u;
    uint32_t e = threadIdx.x >= shift ? threadIdx.x - shift : threadIdx.x + kThreads - shift;
    if (e >= len) return;
    // record e is round j of the CTA's rank number gq / q; round j uses i = j + x: entry
    // k = i mod q of phase floor(i / q), whose block numbers are the entries plus add = q * floor(i / q)
    const uint32_t rank = rank_of(e0 + e);
    uint32_t j = e0 + e - rank * rounds, gq = rank * q;
    // (i is counted from the phase in which the CTA begins, so that it is small: the CTA's first rank may be any number of rounds in)
    const uint32_t phase0 = rank == 0u ? (e0 + x) / q : 0u;
    const uint32_t i = j + x - phase0 * q, phase = phase_of(i);
    int k = (int)(i - phase * q), add = (int)((phase0 + phase) * q);
    const int last = (int)n - 1;
    for (;;) {
        const int4 rec = entries[gq + (uint32_t)k];
        int sb = rec.x + add, rb = rec.y + add;
        sb = sb < 0 ? -1 : (sb > last ? last : sb);
        rb = rb < 0 ? -1 : (rb > last ? last : rb);
        __stcs(out + e, make_int4(sb, rb, rec.z, rec.w));
        e += kThreads;
        if (e >= len) break;
        j += kThreads;
        k += walk.step_k;
        add += walk.step_add;
        if (k >= (int)q) { k -= (int)q; add += (int)q; }
        while (j >= rounds) {                                        // on to the next rank: i falls by `rounds`
            j -= rounds;
            gq += q;
            k -= walk.row_k;
            add -= walk.row_add;
            if (k < 0) { k += (int)q; add -= (int)q; }
        }
    }
}

// ---------------------------------------------------------------- Algorithms 7 and 8: round tables
// One 16-byte record per (rank, round k), q records per rank.  Regular allgather (Algorithm 7):
// {to = r - skips[k], from = r + skips[k] (mod p), blocks exchanged skips[k+1] - skips[k],
// receive offset skips[k]}.  Census (Algorithm 8): when 2 skips[k] > skips[k+1] the edges are one
// shorter and only the partial sum S is sent: {to, from, 1 if x_r is added to what is sent, 0}.
__global__ void __launch_bounds__(256)
circulant_rounds_kernel(PTable tab, uint64_t r_begin, uint64_t n_records, int census,
                        int4 *__restrict__ out)
{
    const uint64_t e = (uint64_t)blockIdx.x * 256 + threadIdx.x;
    if (e >= n_records) return;
    const uint32_t q = (uint32_t)tab.q, p = tab.p;
    const uint64_t j = e / q;
    const uint32_t k = (uint32_t)(e - j * q);
    const uint32_t r = (uint32_t)(r_begin + j);
    const uint32_t lo = tab.s[k], hi = tab.s[k + 1];
    uint32_t step = lo;
    int c = (int)(hi - lo), d = (int)lo;
    if (census) {
        const bool shorter = 2ull * lo > hi;
        step = shorter ? lo - 1u : lo;
        c = shorter ? 0 : 1;
        d = 0;
    }
    const uint32_t to = r >= step ? r - step : r + p - step;
    uint32_t from = r + step;
    if (from >= p) from -= p;
    __stcs(out + e, make_int4((int)to, (int)from, c, d));
}

}  // namespace
}  // namespace bcs

using namespace bcs;

extern "C" {

bcs_status bcs_expand(uint32_t p, uint32_t n, uint64_t r_begin, uint64_t r_end,
                      const int8_t *recv, const int8_t *send, int32_t *table_out,
                      void *cuda_stream)
{
    bcs_status st = check_range(p, r_begin, r_end);
    if (st != BCS_OK) return st;
    if (n == 0) return BCS_ERR_ARG;
    if (n > 0x7fffff00u) return BCS_ERR_UNSUPPORTED;   // block numbers and n-1+q stay in int32
    PTable tab;
    make_table(p, &tab);
    const uint64_t count = r_end - r_begin;
    if (count == 0 || tab.q == 0) return BCS_OK;
    if (table_out == nullptr || (recv == nullptr) != (send == nullptr)) return BCS_ERR_ARG;
    if (!aligned16(table_out)) return BCS_ERR_ALIGN;
    const uint32_t q = (uint32_t)tab.q, rounds = n - 1u + q;
    const uint64_t total = count * rounds;
    const bool few = recv == nullptr || total < kExpandFew;
    uint32_t records = total < kExpandMany ? kExpandFewer : kExpandRecords;
    if (rounds <= kExpandFewer && total > kExpandFewer * kExpandSms) {
        for (uint32_t r = kExpandFewest; r < kExpandFewer && records == kExpandFewer; r += kExpandStep)
            if (total <= (uint64_t)r * kExpandAtOnce) records = r;
    }
    uint64_t ranks = (records + rounds - 2u) / rounds + 1u;          // that a CTA's records can belong to
    uint32_t extra = 0;
    if (recv == nullptr) {                                           // no tables: whole ranks, as far as their entries fit in shared memory
        const uint64_t share = total / kExpandCtas;
        const uint32_t aim = share > kExpandBuilt ? kExpandBuilt : (share < kExpandFewer ? kExpandFewer : (uint32_t)share);
        extra = kRow * 4u;                                           // room for the skips
        const uint32_t fit = (kExpandSharedBytes - extra) / (16u * q);
        ranks = (aim + rounds - 1u) / rounds;
        if (ranks > fit) ranks = fit;
        records = (uint32_t)ranks * rounds;
    }
    const uint64_t blocks = (total + records - 1u) / records;
    if (blocks > 0x7fffffffull) return BCS_ERR_UNSUPPORTED;
    const uint32_t threads = few ? kExpandThreadsFew : kExpandThreads;
    const Walk walk = {~0ull / rounds + 1u, 0xffffffffu / rounds + 1u, 0xffffffffu / q + 1u, rounds, (q - rounds % q) % q,
                       (int)(threads % q), (int)(threads / q * q), (int)(rounds % q), (int)(rounds / q * q)};
    const size_t shared = (size_t)ranks * q * 16u + extra;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    int4 *out = reinterpret_cast<int4 *>(table_out);
    if (recv == nullptr)                               // the kernel builds the rows it needs
        launch_dependent(true, expand_kernel<true, kExpandThreadsFew>, (unsigned)blocks, threads, shared, stream, tab, walk, n, r_begin, total, records, recv, send, out);
    else if (few)
        launch_dependent(true, expand_kernel<false, kExpandThreadsFew>, (unsigned)blocks, threads, shared, stream, tab, walk, n, r_begin, total, records, recv, send, out);
    else
        launch_dependent(true, expand_kernel<false, kExpandThreads>, (unsigned)blocks, threads, shared, stream, tab, walk, n, r_begin, total, records, recv, send, out);
    return launch_status();
}

bcs_status bcs_circulant_rounds(uint32_t p, uint64_t r_begin, uint64_t r_end, int census,
                                int32_t *table_out, void *cuda_stream)
{
    bcs_status st = check_range(p, r_begin, r_end);
    if (st != BCS_OK) return st;
    PTable tab;
    make_table(p, &tab);
    const uint64_t records = (r_end - r_begin) * (uint64_t)tab.q;
    if (records == 0) return BCS_OK;
    if (table_out == nullptr) return BCS_ERR_ARG;
    if (!aligned16(table_out)) return BCS_ERR_ALIGN;
    const uint64_t blocks = (records + 255) / 256;
    if (blocks > 0x7fffffffull) return BCS_ERR_UNSUPPORTED;
    circulant_rounds_kernel<<<(unsigned)blocks, 256, 0, static_cast<cudaStream_t>(cuda_stream)>>>(
        tab, r_begin, records, census != 0, reinterpret_cast<int4 *>(table_out));
    return launch_status();
}

}  // extern "C"
