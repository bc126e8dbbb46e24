// Index tables of the irregular allgather (arXiv 2205.10072, Algorithm 9 without the data
// movement): for one processor r, which block of buffer[j] is packed and which is unpacked in
// every round.  Processor r treats buffer j as virtual processor (r-j) mod p of a broadcast
// rooted at j, so entry [round][j] is the send resp. receive block of that virtual processor's
// round (Algorithm 6's closed form).  A pure store stream: 8 bytes per (round, buffer).
#include "bcs_common.cuh"

namespace bcs {
namespace {

constexpr int kAgThreads = 256;   // threads per CTA; a CTA writes 256 consecutive buffers of a row
constexpr int kAgLine = 32;       // int32 elements per 128-byte line
constexpr int kAgCols = kAgThreads + kAgLine;   // buffers staged per CTA: its window slides by up to 31 from row to row
// Rounds of a CTA.  Memory writes bound it, and as every stream of stores it is fastest with short CTAs, handed out in order; but a CTA copies the schedule
// rows of its 288 buffers first, 2 x 288 q bytes for 2048 bytes of output per round.
constexpr uint32_t kAgFewest = 4;               // while all CTAs run at once like that:
constexpr uint32_t kAgFitBoth = 148 * 6;
constexpr uint32_t kAgFitOne = 148 * 7;
constexpr uint32_t kAgOneTurn = 1000;           // CTAs that a call aims for while they have fewer than
constexpr uint32_t kAgMany = 1350;              // CTAs that are more than those that run at once,
constexpr uint32_t kAgMost = 1000;              // and that nearly fill the card: where the longer ones of the following leave so many
constexpr uint32_t kAgRounds = 32, kAgRoundsEven = 48;                         // both tables (even q: the copy takes longer)
constexpr uint32_t kAgRoundsOne = 48, kAgRoundsTwice = 96, kAgRoundsLong = 128;         // one table (the last: twice as many)

// A CTA's copy of a schedule table: rows of consecutive ranks as they lie there, that of rank number i (from the lowest of the CTA's on, going on at 0 behind
// p - 1) from byte at(i) on.  A thread reads one byte of each of four rows, its neighbours of the next four: the lanes are an odd number of words apart
// if q is odd, and with four bytes between any four rows if it is even (q = 16: 64 bytes apart, 16 lanes would meet in a bank).
template <bool kPad>
struct Staged {
    uint32_t first;                             // place of rank number 0: its byte, or (kPad) its number in the copy
    uint32_t q;
    __device__ __forceinline__ uint32_t at(uint32_t i) const
    {
        if (!kPad) return first + i * q;
        const uint32_t row = first + i;
        return row * q + (row & ~3u);
    }
};

__host__ __device__ constexpr uint32_t staged_bytes(uint32_t q) { return ((kAgCols + 4u) * q + (q % 2u ? 16u : kAgCols + 4u) + 31u) & ~15u; }

// Copies the rows of the n ranks lo, lo + 1, ... (mod p) of `table` ([p][q] int8, 16-byte aligned).  by_q: 2^32 / q, rounded up.  The caller synchronises.
template <bool kPad>
__device__ __forceinline__ Staged<kPad> stage_rows(uint8_t *copy, const int8_t *__restrict__ table, uint32_t p, uint32_t q, uint32_t by_q, uint32_t lo,
                                                   uint32_t n)
{
    const uint32_t whole = n <= p - lo ? n : p - lo;             // (the others are the ranks 0, 1, ...)
    Staged<kPad> st;
    st.q = q;
    if (!kPad) {
        const uint64_t byte = (uint64_t)lo * q;
        st.first = (uint32_t)(byte & 15u);
        load_span(copy, st.first, whole * q, table, byte);
        const uint32_t end = st.first + whole * q;
        for (uint32_t e = threadIdx.x; e < (n - whole) * q; e += kAgThreads) copy[end + e] = (uint8_t)table[e];
    } else {
        // four rows are q words; they begin on one where the rank is a multiple of four
        st.first = lo & 3u;
        const int8_t *from = table + (uint64_t)(lo - st.first) * q;
        const uint32_t bytes = (st.first + whole) * q;
        uint32_t *words = reinterpret_cast<uint32_t *>(copy);
        for (uint32_t w = threadIdx.x; w < bytes / 4u; w += kAgThreads)
            words[w + __umulhi(w, by_q)] = reinterpret_cast<const uint32_t *>(from)[w];
        if ((bytes & 2u) != 0u && threadIdx.x < 2u) {            // (the end of the table, maybe)
            const uint32_t w = bytes / 4u;
            copy[4u * (w + __umulhi(w, by_q)) + threadIdx.x] = (uint8_t)from[4u * w + threadIdx.x];
        }
        for (uint32_t e = threadIdx.x; e < (n - whole) * q; e += kAgThreads) {
            const uint32_t i = __umulhi(e, by_q);
            copy[st.at(whole + i) + e - i * q] = (uint8_t)table[e];
        }
    }
    return st;
}

// Block number of Algorithm 6's closed form: entry + q * floor(i / q) - x (= entry + add); below
// 0 -> -1 (nothing is packed or unpacked), above n-1 -> n-1.
__device__ __forceinline__ int clamp_block(int b, int last) { return max(min(b, last), -1); }

// A thread's share of one output table.  A row of the output is p * 4 bytes long and starts
// wherever the row before it ended, so the 128-byte lines of memory cut every row at different
// buffers.  Stores that do not cover whole lines (even whole 32-byte sectors) cost the memory
// system up to 40 % of its write bandwidth, so in every row the CTA with first buffer j0 writes
// the eight lines that begin at buffers j0 + hd .. j0 + hd + 255, hd in 0..31 being the distance
// from buffer j0 of this row to the next line boundary: a warp's 32 x 16 bytes are then four whole
// lines.  The hd buffers before the first line of a row and the up to three after the last whole
// group of four are written one by one, by the first CTA of the row and the one in whose window it ends.  Thread t takes the rows jr0 + t / 64, +4, +8, ...
// and in each of them the four buffers j0 + hd + 4 * (t % 64) .. +3.
template <bool kPad>
struct QuadStream {
    const uint8_t *copy;     // the rows; buffer j0 + c is rank number top - c
    Staged<kPad> rows;
    int32_t *row;            // &out[jr * p + j0]
    uint32_t phase;          // (element address of row[0]) mod 32
    __device__ __forceinline__ void init(const uint8_t *copy_, const Staged<kPad> &rows_, int32_t *out, uint64_t at)
    {
        copy = copy_;
        rows = rows_;
        row = out + at;
        phase = (uint32_t)(reinterpret_cast<uintptr_t>(row) >> 2) & (kAgLine - 1u);
    }
    __device__ __forceinline__ int entry(uint32_t number, uint32_t k) const
    {
        return (int)reinterpret_cast<const int8_t *>(copy)[rows.at(number) + k];
    }
    // edge: the first CTA of a row, or one in whose window it ends (`avail` buffers from j0 on)
    __device__ __forceinline__ void store(uint32_t slot, uint32_t k, int add, bool clamp, int last, uint32_t p, uint32_t avail, uint32_t top, bool head, bool edge)
    {
        const uint32_t hd = (0u - phase) & (kAgLine - 1u), c = hd + 4u * slot;
        if (c + 4u <= avail) {
            int4 v;
            v.x = entry(top - c, k) + add;
            v.y = entry(top - c - 1u, k) + add;
            v.z = entry(top - c - 2u, k) + add;
            v.w = entry(top - c - 3u, k) + add;
            if (clamp) {
                v.x = clamp_block(v.x, last);
                v.y = clamp_block(v.y, last);
                v.z = clamp_block(v.z, last);
                v.w = clamp_block(v.w, last);
            }
            __stcs(reinterpret_cast<int4 *>(row + c), v);
        }
        if (edge) {
            uint32_t col = 0xffffffffu;
            if (slot < (uint32_t)kAgLine) {
                if (head && slot < hd) col = slot;
            } else if (avail >= hd && avail - hd < (uint32_t)kAgThreads) {
                const uint32_t left = slot - kAgLine;
                if (left < ((avail - hd) & 3u)) col = hd + ((avail - hd) & ~3u) + left;
            }
            if (col < avail) row[col] = clamp_block(entry(top - col, k) + add, last);
        }
        row += 4ull * p;
        phase = (phase + 4u * p) & (kAgLine - 1u);
    }
};

// x: rounds before the first one; by_q: 2^32 / q, rounded up.
// kMany: with both tables eight CTAs per SM, in 32 registers a thread, instead of six; with one table (six are as fast) two rows at a time, which pays
// for long calls (even q, which has the more instructions: p = 150 000, n = 768 73.8 -> 72.2 us, 9000, 12 000 70.8 -> 69.3).  q >= 4.
template <bool kPack, bool kUnpack, bool kPad, bool kMany>
__global__ void __launch_bounds__(kAgThreads, kMany && kPack && kUnpack ? 8 : 6)
allgather_kernel(uint32_t p, uint32_t q, uint32_t by_q, uint32_t n, uint32_t x, uint32_t r, uint32_t rounds_per_cta, const int8_t *__restrict__ recv,
                 const int8_t *__restrict__ send, int32_t *__restrict__ pack_out, int32_t *__restrict__ unpack_out)
{
    extern __shared__ __align__(16) uint8_t copies[];
    uint8_t *send_copy = copies, *recv_copy = copies + (kPack ? staged_bytes(q) : 0u);
    grid_launch_dependents();
    const uint32_t rounds = n - 1u + q;
    const uint32_t j0 = blockIdx.x * kAgThreads;                   // first buffer of the CTA
    const uint32_t avail = p - j0;                                 // buffers from j0 to the end of a row
    const uint32_t cols = avail < (uint32_t)kAgCols ? avail : (uint32_t)kAgCols;   // buffers staged
    // buffer j0 + c: virtual rank (r - j0 - c) mod p; the lowest of them is that of the last buffer staged
    uint32_t lo = r + (p - j0);
    if (lo >= p) lo -= p;
    lo = lo >= cols - 1u ? lo - (cols - 1u) : lo + (p - (cols - 1u));
    grid_dependency_wait();                                        // (the rows may be the work of the kernel before this one)
    Staged<kPad> st = {};
    if (kPack) st = stage_rows<kPad>(send_copy, send, p, q, by_q, lo, cols);
    if (kUnpack) st = stage_rows<kPad>(recv_copy, recv, p, q, by_q, lo, cols);     // the same places for both tables
    const uint32_t jr0 = blockIdx.y * rounds_per_cta;
    const uint32_t jr1 = rounds - jr0 > rounds_per_cta ? jr0 + rounds_per_cta : rounds;
    const int last = (int)n - 1;
    uint32_t jr = jr0 + (threadIdx.x >> 6);
    const uint32_t slot = threadIdx.x & 63u, top = cols - 1u;
    const bool head = j0 == 0u, edge = head || avail < (uint32_t)kAgCols;
    const uint64_t at = (uint64_t)jr * p + j0;                     // element index of the CTA's first buffer in this row
    QuadStream<kPad> ps, us;
    if (kPack) ps.init(send_copy, st, pack_out, at);
    if (kUnpack) us.init(recv_copy, st, unpack_out, at);
    const uint32_t i0 = jr + x, phase = i0 / q;
    uint32_t k = i0 - phase * q;
    int add = (int)(phase * q) - (int)x;                           // q * floor(i / q) - x
    __syncthreads();
#pragma unroll(kMany && !(kPack && kUnpack) ? 2 : 1)
    for (; jr < jr1; jr += 4) {
        // entries are in [-q, q-1]: only rows of the first two and of the last phases can
        // leave 0..n-1 (the same test for all threads of a warp)
        const bool clamp = add < (int)q || add + (int)q - 1 > last;
        if (kPack) ps.store(slot, k, add, clamp, last, p, avail, top, head, edge);
        if (kUnpack) us.store(slot, k, add, clamp, last, p, avail, top, head, edge);
        k += 4u;
        while (k >= q) {                                           // (once at most; written as an `if` both tables took 5 to 7 % longer)
            k -= q;
            add += (int)q;
        }
    }
}

// Up to eight buffers (q < 4): a row per thread.  (By the kernel above, five buffers and 50 000 rounds took 14.2 us.)
__global__ void __launch_bounds__(kAgThreads)
allgather_few_kernel(uint32_t p, uint32_t q, uint32_t n, uint32_t x, uint32_t r, const int8_t *__restrict__ recv, const int8_t *__restrict__ send,
                     int32_t *__restrict__ pack_out, int32_t *__restrict__ unpack_out)
{
    grid_launch_dependents();
    const uint32_t rounds = n - 1u + q, jr = blockIdx.x * kAgThreads + threadIdx.x;
    grid_dependency_wait();                                        // (the rows may be the work of the kernel before this one)
    if (jr >= rounds) return;
    const uint32_t phase = (jr + x) / q, k = jr + x - phase * q;
    const int add = (int)(phase * q) - (int)x;
    for (uint32_t j = 0; j < p; ++j) {
        const uint32_t entry = (r >= j ? r - j : r + p - j) * q + k;
        const uint64_t at = (uint64_t)jr * p + j;
        if (pack_out != nullptr) pack_out[at] = clamp_block((int)send[entry] + add, (int)n - 1);
        if (unpack_out != nullptr) unpack_out[at] = clamp_block((int)recv[entry] + add, (int)n - 1);
    }
}

template <bool kPack, bool kUnpack, bool kPad, bool kMany>
void launch_tables(dim3 grid, uint32_t p, uint32_t q, uint32_t n, uint32_t r, uint32_t per_cta, const int8_t *recv, const int8_t *send, int32_t *pack_out,
                   int32_t *unpack_out, cudaStream_t stream)
{
    const uint32_t by_q = 0xffffffffu / q + 1u, x = (q - (n - 1u + q) % q) % q;
    const size_t shared = (size_t)staged_bytes(q) * ((kPack ? 1u : 0u) + (kUnpack ? 1u : 0u));
    launch_dependent(true, allgather_kernel<kPack, kUnpack, kPad, kMany>, grid, kAgThreads, shared, stream, p, q, by_q, n, x, r, per_cta, recv, send, pack_out,
                     unpack_out);
}

template <bool kPack, bool kUnpack, class... Args>
void launch_allgather(bool many, uint32_t q, Args... args)
{
    if (q % 2u) return many ? launch_tables<kPack, kUnpack, false, true>(args...) : launch_tables<kPack, kUnpack, false, false>(args...);
    return many ? launch_tables<kPack, kUnpack, true, true>(args...) : launch_tables<kPack, kUnpack, true, false>(args...);
}

}  // namespace
}  // namespace bcs

using namespace bcs;

extern "C" {

bcs_status bcs_allgather_tables(uint32_t p, uint32_t n, uint32_t r, const int8_t *recv,
                                const int8_t *send, int32_t *pack_out, int32_t *unpack_out,
                                void *cuda_stream)
{
    PTable tab;
    bcs_status st = make_table(p, &tab);
    if (st != BCS_OK) return st;
    if (r >= p) return BCS_ERR_RANGE;
    if (n == 0) return BCS_ERR_ARG;
    if (n > 0x7fffff00u) return BCS_ERR_UNSUPPORTED;
    if (tab.q == 0) return BCS_OK;
    if (recv == nullptr || send == nullptr || (pack_out == nullptr && unpack_out == nullptr))
        return BCS_ERR_ARG;
    if ((reinterpret_cast<uintptr_t>(pack_out) & 3u) || (reinterpret_cast<uintptr_t>(unpack_out) & 3u) ||
        !aligned16(recv) || !aligned16(send))
        return BCS_ERR_ALIGN;
    // Four rounds per CTA while all of them run at once; then some thousand CTAs; from 30 000 pairs of 256 buffers and a round on (both tables) CTAs of 32
    // or 48 rounds, eight per SM.  us, six per SM and about 1000 CTAs / eight per SM and 32 rounds / 48 rounds (with the rows copied and
    // transposed: some 80 rounds): p = 20 262, n = 116 (10 000 pairs) 7.6/8.3/8.3 (13.0), 20 000, 300 (25 000) 11.6/12.8/12.7 (16.6), 3000, 3000 (36 000)
    // 18.4/15.7/18.4 (24.7), 5000, 5000 (100 000) 35.8/32.3/34.3 (42.2), 100 003, 1000 (397 000) 120/114.8/119 (130); even q: 50 000, 300 (62 000)
    // 23.3/22.0/21.3 (28.8), 150 000, 400 (244 000) 79.9/79.5/74.3 (82.2); but where 48 rounds leave less than kAgMost CTAs, 9000, 1000
    // (792) -/15.0/20.4 (24.7).  One table, six per SM, 48 / 96 / 128 rounds (the rows
    // transposed): 12 000, 1500 (71 000 pairs) 14.3/16.1/20.6 (15.0), 9000, 3000 (108 000) 20.9/21.3/22.1 (22.1), 12 000, 3000 26.4/24.9/26.2 (25.6), 35 000, 1000
    // 25.8/24.7/25.4 (27.1), 9000, 12 000 (432 000) 74.3/69.3/68.2 (66.7), 150 000, 768 79.7/72.2/71.0 (70.5), 262 144, 300 56.9/51.9/50.6 (52.3).
    // Chunks are about equally long with one table, and with both where they all run at once: 150 000, 40, 57 rounds as 48 and 9 20.2, as 32 and 25 14.6 (18.9).
    const uint32_t rounds = n - 1u + (uint32_t)tab.q;
    const uint32_t col_blocks = (p + kAgThreads - 1) / kAgThreads;
    const uint32_t q = (uint32_t)tab.q, tables = pack_out && unpack_out ? 2u : 1u;
    const uint64_t pairs = (uint64_t)col_blocks * rounds;
    const bool many = pairs * tables >= 2u * 30000u;
    uint32_t per_cta = kAgFewest;
    if (many) {
        auto leaves = [&](uint32_t per, uint32_t ctas) { return (uint64_t)col_blocks * ((rounds + per - 1) / per) >= ctas; };
        if (tables == 2u) per_cta = q % 2u == 0u && leaves(kAgRoundsEven, kAgMost) ? kAgRoundsEven : kAgRounds;
        else per_cta = leaves(kAgRoundsLong, 2u * kAgMany) ? kAgRoundsLong : (leaves(kAgRoundsTwice, kAgMany) ? kAgRoundsTwice : kAgRoundsOne);
        const uint32_t chunks = (rounds + per_cta - 1) / per_cta;
        if (tables == 1u || !leaves(per_cta, kAgMany)) per_cta = ((rounds + chunks - 1) / chunks + 3u) & ~3u;
    } else if ((uint64_t)col_blocks * ((rounds + kAgFewest - 1) / kAgFewest) > (tables == 2u ? kAgFitBoth : kAgFitOne)) {
        per_cta = ((uint32_t)pairs / kAgOneTurn + 4u) & ~3u;
    }
    while ((rounds + per_cta - 1) / per_cta > 65535u) per_cta *= 2u;         // (as many as a grid has in y)
    const dim3 grid(col_blocks, (rounds + per_cta - 1) / per_cta);
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    if (q < 4u)
        launch_dependent(true, allgather_few_kernel, (rounds + kAgThreads - 1) / kAgThreads, kAgThreads, 0, stream, p, q, n, (q - rounds % q) % q, r, recv, send,
                         pack_out, unpack_out);
    else if (pack_out && unpack_out)
        launch_allgather<true, true>(many, q, grid, p, q, n, r, per_cta, recv, send, pack_out, unpack_out, stream);
    else if (pack_out)
        launch_allgather<true, false>(many, q, grid, p, q, n, r, per_cta, recv, send, pack_out, unpack_out, stream);
    else
        launch_allgather<false, true>(many, q, grid, p, q, n, r, per_cta, recv, send, pack_out, unpack_out, stream);
    return launch_status();
}

}  // extern "C"
