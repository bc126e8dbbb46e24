// Schedule rows straight from the binary form of a rank (arXiv 2205.10072, Algorithms 1-5 and the
// lookup of Algorithm 9): no table of all ranks, no scratch memory, every stretch of ranks on its own.
//
// Notation: e_t = 2 skips[t-1] - skips[t], which Algorithm 1 makes 0 or 1; C(a, b) = e_{a+1} + ... + e_b.
// The skip code of a rank (bcs_common.cuh) has bit k set iff skips[k] is a term of its greedy sum.
//
// Segments.  Cut the ranks at every rank whose code has no bit below L = min(7, q).  Because
// skips[k] = ceil(p / 2^(q-k)), the part of the codes from bit L up counts these segments in plain
// binary: segment g (0 <= g < 2^(q-L)) starts at the sum of the skips[L+k] over the bits k of g.  Let m be
// the lowest zero bit of g, as a level (L + its position, q if there is none): the segment has
// skips[L] - C(L, m) ranks (65..128 for q > 7, less at most 24).
//
// Rounds from L up.  The window of round i of rank r ends skips[i] ranks below r, so with `low` the part
// of r below its segment's start, and K the lowest set bit of g as a level (K = q: no bit, the root's segment):
//   * bit i of the code set: the window holds the rank with the bits above i only, whose baseblock,
//     the next higher set bit of r, is the largest of the window.  No higher set bit: i is
//     the home round, the entry is the baseblock of r.
//   * bit i not set: the window lies below that rank, and the largest new block in it is i.
// So in these rounds all ranks of a segment have the same entries, and the blocks 0..i-1 and the next set
// bit are the ones taken before round i.  The exceptions are ranks close behind a segment's start (low
// <= C(L, K) <= 24), in the rounds L..K-1: as long as low < C(i+1, K) the window of round i reaches the rank
// with baseblock i+1, and the entry is i+1; the first round after that takes the one block of
// 0..i that is missing by then, and the rounds behind it are as above.
// A send entry is the receive entry of the rank skips[k] further on.  Bit k set: adding skips[k]
// carries, the bit is clear there, the entry is k.  Not set: the bit is set there, the entry is the next
// higher set bit of r (none: the baseblock of r; the root sends block k).  Exceptions: the last C(k, m) ranks
// before a segment whose lowest bit is k (m the lowest zero bit above k): they carry into a rank
// close behind a segment's start.
//
// Rounds below L.  The entries of a rank depend on (K, low) only, low < skips[L] <= 128: a table of at most
// 25 x 128 rows of 8 bytes in the CTA's shared memory.  What lies d ranks below the rank skips[K] is what lies
// d + C(7, K) ranks below skips[7], so there are few shapes of such rows in all: they are kept as constants.
//
// All of this is checked entry by entry against the CPU oracle by the tests.
#pragma once
#include "bcs_common.cuh"

namespace bcs {

constexpr unsigned kSms = 148;
constexpr int kLow = 7;                       // rounds whose entries come from the table
constexpr int kLowRanks = 128;                // skips[7] <= 128
constexpr int kMissRanks = 32;                // ranks behind a segment's start that can be exceptions (<= 25)
constexpr uint32_t kRootMark = 0x7f;          // in place of the root's baseblock in the table
constexpr uint32_t kItemRanks = 128;          // ranks that a warp takes at a time
constexpr uint32_t kHalo = 64;                // and the ranks behind them that their send rows look at (skips[6] <= 64)
constexpr int kItemSegments = 5;              // segments that an item can touch: all but the two at its ends lie
                                              // inside it, a run of c segments has more than 64 c - 25 ranks

// What a p is to the kernels.
struct RowConsts {
    uint32_t s[kRow + kLow + 1];   // skips[0..q], then 0
    uint32_t p;
    int q;
    uint32_t odd;                  // bit t: e_t
    uint32_t inv;                  // floor(2^(q - L + 32) / p)
};

__host__ __device__ constexpr int low_levels(int q) { return q < kLow ? q : kLow; }

// Number of e_t set, a < t <= b.
__device__ __forceinline__ uint32_t count_odd(uint32_t odd, int a, int b)
{
    return (uint32_t)__popc((odd >> (a + 1)) & ((1u << (b - a)) - 1u));
}

// ---------------------------------------------------------------- shared memory of a CTA
// A warp's part: table rows of the item's ranks and of those behind it, a word about each of its ranks, entries of
// its segments from round L up (receive and send, 32 bytes each), its segments, the staged rows.
constexpr uint32_t kWarpNotes = (kItemRanks + kHalo) * 8u;
constexpr uint32_t kWarpEntries = kWarpNotes + kItemRanks * 2u;
constexpr uint32_t kWarpSegments = kWarpEntries + kItemSegments * 64u;
constexpr uint32_t kWarpStage = kWarpSegments + 48u;
static_assert(kItemSegments * 8u <= 48u && kWarpStage % 16u == 0, "layout of a warp's shared memory");

// Byte offsets in the CTA's dynamic shared memory.
struct RowLayout {
    uint32_t miss = 0, s = 0, flags = 0, warps = 0, warp_bytes = 0;
    __host__ __device__ constexpr explicit RowLayout(int q)
    {
        const uint32_t rows = (uint32_t)(q - low_levels(q) + 1);
        miss = rows * kLowRanks * 8u;
        s = miss + rows * kMissRanks;
        flags = s + (kRow + kLow + 1) * 4u;
        warps = flags + 16u + 32u;
        warps = (warps + 127u) & ~127u;
        warp_bytes = kWarpStage + ((kItemRanks * (uint32_t)q + 31u) & ~15u);
    }
    __host__ __device__ constexpr uint32_t total(uint32_t n_warps) const { return warps + n_warps * warp_bytes; }
};

struct RowTable {
    uint2 *rows;          // [K - L][low]: entries of rounds 0..6 as bytes 0..6, baseblock as byte 7
    uint8_t *miss;        // [K - L][low < 32]: the block of 0..7 that is not taken before round 7
    uint32_t *s;
    uint32_t *wanted;     // bit K - L: the rows of K are wanted
    uint8_t *list;        // the wanted K
    __device__ RowTable(uint8_t *sm, const RowLayout &at)
        : rows(reinterpret_cast<uint2 *>(sm)), miss(sm + at.miss), s(reinterpret_cast<uint32_t *>(sm + at.s)),
          wanted(reinterpret_cast<uint32_t *>(sm + at.flags)), list(sm + at.flags + 16)
    {
    }
};

// The rows of all shapes of segments (gen/row_table.c writes them at build time and says how they are packed): 1.7 MB, of which a
// CTA reads 512 bytes for each K that it wants, and the same 512 bytes of row_six each time.
#include "row_table.inc"

// Place of row `low` in a table whose readers are four rows apart: 16 lanes meet in no bank.
__device__ __forceinline__ uint32_t permuted_row(uint32_t low) { return low ^ ((low >> 4) & 3u); }

// A packed row: entries are block - q, K for 8, blocks of 16 and more the rank's own.
__device__ __forceinline__ uint2 unpack_row(unsigned long long v, int q, int K)
{
    auto word = [&](uint32_t x, uint32_t ones) {
        x += ((x >> 3) & 0x01010101u) * (uint32_t)(K - 8) + ((x >> 4) & 0x01010101u) * (uint32_t)(q - 16);
        return ((x | 0x80808080u) - (uint32_t)q * ones) ^ 0x80808080u;          // (no byte borrows)
    };
    return make_uint2(word((uint32_t)v, 0x01010101u), word((uint32_t)(v >> 32) & 0x1fffffffu, 0x00010101u));
}

// Fills the table of a p, for the K whose bits in *t.wanted are set (q > 7); all threads of the CTA call, after a barrier behind the
// writes of t.s (the skips, then zeros) and *t.wanted.  Ends with a barrier.
// (Two loads and some twenty instructions for two rows.  Computed by Algorithm 4 in every CTA it took 5000 cycles before the first row:
// 65 553 ranks 4.2 -> 3.5 us, all ranks of 100 003 5.5 -> 4.8, of about 2^20 15.6 -> 13.6, every p up to 1024 in any order 18.3 -> 16.7, back
// to back; a call alone 2 us less.)
// kJobs: loads in flight per thread.  Their latency is most of the time of a table that a kernel begins with (four: all ranks of 100 003 2.6 -> 2.4 us); the kernels
// for lists, which build one table beside the rows of another or spill, take longer with so many (one p of 200 2.8 -> 3.0 us with four and not one, of 2000 6.45 -> 6.7 with
// four and not two, receive rows of 8 of 2^20 45.6 -> 48.4; 40 of 2^10..2^20 with one, two, four 68.6, 67.1, 67.3).
template <bool kPermuted = false, int kJobs = 4>
__device__ __forceinline__ void build_row_table(const RowTable &t, int q, uint32_t odd)
{
    auto place = [](uint32_t low) { return kPermuted ? permuted_row(low) : low; };
    const int L = low_levels(q);
    const uint32_t lows = t.s[L];
    if (q < kLow) {                                              // one segment, all rounds in the table
        for (uint32_t low = threadIdx.x; low < lows; low += blockDim.x) {
            uint2 row = unpack_row(__ldg(row_small + lows * (lows - 1u) / 2u + low), q, 0x7f);
            row.y &= 0xff000000u | (q > 4 ? (1u << (8 * (q - 4))) - 1u : 0u);
            t.rows[place(low)] = row;                            // (the root's baseblock is 8 in the constants: 0x7f)
        }
        __syncthreads();
        return;
    }
    const uint32_t wanted = q > kLow ? *t.wanted : 1u;
    if (threadIdx.x < 32u && ((wanted >> threadIdx.x) & 1u))     // list of the K
        t.list[__popc(wanted & ((1u << threadIdx.x) - 1u))] = (uint8_t)(L + threadIdx.x);
    __syncthreads();
    const uint32_t six = t.s[6];
    const unsigned long long *shapes = row_shapes + (lows - 65u) * (52u * 64u), *sixes = row_six + (lows - 65u) * 64u;
    const int n = __popc(wanted) * 64;
    for (int job0 = (int)threadIdx.x; job0 < n; job0 += kJobs * (int)blockDim.x) {
        unsigned long long v[kJobs], w[kJobs];
#pragma unroll
        for (int j = 0; j < kJobs; ++j) {
            const int job = job0 + j * (int)blockDim.x;
            v[j] = w[j] = 0;
            if (job < n) {
                const int K = t.list[job >> 6];
                const uint32_t low = (uint32_t)job & 63u, shape = (K == q ? 26u : 0u) + (K == kLow ? 0u : 1u + count_odd(odd, kLow, K));
                v[j] = __ldg(shapes + shape * 64u + low);
                w[j] = __ldg(sixes + low);
            }
        }
#pragma unroll
        for (int j = 0; j < kJobs; ++j) {
            const int job = job0 + j * (int)blockDim.x;
            if (job >= n) break;
            const int K = t.list[job >> 6];
            const uint32_t low = (uint32_t)job & 63u;
            uint2 *rows = t.rows + (K - kLow) * kLowRanks;
            if (low < six) {
                uint2 row = unpack_row(v[j], q, K);
                if (K == q && low == 0u) row.y |= kRootMark << 24;
                rows[place(low)] = row;
                if (low < (uint32_t)kMissRanks) t.miss[(K - kLow) * kMissRanks + (int)low] = (uint8_t)(v[j] >> 61);
            }
            // ranks with bit 6: the rounds before that do not depend on K, round 6 receives the next higher bit
            const uint32_t at = low + six;
            uint2 row = make_uint2(0u, 0u);                      // (read, but not used, behind the last one)
            if (at < lows) {
                row = unpack_row(w[j], q, K);
                row.y = (row.y & 0xff00ffffu) | (uint32_t)(uint8_t)(K < q ? K - q : (int)(row.y >> 24)) << 16;
            }
            if (at < kLowRanks) rows[place(at)] = row;
        }
    }
    __syncthreads();
}

// Bits K - L of the rows that the ranks x0 .. x0+n-1 (mod p; x0 < p, n <= 1000) need: those of their segments, and where
// the send exceptions of these carry to; by one warp, q > 7.
__device__ __forceinline__ uint32_t wanted_rows(int q, uint32_t inv, uint32_t x0, uint32_t n)
{
    const uint32_t lane = threadIdx.x & 31u;
    const int high = q - kLow;
    uint32_t from = __umulhi(x0, inv);                           // one before or behind, at most
    from = from ? from - 1u : 0u;
    uint32_t bits = 0;
    if (lane <= n / 40u + 4u) {                                  // (a segment has more than 40 ranks)
        const uint32_t g = (from + lane) & ((1u << high) - 1u);
        const int z = __ffs(~g) - 1;                             // lowest zero bit, and the next one
        bits = (g ? g & (0u - g) : 1u << high) | 1u << z;
        if (z < high) bits |= 1u << (z + __ffs(~(g >> (z + 1))));
    }
    return __reduce_or_sync(0xffffffffu, bits);
}

// The same for any n < 2^31, into *t.wanted; by the whole CTA.  Starts and ends with a barrier.
__device__ __forceinline__ void want_rows(const RowTable &t, int q, uint32_t inv, uint32_t x0, uint32_t n)
{
    const int high = q - kLow;
    __syncthreads();
    if (threadIdx.x == 0) *t.wanted = 0u;
    // (where a segment has 128 ranks, the first row of the group behind its own is looked at, if not used)
    if ((int)threadIdx.x <= high) t.rows[threadIdx.x * kLowRanks] = make_uint2(0u, 0u);
    __syncthreads();
    uint32_t from = __umulhi(x0, inv);                           // one before or behind, at most
    from = from ? from - 1u : 0u;
    const uint32_t count = __umulhi(n, inv) + 7u;                // (from is up to two before; the ends lie up to n inv / 2^32 + 3 segments apart)
    uint32_t bits = 0;
    for (uint32_t j = threadIdx.x; j < count; j += blockDim.x) {
        const uint32_t g = (from + j) & ((1u << high) - 1u);
        const int z = __ffs(~g) - 1;                             // lowest zero bit, and the next one
        bits |= (g ? g & (0u - g) : 1u << high) | 1u << z;
        if (z < high) bits |= 1u << (z + __ffs(~(g >> (z + 1))));
    }
    bits = __reduce_or_sync(0xffffffffu, bits);
    if ((threadIdx.x & 31u) == 0u && bits != 0u) atomicOr(t.wanted, bits);
    __syncthreads();
}

// ---------------------------------------------------------------- rows of an item, by one warp
// How a lane's rows of q bytes lie in the words of the staging buffer, where the rows of a warp follow one another.
// (The same for every 32 ranks of an item: 32 rows are whole words.)
struct RowPlace {
    uint32_t sh;       // bits by which the row is off a word
    bool longer;       // it ends in or behind word ceil(q / 4), counted from the word it begins in
    uint32_t shared;   // all ones if the next row begins in this row's last word
    __device__ RowPlace(uint32_t first_byte, int q)
    {
        const uint32_t mis = (first_byte + (threadIdx.x & 31u) * (uint32_t)q) & 3u;
        sh = 8u * mis;
        longer = mis + (uint32_t)q >= 4u * (((uint32_t)q + 3u) / 4u);
        shared = ((mis + (uint32_t)q) & 3u) != 0u ? 0xffffffffu : 0u;
    }
};

// Stores the rows (words W, zero beyond byte q) of 32 ranks at once, this lane's at `at`.  A word that two rows share is
// stored by the lane it ends in.  kAligned: the first row begins on a word.  Else the last lane stores what it has of a shared word,
// too, and the first lane of the next 32 ranks (`more`) completes that.  Lanes without a rank store too (the buffer has room for
// them, and nobody reads it).
// (With the words at either end written byte by byte every p up to 1024 took 16.5 us and not 13.8, 1024 p up to 2^20 1257 and not 1250.)
template <int kWords, bool kAligned>
__device__ __forceinline__ void stage_row(uint8_t *at, const uint32_t (&W)[kWords], int q, const RowPlace &pl, bool more)
{
    if (kWords == 1 && q < 4) {
        for (int k = 0; k < q; ++k) at[k] = (uint8_t)(W[0] >> (8 * k));
        return;
    }
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t V[kWords + 1];
#pragma unroll
    for (int w = 0; w <= kWords; ++w) V[w] = __funnelshift_l(w ? W[w - 1] : 0u, w < kWords ? W[w] : 0u, pl.sh);
    uint32_t *words = reinterpret_cast<uint32_t *>(at - (pl.sh >> 3));
    const uint32_t rest = (pl.longer ? V[kWords] : V[kWords - 1]) & pl.shared;
    const uint32_t before = __shfl_sync(0xffffffffu, rest, (lane - 1u) & 31u);
    V[0] |= kAligned || lane != 0u ? before : (more && pl.sh ? words[0] : 0u);       // (aligned: lane 31 shares no word)
#pragma unroll
    for (int w = 0; w < kWords - 1; ++w) words[w] = V[w];
    if (pl.longer) words[kWords - 1] = V[kWords - 1];
    if (!kAligned && lane == 31u && pl.shared) words[pl.longer ? kWords : kWords - 1] = rest;
}

// Row of a rank: its rounds below L from the table, the others from its segment.
template <int kWords>
__device__ __forceinline__ void join_row(uint32_t lo, uint32_t hi, const uint8_t *entries, uint32_t (&W)[kWords])
{
    W[0] = lo;
    if (kWords > 1) {
        const uint4 a = *reinterpret_cast<const uint4 *>(entries);
        W[1 % kWords] = a.y | (hi & 0xffffffu);
        if (kWords > 2) W[2 % kWords] = a.z;
        if (kWords > 3) W[3 % kWords] = a.w;
    }
    if (kWords > 4) {
        const uint4 b = *reinterpret_cast<const uint4 *>(entries + 16);
        W[4 % kWords] = b.x;
        if (kWords > 5) W[5 % kWords] = b.y;
        if (kWords > 6) W[6 % kWords] = b.z;
        if (kWords > 7) W[7 % kWords] = b.w;
    }
}

// The lane that starts a warp's bulk copies and waits for them.  (An elected one is known to be one to the compiler, 32 ranks 1.73 -> 1.69 us; where rows begin at
// any byte the same cost more than lane 0: one p of 200 2.8 -> 2.9 us.)
template <bool kAligned>
__device__ __forceinline__ bool copying_lane()
{
    return kAligned ? elect_one() : (threadIdx.x & 31u) == 0u;
}

// Sends the staged rows out: len bytes for `dst`, staged at the same offset in their 16-byte group.  All but
// the ragged ends go as one bulk copy of the TMA unit.
template <bool kAligned>
__device__ __forceinline__ void flush_item(uint8_t *stage, int8_t *dst, uint32_t len)
{
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t shift = kAligned ? 0u : (uint32_t)(reinterpret_cast<uintptr_t>(dst) & 15u);
    fence_before_bulk();
    grid_dependency_wait();                                      // (the kernel before: not until the first store)
    __syncwarp();
    const uint32_t begin = (shift + 15u) & ~15u, end = shift + len;
    uint8_t *base = reinterpret_cast<uint8_t *>(dst) - shift;
    const uint32_t stop = end & ~15u;
    if (copying_lane<kAligned>() && stop > begin) bulk_store(base + begin, stage + begin, stop - begin);
    if (!kAligned || (end & 15u) != 0u) {                        // bytes [shift, head) and [tail, end) one by one
        const uint32_t head = begin < end ? begin : end;
        if (shift + lane < head) base[shift + lane] = stage[shift + lane];
        const uint32_t tail = stop > begin ? stop : head;
        if (tail + lane < end) base[tail + lane] = stage[tail + lane];
    }
}

// The staging buffer may be written again.  (kAligned: as for the copies.)
template <bool kAligned>
__device__ __forceinline__ void stage_free()
{
    if (copying_lane<kAligned>()) bulk_stores_read();
    __syncwarp();
}

// What the lookup leaves about a rank of the item.
constexpr uint32_t kNoteFrom = 3;        // bits 0..2: its segment, counted from the item's first; 3..7: home round + 1, or L
constexpr uint32_t kNoteRecv = 1u << 8;  // some of its receive entries from round L up are exceptions
constexpr uint32_t kNoteSend = 1u << 9;  // one of its send entries is

// Receive and send rows (either pointer may be null) of the n <= 128 ranks x0, x0+1, ... (mod p; x0 < p, n <= p) by
// one warp.  recv, send: where the row of x0 goes (kAligned: 16-byte aligned).  mine: the warp's shared memory.
template <int kWords, bool kAligned>
__device__ __forceinline__ void warp_rows(const RowTable &t, uint8_t *mine, int q, uint32_t odd, uint32_t inv,
                                          uint32_t x0, uint32_t n, int8_t *recv, int8_t *send)
{
    const uint32_t lane = threadIdx.x & 31u;
    const int L = low_levels(q), high = q - L;
    uint2 *looked = reinterpret_cast<uint2 *>(mine);
    uint16_t *notes = reinterpret_cast<uint16_t *>(mine + kWarpNotes);
    uint8_t *entries = mine + kWarpEntries;
    uint2 *segments = reinterpret_cast<uint2 *>(mine + kWarpSegments);   // start, number
    uint8_t *stage = mine + kWarpStage;
    const uint32_t end = x0 + n;

    // Lane j < 8: segment number gs + j, gs one or two before that of x0 (or the first).  Positions go on
    // counting behind p - 1: the root's segment again.
    uint32_t gs = __umulhi(x0, inv);
    gs = gs ? gs - 1u : 0u;
    const uint32_t at0 =
        __reduce_add_sync(0xffffffffu, (int)lane < high && ((gs >> lane) & 1u) ? t.s[lane + L] : 0u);
    const uint32_t g = (gs + lane) & ((1u << high) - 1u);
    const int tz = __ffs(~g) - 1;                                // L + tz: lowest zero bit, as a level
    const uint32_t len = t.s[L] - count_odd(odd, L, L + tz);
    uint32_t pos = len;
#pragma unroll
    for (uint32_t d = 1; d < 8; d *= 2) {
        const uint32_t up = __shfl_up_sync(0xffffffffu, pos, d);
        if (lane >= d) pos += up;
    }
    pos += at0 - len;
    const int first = __popc(__ballot_sync(0xffffffffu, lane < 8u && pos <= x0)) - 1;
    uint32_t info;
    {
        const int K = g ? __ffs(g) - 1 + L : q;                  // lowest and highest set bit
        const int home = g ? 31 - __clz(g) + L : 0;
        const uint32_t behind = K > L ? count_odd(odd, L, K) + 1u : 0u;       // exceptions at its start
        // and at its end: the next segment's lowest bit is L + tz, the next zero bit of g is m
        const int m = L + tz + __ffs(~(g >> (tz + 1)));
        const uint32_t before = tz < high ? count_odd(odd, L + tz, m) : 0u;
        info = (uint32_t)(K - L) * kLowRanks | (uint32_t)(home ? home + 1 : L) << 12 | behind << 17 | before << 22 |
               (g & 1u) << 27;
        const uint32_t slot = lane - (uint32_t)first;
        if (slot < (uint32_t)kItemSegments) segments[slot] = make_uint2(pos, g);
    }

    // Entries of the segments' rounds from L up, lane = round.
    for (int j = first;; ++j) {
        const uint32_t gj = __shfl_sync(0xffffffffu, g, j);
        const int k = (int)lane;
        const uint32_t bits = k >= L ? gj >> (k - L) : 0u;
        const uint32_t above = bits >> 1;
        const int next = above ? __ffs(above) + k - q : 0;       // 0 where the baseblock goes
        const bool inside = k >= L && k < q;
        uint8_t *e = entries + (j - first) * 64 + k;
        e[0] = (uint8_t)(inside ? ((bits & 1u) ? next : k - q) : 0);
        e[32] = (uint8_t)(inside ? ((bits & 1u) ? k - q : next) : 0);
        if (__shfl_sync(0xffffffffu, pos, j + 1) >= end) break;
    }

    // Table rows of the ranks and of those that their send rows look at.
    {
        const uint32_t total = send != nullptr ? n + t.s[L - 1] : n;
        int j = first;
        uint32_t after = __shfl_sync(0xffffffffu, pos, j + 1);
        for (uint32_t b = 0; b < total; b += 32u) {
            const uint32_t x = x0 + b + lane;
            const uint32_t stop = x0 + (b + 32u < total ? b + 32u : total);
            uint32_t start = __shfl_sync(0xffffffffu, pos, j);
            uint32_t inf = __shfl_sync(0xffffffffu, info, j);
            uint32_t over = after;
            int slot = j - first;
            while (after < stop) {                               // segments that start among these ranks
                ++j;
                const uint32_t begins = after, inf_j = __shfl_sync(0xffffffffu, info, j);
                after = __shfl_sync(0xffffffffu, pos, j + 1);
                if (x >= begins) {
                    start = begins;
                    inf = inf_j;
                    over = after;
                    slot = j - first;
                }
            }
            if (x < stop) looked[b + lane] = t.rows[(inf & 0xfffu) + (x - start)];
            if (b < n) {
                const uint32_t low = x - start;
                uint32_t note = (uint32_t)slot | ((inf >> 12) & 31u) << kNoteFrom;
                if (low < ((inf >> 17) & 31u)) note |= kNoteRecv;
                if (over - x <= ((inf >> 22) & 31u) || (low == 0u && (inf >> 27) != 0u)) note |= kNoteSend;
                notes[b + lane] = (uint16_t)(x < end ? note : (uint32_t)L << kNoteFrom);
            }
        }
    }
    __syncwarp();

    if (recv != nullptr) {
        const uint32_t shift = kAligned ? 0u : (uint32_t)(reinterpret_cast<uintptr_t>(recv) & 15u);
        const RowPlace place(shift, q);
        uint8_t *at = stage + shift + lane * (uint32_t)q;
        stage_free<kAligned>();
        for (uint32_t b = 0; b < n; b += 32u, at += 32 * q) {
            const uint2 row = looked[b + lane];
            const uint32_t note = notes[b + lane];
            uint32_t W[kWords];
            join_row<kWords>(row.x, row.y, entries + (note & 7u) * 64u, W);
            stage_row<kWords, kAligned>(at, W, q, place, b != 0u);
            __syncwarp();
            const uint32_t from = (note >> kNoteFrom) & 31u;
            if (from > (uint32_t)L) at[from - 1u] = (uint8_t)(row.y >> 24);     // home round
            if (note & kNoteRecv) {
                const uint2 seg = segments[note & 7u];
                const int K = seg.y ? __ffs(seg.y) - 1 + L : q;
                const int low = (int)(x0 + b + lane - seg.x);
                int k = L;
                for (; low < (int)count_odd(odd, k + 1, K); ++k) at[k] = (uint8_t)(k + 1 - q);
                at[k] = (uint8_t)((int)t.miss[(K - L) * kMissRanks + low] - q);
            }
            if (!kAligned) __syncwarp();                         // (bytes of a word that the first lane completes next)
        }
        flush_item<kAligned>(stage, recv, n * (uint32_t)q);
    }
    if (send != nullptr) {
        const uint32_t shift = kAligned ? 0u : (uint32_t)(reinterpret_cast<uintptr_t>(send) & 15u);
        const RowPlace place(shift, q);
        uint8_t *at = stage + shift + lane * (uint32_t)q;
        const uint8_t *mine_row = reinterpret_cast<const uint8_t *>(looked + lane);
        const uint8_t *theirs[kLow];                             // entry k of the rank skips[k] further on
#pragma unroll
        for (int k = 0; k < kLow; ++k) theirs[k] = mine_row + (k < L ? t.s[k] * 8u + k : 0u);
        stage_free<kAligned>();
        for (uint32_t b = 0; b < n; b += 32u, at += 32 * q) {
            const uint32_t note = notes[b + lane];
            uint32_t e[kLow];
#pragma unroll
            for (int k = 0; k < kLow; ++k) e[k] = theirs[k][b * 8u];
            const uint32_t bb = mine_row[b * 8u + 7u];
            uint32_t lo = __byte_perm(__byte_perm(e[0], e[1], 0x0040), __byte_perm(e[2], e[3], 0x0040), 0x5410);
            uint32_t hi = __byte_perm(__byte_perm(e[4], e[5], 0x0040), e[6], 0x0410);
            if (kWords <= 2 && q < kLow) {                       // no entries beyond round q
                if (q < 4) lo &= (1u << (8 * q)) - 1u;
                hi &= q > 4 ? (1u << (8 * (q - 4))) - 1u : 0u;
            }
            uint32_t W[kWords];
            join_row<kWords>(lo, hi, entries + (note & 7u) * 64u + 32u, W);
            stage_row<kWords, kAligned>(at, W, q, place, b != 0u);
            __syncwarp();
            const int from = (int)((note >> kNoteFrom) & 31u);
            if (from < q) {                                      // rounds past the home round: the baseblock
                const bool root = bb == kRootMark;
                for (int k = from; k < q; ++k) at[k] = (uint8_t)(root ? (uint32_t)k : bb);
            }
            if (note & kNoteSend) {
                const uint2 seg = segments[note & 7u];
                const uint32_t sg = seg.y;
                const int z = __ffs(~sg) - 1;
                const int low = (int)(x0 + b + lane - seg.x);
                if (low == 0) {
                    // carries into a rank C(L, m) behind the start of a segment
                    if (sg & 1u) at[L] = (uint8_t)((int)t.miss[z * kMissRanks + (int)count_odd(odd, L, L + z)] - q);
                } else {
                    const int k = L + z, m = k + __ffs(~(sg >> (z + 1)));
                    const int behind = (int)count_odd(odd, k, m) - ((int)(t.s[L] - count_odd(odd, L, k)) - low);
                    const int block = behind < (int)count_odd(odd, k + 1, m)
                                          ? k + 1 : (int)t.miss[(m - L) * kMissRanks + behind];
                    at[k] = (uint8_t)(block - q);
                }
            }
            if (!kAligned) __syncwarp();
        }
        flush_item<kAligned>(stage, send, n * (uint32_t)q);
    }
}

}  // namespace bcs
