// Rows of a p with q >= 16 put together 16 output bytes at a time: for the larger p of a list (batch.cuh), and for send rows alone of some million ranks (rows.cu).
//
// The per-rank form (warp_rows) pays for every rank: shifting a row to its place among the words of its neighbours, an
// exchange with the next lane, stores q bytes apart, a copy out of shared memory.  Here a lane makes aligned
// 16-byte vectors of the output.  16 ranks are q vectors, so in steps of 16 ranks a lane's vector always begins
// with the same round k0 of a rank at the same place of the step (the lanes from q on repeat the first ones').  Where fewer
// ranks are whole vectors already, a step takes as many as 32 lanes hold.  A vector holds bytes of two rows at most
// (q >= 16), those of ranks A and A + 1:
//     out = segment part | bytes of A's table row | bytes of (A+1)'s table row,
// the first in registers for as long as the segment lasts, the others by byte permutations whose selectors
// depend on (k0, home round) only.  Send rows work the same way with a row table of their own: what a rank sends in
// the rounds below L depends on (lowest set bit of its segment, lowest set bit of the next one, low), and one of
// the two is always L.
//
// Warps work alone, on one table at a time (both at once, two streams of stores, was slower than one after the other:
// 1600 against 1290 us for 2^27 ranks of q = 30).  In the step in which a segment ends, the lanes whose rank A lies behind that point
// take the next segment's part, and the one vector that holds bytes of both takes each from where it belongs.  The few
// exceptions (rows.cuh) go out as bytes after the vectors that hold their place.
#pragma once
#include "rows.cuh"

namespace bcs {

constexpr int kWideMinQ = 16;

constexpr uint32_t kStep = 16;        // items are multiples of this many ranks

// Ranks of a step: as many as are whole vectors and 32 of these at most, 512 / q rounded down to a multiple of
// 16 / gcd(16, q); and 2^32 divided by it, rounded up.  Two segments never end in the same step: they have 41 ranks or more.
// (16 ranks for all q left 12 of 32 lanes idle for q = 20: 200 p of 2^19..2^20 1341 -> 1224 us, 3000 of 2^15..2^16 1316 -> 1086.)
__host__ __device__ constexpr uint32_t step_ranks(int q)
{
    return q == 16 ? 32u : (q == 18 || q == 20 ? 24u : (q == 24 ? 20u : 16u));
}
__host__ __device__ constexpr uint32_t step_inverse(int q)
{
    return q == 16 ? 1u << 27 : (q == 18 || q == 20 ? 0xffffffffu / 24u + 1u : (q == 24 ? 0xffffffffu / 20u + 1u : 1u << 28));
}

struct WideLayout {
    RowLayout base;                   // (its warps' part is not used)
    uint32_t send, ends, bytes;       // ends: 32 bytes per warp, see below
    __host__ __device__ explicit WideLayout(int q) : base(q)
    {
        send = base.warps;
        ends = send + 2u * (uint32_t)(q - kLow) * kLowRanks * 8u + 128u;     // (one more row than ranks: of zeros)
        bytes = ends + 32u * 32u;
    }
};

// Send table: [u - 1][low], u = K - L (1..q-L) for a segment with bit L clear and lowest bit K, u = q - L + (K2 - L) for
// one with bit L set and K2 the lowest bit of the next segment.  Entries of the rounds 0..6, baseblock as byte 7.
// For the K of *t.wanted; all threads of the CTA call, the row table is complete.  Ends with a barrier.
__device__ __forceinline__ void build_send_table_wide(const RowTable &t, uint2 *send, int q, uint32_t odd)
{
    const int high = q - kLow;
    const uint8_t *bytes = reinterpret_cast<const uint8_t *>(t.rows);
    // (the first row of a group, and of the end, is looked at as the one behind a segment of 128 ranks)
    if ((int)threadIdx.x <= 2 * high && ((int)threadIdx.x == 2 * high || ((*t.wanted >> (threadIdx.x % (uint32_t)high + 1u)) & 1u) == 0u))
        send[threadIdx.x * kLowRanks] = make_uint2(0u, 0u);
    // Rows are 8 bytes apart, so the two halves of a warp would meet in the same banks: the upper half takes the
    // bytes 4..7 (odd words) while the lower half takes 0..3, and the other way round.
    const uint32_t turn = (threadIdx.x & 16u) ? 4u : 0u;
    int skip[8];
#pragma unroll
    for (uint32_t j = 0; j < 8; ++j) skip[j] = (j ^ turn) < 7u ? (int)t.s[j ^ turn] : 0;
    const uint32_t jobs = (uint32_t)__popc(*t.wanted) * 2u * kLowRanks;
    for (uint32_t job = threadIdx.x; job < jobs; job += blockDim.x) {
        const int K = (int)t.list[job / (2u * kLowRanks)] - kLow, low = (int)(job % kLowRanks);
        if (K == 0) continue;                                    // (is one of the two anyway)
        const int own = (job & kLowRanks) ? 0 : K, next = K - own;
        const int len = (int)t.s[kLow] - (int)count_odd(odd, kLow, kLow + next);
        uint2 row = make_uint2(0u, 0u);                          // (read, but not used, behind a segment's last rank)
        if (low < len) {
            uint32_t e[8];
#pragma unroll
            for (uint32_t j = 0; j < 8; ++j) {
                const int to = low + skip[j];
                e[j] = bytes[(uint32_t)(to < len ? own * kLowRanks + to : next * kLowRanks + to - len) * 8u + (j ^ turn)];
            }
            const uint32_t first = e[0] | e[1] << 8 | e[2] << 16 | e[3] << 24;
            const uint32_t second = e[4] | e[5] << 8 | e[6] << 16 | e[7] << 24;
            row = turn ? make_uint2(second, first) : make_uint2(first, second);
        }
        send[(uint32_t)((own ? K : high + K) - 1) * kLowRanks + (uint32_t)low] = row;
    }
    __syncthreads();
}

// Byte selectors of a vector, word by word, for A's row and for the next one's.
struct Pick {
    uint32_t a[4], b[4];
};

// Selectors of a row's bytes in a vector, a nibble per byte, bytes 0..7 and 8..15: its round 0 would be byte `off` of the vector
// (-31..31), its home round is `home`, L - 1 if in the table.  A nibble is the round below L; 7 = baseblock (receive: the home
// round, send: all rounds behind it); 15 = neither (a zero: byte 7 is below 128).
template <bool kSend>
__device__ __forceinline__ uint2 row_pick(int off, int q, int home)
{
    // nibbles n .. 7 of a word (none from n = 8 on, all for n <= 0)
    auto from = [](int n) { return n >= 8 ? 0u : 0xffffffffu << (n > 0 ? 4 * n : 0); };
    constexpr uint32_t low = 0xf6543210u;
    uint32_t a = ~0u, b = ~0u;
    if (off <= 0) {
        if (off > -8) a = __funnelshift_r(low, ~0u, (uint32_t)(-4 * off));
    } else if (off < 8) {
        a = low << (4 * off) | ~from(off);
        b = __funnelshift_l(low, ~0u, (uint32_t)(4 * off));
    } else if (off < 16) {
        b = low << (4 * (off - 8)) | ~from(off - 8);
    }
    // the baseblock's bytes: nibble 15 without its top bit
    const int first = off + (kSend ? home + 1 : home), end = kSend ? off + q : first + (home >= kLow ? 1 : 0);
    a &= ~(0x88888888u & from(first) & ~from(end));
    b &= ~(0x88888888u & from(first - 8) & ~from(end - 8));
    return make_uint2(a, b);
}

// All of a vector's selectors, 16 bits a word: A's row in x and y, the next one's in z and w.  k0: round of the
// vector's first byte; home_a, home_b: home rounds of A and A + 1.  (Out of line: needed where the
// home round changes only, at the skips; inlined, parts of it were computed in every segment.)
template <bool kSend>
__device__ __noinline__ uint4 packed_pick(int k0, int q, int home_a, int home_b)
{
    const uint2 a = row_pick<kSend>(-k0, q, home_a), b = row_pick<kSend>(q - k0, q, home_b);
    return make_uint4(a.x, a.y, b.x, b.y);
}

template <bool kSend>
__device__ __forceinline__ Pick make_pick(int k0, int q, int home_a, int home_b)
{
    const uint4 x = packed_pick<kSend>(k0, q, home_a, home_b);
    Pick pick;
    pick.a[0] = x.x & 0xffffu;
    pick.a[1] = x.x >> 16;
    pick.a[2] = x.y & 0xffffu;
    pick.a[3] = x.y >> 16;
    pick.b[0] = x.z & 0xffffu;
    pick.b[1] = x.z >> 16;
    pick.b[2] = x.w & 0xffffu;
    pick.b[3] = x.w >> 16;
    return pick;
}

// Four words of a vector.
struct Words {
    uint32_t w[4];
};

// The entries of a segment from round L up depend on its number g bit by bit: those from L + 3 up on the bits from 3 up
// only, the same for eight segments in a row.
constexpr int kNear = 3;

// Entry of round k >= L in segment g; 0 where the baseblock goes.
template <bool kSend>
__device__ __forceinline__ uint32_t far_entry(uint32_t g, int k, int q)
{
    const uint32_t bits = g >> (k - kLow);
    const uint32_t above = bits >> 1;
    const uint32_t next = above ? (uint32_t)(__ffs(above) + k - q) & 0xffu : 0u;
    return ((bits & 1u) != 0u) != kSend ? next : (uint32_t)(k - q) & 0xffu;
}

// Those of the rounds from L + 3 up, in the lane's vector: rounds k0 .. k0+15 (mod q).
template <bool kSend>
__device__ __forceinline__ Words far_part(uint32_t g, int q, int k0)
{
    const int k = (int)(threadIdx.x & 31u);
    uint32_t e = k >= kLow + kNear && k < q ? far_entry<kSend>(g, k, q) : 0u;
    auto wrap = [&](int x) { return x >= q ? x - q : x; };
    // lane k: the entries of the rounds k .. k+3 (mod q)
    e |= __shfl_sync(0xffffffffu, e, wrap(k < q ? k + 1 : 0)) << 8;
    e |= __shfl_sync(0xffffffffu, e, wrap(k < q ? k + 2 : 0)) << 16;
    Words part;
#pragma unroll
    for (int w = 0; w < 4; ++w) part.w[w] = __shfl_sync(0xffffffffu, e, wrap(k0 + 4 * w));
    return part;
}

// The bytes of the rows.
__device__ __forceinline__ Words wide_rows_of(const uint2 a, const uint2 b, const Pick &pick)
{
    Words x;
#pragma unroll
    for (int w = 0; w < 4; ++w) x.w[w] = pick_bytes(a.x, a.y, pick.a[w]) | pick_bytes(b.x, b.y, pick.b[w]);
    return x;
}

__device__ __forceinline__ uint4 wide_vector(const uint2 a, const uint2 b, const Words &c, const Pick &pick)
{
    uint32_t x[4];
#pragma unroll
    for (int w = 0; w < 4; ++w)
        x[w] = c.w[w] | pick_bytes(a.x, a.y, pick.a[w]) | pick_bytes(b.x, b.y, pick.b[w]);
    return make_uint4(x[0], x[1], x[2], x[3]);
}

// What a lane knows of its vector, for all items of a table that begin at the same place of a 16-byte group: byte
// 16 v - shift of a step is round k0 of its rank a (-1: the rank before it).
struct WideLane {
    uint32_t v;
    int a, k0;
    uint32_t own[4];                                             // bytes of A's row
    uint32_t near[4];                                            // selectors of the rounds L .. L+2
    Pick pick;
    int home;                                                    // home round that it is for, -1: none
    template <bool kAnyStep>
    __device__ __forceinline__ void init(int q, uint32_t shift)
    {
        const uint32_t lane = threadIdx.x & 31u;
        const uint32_t vectors = kAnyStep ? step_ranks(q) * (uint32_t)q / 16u : (uint32_t)q;
        v = lane < vectors ? lane : lane - vectors;
        const int byte = (int)(16u * v + (uint32_t)q - shift);   // shift < 16 <= q
        a = byte / q - 1;
        k0 = byte - byte / q * q;
        home = -1;
        const int to_low = (k0 <= kLow ? kLow : kLow + q) - k0;  // where round L is, or would be
        // nibbles 4 (a zero) but for 0, 1, 2 there
        uint64_t n = 0x4444444444444444ull;
#pragma unroll
        for (int i = 0; i < kNear; ++i) {
            int b = to_low + i;                                  // k0 = L + 1 or L + 2: a round before L + 2 is q behind
            b = b >= q ? b - q : b;
            if (b < 16) n = (n & ~(15ull << (4 * b))) | (uint64_t)i << (4 * b);
        }
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const int n_own = q - k0 - 4 * w;
            own[w] = n_own >= 4 ? 0xffffffffu : (n_own <= 0 ? 0u : (1u << (8 * n_own)) - 1u);
            near[w] = (uint32_t)(n >> (16 * w)) & 0xffffu;
        }
    }
    // The whole part of a segment: `far` and the entries of the rounds L .. L+2, bytes 0..2 of `three`.
    __device__ __forceinline__ Words part(const Words &far, uint32_t three) const
    {
        Words c;
#pragma unroll
        for (int w = 0; w < 4; ++w) c.w[w] = far.w[w] | pick_bytes(three, 0u, near[w]);
        return c;
    }
};

// Receive (send) rows of the n ranks x0, x0 + 1, ... (mod p; x0 < p, n <= p) by one warp.  dst: where the row of x0
// goes, any address.  The warp writes whole aligned vectors, from the one that holds the row's first byte on; `head`:
// these are the first ranks, nothing in front of them is written; `tail`: the last ones, the end is
// theirs too (else n is a multiple of 16).
// sm: the CTA's shared memory, the row table at 0, the send table at send_at; ends: 32 bytes for the two vectors that are
// not written as a whole.
// Waits for the kernel before (dependent launches) in front of the first store: where the run starts, some 2400 cycles, does not
// depend on it (all ranks of 100 003 6.0 -> 5.5 us).
// kRoom: the kernel has registers left for one computation of selectors per change of the home round instead of two (some 700 cycles each,
// and the warp that has the first ranks has four or five such changes); the middle kernel of a batch would spill (1320 -> 1350 us).
// kAnyStep: false where step_ranks(q) is known to be 16 (a constant: 0.2-0.3 us less for tables of up to 2 million ranks).
template <bool kSend, bool kAnyStep, bool kRoom>
__device__ __forceinline__ void wide_rows(const RowTable &t, const uint8_t *sm, uint32_t send_at, uint8_t *ends, uint32_t p,
                                          int q, uint32_t odd, uint32_t inv, WideLane &mine, uint32_t x0, uint32_t n,
                                          bool head, bool tail, int8_t *dst)
{
    constexpr uint32_t kRowStride = kLowRanks * 8u;
    const uint32_t lane = threadIdx.x & 31u;
    const int high = q - kLow;
    const uint32_t shift = (uint32_t)(reinterpret_cast<uintptr_t>(dst) & 15u);
    // window: bytes [skip, len) from there; the row of rank x0 + r starts at byte shift + r q
    uint8_t *out = reinterpret_cast<uint8_t *>(dst) - shift;
    const uint32_t len = n * (uint32_t)q + (tail ? shift : 0u);
    const uint32_t skip = head ? shift : 0u;
    const bool ragged = skip != 0u || (len & 15u) != 0u;
    const uint32_t ranks = kAnyStep ? step_ranks(q) : 16u, step_bytes = ranks * (uint32_t)q;     // of a step
    const uint32_t by_ranks = step_inverse(q);

    // Ranks are counted from x0 on; y: the first one that the window shows.
    const uint32_t lead = shift != 0u ? 1u : 0u;
    const uint32_t y = x0 >= lead ? x0 - lead : p - 1u;
    uint32_t gs = __umulhi(y, inv);
    gs = gs ? gs - 1u : 0u;                                      // the segment of y, or one or two before
    bool begun = false, head_left = skip != 0u;
    int start = 0, next = 0;                                     // first rank of the segment, of the next one
    Words far, part;
    uint32_t at = 0;                                             // shared-memory offset of A's row
    uint32_t to = 16u * mine.v;                                  // byte of the vector in the window
    int step = 0;                                                // its first rank

    auto store = [&](uint32_t b, const uint4 x) {
        if (!ragged || (b >= skip && b + 16u <= len)) *reinterpret_cast<uint4 *>(out + b) = x;
        else *reinterpret_cast<uint4 *>(ends + (b < skip ? 0 : 16)) = x;
    };
    // what a window shows of a vector that it does not hold as a whole
    auto store_end = [&](uint32_t vector, const uint8_t *bytes) {
        const uint32_t b = vector + lane;
        if (lane < 16u && b >= skip && b < len) out[b] = bytes[lane];
    };
    auto put = [&](int b, uint32_t value) {
        if (b >= (int)skip && b < (int)len) out[b] = (uint8_t)value;
    };
    // Receive exceptions of the segment with lowest bit K whose first row starts at byte row0.  With t(0) > t(1) > ... the levels
    // t = 8 .. K of which e_t is set, rank `low` receives block k + 1 in the rounds k = L .. t(low) - 2, then the missing one;
    // the rank behind the last such level has the missing one in round L.
    auto receive_ahead = [&](int K, int row0) {
        uint32_t levels = odd & ((2u << K) - 1u) & ~((2u << kLow) - 1u);
        for (int low = 0;; ++low) {
            const int top = top_bit(levels);                     // -1 behind the last one
            const int row = row0 + low * q;
            int k = kLow;
            for (; k <= top - 2; ++k) put(row + k, (uint32_t)(k + 1 - q));
            put(row + k, (uint32_t)((int)t.miss[(K - kLow) * kMissRanks + low] - q));
            if (levels == 0u) break;
            levels &= ~(1u << top);
        }
    };
    // Exceptions of the lanes' segments: g, its first row's byte, that of the next one's first row, whether it counts.  A few
    // bytes each, so all the segments of an item at once, one by lane (the whole warp on one segment after another took a
    // fifth more instructions in all); but those with hundreds, near multiples of large skips, by the warp.
    constexpr int kAlone = kLow + 4;
    auto exceptions = [&](uint32_t g, int row0, int row1, bool counts) {
        if (!kSend) {
            const int K = g ? __ffs(g) - 1 + kLow : q;           // its first ranks receive ahead
            if (counts && !(g & 1u) && K <= kAlone) receive_ahead(K, row0);
            uint32_t heavy = __ballot_sync(0xffffffffu, counts && K > kAlone);
            for (; heavy != 0u; heavy &= heavy - 1u) {
                const int j = __ffs(heavy) - 1;
                const int heavy_k = __shfl_sync(0xffffffffu, K, j);
                const int row = __shfl_sync(0xffffffffu, row0, j) + (int)lane * q;
                int missing = kLow;                              // round of the lane's missing block
                for (int k = kLow; k <= heavy_k - 2; ++k) {
                    if ((int)lane >= (int)count_odd(odd, k + 1, heavy_k)) continue;
                    put(row + k, (uint32_t)(k + 1 - q));
                    missing = k + 1;
                }
                if ((int)lane <= (int)count_odd(odd, kLow, heavy_k))
                    put(row + missing, (uint32_t)((int)t.miss[(heavy_k - kLow) * kMissRanks + (int)lane] - q));
            }
        } else if (counts) {
            const int z = __ffs(~g) - 1;
            if (g & 1u) {                                        // the first rank carries into one that does
                put(row0 + kLow, (uint32_t)((int)t.miss[z * kMissRanks + (int)count_odd(odd, kLow, kLow + z)] - q));
            } else if (g == 0u) {                                // the root sends block k in round k
                for (int k = kLow; k < q; ++k) put(row0 + k, (uint32_t)k);
            }
            if (z < high) {                                      // so do the last ones
                const int k = kLow + z, m = k + __ffs(~(g >> (z + 1)));
                const int before = (int)count_odd(odd, k, m), deeper = (int)count_odd(odd, k + 1, m);
                for (int d = 1; d <= before; ++d) {
                    const int behind = before - d;
                    const int block = behind < deeper ? k + 1 : (int)t.miss[(m - kLow) * kMissRanks + behind];
                    put(row1 - d * q + k, (uint32_t)(block - q));
                }
            }
        }
    };

    for (;;) {
        // lane j: segment gs + j.  Positions go on counting behind p - 1: the root's segment again.
        gs &= (1u << high) - 1u;
        const uint32_t at0 =
            __reduce_add_sync(0xffffffffu, (int)lane < high && ((gs >> lane) & 1u) ? t.s[lane + kLow] : 0u);
        const uint32_t g = (gs + lane) & ((1u << high) - 1u);
        const int tz = __ffs(~g) - 1;
        const uint32_t seg_len = t.s[kLow] - count_odd(odd, kLow, kLow + tz);
        uint32_t pos = seg_len;
#pragma unroll
        for (uint32_t d = 1; d < 32; d *= 2) {
            const uint32_t up = __shfl_up_sync(0xffffffffu, pos, d);
            if (lane >= d) pos += up;
        }
        pos += at0 - seg_len;
        const uint32_t own = g ? (uint32_t)__ffs(g) - 1u : (uint32_t)high;
        // its rows, and the home round
        const uint32_t rows = kSend ? send_at + (((g & 1u) ? (uint32_t)(high + tz) : own) - 1u) * kRowStride : own * kRowStride;
        const uint32_t info = rows | (uint32_t)(g ? 31 - __clz(g) + kLow : kLow - 1) << 24;
        // its entries in the rounds L .. L+2, and whether it begins eight segments
        uint32_t three = (g & ((1u << kNear) - 1u)) == 0u ? 1u << 24 : 0u;
#pragma unroll
        for (int i = 0; i < kNear; ++i) three |= far_entry<kSend>(g, kLow + i, q) << (8 * i);
        int j = 0, j0;                                           // segments j0 .. j have been gone through
        uint32_t base;                                           // position of rank x0
        if (!begun) {
            j = __popc(__ballot_sync(0xffffffffu, pos <= y)) - 1;
            base = y + lead;
            const uint32_t inf = __shfl_sync(0xffffffffu, info, j);
            start = (int)(__shfl_sync(0xffffffffu, pos, j) - base);
            next = (int)(__shfl_sync(0xffffffffu, pos, j + 1) - base);
            far = far_part<kSend>(__shfl_sync(0xffffffffu, g, j), q, mine.k0);
            part = mine.part(far, __shfl_sync(0xffffffffu, three, j));
            const int home = (int)(inf >> 24);
            at = (inf & 0xffffffu) + (uint32_t)((mine.a - start) * 8);
            if (home != mine.home) mine.pick = make_pick<kSend>(mine.k0, q, home, home);
            mine.home = home;
            begun = true;
            grid_dependency_wait();                              // (the kernel before: not until the first store)
        } else {
            base = __shfl_sync(0xffffffffu, pos, 0) - (uint32_t)start;
            next = (int)(__shfl_sync(0xffffffffu, pos, 1) - base);
        }
        j0 = j;
        bool done = false;
        for (;;) {
            // steps inside the segment
            const int room = (next < (int)n ? next : (int)n) - step;
            const int steps = kAnyStep ? (int)__umulhi(room > 0 ? (uint32_t)room : 0u, by_ranks) : room / 16;
            if (!ragged) {
                uint8_t *o = out + to;
#pragma unroll 1                                                 // (a handful: 1024 p of 2^10..2^20 1330 us unrolled, 1295 not)
                for (int i = 0; i < steps; ++i) {
                    const uint2 ra = *reinterpret_cast<const uint2 *>(sm + at);
                    const uint2 rb = *reinterpret_cast<const uint2 *>(sm + at + 8);
                    *reinterpret_cast<uint4 *>(o) = wide_vector(ra, rb, part, mine.pick);
                    at += 8u * ranks;
                    o += step_bytes;
                }
            } else {
                for (int i = 0; i < steps; ++i) {
                    const uint2 ra = *reinterpret_cast<const uint2 *>(sm + at);
                    const uint2 rb = *reinterpret_cast<const uint2 *>(sm + at + 8);
                    store(to + (uint32_t)i * step_bytes, wide_vector(ra, rb, part, mine.pick));
                    at += 8u * ranks;
                }
            }
            to += (uint32_t)steps * step_bytes;
            step += steps * (int)ranks;
            // the step in which it ends, or the last one of the item
            const uint32_t inf2 = __shfl_sync(0xffffffffu, info, j + 1), three2 = __shfl_sync(0xffffffffu, three, j + 1);
            const int home2 = (int)(inf2 >> 24);
            if ((three2 >> 24) != 0u) far = far_part<kSend>(__shfl_sync(0xffffffffu, g, j + 1), q, mine.k0);
            const Words coming = mine.part(far, three2);
            const int A = step + mine.a;
            const uint32_t new_at = (inf2 & 0xffffffu) + (uint32_t)((A - next) * 8);
            const bool behind = A >= next, behind_b = A + 1 >= next;
            auto segment_part = [&](int w) {                     // of the two segments
                const uint32_t keep = behind_b ? (behind ? 0u : mine.own[w]) : 0xffffffffu;
                return (part.w[w] & keep) | (coming.w[w] & ~keep);
            };
            if (kRoom && mine.home != home2) {
                // the rows in front by the selectors so far, those behind by the new ones
                const uint2 none = make_uint2(0u, 0u);
                const uint2 ra = *reinterpret_cast<const uint2 *>(sm + (behind ? new_at : at));
                const uint2 rb = *reinterpret_cast<const uint2 *>(sm + (uint32_t)((behind_b ? new_at : at) + 8u));
                Words c = wide_rows_of(behind ? none : ra, behind_b ? none : rb, mine.pick);
                mine.pick = make_pick<kSend>(mine.k0, q, home2, home2);
                const Words d = wide_rows_of(behind ? ra : none, behind_b ? rb : none, mine.pick);
#pragma unroll
                for (int w = 0; w < 4; ++w) c.w[w] |= d.w[w] | segment_part(w);
                if (to < len) store(to, make_uint4(c.w[0], c.w[1], c.w[2], c.w[3]));
            } else {
                if (!kRoom && mine.home != home2)
                    mine.pick = make_pick<kSend>(mine.k0, q, behind ? home2 : mine.home, behind_b ? home2 : mine.home);
                if (to < len) {
                    Words c;
#pragma unroll
                    for (int w = 0; w < 4; ++w) c.w[w] = segment_part(w);
                    const uint2 ra = *reinterpret_cast<const uint2 *>(sm + (behind ? new_at : at));
                    const uint2 rb = *reinterpret_cast<const uint2 *>(sm + (uint32_t)((behind_b ? new_at : at) + 8u));
                    store(to, wide_vector(ra, rb, c, mine.pick));
                }
                if (!kRoom && mine.home != home2) mine.pick = make_pick<kSend>(mine.k0, q, home2, home2);
            }
            mine.home = home2;
            part = coming;
            at = new_at + 8u * ranks;
            to += step_bytes;
            step += (int)ranks;
            done = step * q >= (int)len;
            start = next;
            ++j;
            next = (int)(__shfl_sync(0xffffffffu, pos, j + 1) - base);
            // (lane 31 is known as the next one only; the last step may hold the first ranks of segment j)
            if (done || j == 30) break;
        }
        __syncwarp();                                            // the vectors come first
        if (ragged) {
            if (head_left) store_end(0u, ends);
            head_left = false;
            if (done && (len & 15u) != 0u && (len >= 16u || skip == 0u)) store_end(len & ~15u, ends + 16);
            __syncwarp();
        }
        {
            const uint32_t after = __shfl_down_sync(0xffffffffu, pos, 1);
            exceptions(g, (int)shift + (int)(pos - base) * q, (int)shift + (int)(after - base) * q,
                       (int)lane >= j0 && (int)lane < j + (done ? 1 : 0));
        }
        if (done) return;
        gs += 30u;
    }
}

}  // namespace bcs
