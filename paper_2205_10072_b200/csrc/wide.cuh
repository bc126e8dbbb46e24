// Large tables of a p with q >= 16: rows put together 16 output bytes at a time.
//
// The per-rank form (warp_rows) pays for every rank: shifting a row to its place among the words of its neighbours, an
// exchange with the next lane, stores q bytes apart, a copy out of shared memory.  Here a lane makes aligned
// 16-byte vectors of the output.  16 ranks are q vectors, so in steps of 16, 32 or 48 ranks a lane's vector
// always begins with the same round k0 of a rank at the same place of the step.  It holds bytes of two rows at most
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

// Vectors of a lane per step, and 16-rank groups of a step: q <= 21 has three groups on two vectors (80 to 98 % of
// the lanes' vectors in use, q = 16: 75 %), a larger q one group on one (69 to 97 %).  Two segments never end in the
// same step: for q <= 21 they have at least 65 - 14 ranks, for any q at least 65 - 24.
__host__ __device__ constexpr int wide_vectors(int q) { return q <= 21 ? 2 : 1; }
__host__ __device__ constexpr int wide_groups(int vectors) { return vectors == 2 ? 3 : 1; }

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
// All threads of the CTA call, the row table is complete.  Ends with a barrier.
__device__ __forceinline__ void build_send_table(const RowTable &t, uint2 *send, int q, uint32_t odd)
{
    const int high = q - kLow;
    const uint8_t *bytes = reinterpret_cast<const uint8_t *>(t.rows);
    if (threadIdx.x == 0) send[2 * high * kLowRanks] = make_uint2(0u, 0u);
    // Rows are 8 bytes apart, so the two halves of a warp would meet in the same banks: the upper half takes the
    // bytes 4..7 (odd words) while the lower half takes 0..3, and the other way round.
    const uint32_t turn = (threadIdx.x & 16u) ? 4u : 0u;
    int skip[8];
#pragma unroll
    for (uint32_t j = 0; j < 8; ++j) skip[j] = (j ^ turn) < 7u ? (int)t.s[j ^ turn] : 0;
    for (uint32_t job = threadIdx.x; job < 2u * (uint32_t)high * kLowRanks; job += blockDim.x) {
        const int u = (int)(job / kLowRanks) + 1, low = (int)(job % kLowRanks);
        const int own = u <= high ? u : 0, next = u <= high ? 0 : u - high;
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
        send[job] = row;
    }
    __syncthreads();
}

// Byte selectors of a vector, word by word, for A's row and for the next one's.
struct Pick {
    uint32_t a[4], b[4];
};

// All of a vector's selectors, 16 bits a word: A's row in x and y, the next one's in z and w.  k0: round of the
// vector's first byte; home_a, home_b: home rounds of A and A + 1, L - 1 if in the table.  (Out of line: needed where the
// home round changes only, at the skips; inlined, parts of it were computed in every segment.)
template <bool kSend>
__device__ __noinline__ uint4 packed_pick(int k0, int q, int home_a, int home_b)
{
    // The nibbles of a row: its round below L; 7 = baseblock (receive: the home round, send: all
    // rounds behind it); 15 = neither (a zero: byte 7 is below 128).
    auto nibbles = [&](int home, uint64_t &lo, uint64_t &hi) {
        lo = 0xfffffffff6543210ull;
        hi = ~0ull;
        if (kSend) {
            const int from = home + 1;                           // L..q
            if (from < 16) lo &= ~(0x8888888888888888ull << (4 * from));
            hi &= from < 16 ? ~0x8888888888888888ull : (from < 32 ? ~(0x8888888888888888ull << (4 * (from - 16))) : ~0ull);
        } else if (home >= kLow) {
            if (home < 16) lo &= ~(8ull << (4 * home));
            else hi &= ~(8ull << (4 * (home - 16)));
        }
    };
    uint64_t lo, hi;
    nibbles(home_a, lo, hi);
    uint64_t a = hi >> (4 * (k0 & 15)), b = ~0ull;
    if (k0 < 16) a = k0 ? lo >> (4 * k0) | hi << (64 - 4 * k0) : lo;
    const int n = q - k0;                                        // bytes of A's row
    if (n < 16) {
        a |= ~0ull << (4 * n);
        nibbles(home_b, lo, hi);
        b = lo << (4 * n) | ~(~0ull << (4 * n));
    }
    return make_uint4((uint32_t)a, (uint32_t)(a >> 32), (uint32_t)b, (uint32_t)(b >> 32));
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

// The entries of segment g from round L up, in the lanes' vectors: rounds k0 .. k0+15 (mod q).
template <int kVec, bool kSend>
__device__ __forceinline__ void segment_part(uint32_t g, int q, const int (&k0)[kVec], Words (&part)[kVec])
{
    const int k = (int)(threadIdx.x & 31u);
    const bool inside = k >= kLow && k < q;
    const uint32_t bits = inside ? g >> (k - kLow) : 0u;
    const uint32_t above = bits >> 1;
    const uint32_t next = above ? (uint32_t)(__ffs(above) + k - q) & 0xffu : 0u;     // 0 where the baseblock goes
    const uint32_t own = inside ? (uint32_t)(k - q) & 0xffu : 0u;
    auto wrap = [&](int x) { return x >= q ? x - q : x; };
    // lane k: the entries of the rounds k .. k+3 (mod q)
    uint32_t e = ((bits & 1u) != 0u) != kSend ? next : own;
    e |= __shfl_sync(0xffffffffu, e, wrap(k + 1)) << 8;
    e |= __shfl_sync(0xffffffffu, e, wrap(k + 2)) << 16;
#pragma unroll
    for (int i = 0; i < kVec; ++i)
#pragma unroll
        for (int w = 0; w < 4; ++w) part[i].w[w] = __shfl_sync(0xffffffffu, e, wrap(k0[i] + 4 * w));
}

__device__ __forceinline__ uint4 wide_vector(const uint2 a, const uint2 b, const Words &c, const Pick &pick)
{
    uint32_t x[4];
#pragma unroll
    for (int w = 0; w < 4; ++w)
        x[w] = c.w[w] | pick_bytes(a.x, a.y, pick.a[w]) | pick_bytes(b.x, b.y, pick.b[w]);
    return make_uint4(x[0], x[1], x[2], x[3]);
}

// What a lane knows of its vectors, for all items of a table that begin at the same place of a 16-byte group: byte
// 16 v - shift of a step is round k0 of its rank a (-1: the rank before it).
template <int kVec>
struct WideLane {
    int a[kVec], k0[kVec];
    uint32_t own[kVec][4];                                       // bytes of A's row
    Pick pick[kVec];
    int home;                                                    // home round that they are for, -1: none
    __device__ __forceinline__ void init(int q, uint32_t shift)
    {
        home = -1;
#pragma unroll
        for (int i = 0; i < kVec; ++i) {
            const int byte = (int)(16u * ((threadIdx.x & 31u) + 32u * (uint32_t)i) + (uint32_t)q - shift);   // shift < 16 <= q
            a[i] = byte / q - 1;
            k0[i] = byte - byte / q * q;
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                const int n = q - k0[i] - 4 * w;
                own[i][w] = n >= 4 ? 0xffffffffu : (n <= 0 ? 0u : (1u << (8 * n)) - 1u);
            }
        }
    }
};

// Receive (send) rows of the n ranks x0, x0 + 1, ... (mod p; x0 < p, n <= p) by one warp.  dst: where the row of x0
// goes, any address.  The warp writes whole aligned vectors, from the one that holds the row's first byte on; `head`:
// these are the first ranks, nothing in front of them is written; `tail`: the last ones, the end is
// theirs too (else n is a multiple of 16).
// sm: the CTA's shared memory, the row table at 0, the send table at send_at; ends: 32 bytes for the two vectors that are
// not written as a whole.
template <int kVec, bool kSend>
__device__ __forceinline__ void wide_rows(const RowTable &t, const uint8_t *sm, uint32_t send_at, uint8_t *ends, uint32_t p,
                                          int q, uint32_t odd, uint32_t inv, WideLane<kVec> &mine, uint32_t x0, uint32_t n,
                                          bool head, bool tail, int8_t *dst)
{
    constexpr uint32_t kGroups = (uint32_t)wide_groups(kVec), kStep = 16u * kGroups;     // ranks of a step
    constexpr uint32_t kRowStride = kLowRanks * 8u;
    const uint32_t lane = threadIdx.x & 31u;
    const int high = q - kLow;
    const uint32_t shift = (uint32_t)(reinterpret_cast<uintptr_t>(dst) & 15u);
    // window: bytes [skip, len) from there; the row of rank x0 + r starts at byte shift + r q
    uint8_t *out = reinterpret_cast<uint8_t *>(dst) - shift;
    const uint32_t len = n * (uint32_t)q + (tail ? shift : 0u);
    const uint32_t skip = head ? shift : 0u;
    const bool ragged = skip != 0u || (len & 15u) != 0u;
    const uint32_t step_bytes = kStep * (uint32_t)q;

    // Ranks are counted from x0 on; y: the first one that the window shows.
    const uint32_t lead = shift != 0u ? 1u : 0u;
    const uint32_t y = x0 >= lead ? x0 - lead : p - 1u;
    uint32_t gs = __umulhi(y, inv);
    gs = gs ? gs - 1u : 0u;                                      // the segment of y, or one or two before
    bool begun = false, head_left = skip != 0u;
    int start = 0, next = 0;                                     // first rank of the segment, of the next one
    Words part[kVec];
    uint32_t at[kVec];                                           // shared-memory offset of A's row
    uint32_t to[kVec], until[kVec];                              // byte of the vector in the window; end of what the lane writes
#pragma unroll
    for (int i = 0; i < kVec; ++i) {
        to[i] = 16u * (lane + 32u * (uint32_t)i);
        until[i] = to[i] < step_bytes ? len : 0u;
    }
    int step = 0;                                                // its first rank

    auto store = [&](uint32_t b, const uint4 x) {
        if (!ragged || (b >= skip && b + 16u <= len)) *reinterpret_cast<uint4 *>(out + b) = x;
        else *reinterpret_cast<uint4 *>(ends + (b < skip ? 0 : 16)) = x;
    };
    // bytes [from, until) of a vector that the window shows in part
    auto store_end = [&](uint32_t vector, const uint8_t *bytes) {
        const uint32_t b = vector + lane;
        if (lane < 16u && b >= skip && b < len) out[b] = bytes[lane];
    };
    auto put = [&](int b, uint32_t value) {
        if (b >= (int)skip && b < (int)len) out[b] = (uint8_t)value;
    };
    // Exceptions of the segment with ranks start .. next-1.  x: what its lane packed (below).
    auto exceptions = [&](uint32_t x) {
        const int row0 = (int)shift + start * q;
        if (!kSend) {
            if (lane < (x & 31u)) {                              // its first ranks receive ahead
                const int K = (int)(x >> 8);
                const int row = row0 + (int)lane * q;
                int k = kLow;
                for (; (int)lane < (int)count_odd(odd, k + 1, K); ++k) put(row + k, (uint32_t)(k + 1 - q));
                put(row + k, (uint32_t)((int)t.miss[(K - kLow) * kMissRanks + (int)lane] - q));
            }
        } else {
            const uint32_t before = x & 31u;
            if (lane - 1u < before) {                            // the last ranks carry into ones that do
                const int k = (int)((x >> 5) & 31u), m = (int)((x >> 10) & 31u);
                const uint32_t behind = before - lane;
                const int block = behind < ((x >> 15) & 31u) ? k + 1 : (int)t.miss[(m - kLow) * kMissRanks + (int)behind];
                put((int)shift + (next - (int)lane) * q + k, (uint32_t)(block - q));
            }
            if ((x >> 30) != 0u) {
                if ((x >> 31) != 0u) {                           // so does the first one, into the block kept in bits 20..27
                    if (lane == 0u) put(row0 + kLow, (x >> 20) & 0xffu);
                } else if ((int)lane >= kLow && (int)lane < q) { // the root sends block k in round k
                    put(row0 + (int)lane, lane);
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
        uint32_t extra;                                          // its exceptions
        if (!kSend) {
            const int K = kLow + (int)own;
            extra = (g & 1u) ? 0u : (count_odd(odd, kLow, K) + 1u) | (uint32_t)K << 8;
        } else {
            extra = g == 0u ? 1u << 30 : 0u;
            if (g & 1u)
                extra = 1u << 31 | ((uint32_t)t.miss[tz * kMissRanks + (int)count_odd(odd, kLow, kLow + tz)] - (uint32_t)q & 0xffu) << 20;
            if (tz < high) {
                const int k = kLow + tz, m = k + __ffs(~(g >> (tz + 1)));
                extra |= count_odd(odd, k, m) | (uint32_t)k << 5 | (uint32_t)m << 10 | count_odd(odd, k + 1, m) << 15;
            }
        }
        int j = 0;
        uint32_t base;                                           // position of rank x0
        if (!begun) {
            j = __popc(__ballot_sync(0xffffffffu, pos <= y)) - 1;
            base = y + lead;
            const uint32_t inf = __shfl_sync(0xffffffffu, info, j);
            start = (int)(__shfl_sync(0xffffffffu, pos, j) - base);
            next = (int)(__shfl_sync(0xffffffffu, pos, j + 1) - base);
            segment_part<kVec, kSend>(__shfl_sync(0xffffffffu, g, j), q, mine.k0, part);
            const int home = (int)(inf >> 24);
#pragma unroll
            for (int i = 0; i < kVec; ++i) {
                at[i] = (inf & 0xffffffu) + (uint32_t)((mine.a[i] - start) * 8);
                if (home != mine.home) mine.pick[i] = make_pick<kSend>(mine.k0[i], q, home, home);
            }
            mine.home = home;
            begun = true;
        } else {
            base = __shfl_sync(0xffffffffu, pos, 0) - (uint32_t)start;
            next = (int)(__shfl_sync(0xffffffffu, pos, 1) - base);
        }
        for (;;) {
            // steps inside the segment
            const int end = next < (int)n ? next : (int)n;
            for (; step + (int)kStep <= end; step += (int)kStep) {
#pragma unroll
                for (int i = 0; i < kVec; ++i) {
                    if (until[i] != 0u) {
                        const uint2 ra = *reinterpret_cast<const uint2 *>(sm + at[i]);
                        const uint2 rb = *reinterpret_cast<const uint2 *>(sm + at[i] + 8);
                        store(to[i], wide_vector(ra, rb, part[i], mine.pick[i]));
                    }
                    at[i] += 8u * kStep;
                    to[i] += step_bytes;
                }
            }
            // the step in which it ends, or the last one of the item
            const uint32_t inf2 = __shfl_sync(0xffffffffu, info, j + 1);
            const int home2 = (int)(inf2 >> 24);
            Words coming[kVec];
            segment_part<kVec, kSend>(__shfl_sync(0xffffffffu, g, j + 1), q, mine.k0, coming);
#pragma unroll
            for (int i = 0; i < kVec; ++i) {
                const int A = step + mine.a[i];
                const uint32_t new_at = (inf2 & 0xffffffu) + (uint32_t)((A - next) * 8);
                const bool behind = A >= next, behind_b = A + 1 >= next;
                if (mine.home != home2)
                    mine.pick[i] = make_pick<kSend>(mine.k0[i], q, behind ? home2 : mine.home, behind_b ? home2 : mine.home);
                if (to[i] < until[i]) {
                    Words c;
#pragma unroll
                    for (int w = 0; w < 4; ++w) {
                        const uint32_t keep = behind_b ? (behind ? 0u : mine.own[i][w]) : 0xffffffffu;
                        c.w[w] = (part[i].w[w] & keep) | (coming[i].w[w] & ~keep);
                    }
                    const uint2 ra = *reinterpret_cast<const uint2 *>(sm + (behind ? new_at : at[i]));
                    const uint2 rb = *reinterpret_cast<const uint2 *>(sm + (uint32_t)((behind_b ? new_at : at[i]) + 8u));
                    store(to[i], wide_vector(ra, rb, c, mine.pick[i]));
                }
                part[i] = coming[i];
                if (mine.home != home2) mine.pick[i] = make_pick<kSend>(mine.k0[i], q, home2, home2);
                at[i] = new_at + 8u * kStep;
                to[i] += step_bytes;
            }
            mine.home = home2;
            step += (int)kStep;
            const bool done = step * q >= (int)len;
            __syncwarp();                                        // the vectors come first
            if (ragged) {
                if (head_left) store_end(0u, ends);
                head_left = false;
                if (done && (len & 15u) != 0u && (len >= 16u || skip == 0u)) store_end(len & ~15u, ends + 16);
                __syncwarp();
            }
            exceptions(__shfl_sync(0xffffffffu, extra, j));
            start = next;
            ++j;
            if ((int)shift + start * q >= (int)len) return;
            next = (int)(__shfl_sync(0xffffffffu, pos, j + 1) - base);
            if (done) {                                          // its first ranks were in that step
                exceptions(__shfl_sync(0xffffffffu, extra, j));
                return;
            }
            if (j == 30) break;                                  // (lane 31 is known as the next one only)
        }
        gs += 30u;
    }
}

}  // namespace bcs
