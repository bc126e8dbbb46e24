// Larger tables of a p with q >= 17, and lists of p up to 1024 (q = 8..10): four consecutive ranks per lane.
//
// Four rows of q bytes are q words, so what a lane writes begins and ends on words, for every q: the four rows are joined in registers by
// funnel shifts and byte permutations that are constants of q, without a word that two lanes share.  A warp makes the rows of 256
// ranks (a pass: two look-ups of 128) in shared memory and sends them out as one bulk copy of the TMA unit; the few exceptions (rows.cuh) are written as bytes
// in between.
//
//   * Receive rows: a lane looks its four table rows up and joins them with the entries of their segment.
//   * Send rows: entry k < L of a rank is the receive entry of the rank skips[k] <= 64 further on.  The rows of a pass and of the 64 ranks behind are
//     transposed (sixteen byte permutations for four ranks) and kept as columns, a byte per rank, one column per round; four consecutive bytes
//     of column k from skips[k] further on are the entries of a lane's four ranks.  Transposed back they are their rows.  Long ranges look
//     them up in a table of send rows (kTable).
//
// Some 700 warp instructions for both rows of 128 ranks of q = 21, 520 where send rows come from their table (1000 with 128 ranks a pass and the exceptions segment after segment; 1230 by vectors of
// 16 output bytes), of which the integer pipe takes half at half rate: that and the issue slots bound the kernel until memory does.  The exceptions take
// 85, the transpositions and the ranks behind 120, the packing and staging of rows 150, a bulk copy some 20.
#pragma once
#include "rows.cuh"

namespace bcs {

constexpr int kQuadMinQ = 17;

// Table of send rows: [u - 1][low], u = K - L (1..7) for a segment with bit L clear and lowest bit K, u = 7 + (K2 - L) for one with bit L
// set and K2 the lowest bit of the next segment.  Entries of the rounds 0..6, baseblock as byte 7.  Segments with a larger K or K2, one in 64, have
// their send rows put together from the row table (42 groups of rows for q = 28 take 3 us to build, 14 take 1).
constexpr int kSendDepth = 7;
__host__ __device__ constexpr int send_groups(int q) { return q - kLow < kSendDepth ? q - kLow : kSendDepth; }

// All threads of the CTA call, the row table is complete (its rows permuted, as these).  Ends with a barrier.
__device__ __forceinline__ void build_send_table(const RowTable &t, uint2 *send, int q, uint32_t odd)
{
    const int groups = send_groups(q);
    const uint8_t *bytes = reinterpret_cast<const uint8_t *>(t.rows);
    // Rows are 8 bytes apart, so the two halves of a warp would meet in the same banks: the upper half takes the
    // bytes 4..7 (odd words) while the lower half takes 0..3, and the other way round.
    const uint32_t turn = (threadIdx.x & 16u) ? 4u : 0u;
    int skip[8];
#pragma unroll
    for (uint32_t j = 0; j < 8; ++j) skip[j] = (j ^ turn) < 7u ? (int)t.s[j ^ turn] : 0;
    const uint32_t jobs = (uint32_t)groups * 2u * kLowRanks;
    for (uint32_t job = threadIdx.x; job < jobs; job += blockDim.x) {
        const int K = (int)(job / (2u * kLowRanks)) + 1, low = (int)(job % kLowRanks);
        const int own = (job & kLowRanks) ? 0 : K, next = K - own;
        const int len = (int)t.s[kLow] - (int)count_odd(odd, kLow, kLow + next);
        if (low >= len) continue;
        uint32_t e[8];
#pragma unroll
        for (uint32_t j = 0; j < 8; ++j) {
            const int to = low + skip[j];
            const uint32_t row = to < len ? own * kLowRanks + permuted_row((uint32_t)to) : next * kLowRanks + permuted_row((uint32_t)(to - len));
            e[j] = bytes[row * 8u + (j ^ turn)];
        }
        const uint32_t first = e[0] | e[1] << 8 | e[2] << 16 | e[3] << 24;
        const uint32_t second = e[4] | e[5] << 8 | e[6] << 16 | e[7] << 24;
        send[(uint32_t)((own ? K : groups + K) - 1) * kLowRanks + permuted_row((uint32_t)low)] = turn ? make_uint2(second, first) : make_uint2(first, second);
    }
    __syncthreads();
}

constexpr uint32_t kQuads = 128;                       // ranks that a warp looks up at a time, four a lane

constexpr int kTurns = 2;                              // look-ups of a pass: its rows are staged and sent out together
constexpr uint32_t kPass = kTurns * kQuads;
constexpr uint32_t kMostRun = 896;                     // ranks of a run

// A warp's segments lie in shared memory: all that the look-ups of a run can touch, and one more.  Looked up are the ranks of whole passes (of a last one
// that is half full, fewer) and 128 behind.  c segments in a row have more than 64 c - 25 ranks, so r ranks touch (r + 22) / 64 + 2 segments at most.
__host__ __device__ constexpr uint32_t run_segments(uint32_t run) { return ((run + kPass - 1u) / kPass * kPass + kQuads + 22u) / 64u + 3u; }
static_assert(run_segments(kMostRun) <= 30u, "located by one warp, the first of them up to two lanes behind the first");
// Room for them in the kernel for one p, which takes 1 to 5 % longer with less (q = 30: 83 000 receive rows 1.98 us, with what they need 2.05).
__host__ __device__ constexpr uint32_t roomy_segments(uint32_t run) { return ((run + kPass - 1u) / kPass * kPass + kQuads) / 41u + 4u; }
static_assert(roomy_segments(kQuads) >= run_segments(kQuads) && roomy_segments(kMostRun) >= run_segments(kMostRun), "the steps between are larger, too");
constexpr uint32_t kColumn = kPass + kHalo + 8u;       // bytes of a column

// Byte offsets in the CTA's shared memory: the row table, with kTable that of send rows, and a warp's part (with columns otherwise).
template <bool kTable>
struct QuadLayout {
    RowLayout base;                                    // (its warps' part is not used)
    uint32_t segments;                                 // of a run
    uint32_t table = 0, warps = 0, entries = 0, columns = 0, stage = 0, warp_bytes = 0;
    __host__ __device__ constexpr QuadLayout(int q, uint32_t segments_of_run) : base(q), segments(segments_of_run)
    {
        table = base.warps;
        warps = table + (kTable ? 2u * (uint32_t)send_groups(q) * kLowRanks * 8u : 0u);
        entries = segments * 16u;
        columns = entries + segments * 64u;
        stage = (columns + (kTable ? 0u : kLow * kColumn) + 15u) & ~15u;
        warp_bytes = stage + kPass * (uint32_t)q + 16u;      // (rows that are shifted end in the last 16 bytes)
    }
    __host__ __device__ constexpr uint32_t total(uint32_t n_warps) const { return warps + n_warps * warp_bytes; }
};

// What the run's look-up knows of a segment.
struct Segment {
    int start;             // its first rank, counted from the run's first
    int key;               // byte of its first table row, less 8 start
    uint32_t recv;         // bits 0..4: ranks behind its start that can be receive exceptions; 5..9: K - L; 10..14: home round, 0 if below L;
                           // 15: that is not in the last two words of a row; 16..: its group in the table of send rows, less K - L
    uint32_t send;         // bits 0..4: ranks before its end whose entry in round L + (10..14) is an exception, 5..9: those of them that send the next
                           // block, 15..19: the segment whose missing blocks the others send; 20: its first rank's entry L is bits 24..31; 21: the
                           // root's; 22: it has no group in the table of send rows
};

// Rows of four ranks a lane are 32 bytes apart: permuted like this, 16 lanes meet in no bank.  (Byte offset of a row in the table.)
__device__ __forceinline__ uint32_t row_at(uint32_t at) { return at ^ ((at >> 4) & 0x18u); }

// Segments of the run that begins at rank x0 (mod p), all that it can touch, and the entries of those that start in front of rank n.  Returns the
// start of segment `lane` of these (counted from the run's first rank), 0x7fffffff if there is none.  By a warp.
template <int Q, bool kTable>
__device__ __forceinline__ int locate_run(const RowTable &t, Segment *segments, uint8_t *entries, uint32_t odd, uint32_t inv,
                                          uint32_t x0, uint32_t n, uint32_t most)
{
    constexpr int high = Q - kLow;
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t gs = __umulhi(x0, inv);
    gs = gs ? gs - 1u : 0u;                                      // the segment of x0, or one or two before
    const uint32_t at0 = __reduce_add_sync(0xffffffffu, (int)lane < high && ((gs >> lane) & 1u) ? t.s[lane + kLow] : 0u);
    const uint32_t g = (gs + lane) & ((1u << high) - 1u);        // (positions go on counting behind p - 1: the root's segment again)
    const int tz = __ffs(~g) - 1;                                // lowest zero bit
    const uint32_t len = t.s[kLow] - count_odd(odd, kLow, kLow + tz);
    uint32_t pos = len;
#pragma unroll
    for (uint32_t d = 1; d < 32; d *= 2) {
        const uint32_t up = __shfl_up_sync(0xffffffffu, pos, d);
        if (lane >= d) pos += up;
    }
    pos += at0 - len;
    const uint32_t first = __popc(__ballot_sync(0xffffffffu, pos <= x0)) - 1u;
    const int start = (int)(pos - x0);
    const uint32_t slot = lane - first;
    if (slot < most) {
        Segment seg;
        const int K = g ? __ffs(g) - 1 : high;
        seg.start = start;
        seg.key = (K * kLowRanks - start) * 8;
        const uint32_t home = g ? (uint32_t)(31 - __clz(g) + kLow) : 0u;
        seg.recv = (K ? count_odd(odd, kLow, kLow + K) + 1u : 0u) | (uint32_t)K << 5 | home << 10 | ((int)(home ? home : kLow) < 4 * ((Q + 3) / 4 - 2) ? 1u << 15 : 0u);
        seg.send = g ? 0u : 1u << 21;
        if (g & 1u)                                              // its first rank carries into one close behind a start
            seg.send = 1u << 20 | (uint32_t)((int)t.miss[tz * kMissRanks + (int)count_odd(odd, kLow, kLow + tz)] - Q) << 24;
        if (tz < high) {                                         // so do its last ones
            const int m = tz + __ffs(~(g >> (tz + 1)));
            seg.send |= count_odd(odd, kLow + tz, kLow + m) | count_odd(odd, kLow + tz + 1, kLow + m) << 5 | (uint32_t)tz << 10 | (uint32_t)m << 15;
        }
        if constexpr (kTable) {
            const int level = (g & 1u) ? tz : K, group = level > kSendDepth ? 0 : ((g & 1u) ? send_groups(Q) + tz : K) - 1;
            if (level > kSendDepth) seg.send |= 1u << 22;
            seg.recv |= (uint32_t)(group - K) << 16;
        }
        segments[slot] = seg;
    }
    // Entries of the rounds from L up, 32 bytes for receive rows and 32 for send rows: four segments at a time, a word of each per lane.
    // Word 0 of either: where the baseblock goes in the last two words of a row, as selectors of byte permutations (round `tail` and those behind it).
    constexpr int tail = 4 * ((Q + 3) / 4 - 2);
    const uint32_t some = __popc(__ballot_sync(0xffffffffu, lane >= first && start < (int)n));
    const int word = (int)(lane & 7u), round = 4 * word;
    uint32_t same = 0, inside = 0;                               // k - q in byte k, and where k is from L up
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        if (round + b < kLow || round + b >= Q) continue;
        same |= (uint32_t)(uint8_t)(round + b - Q) << (8 * b);
        inside |= 0xffu << (8 * b);
    }
    for (uint32_t j = 0; j < some; j += 4u) {
        const uint32_t of = j + (lane >> 3);
        const uint32_t code = (__shfl_sync(0xffffffffu, g, (first + of) & 31u) << kLow) >> round;
        // the next higher set bit of round + 3, + 2, + 1, + 0; 0 where the baseblock goes
        const uint32_t above = code >> 4;
        const uint32_t three = above ? (uint32_t)(round + 3 - Q + __ffs(above)) : 0u;
        const uint32_t two = (code & 8u) ? (uint32_t)(round + 3 - Q) : three;
        const uint32_t one = (code & 4u) ? (uint32_t)(round + 2 - Q) : two;
        const uint32_t zero = (code & 2u) ? (uint32_t)(round + 1 - Q) : one;
        const uint32_t next = __byte_perm(__byte_perm(zero, one, 0x0040), __byte_perm(two, three, 0x0040), 0x5410);
        const uint32_t set = (((code & 15u) * 0x00204081u) & 0x01010101u) * 0xffu;
        if (of < some) {
            uint32_t *e = reinterpret_cast<uint32_t *>(entries + of * 64u) + word;
            uint32_t received = ((set & next) | (~set & same)) & inside, sent = ((set & same) | (~set & next)) & inside;
            if (word == 0) {                                     // (the code from bit 0 on)
                const int home = code ? 31 - __clz(code) - tail : -1;
                received = sent = 0x32103210u;
                if (home >= 0) {
                    received |= 7u << (4 * home);
                    sent |= home < 7 ? 0x77777777u << (4 * home + 4) : 0u;
                } else if constexpr (kLow >= tail) {             // the root's segment, rounds from L on
                    if (code == 0u) sent |= 0x77777777u << (4 * (kLow - tail));
                }
            }
            e[0] = received;
            e[8] = sent;
        }
    }
    __syncwarp();
    const int behind = __shfl_sync(0xffffffffu, start, (lane + first) & 31u);
    return lane + first < 32u ? behind : 0x7fffffff;
}

// 4 x 4 bytes: word i of the result holds the bytes i of a, b, c, d.
__device__ __forceinline__ void transpose(uint32_t a, uint32_t b, uint32_t c, uint32_t d, uint32_t &w0, uint32_t &w1, uint32_t &w2, uint32_t &w3)
{
    const uint32_t ab = __byte_perm(a, b, 0x5140), cd = __byte_perm(c, d, 0x5140);
    const uint32_t ab2 = __byte_perm(a, b, 0x7362), cd2 = __byte_perm(c, d, 0x7362);
    w0 = __byte_perm(ab, cd, 0x5410);
    w1 = __byte_perm(ab, cd, 0x7632);
    w2 = __byte_perm(ab2, cd2, 0x5410);
    w3 = __byte_perm(ab2, cd2, 0x7632);
}

// Word o of four rows of Q bytes one behind the other; R[i]: the words of row i.
template <int Q, int o, int kWords>
__device__ __forceinline__ uint32_t joined(const uint32_t (&R)[4][kWords])
{
    constexpr int i = 4 * o / Q, k = 4 * o % Q, w = k / 4, off = k % 4, n = Q - k;       // row, byte and the bytes that are left of it
    static_assert(Q >= 4, "bytes of two rows at most");
    const uint32_t a = R[i][w];
    if constexpr (n >= 4) {
        if constexpr (off == 0) return a;
        else return __funnelshift_r(a, R[i][w + 1], 8 * off);
    } else {
        const uint32_t next = R[i + 1][0];
        constexpr uint32_t from = 0x76543210u >> (4 * off);      // bytes off, off + 1, .. of (a, ...)
        if constexpr (off + n <= 4) {
            constexpr uint32_t pick = (from & ((1u << (4 * n)) - 1u)) | (0x7654u << (4 * n) & 0xffffu);
            return __byte_perm(a, next, pick);
        } else {
            const uint32_t tail = __funnelshift_r(a, R[i][w + 1], 8 * off);
            constexpr uint32_t pick = (0x3210u & ((1u << (4 * n)) - 1u)) | (0x7654u << (4 * n) & 0xffffu);
            return __byte_perm(tail, next, pick);
        }
    }
}

// Stores the lane's four rows, Q words, at `at` (16-byte aligned where Q is a multiple of 4, 8-byte where it is even): the widest stores
// that keep the lanes, Q words apart, in different banks (but for Q = 16 and 24).
template <int Q, int o, int kWords>
__device__ __forceinline__ void stage_words(uint8_t *at, const uint32_t (&R)[4][kWords])
{
    if constexpr (o < Q) {
        constexpr int step = Q % 4 == 0 ? 4 : (Q % 2 == 0 ? 2 : 1);
        if constexpr (step == 4)
            *reinterpret_cast<uint4 *>(at + 4 * o) = make_uint4(joined<Q, o>(R), joined<Q, o + 1>(R), joined<Q, o + 2>(R), joined<Q, o + 3>(R));
        else if constexpr (step == 2)
            *reinterpret_cast<uint2 *>(at + 4 * o) = make_uint2(joined<Q, o>(R), joined<Q, o + 1>(R));
        else
            *reinterpret_cast<uint32_t *>(at + 4 * o) = joined<Q, o>(R);
        stage_words<Q, o + step>(at, R);
    }
}

// The same for rows that begin `bits` / 8 bytes behind `at`, 3 at most: the words are shifted, the last one runs into the next lane's first.
// prev: the word in front of the lane's.
template <int Q, int o, int kWords>
__device__ __forceinline__ void stage_words_shifted(uint8_t *at, const uint32_t (&R)[4][kWords], uint32_t prev, uint32_t bits)
{
    if constexpr (o < Q) {
        constexpr int step = Q % 4 == 0 ? 4 : (Q % 2 == 0 ? 2 : 1);
        const uint32_t a = joined<Q, o>(R);
        if constexpr (step == 4) {
            const uint32_t b = joined<Q, o + 1>(R), c = joined<Q, o + 2>(R), d = joined<Q, o + 3>(R);
            *reinterpret_cast<uint4 *>(at + 4 * o) = make_uint4(__funnelshift_l(prev, a, bits), __funnelshift_l(a, b, bits),
                                                                __funnelshift_l(b, c, bits), __funnelshift_l(c, d, bits));
            stage_words_shifted<Q, o + 4>(at, R, d, bits);
        } else if constexpr (step == 2) {
            const uint32_t b = joined<Q, o + 1>(R);
            *reinterpret_cast<uint2 *>(at + 4 * o) = make_uint2(__funnelshift_l(prev, a, bits), __funnelshift_l(a, b, bits));
            stage_words_shifted<Q, o + 2>(at, R, b, bits);
        } else {
            *reinterpret_cast<uint32_t *>(at + 4 * o) = __funnelshift_l(prev, a, bits);
            stage_words_shifted<Q, o + 1>(at, R, a, bits);
        }
    }
}

// How the rows of a run lie in memory, and the words that a lane hands on.  Where q is 8 (mod 16) rows begin at one of two places of a 16-byte group, so up to 7 bytes of
// shift are left, else 3 (quad_shift()).
template <int Q>
struct Shifted {
    static constexpr int kCarry = Q % 8 == 0 ? 2 : 1;
    uint32_t bytes;                                    // by which the run's first row is off a 16-byte group
    uint32_t carry[kCarry];                            // the last words of the 128 ranks before, the last one first
};

template <int Q, int o, int kWords>
__device__ __forceinline__ void join_words(const uint32_t (&R)[4][kWords], uint32_t (&V)[Q + 2])
{
    if constexpr (o < Q) {
        V[o + 2] = joined<Q, o>(R);
        join_words<Q, o + 1>(R, V);
    }
}

template <int Q, int kWords>
__device__ __forceinline__ void stage_shifted(uint8_t *at, const uint32_t (&R)[4][kWords], Shifted<Q> &sh)
{
    const uint32_t lane = threadIdx.x & 31u;
    if constexpr (Q % 8 == 0) {
        static_assert(Q % 16 != 0, "7 bytes of shift at most");
        uint32_t V[Q + 2];                             // V[w + 2]: word w
        join_words<Q, 0>(R, V);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const uint32_t before = __shfl_up_sync(0xffffffffu, V[Q + 1 - j], 1);
            V[1 - j] = lane ? before : sh.carry[j];
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) sh.carry[j] = __shfl_sync(0xffffffffu, V[Q + 1 - j], 31);
        const uint32_t bits = 8u * (sh.bytes & 3u);
#pragma unroll
        for (int w = Q + 1; w > 0; --w) V[w] = __funnelshift_l(V[w - 1], V[w], bits);
        if (sh.bytes & 4u) {
#pragma unroll
            for (int w = Q + 1; w > 1; --w) V[w] = V[w - 1];
        }
#pragma unroll
        for (int w = 0; w < Q; w += 4) *reinterpret_cast<uint4 *>(at + 4 * w) = make_uint4(V[w + 2], V[w + 3], V[w + 4], V[w + 5]);
    } else {
        const uint32_t last = joined<Q, Q - 1>(R), before = __shfl_up_sync(0xffffffffu, last, 1);
        stage_words_shifted<Q, 0>(at, R, lane ? before : sh.carry[0], 8u * sh.bytes);
        sh.carry[0] = __shfl_sync(0xffffffffu, last, 31);
    }
}

// What the rows of the last lane leave for the 16 bytes behind them.
template <int Q>
__device__ __forceinline__ void stage_rest(uint8_t *at, const Shifted<Q> &sh)
{
    if ((threadIdx.x & 31u) != 0u || sh.bytes == 0u) return;
    if constexpr (Q % 8 == 0) {
        const uint32_t bits = 8u * (sh.bytes & 3u);
        const uint32_t one = __funnelshift_l(sh.carry[1], sh.carry[0], bits), two = __funnelshift_l(sh.carry[0], 0u, bits);
        *reinterpret_cast<uint2 *>(at) = sh.bytes & 4u ? make_uint2(one, two) : make_uint2(two, 0u);
    } else {
        *reinterpret_cast<uint32_t *>(at) = __funnelshift_l(sh.carry[0], 0u, 8u * sh.bytes);
    }
}

// Of 16 consecutive ranks of a p whose rows begin at byte `entry`, one whose row begins the least behind a 16-byte boundary: 0 bytes for odd q, 1 at most
// for q = 2 (mod 4), 3 for 4 (mod 8), 7 for 8 (mod 16).  Returns rank + 16 bytes.  By a warp.
__device__ __forceinline__ uint32_t quad_shift(uint64_t entry, int q)
{
    const uint32_t rank = threadIdx.x & 15u;
    return __reduce_min_sync(0xffffffffu, (((uint32_t)entry + rank * (uint32_t)q) & 15u) << 4 | rank);
}

// What a look-up leaves about four ranks for the rows that are made from them.
struct QuadState {
    uint32_t slot;         // segment of the first of them
    int room;              // how many are in that segment, 4 or more if all
    uint32_t here, next;   // Segment::recv of that segment and of the one behind
    uint32_t bases;        // baseblocks, a byte each
};

// Stages four rows at `at`: words 0 and 1 from the rounds below L (eight bytes a row, the last one the baseblock), the others from the entries of
// their segment and of the next one; in the home round (kSend: in all rounds behind it) the baseblock.
template <int Q, bool kSend, bool kAligned>
__device__ __forceinline__ void stage_quad(uint8_t *at, const uint32_t (&lo)[4], const uint32_t (&hi)[4], const uint8_t *entries, const QuadState &s,
                                           Shifted<Q> &shifted)
{
    constexpr int kWords = (Q + 3) / 4;
    // The baseblock's bytes: of nearly all ranks in the last two words, of those below some 2^(q - 5) anywhere.  (Small q have no other words.)
    constexpr bool kAnywhere = 4 * (kWords - 2) > kLow;
    uint32_t R[4][kWords], S[8];
    auto load = [&](uint32_t (&X)[8], const uint8_t *from) {
        const uint4 a = *reinterpret_cast<const uint4 *>(from);
        X[0] = a.x;
        X[1] = a.y;
        X[2] = a.z;
        X[3] = a.w;
        if constexpr (kWords > 6) {
            const uint4 b = *reinterpret_cast<const uint4 *>(from + 16);
            X[4] = b.x;
            X[5] = b.y;
            X[6] = b.z;
            X[7] = b.w;
        } else if constexpr (kWords > 5) {
            const uint2 b = *reinterpret_cast<const uint2 *>(from + 16);
            X[4] = b.x;
            X[5] = b.y;
        } else if constexpr (kWords > 4) {
            X[4] = *reinterpret_cast<const uint32_t *>(from + 16);
        }
    };
    const uint8_t *from = entries + s.slot * 64u + (kSend ? 32u : 0u);
    uint32_t picks_of[4];
    auto pick = [&](int i) {
        R[i][kWords - 2] = __byte_perm(R[i][kWords - 2], hi[i], picks_of[i]);
        R[i][kWords - 1] = __byte_perm(R[i][kWords - 1], hi[i], picks_of[i] >> 16);
    };
    if constexpr (Q % 8 != 0) {
        // (loaded once more for each rank rather than selected, word by word, from those of two segments: the integer pipe has more to do than shared
        // memory, 1.06 million ranks of q = 21 0.2 us less, of about 10; but q = 24, whose rows meet in banks, 12 million ranks 88.4 -> 91.4)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            load(S, i == 0 || i < s.room ? from : from + 64);
            picks_of[i] = S[0];
            R[i][0] = lo[i];
            R[i][1] = (hi[i] & 0xffffffu) | S[1];
#pragma unroll
            for (int w = 2; w < kWords; ++w) R[i][w] = S[w];
            if constexpr (!kAnywhere) pick(i);                   // (here, or the kernel of eight CTAs per SM spills)
        }
    } else {
        uint32_t T[8];
        load(S, from);
#pragma unroll
        for (int w = 0; w < 8; ++w) T[w] = S[w];
        if (s.room < 4) load(T, from + 64);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const bool mine = i == 0 || i < s.room;
            R[i][0] = lo[i];
            picks_of[i] = mine ? S[0] : T[0];
            R[i][1] = (hi[i] & 0xffffffu) | (mine ? S[1] : T[1]);
#pragma unroll
            for (int w = 2; w < kWords; ++w) R[i][w] = mine ? S[w] : T[w];
            if constexpr (!kAnywhere) pick(i);
        }
    }
    if constexpr (!kAnywhere) {
    } else if (!__any_sync(0xffffffffu, ((s.here | (s.room < 4 ? s.next : 0u)) >> 15) & 1u)) {
#pragma unroll
        for (int i = 0; i < 4; ++i) pick(i);
    } else {
        // They are the zero bytes of the entries (all others are negative): look at those of the last four words, and of the words before where a home round
        // is among them (or none there, the root's segment).  Two instructions a word and rank; a selector for each word from the home rounds of both segments
        // took five: a million ranks from 0 on, q = 27, 29, 31: 12.2, 12.8, 12.8 -> 10.8, 11.4, 11.0 us.
        constexpr int kFirst = kWords > 5 ? kWords - 4 : 1;
        auto fill = [&](int i, int w) {                          // (word 1: round L, the others are from the table)
            const uint32_t others = w == 1 ? sign_bytes<0xb444>(R[i][w], 0xffffffffu) : sign_bytes<0xba98>(R[i][w], 0u);
            R[i][w] |= __byte_perm(hi[i], 0u, 0x3333) & ~others;
        };
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int w = kFirst; w < kWords; ++w) fill(i, w);
        if constexpr (kFirst > 1) {
            const uint32_t here = (s.here >> 10) & 31u, next = s.room < 4 ? (s.next >> 10) & 31u : here;
            if (__any_sync(0xffffffffu, (here < next ? here : next) < 4u * kFirst)) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int w = 1; w < kFirst; ++w) fill(i, w);
            }
        }
    }
    if constexpr (kAligned) stage_words<Q, 0>(at, R);
    else stage_shifted<Q>(at, R, shifted);
}

// Receive and send rows (either pointer may be null) of the n ranks x0, x0 + 1, ... (mod p; x0 < p, n <= the run of `at`, n <= p) by one warp.
// recv, send: where the row of x0 goes: kAligned, on a 16-byte boundary; else `bytes` behind one (quad_shift()), and the first `lead` ranks are not written.
// mine: the warp's shared memory; skips: those of p.  kTable: send rows from their table, at send_rows.
template <int Q, bool kTable, bool kAligned>
__device__ __forceinline__ void quad_run(const RowTable &t, const uint8_t *send_rows, uint8_t *mine, const QuadLayout<kTable> &at, const uint32_t *skips,
                                         uint32_t odd, uint32_t inv, uint32_t x0, uint32_t n, uint32_t lead, uint32_t shift,
                                         int8_t *recv, int8_t *send)
{
    const uint32_t lane = threadIdx.x & 31u;
    Segment *segments = reinterpret_cast<Segment *>(mine);
    uint8_t *entries = mine + at.entries, *columns = mine + at.columns, *staged = mine + at.stage;
    uint8_t *own = staged + lane * (4u * Q), *stage = staged + (kAligned ? 0u : shift);       // the lane's words, the first row
    const uint8_t *table = reinterpret_cast<const uint8_t *>(t.rows);
    const int starts = locate_run<Q, kTable>(t, segments, entries, odd, inv, x0, n, at.segments);

    for (uint32_t b = 0; b < n; b += kPass) {
        const uint32_t ranks = n - b < kPass ? n - b : kPass, bytes = ranks * Q;
        const uint32_t turns = ranks > kQuads ? 2u : 1u;
        // segments of the pass: from slot0 on, those that start in front of its end; four lanes each for their exceptions
        const uint32_t slot0 = __popc(__ballot_sync(0xffffffffu, starts <= (int)b)) - 1u;
        const uint32_t slots = __popc(__ballot_sync(0xffffffffu, starts < (int)(b + ranks)));
        const uint32_t slot = slot0 + (lane >> 2), low0 = lane & 3u;

        // Segments of the 128 ranks from rank `from` on.
        auto find = [&](uint32_t from, QuadState &s, int2 &keys) {
            const uint32_t first = __popc(__ballot_sync(0xffffffffu, starts <= (int)from)) - 1u;
            // the first lane whose first rank is in that segment (unsigned: the sum may wrap, to something negative, where there is none)
            const int quad = (int)((uint32_t)starts - from + 3u) >> 2;
            const uint32_t begin = __reduce_or_sync(0xffffffffu, quad > 0 && quad < 32 ? 1u << quad : 0u);
            s.slot = first + __popc(begin & ((2u << lane) - 1u));
            const Segment here = segments[s.slot], next = segments[s.slot + 1u];
            const int x = (int)(from + 4u * lane);
            s.room = next.start - x;
            s.here = here.recv;
            s.next = next.recv;
            keys = make_int2(here.key + 8 * x, next.key + 8 * x);
        };
        // Their rows in a table.
        auto look_up = [&](const uint8_t *rows, const QuadState &s, int2 keys, uint32_t (&lo)[4], uint32_t (&hi)[4]) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint2 row = *reinterpret_cast<const uint2 *>(rows + row_at((uint32_t)((i < s.room ? keys.x : keys.y) + 8 * i)));
                lo[i] = row.x;
                hi[i] = row.y;
            }
        };
        // Send rows by their table, or put together where a segment has no group there.
        auto look_up_sends = [&](uint32_t from, const QuadState &s, int2 keys, uint32_t (&lo)[4], uint32_t (&hi)[4]) {
            look_up(send_rows, s, make_int2(keys.x + (((int)s.here >> 6) & ~1023), keys.y + (((int)s.next >> 6) & ~1023)), lo, hi);
            const bool deep = ((segments[s.slot].send | (s.room < 4 ? segments[s.slot + 1u].send : 0u)) >> 22) & 1u;
            if (!__any_sync(0xffffffffu, deep)) return;
            if (!deep) return;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const Segment *seg = segments + s.slot + (i < s.room ? 0u : 1u);
                const int low = (int)(from + 4u * lane) + i - seg->start, len = seg[1].start - seg->start;
                if (((seg->send >> 22) & 1u) == 0u || low >= len) continue;
                const uint32_t own = ((seg[0].recv >> 5) & 31u) * kLowRanks, next = ((seg[1].recv >> 5) & 31u) * kLowRanks;
                uint32_t e[8];
#pragma unroll
                for (int k = 0; k < kLow; ++k) {
                    const int to = low + (int)skips[k];
                    e[k] = table[(to < len ? own + permuted_row((uint32_t)to) : next + permuted_row((uint32_t)(to - len))) * 8u + k];
                }
                e[7] = table[(own + permuted_row((uint32_t)low)) * 8u + 7u];
                lo[i] = e[0] | e[1] << 8 | e[2] << 16 | e[3] << 24;
                hi[i] = e[4] | e[5] << 8 | e[6] << 16 | e[7] << 24;
            }
        };
        // and their columns, of the first `lanes` lanes
        auto put_columns = [&](uint32_t from, uint32_t lanes, QuadState &s, const uint32_t (&lo)[4], const uint32_t (&hi)[4]) {
            uint32_t c[8];
            transpose(lo[0], lo[1], lo[2], lo[3], c[0], c[1], c[2], c[3]);
            transpose(hi[0], hi[1], hi[2], hi[3], c[4], c[5], c[6], c[7]);
            s.bases = c[7];
            if (lane >= lanes) return;
            uint32_t *column = reinterpret_cast<uint32_t *>(columns + from) + lane;
#pragma unroll
            for (int k = 0; k < kLow; ++k) column[k * (int)(kColumn / 4u)] = c[k];
        };
        // Sends the staged rows out.
        auto flush = [&](int8_t *out) {
            fence_before_bulk();
            if (b == 0u) grid_dependency_wait();                 // (the kernel before: not until the first store)
            __syncwarp();
            if constexpr (kAligned) {
                int8_t *dst = out + b * Q;
                if (elect_one() && bytes >= 16u) bulk_store(dst, stage, bytes & ~15u);
                if (ranks != kPass && lane < (bytes & 15u)) dst[(bytes & ~15u) + lane] = (int8_t)stage[(bytes & ~15u) + lane];
            } else {                                             // bytes [begin, end) from a 16-byte boundary on, the ragged ends one by one
                int8_t *dst = out + (int64_t)b * Q - shift;
                const uint32_t begin = shift + (b == 0u ? lead * Q : 0u), end = shift + bytes;
                const uint32_t head = (begin + 15u) & ~15u, tail = end & ~15u;
                if (elect_one() && tail > head) bulk_store(dst + head, staged + head, tail - head);
                const uint32_t stop = head < end ? head : end, rest = tail > head ? tail : stop;
                if (begin + lane < stop) dst[begin + lane] = (int8_t)staged[begin + lane];
                if (rest + lane < end) dst[rest + lane] = (int8_t)staged[rest + lane];
            }
        };

        QuadState states[kTurns];
        int2 keys[kTurns];
        Shifted<Q> shifted = {kAligned ? 0u : shift, {}};
        stage_free<true>();
#pragma unroll
        for (int j = 0; j < kTurns; ++j) {
            if (j != 0 && turns == 1u) break;
            uint32_t lo[4], hi[4];
            find(b + j * kQuads, states[j], keys[j]);
            if (kTable && recv == nullptr) continue;
            look_up(table, states[j], keys[j], lo, hi);
            if (!kTable && send != nullptr) put_columns(j * kQuads, 32u, states[j], lo, hi);
            if (recv != nullptr) stage_quad<Q, false, kAligned>(own + j * (int)(kQuads * Q), lo, hi, entries, states[j], shifted);
        }
        if (!kTable && send != nullptr) {                        // and the ranks behind
            QuadState s;
            int2 k;
            uint32_t lo[4], hi[4];
            find(b + turns * kQuads, s, k);
            look_up(table, s, k, lo, hi);
            put_columns(turns * kQuads, (kHalo + 8u) / 4u, s, lo, hi);
        }
        if (!kAligned && recv != nullptr) stage_rest<Q>(staged + turns * (kQuads * Q), shifted);
        __syncwarp();
        if (recv != nullptr) {
            for (uint32_t j = slot; j < slots; j += 8u) {
                const Segment seg = segments[j];
                const uint32_t behind = seg.recv & 31u, K = (seg.recv >> 5) & 31u;
                for (uint32_t low = low0; low < behind; low += 4u) {
                    const uint32_t row = (uint32_t)seg.start + low - b;
                    if (row >= ranks) continue;
                    uint32_t levels = (odd & ((2u << (kLow + K)) - 1u)) >> (kLow + 2);      // C(k + 1, K) are set from round k = L on
                    uint8_t *e = stage + row * Q + kLow;
                    int block = kLow + 1 - Q;
                    for (; low < (uint32_t)__popc(levels); levels >>= 1, ++block) *e++ = (uint8_t)block;
                    *e = (uint8_t)((int)t.miss[K * kMissRanks + low] - Q);
                }
            }
            flush(recv);
        }
        if (send == nullptr) continue;
        if (recv != nullptr) stage_free<true>();
        if (!kAligned) shifted = {shift, {}};
#pragma unroll
        for (int j = 0; j < kTurns; ++j) {
            if (j != 0 && turns == 1u) break;
            uint32_t lo[4], hi[4];
            if constexpr (kTable) {
                look_up_sends(b + j * kQuads, states[j], keys[j], lo, hi);
            } else {
                const uint8_t *column = columns + j * kQuads + 4u * lane;
                uint32_t c[kLow];
#pragma unroll
                for (int k = 0; k < kLow; ++k) {
                    const uint32_t *w = reinterpret_cast<const uint32_t *>(column + (k * kColumn + (skips[k] & ~3u)));
                    c[k] = __funnelshift_r(w[0], w[1], skips[k] * 8u);
                }
                transpose(c[0], c[1], c[2], c[3], lo[0], lo[1], lo[2], lo[3]);
                transpose(c[4], c[5], c[6], states[j].bases, hi[0], hi[1], hi[2], hi[3]);
            }
            stage_quad<Q, true, kAligned>(own + j * (int)(kQuads * Q), lo, hi, entries, states[j], shifted);
        }
        if (!kAligned) stage_rest<Q>(staged + turns * (kQuads * Q), shifted);
        __syncwarp();
        for (uint32_t j = slot; j < slots; j += 8u) {
            const Segment seg = segments[j];
            const uint32_t before = seg.send & 31u, row0 = (uint32_t)seg.start - b;
            if (((seg.send >> 20) & 3u) != 0u && row0 < ranks) {        // its first rank, or the root
                if ((seg.send >> 20) & 1u) stage[row0 * Q + kLow] = (uint8_t)(seg.send >> 24);
                else for (uint32_t k = kLow + low0; k < (uint32_t)Q; k += 4u) stage[row0 * Q + k] = (uint8_t)k;
            }
            const uint32_t row1 = (uint32_t)segments[j + 1].start - b - before;
            for (uint32_t low = low0; low < before; low += 4u) { // its last ranks
                if (row1 + low >= ranks) continue;
                const uint32_t deeper = (seg.send >> 5) & 31u, k = kLow + ((seg.send >> 10) & 31u), m = (seg.send >> 15) & 31u;
                const uint32_t block = low < deeper ? k + 1u : t.miss[m * kMissRanks + low];
                stage[(row1 + low) * Q + k] = (uint8_t)(block - Q);
            }
        }
        flush(send);
    }
}

}  // namespace bcs
