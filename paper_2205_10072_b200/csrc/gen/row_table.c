/* Writes the rows of the row table (csrc/rows.cuh) for every shape of segment as initialisers of arrays, for build_ext.py.
 *
 * The entries of the rounds 0..6 of a rank depend on its place `low` in its segment, on skips[7] (65..128, which gives the skips below
 * it), and on the segment's lowest set bit K by way of three things: the number c = C(7, K) of halvings that rounded up between 7 and
 * K, whether K is 7, and whether it is the root's segment (K = q).  The rounds 0..5 in which the rank's skip code has no bit are
 * computed here by Algorithm 4 (arXiv 2205.10072) as it is written: windows of baseblocks, the largest new one.  Where the code has the bit,
 * and in round 6, it is the closed form of csrc/rows.cuh: the next higher bit, or the block that is left, with the exceptions behind a
 * segment's start.  Baseblock K stands for itself as 8.
 *
 * A row is 8 bytes.  Rounds 0..6: the block, 8 for K, 16 + the block where it is the rank's own (the home round, entry without
 * - q).  Byte 7: baseblock (8 for K, 0 for the root) in bits 0..3, and in bits 5..7 the block of 0..7 that is not taken before round 7.
 *   row_shapes[s7 - 65][shape][low < 64]: ranks without bit 6 (low < skips[6])
 *   row_six[s7 - 65][low]: rounds 0..5 and the baseblock of the ranks skips[6] + low
 *   row_small[p (p - 1) / 2 + rank]: all rounds of p <= 64, 7 rounds at most; byte 7: the baseblock, 8 for the root
 */
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

enum { BEHIND = 160, MOST = 400 };

static int s[9], e7;

static void skips_of(int top, int q)
{
    s[q] = top;
    for (int k = q - 1; k >= 0; --k) s[k] = (s[k + 1] + 1) / 2;
}

/* greedy sum of x over the skips below `levels` */
static int code_of(int x, int levels)
{
    int c = 0;
    for (int k = levels - 1; k >= 0; --k)
        if (x >= s[k]) {
            x -= s[k];
            c |= 1 << k;
        }
    return c;
}

static int lowest(int v) { return v ? __builtin_ctz((unsigned)v) : -1; }

/* Rounds 0 .. n-1 of the rank `low` with the given code; around[BEHIND + x]: baseblock of the rank x behind the segment's start as a
 * bit.  own: the segment's lowest bit, which is the baseblock of a rank without bits (-1: the root); root: the home round is in here.
 * Returns the blocks taken. */
static int rounds(const int *around, int low, int code, int n, int own, int root, uint8_t *row)
{
    int taken = code ? code & -code : (own >= 0 ? 1 << own : 0);
    int sum = 0;
    for (int i = 0; i < n; ++i) {
        sum += s[i];
        int above = code >> (i + 1), set = (code >> i) & 1;
        if (root && set && above == 0) {
            row[i] = (uint8_t)(16 + lowest(code));
            continue;
        }
        int u = 0;
        if (set) {
            u = above ? (above & -above) << (i + 1) : 1 << own;
        } else {
            for (int d = s[i]; d < s[i + 1]; ++d) u |= around[BEHIND + low - d];
            u &= ~taken;
            if (u == 0)
                for (int d = s[i + 1]; d <= sum; ++d) u |= around[BEHIND + low - d];
            u &= ~taken;
        }
        if (u == 0) {
            fprintf(stderr, "no block: skips[7] %d, rank %d, round %d\n", s[7], low, i);
            exit(1);
        }
        int block = 31 - __builtin_clz((unsigned)u);
        taken |= 1 << block;
        row[i] = (uint8_t)block;
    }
    return taken;
}

static void print_row(const uint8_t *row)
{
    uint64_t v = 0;
    for (int i = 7; i >= 0; --i) v = v << 8 | row[i];
    printf("0x%llxull,", (unsigned long long)v);
}

/* around a segment's start: the segment before ends with the ranks below `top`, behind the start the ranks of a first segment */
static void surround(int *around, int lows, int levels, int top, int own)
{
    memset(around, 0, sizeof(int) * MOST);
    for (int x = -BEHIND; x < lows; ++x) {
        int z = x < 0 ? top + x : x;
        int c = z >= 1 && z < lows ? code_of(z, levels) : 0;
        around[BEHIND + x] = c & -c;
    }
    if (own >= 0) around[BEHIND] = 1 << own;
}

int main(void)
{
    int around[MOST];
    printf("static __device__ const unsigned long long row_shapes[64 * 52 * 64] = {\n");
    for (int s7 = 65; s7 <= 128; ++s7) {
        skips_of(s7, 7);
        e7 = 2 * s[6] - s7;
        for (int shape = 0; shape < 52; ++shape) {
            int root = shape >= 26, c = shape % 26 ? shape % 26 - 1 : 0, seven_itself = shape % 26 == 0;
            surround(around, s7, 7, s7 - c, root ? -1 : 8);
            for (int low = 0; low < 64; ++low) {
                uint8_t row[8] = {0};
                if (low < s[6]) {
                    int code = code_of(low, 7);
                    int taken = rounds(around, low, code, 6, root ? -1 : 8, root, row);
                    int m = lowest(~taken & 0x7f);                        /* the block of 0..6 not taken so far */
                    if (m < 0) m = 7;
                    int ahead = low < c || (m == 6 && !seven_itself && low < e7 + c);
                    row[6] = (uint8_t)(ahead ? 7 : m);
                    row[7] = (uint8_t)((code ? lowest(code) : (root ? 0 : 8)) | (ahead ? m : 7) << 5);
                }
                print_row(row);
            }
            printf("\n");
        }
    }
    printf("};\nstatic __device__ const unsigned long long row_six[64 * 64] = {\n");
    for (int s7 = 65; s7 <= 128; ++s7) {
        skips_of(s7, 7);
        surround(around, s7, 7, s[6], 6);                                 /* a segment whose lowest bit is 6 */
        for (int low = 0; low < 64; ++low) {
            uint8_t row[8] = {0};
            if (low < s[6]) {
                int code = code_of(low, 6);
                rounds(around, low, code, 6, 6, 0, row);
                row[7] = (uint8_t)(code ? lowest(code) : 6);
            }
            print_row(row);
        }
        printf("\n");
    }
    printf("};\nstatic __device__ const unsigned long long row_small[64 * 65 / 2] = {\n");
    for (int p = 1; p <= 64; ++p) {
        int q = 0;
        while (1 << q < p) ++q;
        skips_of(p, q);
        s[q + 1] = 0;
        surround(around, p, q, p, -1);
        for (int r = 0; r < p; ++r) {
            uint8_t row[8] = {0};
            int code = code_of(r, q);
            rounds(around, r, code, q, -1, 1, row);
            row[7] = (uint8_t)(code ? lowest(code) : 8);
            print_row(row);
        }
        printf("\n");
    }
    printf("};\n");
    return 0;
}
