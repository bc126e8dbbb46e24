"""The rows of a rank from the binary form of its segment, restated with numpy (test infrastructure: the rule that the comment
in front of csrc/rows.cuh states, sharing no code with the kernels or the oracle).

Notation as there: e_t = 2 skips[t-1] - skips[t]; C(a, b) = e_{a+1} + ... + e_b; L = min(7, q); a segment is the run of ranks whose
skip codes agree from bit L up, g that part of the code; K the lowest set bit of g as a level (q if there is none), `low` the
place in the segment, m the lowest zero bit of g as a level.
"""
from __future__ import annotations

import numpy as np

BEHIND, AROUND = 80, 208


def _ctz(v, none):
    v = np.asarray(v, dtype=np.int64)
    low = np.where(v == 0, 1, v & -v)
    return np.where(v == 0, none, np.log2(low.astype(np.float64)).astype(np.int64))


class Form:
    def __init__(self, p: int):
        self.p, self.q = p, max(p - 1, 0).bit_length()
        s = [p]
        for _ in range(self.q):                                  # Algorithm 1
            s.append((s[-1] + 1) // 2)
        self.s = s[::-1]
        self.L = min(7, self.q)
        self.e = [0] + [2 * self.s[t - 1] - self.s[t] for t in range(1, self.q + 1)]
        assert set(self.e) <= {0, 1}
        self.sum = np.concatenate([[0], np.cumsum(self.e)])      # C(a, b) = sum[b+1] - sum[a+1]
        lows = np.arange(self.s[self.L])
        self.codes = np.zeros(len(lows), dtype=np.int64)
        rest = lows.copy()
        for k in range(self.L - 1, -1, -1):
            take = rest >= self.s[k]
            rest = np.where(take, rest - self.s[k], rest)
            self.codes |= take.astype(np.int64) << k
        self.bits = self.codes & -self.codes                     # baseblock, as a bit
        self.rows = {}                                           # K -> rounds below L, baseblock (root: 0), missing block

    def C(self, a, b):
        return self.sum[np.asarray(b) + 1] - self.sum[np.asarray(a) + 1]

    def locate(self, x):
        """(g, low, length) of the ranks x."""
        x = np.asarray(x, dtype=np.int64)
        g, low = np.zeros_like(x), x.copy()
        for k in range(self.q - 1, self.L - 1, -1):
            take = low >= self.s[k]
            low = np.where(take, low - self.s[k], low)
            g |= take.astype(np.int64) << (k - self.L)
        m = self.L + _ctz(~g, 0)
        return g, low, self.s[self.L] - self.C(self.L, m)

    def table(self, K: int):
        """Rows of the ranks of a segment with lowest bit K: Algorithm 4 on the rounds below L, its windows read from the
        baseblocks of the ranks around the segment's start.  Block K is bit 7 (bit K, K < 7)."""
        if K in self.rows:
            return self.rows[K]
        s, q, L = self.s, self.q, self.L
        top = int(s[7] - self.C(7, K)) if K >= 7 else s[K]
        flag = min(K, 7)
        around = np.zeros(BEHIND + AROUND, dtype=np.int64)
        for x in range(-BEHIND, AROUND):
            z = top + x if x < 0 else x
            around[x + BEHIND] = self.bits[z] if 1 <= z < len(self.bits) else 0
        around[BEHIND] = 1 << flag if K < q else 0
        n = len(self.codes)
        low = np.arange(n)

        def window(end, length):                                 # the ranks end .. end + length - 1 below
            got = np.zeros(n, dtype=np.int64)
            for d in range(end, end + length):
                inside = low - d >= -BEHIND
                got |= np.where(inside, around[np.maximum(low - d + BEHIND, 0)], 0)
            return got
        base = np.where(self.codes != 0, _ctz(self.codes, 0), K)
        B = np.where(self.codes != 0, self.bits, (1 << flag) if K < q else 0)
        out = np.zeros((n, max(L, 1)), dtype=np.int64)
        for i in range(min(L, 6)):
            lo, hi, total = s[i], s[i + 1], sum(s[:i + 1])
            U = window(lo, max(hi - lo, 1)) & ~B
            U = np.where(U == 0, (window(hi, total - hi + 1) if total >= hi else 0) & ~B, U)
            above = self.codes >> (i + 1)
            is_set = (self.codes >> i) & 1 == 1
            U = np.where(is_set, np.where(above != 0, (above & -above) << (i + 1), 1 << flag), U)
            home = is_set & (above == 0) & (K == q)
            assert np.all(U != 0)
            blk = np.log2(U.astype(np.float64)).astype(np.int64)
            B = np.where(home, B, B | 1 << blk)
            out[:, i] = np.where(home, base, np.where(blk == 7, K, blk) - q)
        missing = np.full(n, 7)
        if L == 7:
            without = low < s[6]                                 # ranks without bit 6
            m = _ctz(~B, 0)
            seven = (low < self.C(7, K)) | ((m == 6) & (K > 7) & (low < self.C(6, K)))
            six = np.where(without, np.where(seven, 7, m) - q, K - q if K < q else base)
            missing = np.where(seven, m, 7)
            # those with it: rounds 0..5 are the ones of the rank s[6] further down behind bit 6
            if not np.all(without):
                deep = Form.table(self, 6) if K != 6 else None
                if deep is not None:
                    at = low[~without]
                    out[at, :6] = deep[0][at - s[6], :6]
            out[:, 6] = six
        self.rows[K] = out, base if K < q else np.where(self.codes != 0, base, 0), missing
        return self.rows[K]

    def receive(self, x):
        q, L = self.q, self.L
        g, low, _ = self.locate(x)
        K = L + _ctz(g, q - L)
        out = np.zeros((len(g), q), dtype=np.int64)
        for level in np.unique(K):
            at = np.nonzero(K == level)[0]
            rows, base, missing = self.table(int(level))
            out[at, :L] = rows[low[at], :L]
            for k in range(L, q):
                bits = g[at] >> (k - L)
                above = bits >> 1
                nxt = np.where(above != 0, _ctz(above, 0) + k + 1 - q, base[low[at]])
                out[at, k] = np.where(bits & 1, nxt, k - q)
            if level == L:
                continue
            for i in at[low[at] <= self.C(L, level)]:            # close behind the start
                k = L
                while low[i] < self.C(k + 1, level):
                    out[i, k] = k + 1 - q
                    k += 1
                out[i, k] = missing[low[i]] - q
        return out

    def send(self, x):
        q, L, s = self.q, self.L, self.s
        g, low, length = self.locate(x)
        out = np.zeros((len(g), q), dtype=np.int64)
        full = (1 << (q - L)) - 1
        K, K2 = L + _ctz(g, q - L), L + _ctz((g + 1) & full, q - L)
        for i in range(len(g)):
            gi, li, n = int(g[i]), int(low[i]), int(length[i])
            own = self.table(int(K[i]))
            for k in range(L):
                to = li + s[k]
                out[i, k] = own[0][to, k] if to < n else self.table(int(K2[i]))[0][to - n, k]
            for k in range(L, q):
                above = gi >> (k - L + 1)
                if (gi >> (k - L)) & 1:
                    out[i, k] = k - q
                elif above:
                    out[i, k] = (above & -above).bit_length() + k - q
                else:
                    out[i, k] = own[1][li] if gi or li else k
            z = (~gi & (gi + 1)).bit_length() - 1                # lowest zero bit
            if gi & 1 and li == 0:                               # carries into a rank close behind a start
                out[i, L] = self.table(L + z)[2][self.C(L, L + z)] - q
            if gi < full:
                k = L + z
                rest = gi >> (z + 1)
                m = k + (~rest & (rest + 1)).bit_length()
                behind = int(self.C(k, m)) - (n - li)
                if behind >= 0:
                    out[i, k] = (k + 1 if behind < self.C(k + 1, m) else self.table(m)[2][behind]) - q
        return out
