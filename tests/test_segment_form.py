"""The rule by which the kernels compute a row (tests/segment_form.py) gives the oracle's rows, and the bounds that their shared
memory and searches are laid out for hold."""
import numpy as np
import pytest

import oracle
from tests.segment_form import Form


def _compare(p, ranks):
    form = Form(p)
    ranks = np.unique(np.asarray(ranks, dtype=np.int64))
    want = oracle.build_ranks(p, ranks.astype(np.uint32))
    assert np.array_equal(form.receive(ranks), want[0]), p
    assert np.array_equal(form.send(ranks), want[1]), p


def _near(p, rng, count):
    """Ranks around the skips and their sums of two, the ends, and some more."""
    s = oracle.skips(p).tolist()
    heads = s + [s[i] + s[j] for i in range(len(s)) for j in range(max(0, i - 4), i)]
    return [(h + d) % p for h in heads for d in range(-3, 4)] + [int(v) for v in rng.integers(0, p, count)]


@pytest.mark.parametrize("first", range(8))
def test_every_rank_of_small_p(first):
    for p in range(2 + first, 1400, 8):
        _compare(p, np.arange(p))


def test_sampled_ranks_of_larger_p():
    rng = np.random.default_rng(7)
    edges = [(1 << k) + d for k in (10, 13, 16, 20, 23, 28, 30) for d in (-1, 0, 1)] + [65 << 9, (97 << 17) + 5, (1 << 31) - 1]
    for p in edges + [int(2 ** e) for e in rng.uniform(9.5, 31, 60)]:
        _compare(p, _near(p, rng, 150))


def test_bounds_of_the_layout():
    """A segment has 41 ranks or more, the exceptions behind a start are the first 25 of them, and segment floor(x inv / 2^32) is
    the one of rank x or next to it."""
    rng = np.random.default_rng(8)
    for p in [129, 255, 256, 257, (1 << 31) - 1, (1 << 30) + 1, (1 << 23) + 1] + [int(2 ** e) for e in rng.uniform(7.1, 31, 300)]:
        form = Form(p)
        q, L = form.q, form.L
        assert form.C(L, q) <= 24 and form.s[L] - form.C(L, q) >= 41, p
        x = np.array(_near(p, rng, 300), dtype=np.int64)
        inv = (1 << (q - L + 32)) // p
        guess = x * inv >> 32
        g, low, length = form.locate(x)
        assert np.all(np.abs(guess - g) <= 1), p
        assert np.all(low < length) and np.all(length >= 41), p


def test_segments_that_a_run_touches():
    """r consecutive ranks, also those that go on at 0 behind p - 1, touch (r + 22) / 64 + 2 segments at most: what the warps' shared memory is laid out for."""
    rng = np.random.default_rng(9)
    most = {}
    for p in [129, 130, 255, 256, 257, 511, 513, 1023, 1024, (1 << 16) + 1, (1 << 17) - 1, (1 << 20) + 1, 65 << 9] + [int(2 ** e) for e in rng.uniform(7.1, 20, 120)]:
        form = Form(p)
        x = np.arange(p)
        starts = x[form.locate(x)[1] == 0]
        starts = np.concatenate([starts + turn * p for turn in range(20 if p < 1100 else 2)])
        for r in (128, 192, 384, 512, 640, 1024):
            begin = starts[1:len(starts) // 2] - 1                   # (the last rank of a segment: as many as can be)
            touched = np.searchsorted(starts, begin + r) - np.arange(len(begin))
            most[r] = max(most.get(r, 0), int(touched.max()))
    for p in [(1 << 31) - 1, (1 << 30) + 1, (1 << 25) - 1] + [int(2 ** e) for e in rng.uniform(20, 31, 60)]:
        form = Form(p)
        for head in form.s[8:form.q + 1]:
            for r in (384, 1024):
                x = (np.arange(int(head) - r, int(head) + r)) % p
                new = np.concatenate([[0], np.cumsum(form.locate(x)[1][1:] == 0)])
                most[r] = max(most[r], int((new[r - 1:] - new[:len(new) - r + 1]).max()) + 1)
    assert all(n <= (r + 22) // 64 + 2 for r, n in most.items()), most


def test_rows_wanted_for_a_stretch():
    """The kernels that build table rows for a stretch of ranks only name all that these need: the segments' own lowest bits, those of
    the segments behind them, and where the send exceptions carry to."""
    rng = np.random.default_rng(10)
    for p in [129, 257, 1000, (1 << 14) + 1, (1 << 21) - 1, (1 << 23) + 1, (1 << 31) - 1] + [int(2 ** e) for e in rng.uniform(7.1, 31, 200)]:
        form = Form(p)
        high, inv = form.q - form.L, (1 << (form.q - form.L + 32)) // p
        tz = lambda v: high if v == 0 else (v & -v).bit_length() - 1
        for _ in range(8):
            x0, n = int(rng.integers(0, p)), min(p, int(2 ** rng.uniform(0, 15)))
            start = max((x0 * inv >> 32) - 1, 0)
            named = 0
            for g in range(start, start + (n * inv >> 32) + 7):
                g &= (1 << high) - 1
                z = tz(~g & (1 << high) - 1)
                named |= 1 << tz(g) | 1 << z
                if z < high:
                    named |= 1 << z + 1 + tz(~(g >> z + 1) & (1 << high) - 1)
            g = np.unique(form.locate(np.arange(x0, x0 + n) % p)[0]).tolist()
            for v in g:
                z = tz(~v & (1 << high) - 1)
                need = 1 << tz(v) | 1 << tz(v + 1 & (1 << high) - 1)
                if z < high:                                     # the next zero bit, a segment that the last ranks carry to
                    need |= 1 << tz((v + 1 + (1 << z)) & (1 << high) - 1)
                assert need & ~named == 0, (p, x0, n, v)
