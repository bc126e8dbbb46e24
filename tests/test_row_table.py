"""The constants that the row kernels include (written by csrc/gen/row_table.c when the library is built), unpacked as the kernels
do it, are the rows of the rule restated in tests/segment_form.py and, for the smallest p, of the oracle."""
import re

import numpy as np
import pytest

import oracle
from paper_2205_10072_b200 import build_ext
from tests.segment_form import Form


@pytest.fixture(scope="module")
def packed():
    with open(build_ext.build_row_table()) as f:
        parts = re.split(r"static __device__ const unsigned long long (\w+)", f.read())[1:]
    return {name: np.array([int(v, 16) for v in re.findall(r"0x[0-9a-f]+", body)], dtype=np.uint64).view(np.uint8).reshape(-1, 8).astype(int)
            for name, body in zip(parts[::2], parts[1::2])}


def _unpack(rows, q, K):
    """Entries of the rounds 0..6, baseblock, missing block."""
    block, own = np.where(rows == 8, K, rows & 15), rows >= 16
    base = rows[:, 7] & 15
    return np.where(own, block, block - q)[:, :7], np.where(base == 8, K, base), rows[:, 7] >> 5


def _every_shape():
    """Counts p that between them have segments of every kind: for each skips[7], all halvings above it rounding up, for every q, and none."""
    for s7 in range(65, 129):
        yield s7 << 2
        p = s7
        while p < 1 << 31:
            yield p
            p = 2 * p - 1


def test_rows_of_every_shape(packed):
    shapes = packed["row_shapes"].reshape(64, 52, 64, 8)
    sixes = packed["row_six"].reshape(64, 64, 8)
    seen = set()
    for p in _every_shape():
        form = Form(p)
        q, six, lows = form.q, form.s[6], form.s[7]
        for K in range(7, q + 1):
            shape = (26 if K == q else 0) + (0 if K == 7 else 1 + int(form.C(7, K)))
            if (lows, shape) in seen:
                continue
            seen.add((lows, shape))
            want, base, missing = form.table(K)
            got, bb, miss = _unpack(shapes[lows - 65, shape, :six], q, K)
            assert np.array_equal(got, want[:six]) and np.array_equal(miss, missing[:six]), (p, K)
            if K == q:
                base, bb = base[1:], bb[1:]                      # (the root has none)
            assert np.array_equal(bb, base[:six - (K == q)]), (p, K)
            got, bb, _ = _unpack(sixes[lows - 65, :lows - six], q, K)
            assert np.array_equal(got[:, :6], want[six:, :6]) and np.array_equal(bb, form.table(K)[1][six:]), (p, K)
    assert len(seen) == 64 * 51                                  # 25 kinds of segments and the root's 26 for each skips[7]


def test_rows_of_every_shape_against_the_oracle(packed):
    """The rounds 0..6 of the ranks of one segment of each kind, as the oracle computes them rank by rank."""
    shapes = packed["row_shapes"].reshape(64, 52, 64, 8)
    sixes = packed["row_six"].reshape(64, 64, 8)
    seen = set()
    for p in _every_shape():
        q = (p - 1).bit_length()
        s = oracle.skips(p).tolist()
        odd = [0] + [2 * s[t - 1] - s[t] for t in range(1, q + 1)]
        lows, six, ranks, kinds = s[7], s[6], [], []
        for K in range(7, q + 1):
            shape = (26 if K == q else 0) + (0 if K == 7 else 1 + sum(odd[8:K + 1]))
            if (lows, shape) in seen:
                continue
            seen.add((lows, shape))
            # the segment of the rank skips[K] (rank 0) ends where the next one starts: bit 7 is clear unless K = 7
            n = lows - (sum(odd[8:9]) if K == 7 and q > 7 else 0)
            kinds.append((K, shape, n))
            ranks += [(0 if K == q else s[K]) + low for low in range(n)]
        got = oracle.build_ranks(p, np.array(ranks, dtype=np.uint32))[0][:, :7]
        for K, shape, n in kinds:
            rows, got = got[:n], got[n:]
            want = _unpack(shapes[lows - 65, shape, :six], q, K)[0]
            assert np.array_equal(rows[:six], want), (p, K)
            want = _unpack(sixes[lows - 65, :n - six], q, K)[0][:, :6]
            assert np.array_equal(rows[six:, :6], want), (p, K)
    assert len(seen) == 64 * 51


def test_rows_of_small_p(packed):
    rows = packed["row_small"]
    for p in range(2, 65):
        q = Form(p).q
        got, _, _ = _unpack(rows[p * (p - 1) // 2:p * (p + 1) // 2], q, 0)
        assert np.array_equal(got[:, :q], oracle.full_table(p)[0]), p


def test_a_failed_generator_leaves_nothing_behind(tmp_path, monkeypatch):
    """The constants as they were, and no part of others beside them."""
    import os
    import subprocess
    compiler = tmp_path / "cc"
    compiler.write_text('#!/bin/sh\nfor a; do [ "$was" = -o ] && out=$a; was=$a; done\n'
                        'printf "#!/bin/sh\\necho half of it\\nexit 3\\n" > "$out"; chmod +x "$out"\n')
    compiler.chmod(0o755)
    monkeypatch.setattr(build_ext, "ROW_TABLE", str(tmp_path / "row_table.inc"))
    (tmp_path / "row_table.inc").write_text("as it was")
    monkeypatch.setenv("CC", str(compiler))
    with pytest.raises(subprocess.CalledProcessError):
        build_ext.build_row_table(force=True)
    assert sorted(os.listdir(tmp_path)) == ["cc", "row_table.inc"]
    assert (tmp_path / "row_table.inc").read_text() == "as it was"
