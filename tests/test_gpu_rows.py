"""Rows of a range straight from the binary form of its ranks, where that construction can go wrong: the ends of
items and tiles, segments next to heads of every depth, the exceptions behind a segment's start, counts
whose halvings all round up or never do.  Whole numbers, compared with the CPU oracle entry by entry."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bcs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2205_10072_b200 as lib
    lib.lib()
    torch.cuda.set_device(0)
    return lib


def _buffer(n):
    raw = torch.full((n + 64,), 99, dtype=torch.int8, device="cuda")
    return raw, raw[32:32 + n]


def _check(bcs, p, r0, r1, recv=True, send=True):
    q, n = bcs.bcs_q(p), r1 - r0
    raw_r, out_r = _buffer(n * q)
    raw_s, out_s = _buffer(n * q)
    bcs.bcs_build(p, r0, r1, out_r if recv else None, out_s if send else None)
    torch.cuda.synchronize()
    # at most 3000 ranks of a long range: both ends, and some between
    at = np.arange(n) if n <= 3000 else np.unique(np.concatenate([
        np.arange(700), n - 1 - np.arange(700), np.random.default_rng(p).integers(0, n, 1500)]))
    want = oracle.build_ranks(p, (at + r0).astype(np.uint32))
    rows = torch.from_numpy(at).cuda()
    for raw, out, asked, expect in ((raw_r, out_r, recv, want[0]), (raw_s, out_s, send, want[1])):
        if asked:
            got = out.view(n, q)[rows].cpu().numpy()
            bad = np.argwhere(got != expect)
            assert bad.size == 0, (p, r0, r1, "rank %d entry %d" % (at[bad[0][0]] + r0, bad[0][1]))
            assert bool((raw[:32] == 99).all()) and bool((raw[32 + n * q:] == 99).all()), (p, r0, r1)
        else:
            assert bool((raw == 99).all())


# counts with skips[7] = 65 and 128, all halvings above it rounding up, or none
EDGES = [2, 3, 5, 63, 64, 65, 100, 127, 128, 129, 130, 255, 256, 257, 65 << 9, (64 << 9) + 1, (1 << 16) + 1, 1 << 16,
         (1 << 20) + 1, (1 << 23) - 1, (1 << 23) + 1, 100 << 13, (97 << 17) + 5, (1 << 28) + 1, (1 << 30) - 1,
         (1 << 30) + 20, (1 << 31) - 1]


@pytest.mark.parametrize("p", EDGES)
def test_rows_of_ranges(bcs, p):
    s = bcs.bcs_skips(p)
    q = len(s) - 1
    starts = {0, max(p - 300, 0)} | {max(s[k] - 150, 0) for k in (q, q - 1, q - 2, q // 2 + 1) if 0 <= k <= q}
    starts |= {max(s[q - 1] + (s[q - 3] if q > 3 else 0) - 64, 0)}
    for i, r0 in enumerate(sorted(starts)):
        n = min((1, 31, 33, 127, 129, 300, 700)[i % 7], p - r0)
        _check(bcs, p, r0, r0 + n, recv=i % 4 != 1, send=i % 4 != 2)
        _check(bcs, p, r0, min(r0 + 700, p))


@pytest.mark.parametrize("n", [98303, 98304, 1 << 20, (1 << 20) + 1, 148 * 32 * 32 - 1, 148 * 32 * 32 + 1, 148 * 32 * 64, 148 * 32 * 128 + 77])
@pytest.mark.parametrize("p", [(1 << 20) + 1, 3000017, (1 << 22) + 1, 40000003])
def test_rows_where_the_split_changes(bcs, p, n):
    r0 = 1234567 % (p - n + 1)
    _check(bcs, p, r0, r0 + n)


# one table alone, at the line between a rank and four ranks per lane
@pytest.mark.parametrize("n", [148 * 16 * 32, 148 * 16 * 32 + 1, 90001])
@pytest.mark.parametrize("p", [148 * 16 * 32 + 15000, (1 << 20) + 1, (1 << 23) - 1, 40000003])
def test_rows_of_one_table_where_the_split_changes(bcs, p, n):
    r0 = 1234567 % (p - n + 1)
    _check(bcs, p, r0, r0 + n, send=False)
    _check(bcs, p, r0, r0 + n, recv=False)


# four ranks per lane for multiples of 2, 4 and 8 and odd q, runs that end inside a look-up (steps of 16 to 32 ranks, by vectors: the batches below)
@pytest.mark.parametrize("p,r0,n", [(140001, 0, 140001), (262144, 100000, 98311), (600011, 0, 600011), (1 << 20, 777, 98304 + 24),
                                    ((1 << 23) + 1, (1 << 22) + 12345, 100001), (1 << 24, (1 << 23) - 200000, 400009)])
def test_rows_of_other_steps(bcs, p, r0, n):
    _check(bcs, p, r0, r0 + n)


# each q that the tests above leave out, skips that are all odd but the first ones or all even or neither, from an odd rank on, with runs of one or two look-ups per
# warp and of more
@pytest.mark.parametrize("p", [(1 << q - 1) + 1 for q in (23, 24, 25, 26, 27, 28, 29)] + [(1 << q) - 1 for q in (23, 25, 26, 27, 28, 29)] +
                              [(3 << q - 2) + 12345 for q in (23, 24, 25, 26, 27, 28, 29)])
def test_wide_rows_of_every_q(bcs, p):
    for n in (151553, (1 << 20) + 77):
        for r0 in ((p - n) // 2 | 1, p - n):
            _check(bcs, p, r0, r0 + n)


# turns that CTAs take from one another, send rows by their table
@pytest.mark.parametrize("p,r0,n", [((1 << 23) + 1, 0, (1 << 23) + 1), (100 << 17, 4000003, (1 << 23) + 385),
                                    ((1 << 24) - 1, 0, (1 << 24) - 1), ((1 << 30) + 20, (1 << 29) - 777777, (1 << 23) + 1),
                                    ((1 << 31) - 1, (1 << 31) - 1 - (1 << 23) - 15, (1 << 23) + 15)])
def test_rows_of_many_ranks(bcs, p, r0, n):
    _check(bcs, p, r0, r0 + n, send=False)
    _check(bcs, p, r0, r0 + n, recv=False)
    q = bcs.bcs_q(p)
    recv = torch.empty(n * q, dtype=torch.int8, device="cuda")
    send = torch.empty(n * q, dtype=torch.int8, device="cuda")
    bcs.bcs_build(p, r0, r0 + n, recv, send)
    counts = torch.ones(3, dtype=torch.int64, device="cuda")
    bcs.bcs_validate(p, r0, r0 + n, recv, send, counts)      # every row and every pair inside the range
    assert counts.tolist() == [0, 0, 0]


def test_many_ranks_rooted(bcs):
    p, root = (1 << 23) + 12345, 5000001                       # the ranks pass p - 1 inside an item
    q = bcs.bcs_q(p)
    recv = torch.empty(p * q, dtype=torch.int8, device="cuda")
    send = torch.empty(p * q, dtype=torch.int8, device="cuda")
    ws = torch.empty(bcs.bcs_build_rooted_workspace_bytes(p, root, 0, p), dtype=torch.int8, device="cuda")
    bcs.bcs_build_rooted(p, root, 0, p, recv, send, ws)
    at = np.concatenate([np.arange(600), root - 600 + np.arange(1200), p - 1 - np.arange(600)])
    want = oracle.build_ranks(p, ((at - root) % p).astype(np.uint32))
    rows = torch.from_numpy(at).cuda()
    for out, expect in ((recv, want[0]), (send, want[1])):
        assert np.array_equal(out.view(p, q)[rows].cpu().numpy(), expect)


def _batch(bcs, plist, send=True):
    plan = bcs.bcs_batch_plan(plist)
    raw_r, recv = _buffer(plan.total_entries)
    raw_s, out_s = _buffer(plan.total_entries)
    bcs.bcs_build_batch(plan.to("cuda"), recv, out_s if send else None)
    torch.cuda.synchronize()
    assert bool((raw_r[:32] == 99).all()) and bool((raw_r[32 + plan.total_entries:] == 99).all())
    assert bool((raw_s[:32] == 99).all()) and bool((raw_s[32 + plan.total_entries:] == 99).all())
    assert send or bool((raw_s == 99).all())
    tables = {}
    for p, lo, hi in zip(plist, plan.entry_off[:-1].tolist(), plan.entry_off[1:].tolist()):
        if p == 1:
            continue
        q = bcs.bcs_q(p)
        got = [out[lo:hi] for out in ((recv, out_s) if send else (recv,))]
        if p <= 1 << 21:
            if p not in tables:
                tables[p] = [torch.from_numpy(t).cuda().view(-1) for t in oracle.full_table(p)]
            assert all(torch.equal(g, w) for g, w in zip(got, tables[p])), p
            continue
        # ranks around every skip, the ends and some more; the properties and pairs of all ranks
        near = [s + d for s in bcs.bcs_skips(p) for d in range(-40, 41)]
        at = np.unique(np.array(near + np.random.default_rng(p).integers(0, p, 2000).tolist()) % p)
        rows = torch.from_numpy(at).cuda()
        for g, w in zip(got, oracle.build_ranks(p, at.astype(np.uint32))):
            assert np.array_equal(g.view(p, q)[rows].cpu().numpy(), w), p
        counts = torch.ones(3, dtype=torch.int64, device="cuda")
        bcs.bcs_validate(p, 0, p, got[0].clone(), got[1].clone() if send else None, counts)
        assert counts.tolist() == [0, 0, 0], p


# the sizes at which a batch changes kernels and row forms (1024, 2^15, 2^21), tables that start at any byte, shares that
# end inside a p, lists of one p
@pytest.mark.parametrize("plist", [[1024, 1025, 3, 32768, 1, 32769, 65537, 1023, 40001, 2, 65535],
                                   [(1 << 21) + 1, 5, (1 << 21), 1, (1 << 21) - 1, 77, (1 << 22) + 5],
                                   [33333], [65536, 140001, 600011, 1 << 20], [1], [2, 1], [(1 << 20) + 1] * 3, [1025] * 40, [127, 128, 129, 130] * 30])
@pytest.mark.parametrize("send", [True, False])
def test_batches(bcs, plist, send):
    _batch(bcs, plist, send)


# lists of small p that are spread over the SMs or not, with CTAs of 256 and of 128 threads; a share per CTA or several
@pytest.mark.parametrize("plist", [range(500, 560), range(3, 593), range(200, 940), range(200, 941), range(1, 1025), [777] * 1200,
                                   [1 << 20] * 8, [1 << 20] * 8 + [1025, 9]])
def test_batch_splits(bcs, plist):
    _batch(bcs, list(plist))


# Four ranks per lane for lists of small p: tables that begin at any byte of a 16-byte group (rows of q = 8 at any of its bytes, of q = 10 one byte off, of q = 9
# always on one with some rank), runs of a warp that begin in front of rank 0, in CTAs of 256 threads and of 128
@pytest.mark.parametrize("first", [1, 2, 3, 5, 7, 9, 17, 33])
@pytest.mark.parametrize("times", [3, 40])
def test_batches_of_small_p_at_any_byte(bcs, first, times):
    _batch(bcs, [first] + [1024, 1023, 513, 512, 511, 700, 129, 257, 256, 255, 1000, 130, 641] * times)


# The plan of a batch as the work of the kernel before it on the stream, one that lets its successors start early: the list of p
# is a stretch of a row of allgather tables, block numbers of about `row` each.  Nothing of what its memory held before may
# reach the tables, be it another p of the kernel's range or none.
@pytest.mark.parametrize("n,row,count", [(700, 600, 500), (700, 150, 1000), (3000, 2500, 300), (12000, 10000, 40)])
@pytest.mark.parametrize("old", [0, 1, 1024, 1031, -1])
def test_batch_of_a_plan_written_by_the_kernel_before(bcs, n, row, count, old):
    agents = 1000
    q = bcs.bcs_q(agents)
    tables = oracle.full_table(agents)
    recv, send = (torch.from_numpy(t).cuda().view(-1) for t in tables)
    # processor 0 handles buffer j as virtual processor -j: Algorithm 6's closed form
    virtual = -np.arange(count) % agents
    plist = oracle.expand(agents, n, *tables)[virtual, row, 0].tolist()
    assert min(plist) > 1
    plan = bcs.bcs_batch_plan(plist)
    dev = plan.to("cuda")
    want = [np.concatenate(t) for t in zip(*(tuple(x.reshape(-1) for x in oracle.full_table(p)) for p in plist))]
    pack = torch.empty((n - 1 + q) * agents, dtype=torch.int32, device="cuda")
    busy = torch.empty(1 << 29, dtype=torch.int8, device="cuda")
    dev.p_list = pack[row * agents:row * agents + count]
    for _ in range(4):
        raw_r, out_r = _buffer(plan.total_entries)
        raw_s, out_s = _buffer(plan.total_entries)
        torch.cuda.synchronize()
        busy.zero_()                                             # (all that follows is enqueued while this lasts)
        pack.fill_(old)
        bcs.bcs_allgather_tables(agents, n, 0, recv, send, pack, None)
        bcs.bcs_build_batch(dev, out_r, out_s)
        torch.cuda.synchronize()
        assert dev.p_list.tolist() == plist
        for raw, out, expect in ((raw_r, out_r, want[0]), (raw_s, out_s, want[1])):
            assert np.array_equal(out.cpu().numpy(), expect)
            assert bool((raw[:32] == 99).all()) and bool((raw[32 + plan.total_entries:] == 99).all())


def _back_to_back(bcs, p, n, recv=True, send=True, calls=200):
    """Microseconds a call, calls one behind the other: all are enqueued while the card is busy with something else."""
    q, r0 = bcs.bcs_q(p), min(12345, p - n)
    out_r, out_s = (torch.empty(n * q, dtype=torch.int8, device="cuda") if asked else None for asked in (recv, send))
    busy = torch.empty(1 << 30, dtype=torch.int8, device="cuda")
    begin, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    times = []
    for _ in range(5):
        torch.cuda.synchronize()
        for _ in range(10):
            busy.zero_()
        begin.record()
        for _ in range(calls):
            bcs.bcs_build(p, r0, r0 + n, out_r, out_s)
        end.record()
        torch.cuda.synchronize()
        times.append(begin.elapsed_time(end) * 1000 / calls)
    return min(times)


# Fewer ranks do not take longer because some CTAs of the launch have none: by vectors, 1 000 003 ranks (147 of 148 CTAs had some) took 1.34 times
# as long as 2^20 (all had), receive rows alone 1.33 and send rows 1.21 times, when those CTAs left at once; 0.97 and 1.01 since they waited.  (Four ranks per lane: no CTA is without
# ranks.  Send rows alone of 1.9 million ranks have such CTAs.)
@pytest.mark.parametrize("recv,send", [(True, True), (True, False), (False, True)])
def test_ctas_without_ranks_do_not_hold_up_a_row_of_calls(bcs, recv, send):
    p = 1398101
    assert _back_to_back(bcs, p, 1000003, recv, send) < 1.1 * _back_to_back(bcs, p, 1 << 20, recv, send)


# One table alone does not take much longer where the form changes: 80 000 ranks of q = 21 took 3.5 us (send rows 3.4) by vectors, 75 776 a rank per lane 2.3 (2.7); four ranks per
# lane 1.8 (1.9).
@pytest.mark.parametrize("recv", [True, False])
def test_one_table_keeps_the_faster_form(bcs, recv):
    assert _back_to_back(bcs, 1398101, 80000, recv, not recv) < 1.15 * _back_to_back(bcs, 1398101, 75776, recv, not recv)


@pytest.mark.parametrize("p,n", [((1 << 20) + 1, 148 * 18 * 32), ((1 << 20) + 1, 148 * 18 * 32 + 1), (100001, 148 * 18 * 32),
                                 ((1 << 24) - 1, 148 * 18 * 32 + 1), (40000003, 148 * 17 * 32), (40000003, 148 * 17 * 32 + 1)])
def test_rows_of_one_table_at_the_end_of_pairs(bcs, p, n):
    r0 = 1234567 % (p - n + 1)
    _check(bcs, p, r0, r0 + n, send=False)
    _check(bcs, p, r0, r0 + n, recv=False)


# Four ranks per lane: every q, ranges with one run per warp, longer runs, and turns that CTAs take from one another (with the table of send rows); from
# rank 0 on (home rounds in any word of a row) and to the last one; each table alone, and every row and pair of both.
@pytest.mark.parametrize("q", range(17, 32))
def test_four_ranks_per_lane(bcs, q):
    p = min((3 << q - 2) + 12345, (1 << 31) - 1)
    for i, n in enumerate((148 * 16 * 32 + 1, 148 * 10 * 128 + 1, 148 * 20 * 256 + 129, (1 << 22) + 77)):
        if n > p:
            continue
        for r0 in (0, p - n):
            _check(bcs, p, r0, r0 + n, recv=i % 2 == 0 or r0 == 0, send=i % 2 == 1 or r0 == 0)
        recv, send = (torch.empty(n * q, dtype=torch.int8, device="cuda") for _ in range(2))
        counts = torch.ones(3, dtype=torch.int64, device="cuda")
        bcs.bcs_build(p, p - n, p, recv, send)
        bcs.bcs_validate(p, p - n, p, recv, send, counts)
        assert counts.tolist() == [0, 0, 0], n
    assert bcs.bcs_wait_expired() == 0


# Send rows alone of some million ranks take another kernel: around its lines, runs that end inside the last CTA, steps of 16, 20 and 24 ranks
@pytest.mark.parametrize("n", [1899999, 1900000, 2500001, 5999999, 6000000])
@pytest.mark.parametrize("p", [6000001, (1 << 24) - 5, (1 << 28) - 1, (1 << 31) - 1])
def test_send_rows_alone_of_some_million_ranks(bcs, p, n):
    _check(bcs, p, 0, n, recv=False)
    _check(bcs, p, p - n, p, recv=False)


# A call into tables that the kernel in front of it still reads: the row kernels are launched while that one runs, and wait for it in
# front of their first store, warp by warp; warps and CTAs without ranks need not.  `between`: with a call of one CTA into other
# tables in the middle, which must not be done before the one in front of it is.
@pytest.mark.parametrize("between", [False, True])
@pytest.mark.parametrize("n", [32, 20000, 100003, 700001])
@pytest.mark.parametrize("reader", ["expand", "allgather"])
def test_tables_are_not_written_before_they_are_read(bcs, reader, n, between):
    p, blocks, next_p = 100003, 150, 1398101
    q, next_q = bcs.bcs_q(p), bcs.bcs_q(next_p)
    tables = [torch.from_numpy(t).cuda().view(-1) for t in oracle.full_table(p)]
    size, written = p * q, n * next_q
    at = max(size - written, 0) // 16 * 16                       # over the end of the tables, where reading ends
    memory = [torch.empty(max(size, at + written), dtype=torch.int8, device="cuda") for _ in range(2)]
    other = [torch.empty(32 * next_q, dtype=torch.int8, device="cuda") for _ in range(2)]
    out = torch.empty(4 * p * (blocks - 1 + q), dtype=torch.int32, device="cuda")
    busy = torch.empty(1 << 29, dtype=torch.int8, device="cuda")
    rows = [torch.empty(written, dtype=torch.int8, device="cuda") for _ in range(2)]
    bcs.bcs_build(next_p, 0, n, *rows)

    def read():
        if reader == "expand":
            bcs.bcs_expand(p, blocks, 0, p, memory[0][:size], memory[1][:size], out.view(p, -1, 4))
        else:
            half = len(out) // 4
            bcs.bcs_allgather_tables(p, blocks, 7, memory[0][:size], memory[1][:size], out[:half], out[half:2 * half])

    want = None
    for _ in range(5):
        for m, t in zip(memory, tables):
            m[:size] = t
        out.fill_(-9)
        torch.cuda.synchronize()
        if want is None:                                         # nothing behind it
            read()
            want = out.clone()
            continue
        for _ in range(4):
            busy.zero_()                                         # (all that follows is enqueued while this lasts)
        read()
        if between:
            bcs.bcs_build(next_p, 0, 32, *other)
        bcs.bcs_build(next_p, 0, n, memory[0][at:at + written], memory[1][at:at + written])
        torch.cuda.synchronize()
        assert torch.equal(out, want)
        assert all(torch.equal(m[at:at + written], r) for m, r in zip(memory, rows))


def _probe():
    import ctypes
    from paper_2205_10072_b200 import build_ext
    probe = ctypes.CDLL(build_ext.build_probe())
    probe.bcs_probe_turns.argtypes = [ctypes.c_uint32, ctypes.c_void_p, ctypes.c_void_p]
    probe.bcs_probe_unanswered.argtypes = [ctypes.c_uint64, ctypes.c_void_p, ctypes.c_void_p]
    return probe


# Turns that CTAs take from one another: each is taken once, by all threads of one CTA, whether all CTAs run at once or some thousand wait.
@pytest.mark.parametrize("ctas", [1, 2, 148, 3000, 100003])
def test_turns_are_taken_once(bcs, ctas):
    taken = torch.zeros(ctas, dtype=torch.int32, device="cuda")
    assert _probe().bcs_probe_turns(ctas, taken.data_ptr(), torch.cuda.current_stream().cuda_stream or None) == 0
    torch.cuda.synchronize()
    assert bool((taken == 96).all())


# An answer that never comes (none was asked for): all threads of the CTA are told so, not before the limit, and the context goes on.
def test_a_wait_that_runs_out_ends(bcs):
    results = torch.zeros(96, dtype=torch.int32, device="cuda")
    begin, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    begin.record()
    assert _probe().bcs_probe_unanswered(3000000, results.data_ptr(), torch.cuda.current_stream().cuda_stream or None) == 0
    end.record()
    torch.cuda.synchronize()
    assert bool((results == 1).all()) and 3.0 <= begin.elapsed_time(end) < 1000.0


def _us_of_range(bcs, p, r0, r1, recv=True, send=True, calls=200):
    """Microseconds a call for the ranks r0..r1-1, calls one behind the other as in _back_to_back."""
    n = (r1 - r0) * bcs.bcs_q(p)
    out_r, out_s = (torch.empty(n, dtype=torch.int8, device="cuda") if asked else None for asked in (recv, send))
    busy = torch.empty(1 << 30, dtype=torch.int8, device="cuda")
    begin, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    times = []
    for _ in range(7):
        torch.cuda.synchronize()
        for _ in range(10):
            busy.zero_()
        begin.record()
        for _ in range(calls):
            bcs.bcs_build(p, r0, r1, out_r, out_s)
        end.record()
        torch.cuda.synchronize()
        times.append(begin.elapsed_time(end) * 1000 / calls)
    return min(times)


# The ranks below 2^(q - 5) have their home round in any word of a row, and take as long as others: a million ranks of q = 27 from 0 on took 12.2 us, in the middle 10.8;
# of q = 29 12.8 and 11.3.
@pytest.mark.parametrize("q", [27, 29])
def test_low_ranks_take_no_longer(bcs, q):
    p = (1 << q) - 1
    assert _us_of_range(bcs, p, 0, 1000000) < 1.06 * _us_of_range(bcs, p, p // 3, p // 3 + 1000000)


# Home rounds in every word of a row, one run per warp: ranks around each power of two, with the root's segment and without.
@pytest.mark.parametrize("q", range(17, 32))
def test_home_rounds_in_any_word(bcs, q):
    p = min((3 << q - 2) + 12345, (1 << 31) - 1)
    n = 148 * 16 * 32 + 1
    for k in range(8, q):
        middle = bcs.bcs_skips(p)[k]
        for r0 in {0, max(middle - n // 2, 0), max(middle - 300, 0)}:
            if r0 + n <= p and (r0 == 0 or middle > 300):
                _check(bcs, p, r0, r0 + n, recv=k % 3 != 1 or r0 == 0, send=k % 3 != 2 or r0 == 0)


# Larger p of a list, each q whose tables fit: the steps of 16, 20 and 24 ranks for receive and send rows, in tables that begin off a 16-byte boundary
@pytest.mark.parametrize("p", [(1 << 23) + 1, (1 << 24) - 3, (1 << 24) + 1, (3 << 24) + 7, (1 << 26) - 1, (1 << 26) + 1, (1 << 27) + 1, (1 << 28) + 1])
def test_batches_of_large_p(bcs, p):
    _batch(bcs, [7, p, 129])


def _check_rooted(bcs, p, root, r0, r1, recv, send):
    q, n = bcs.bcs_q(p), r1 - r0
    buffers = [_buffer(n * q) for _ in range(2)]
    ws = torch.empty(bcs.bcs_build_rooted_workspace_bytes(p, root, r0, r1), dtype=torch.int8, device="cuda")
    bcs.bcs_build_rooted(p, root, r0, r1, *(out if asked else None for (_, out), asked in zip(buffers, (recv, send))), ws)
    torch.cuda.synchronize()
    passed = root - r0                                           # the row of rank 0, behind that of p - 1
    at = np.unique(np.concatenate([np.arange(300), n - 1 - np.arange(300), np.arange(passed - 600, passed + 600), np.random.default_rng(p).integers(0, n, 1000)]))
    want = oracle.build_ranks(p, ((at + r0 - root) % p).astype(np.uint32))
    rows = torch.from_numpy(at).cuda()
    for (raw, out), asked, expect in zip(buffers, (recv, send), want):
        assert np.array_equal(out.view(n, q)[rows].cpu().numpy(), expect) if asked else bool((raw == 99).all())
        assert bool((raw[:32] == 99).all()) and bool((raw[32 + n * q:] == 99).all())


# Ranges that pass p - 1 in the middle of a run, with one run per warp: even and odd q, multiples of 4 and of 8
@pytest.mark.parametrize("q", [17, 18, 19, 20, 21, 22, 24, 26, 28, 31])
def test_one_run_per_warp_rooted(bcs, q):
    p = min((3 << q - 2) + 12345, (1 << 31) - 1)
    for n in (80003, 300001):
        n = min(n, p)
        r0 = (p - n) // 2
        for root in (r0 + n // 2, r0 + n - 700):
            _check_rooted(bcs, p, root, r0, r0 + n, True, True)
    _check_rooted(bcs, p, root, r0, r0 + n, True, False)
    _check_rooted(bcs, p, root, r0, r0 + n, False, True)


# The same for send rows alone, by vectors of 16 bytes from 1.9 million ranks on
@pytest.mark.parametrize("p,n", [(1000003, 1000003), ((1 << 24) - 5, 700001), ((1 << 24) + 1, 1 << 20), (2000003, 2000003), (5000011, 5000011), (3 << 28, 1900001)])
def test_send_rows_alone_rooted(bcs, p, n):
    r0 = (p - n) // 2
    for root in (r0 + n // 2, r0 + 601, r0 + n - 601):
        _check_rooted(bcs, p, root, r0, r0 + n, False, True)


@pytest.mark.parametrize("p,n", [(3000017, 3000017), ((1 << 28) + 1, 5000001)])
def test_turns_rooted(bcs, p, n):
    r0 = (p - n) // 2
    for recv, send in ((True, True), (True, False)):
        _check_rooted(bcs, p, r0 + n // 2, r0, r0 + n, recv, send)


# Lines of the kernel of four ranks per lane, both sides: runs of one to seven look-ups in 148 or 296 CTAs of ten warps (q = 28: eight), the longest that have one run per
# warp, turns of 768 ranks, the table of send rows; `tables`: both, receive rows, send rows.
@pytest.mark.parametrize("p,n,tables", [(2000003, 148 * 10 * 128, "brs"), (2000003, 296 * 10 * 128, "brs"), (2000003, 296 * 10 * 256, "br"), (2000003, 296 * 10 * 384, "brs"),
                                        (2000003, 296 * 10 * 640, "brs"), ((1 << 22) - 3, 296 * 9 * 896, "br"), (1 << 28, 296 * 8 * 128, "brs"),
                                        (1 << 28, 296 * 8 * 512, "br"), (1 << 28, 296 * 7 * 896, "br"), ((1 << 24) - 1, 3500000, "r"), ((1 << 23) + 1, 1 << 22, "b")])
def test_four_ranks_per_lane_on_both_sides_of_its_lines(bcs, p, n, tables):
    for count in (n, n + 1):
        for r0 in (0, (p - count) // 2 | 1):
            for which in tables:
                _check(bcs, p, r0, r0 + count, recv=which != "s", send=which != "r")
    assert bcs.bcs_wait_expired() == 0


# As test_tables_are_not_written_before_they_are_read, with turns that CTAs take from one another (the wait is in each of them), and with send rows by vectors,
# some CTAs of which have no ranks.
@pytest.mark.parametrize("n,which", [(2700001, "both"), (4300001, "both"), (3000001, "recv"), (1000003, "send"), (1900001, "send")])
@pytest.mark.parametrize("between", [False, True])
def test_long_tables_are_not_written_before_they_are_read(bcs, n, which, between):
    p, blocks, next_p = 100003, 150, 6000011
    q, next_q = bcs.bcs_q(p), bcs.bcs_q(next_p)
    tables = [torch.from_numpy(t).cuda().view(-1) for t in oracle.full_table(p)]
    size, written = p * q, n * next_q
    memory = [torch.empty(written, dtype=torch.int8, device="cuda") for _ in range(2)]         # (longer than the tables: turns in front of, over and behind them)
    other = [torch.empty(32 * next_q, dtype=torch.int8, device="cuda") for _ in range(2)]
    out = torch.empty((p, blocks - 1 + q, 4), dtype=torch.int32, device="cuda")
    busy = torch.empty(1 << 29, dtype=torch.int8, device="cuda")
    asked = [which != "send", which != "recv"]
    rows = [torch.empty(written, dtype=torch.int8, device="cuda") if a else None for a in asked]
    bcs.bcs_build(next_p, 77, 77 + n, *rows)
    bcs.bcs_expand(p, blocks, 0, p, *tables, out)
    want = out.clone()
    for at in (0, (written - size) // 32 * 16, (written - size) // 16 * 16):
        lie = [m[at:at + size] for m in memory]
        for m, t in zip(lie, tables):
            m.copy_(t)
        out.fill_(-9)
        torch.cuda.synchronize()
        for _ in range(4):
            busy.zero_()                                         # (all that follows is enqueued while this lasts)
        bcs.bcs_expand(p, blocks, 0, p, *lie, out)
        if between:
            bcs.bcs_build(next_p, 0, 32, *other)
        bcs.bcs_build(next_p, 77, 77 + n, *(m if a else None for m, a in zip(memory, asked)))
        torch.cuda.synchronize()
        assert torch.equal(out, want)
        assert all(torch.equal(m, r) for m, r, a in zip(memory, rows, asked) if a)
    assert bcs.bcs_wait_expired() == 0


# Send rows alone that the kernel of four ranks per lane would make in turns are made by vectors from there on, both sides of the line: 1.6 million of q = 31 took 1.22 times as
# long as 1.58 million (12.6 us), 1.7 million 1.25 times (12.9); 1.10 and 1.16 now.
@pytest.mark.parametrize("q", [27, 28, 29, 30, 31])
def test_send_rows_alone_where_turns_begin(bcs, q):
    p = min((3 << q - 2) + 12345, (1 << 31) - 1)
    line = (6 if q == 31 else 7) * 7 * 296 * 128
    for n in (line, line + 1):
        for r0 in (0, (p - n) // 2 | 1, p - n):
            _check(bcs, p, r0, r0 + n, recv=False)


def test_send_rows_alone_keep_the_faster_form(bcs):
    p, r0 = (1 << 31) - 1, 306783378
    fewer, more = (_us_of_range(bcs, p, r0, r0 + n, recv=False) for n in (1580000, 1600000))
    assert more < 1.17 * fewer


# Send rows alone of 1.9 million ranks (145 of 148 CTAs have some), made by vectors, take no longer than 1 894 400 and 1 941 760 (148 have, runs of 640 and 656 ranks)
def test_send_rows_with_ctas_without_ranks_take_no_longer(bcs):
    p = (1 << 24) - 5
    some, all_ = (_us_of_range(bcs, p, 12345, 12345 + n, recv=False) for n in (1900001, 148 * 20 * 656))
    assert some < 1.1 * all_
