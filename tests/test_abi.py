"""CPU-only checks of the boundary: the shared library loads, exports every symbol that
include/bcs.h declares, and its host-side entry points (no kernel launch) behave."""
import ctypes
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    from paper_2205_10072_b200 import build_ext
    build_ext.build()
    import paper_2205_10072_b200 as bcs
    return bcs


def test_the_library_holds_its_constants_once(lib):
    """1.75 MB of row constants, once for the device and once for the host, and kernels: 5.8 MB.  In two units, with line information
    (nvcc adds the constants as text) it was 23 MB, and a process's first calls took twice as long."""
    assert os.path.getsize(lib.lib_path()) < 8 << 20


def _declared_symbols():
    names = set()
    for fn in os.listdir(os.path.join(ROOT, "include")):
        if fn.endswith(".h"):
            text = open(os.path.join(ROOT, "include", fn)).read()
            text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
            names |= set(re.findall(r"\b(bcs_[a-z_0-9]+)\s*\(", text))
    return sorted(names)


def test_every_declared_symbol_is_exported(lib):
    names = _declared_symbols()
    assert {"bcs_build", "bcs_build_batch", "bcs_expand", "bcs_checksum", "bcs_skips", "bcs_q",
            "bcs_batch_plan", "bcs_status_str", "bcs_build_to_host", "bcs_build_workspace_bytes",
            "bcs_build_batch_workspace_bytes", "bcs_validate", "bcs_build_static", "bcs_simulate", "bcs_prepare",
            "bcs_build_prepared", "bcs_prepare_workspace_bytes", "bcs_prepare_codes", "bcs_prepare_rows", "bcs_allgather_tables", "bcs_circulant_rounds"} <= set(names)
    dll = ctypes.CDLL(lib.lib_path())
    for n in names:
        assert hasattr(dll, n), n
        assert callable(getattr(lib, n)), "binding lacks %s" % n


def test_q_and_skips_host_side(lib):
    assert lib.bcs_q(0) == -1 and lib.bcs_q(1) == 0 and lib.bcs_q(2) == 1
    assert lib.bcs_q(1024) == 10 and lib.bcs_q(1025) == 11 and lib.bcs_q(2**31 - 1) == 31
    assert lib.bcs_skips(1) == [1]
    assert lib.bcs_skips(20) == [1, 2, 3, 5, 10, 20]            # caption of Table 1
    assert lib.bcs_skips(33) == [1, 2, 3, 5, 9, 17, 33]         # caption of Table 2
    assert lib.bcs_skips(31) == [1, 2, 4, 8, 16, 31]            # caption of Table 4
    assert lib.bcs_skips(2**30 - 1) == [2**k for k in range(30)] + [2**30 - 1]
    with pytest.raises(lib.BcsError) as e:
        lib.bcs_skips(0)
    assert e.value.status == 2
    with pytest.raises(lib.BcsError) as e:
        lib.bcs_skips(2**31)
    assert e.value.status == 4


def test_status_strings(lib):
    assert [lib.bcs_status_str(i) for i in range(6)] == [
        "BCS_OK", "BCS_ERR_ARG", "BCS_ERR_RANGE", "BCS_ERR_ALIGN", "BCS_ERR_UNSUPPORTED",
        "BCS_ERR_CUDA"]
    assert lib.bcs_status_str(99) == "BCS_ERR_UNKNOWN"


def test_batch_plan_host_side(lib):
    plan = lib.bcs_batch_plan([2, 3, 20, 1, 1025])
    assert plan.rank_off.tolist() == [0, 2, 5, 25, 26, 1051]
    assert plan.entry_off.tolist() == [0, 2, 8, 108, 108, 108 + 1025 * 11]
    # tiles of 512 ranks and q rounds of align16(p) bytes of scratch for a p above 1024 only: a
    # smaller p is built by one CTA that keeps everything in shared memory
    assert plan.tile_off.tolist() == [0, 0, 0, 0, 0, 3]
    assert plan.copy_off.tolist() == [0, 0, 0, 0, 0, 11 * 1040]
    assert plan.total_tiles == 3 and plan.workspace_bytes() == 4352 + 11 * 1040
    small = lib.bcs_batch_plan([1024, 7, 1])
    assert small.total_tiles == 0 and small.total_copy == 0 and small.workspace_bytes() == 256
    assert plan.skips_tab[2].tolist()[:6] == [1, 2, 3, 5, 10, 20]
    assert plan.skips_tab[3].tolist()[:2] == [1, 0]
    # full_tab[d] = skip code of rank skips[d]-1: p = 20, skips 1 2 3 5 10 20:
    # 0 -> {}, 1 -> {0}, 2 -> {1}, 4 = 3+1 -> {2,0}, 9 = 5+3+1 -> {3,2,0}, 19 = 10+5+3+1
    assert plan.full_tab[2].tolist()[:6] == [0, 1, 2, 5, 13, 29]
    assert plan.total_ranks == 1051
    with pytest.raises(lib.BcsError):
        lib.bcs_batch_plan([5, 0])


def test_argument_errors_need_no_gpu(lib):
    """Validation happens before any CUDA call: these return an error code on a CPU-only box."""
    L = lib.lib()
    assert L.bcs_build(0, 0, 0, None, None, None, 0, None) == 2
    assert L.bcs_build(2**31, 0, 1, None, None, None, 0, None) == 4
    assert L.bcs_build(10, 5, 4, None, None, None, 0, None) == 2
    assert L.bcs_build(10, 0, 11, None, None, None, 0, None) == 2
    assert L.bcs_build(10, 0, 10, None, None, None, 0, None) == 1
    assert L.bcs_build(10, 0, 10, 8, None, None, 0, None) == 3   # misaligned pointer
    assert L.bcs_build(1, 0, 1, None, None, None, 0, None) == 0  # q == 0: nothing to do
    assert L.bcs_build(10, 3, 3, None, None, None, 0, None) == 0 # empty range
    assert L.bcs_build_workspace_bytes(2**20 + 1, 0, 2**20 + 1) == 4194560 + 21 * 1048592
    assert L.bcs_build_workspace_bytes(0, 0, 0) == 0
    assert L.bcs_build_batch_workspace_bytes(1000, 9008) == 4096 + 9008
    assert L.bcs_expand(10, 0, 0, 10, 16, 16, 16, None) == 1     # n == 0
    assert L.bcs_expand(10, 4, 0, 10, None, 16, 16, None) == 1
    assert L.bcs_expand(10, 4, 0, 10, 16, 16, 8, None) == 3
    assert L.bcs_checksum(16, 8, 2, 16, None) == 3               # first index not a multiple of 4
    assert L.bcs_checksum(16, 8, 0, None, None) == 1
    assert L.bcs_build_batch(None, None, None, None, None, None, None, 3, 10, 40, 1, 48, 16, None, None, 0,
                             None) == 1
    assert L.bcs_prepare_codes(0, 16, 1 << 20, None) == 2
    assert L.bcs_prepare_codes(1000, None, 0, None) == 1
    assert L.bcs_prepare_codes(1000, 16, 64, None) == 1                       # workspace too small
    assert L.bcs_prepare_codes(1000, 8, 1 << 20, None) == 3                    # misaligned workspace
    assert L.bcs_prepare_rows(1000, 8, 100, 16, 16, 1 << 20, None) == 3        # r_begin not a multiple of 16
    assert L.bcs_prepare_rows(1000, 16, 1001, 16, 16, 1 << 20, None) == 2
    assert L.bcs_prepare_rows(1000, 16, 100, 24, 16, 1 << 20, None) == 3       # misaligned rows
    assert L.bcs_prepare_rows(1000, 16, 16, None, 16, 1 << 20, None) == 0      # empty range
    assert L.bcs_prepare_workspace_bytes(1000) == 4096 + 10 * 1008
    assert L.bcs_expand(10, 4, 0, 10, None, None, None, None) == 1             # no table to write to
    assert L.bcs_build_to_host(10, 0, 10, None, None, 16, 1024, None) == 1
    assert L.bcs_build_to_host(10, 0, 10, 16, None, 16, 16, None) == 1   # staging too small


def test_arguments_that_the_fast_calls_take_are_those_of_ctypes(lib):
    """The calls through the extension module refuse what ctypes refuses (None or a fraction as a number) and take what it
    takes (its own integers and pointers); empty ranges, so that nothing is enqueued."""
    import ctypes
    from types import SimpleNamespace
    from paper_2205_10072_b200 import binding
    stream = SimpleNamespace(cuda_stream=0)
    at = SimpleNamespace(data_ptr=lambda: ctypes.c_void_p(0), nbytes=0)
    for p in (10, True, ctypes.c_uint32(10)):
        lib.bcs_build(p, 0, 0, None, None, stream=stream)
    lib.bcs_build(10, ctypes.c_uint64(3), 3, at, at, at, stream=stream)
    lib.bcs_expand(10, 4, 3, 3, at, None, None, stream=stream)
    lib.bcs_build_rooted(10, 3, 3, 3, None, at, stream=stream)
    for number in (None, 3.0, "3"):
        for call in (lambda: lib.bcs_build(10, number, 3, None, None, stream=stream),
                     lambda: lib.bcs_build(number, 0, 0, None, None, stream=stream),
                     lambda: lib.bcs_build_rooted(10, number, 3, 3, None, None, stream=stream),
                     lambda: lib.bcs_build_static(10, 0, number, None, None, stream=stream),
                     lambda: lib.bcs_prepare(number, None, stream=stream),
                     lambda: lib.bcs_prepare_codes(number, None, stream=stream),
                     lambda: lib.bcs_prepare_rows(10, number, 0, None, at, stream=stream),
                     lambda: lib.bcs_build_prepared(10, number, 0, None, None, at, stream=stream),
                     lambda: lib.bcs_expand(10, 4, number, 0, None, None, None, stream=stream),
                     lambda: lib.bcs_allgather_tables(1, 4, number, None, None, None, None, stream=stream),
                     lambda: binding._call.build_batch(0, 0, 0, 0, 0, 0, 0, number, 0, 0, 0, 0, None, None, None, 0, None)):
            with pytest.raises(ctypes.ArgumentError):
                call()
    with pytest.raises(TypeError):                               # too few
        binding._call.build(10, 0, 0)


def test_calls_with_tensors_are_those_with_numbers(lib):
    """What the extension module makes of tensors and streams is what binding.py makes of them: each argument in its place (told by the
    refusals), the errors of a tensor, and the workspace's size."""
    from types import SimpleNamespace
    from paper_2205_10072_b200 import binding
    stream = SimpleNamespace(cuda_stream=0)
    at = lambda address, size=0: SimpleNamespace(data_ptr=lambda: address, nbytes=size)
    good, off, ws, small = at(64), at(72), at(64, 1 << 20), at(64, 64)
    cases = [("build", (10, 0, 10, None, None, None, stream)), ("build", (10, 0, 10, off, None, None, stream)), ("build", (10, 0, 10, good, off, None, stream)),
             ("build", (10, 0, 10, good, None, off, stream)), ("build", (10, 3, 2, good, good, good, stream)), ("build", (10, 3, 3, None, None, None, stream)),
             ("build_rooted", (10, 10, 0, 10, good, good, None, stream)), ("build_rooted", (10, 3, 0, 11, good, good, None, stream)),
             ("build_rooted", (1001, 3, 0, 1001, good, good, small, stream)), ("prepare_rows", (1000, 16, 100, good, small, stream)),
             ("prepare_rows", (1000, 16, 100, off, ws, stream)), ("prepare_rows", (1000, 8, 100, good, ws, stream)),
             ("build_prepared", (1000, 0, 100, good, off, ws, stream)), ("build_prepared", (1000, 0, 100, good, good, small, stream)),
             ("build_prepared", (1000, 0, 100, None, None, ws, stream)), ("build_static", (10, 0, 10, None, off, stream)),
             ("build_static", (10, 0, 11, good, good, stream)), ("expand", (10, 4, 0, 10, good, None, good, stream)), ("expand", (10, 4, 0, 10, good, good, off, stream)),
             ("expand", (10, 0, 0, 10, good, good, good, stream)), ("allgather_tables", (10, 4, 10, good, good, good, good, stream)),
             ("allgather_tables", (10, 4, 3, off, good, good, None, stream)), ("allgather_tables", (10, 4, 3, good, off, None, good, stream)),
             ("allgather_tables", (10, 4, 3, good, good, at(66), None, stream)), ("allgather_tables", (10, 4, 3, good, good, None, None, stream))]
    statuses = set()
    for name, args in cases:
        status = getattr(binding._call, "on_" + name)(*args)
        assert status == binding._PLAIN[name](*args), (name, args)
        statuses.add(status)
    assert statuses == {0, 1, 2, 3}
    for bad in (3, SimpleNamespace(), "x"):
        with pytest.raises(AttributeError):
            lib.bcs_build(10, 0, 10, good, bad, stream=stream)
    with pytest.raises(AttributeError):                          # a workspace without a size
        lib.bcs_build(10, 0, 10, good, good, SimpleNamespace(data_ptr=lambda: 64), stream=stream)
    with pytest.raises(ZeroDivisionError):
        lib.bcs_build(10, 0, 10, SimpleNamespace(data_ptr=lambda: 1 // 0), good, stream=stream)
    with pytest.raises(AttributeError):
        lib.bcs_build(10, 0, 10, good, good, stream=3)


def test_unknown_calls_are_attribute_errors(lib):
    """Names that are no calls, with tensors or without, are missing attributes."""
    from paper_2205_10072_b200 import binding
    for name in ("nothing", "on_nothing", "on_", "on_prepare"):
        assert not hasattr(binding._call, name)
        with pytest.raises(AttributeError):
            getattr(binding._call, name)
    assert callable(binding._call.on_build)


WAITS = r"""
#include <stdint.h>
#include <stdio.h>
#include "ptx.cuh"
// A clock and an event on a time line: polls take `poll` each, between poll number `away` and the look at the clock behind it the context is away for `gone`.
struct Line {
    uint64_t now = 5000000000ull, comes, poll, gone;
    int polls = 0, away;
};
struct Came {
    Line *line;
    bool operator()() const
    {
        const bool there = line->now >= line->comes;
        line->now += line->poll;
        if (++line->polls == line->away) line->now += line->gone;
        return there;
    }
};
struct Clock {
    Line *line;
    uint64_t operator()() const { return line->now; }
};
int main()
{
    unsigned long long comes, poll, gone, limit;
    int away;
    while (scanf("%llu %llu %d %llu %llu", &comes, &poll, &away, &gone, &limit) == 5) {
        Line line;
        const uint64_t begin = line.now;
        line.comes = begin + comes, line.poll = poll, line.away = away, line.gone = gone;
        const bool came = bcs::wait_with_limit(Came{&line}, Clock{&line}, limit);
        printf("%d %llu %d\n", (int)came, (unsigned long long)(line.now - begin), line.polls);
    }
}
"""


def test_a_wait_does_not_give_up_on_what_has_come(tmp_path):
    """The wait of the row kernels for an answer, on a time line (no GPU): time in which the context is away is not time spent waiting, what has come meanwhile
    is found, and what never comes ends the wait within its limit and a few polls."""
    import subprocess
    from paper_2205_10072_b200 import build_ext
    source = tmp_path / "waits.cu"
    source.write_text(WAITS)
    flags = [f for f in build_ext.NVCC_FLAGS if f != "--shared"]
    subprocess.check_call([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")] + flags +
                          ["-I", os.path.join(os.path.dirname(build_ext.LIB_PATH), "csrc"), "-o", str(tmp_path / "waits"), str(source)])
    s, never = 10**9, 10**15
    cases = [(0, 100, 0, 0, 2 * s), (800, 100, 0, 0, 2 * s),             # there, or soon
             (800, 100, 1, 3 * s, 2 * s), (800, 100, 3, 3 * s, 2 * s),   # comes while the context is away, for longer than the limit
             (s, 1000, 5, 100 * s, 2 * s),
             (100 * s + 500000, 1000, 5, 100 * s, 2 * s),                # comes a while after it is back
             (never, 1000, 0, 0, s // 1000), (never, 5 * 10**6, 0, 0, s // 10), (never, 1000, 7, 50 * s, s // 1000)]
    out = subprocess.run([str(tmp_path / "waits")], input="".join("%d %d %d %d %d\n" % c for c in cases), text=True, check=True, capture_output=True)
    got = [tuple(map(int, line.split())) for line in out.stdout.splitlines()]
    assert [came for came, _, _ in got] == [1] * 6 + [0] * 3
    assert all(polls <= 2 for _, _, polls in got[:1])
    for (_, poll, _, gone, limit), (_, took, polls) in list(zip(cases, got))[6:]:
        counted = min(poll, 10**6)                                       # what a poll counts as
        assert limit <= polls * counted + (10**6 if gone else 0)
        assert polls <= limit // counted + 3 and took <= polls * poll + gone


FAKE_RUNTIME = r"""
#include <cuda_runtime.h>
#include <stdio.h>
static cudaError_t last = cudaSuccess;
static bool device = false;
static cudaError_t fail(cudaError_t e) { return last = e; }
static cudaError_t fake_device(int *dev) { *dev = 0; return device ? cudaSuccess : fail(cudaErrorNoDevice); }
template <class T> static cudaError_t fake_attribute(T, cudaFuncAttribute, int) { return fail(cudaErrorInvalidValue); }
static cudaError_t fake_last() { const cudaError_t e = last; last = cudaSuccess; return e; }
#define cudaGetDevice fake_device
#define cudaFuncSetAttribute fake_attribute
#define cudaGetLastError fake_last
#include "bcs_common.cuh"
__global__ void kernel() {}
int main()
{
    for (int i = 0; i < 2; ++i) {
        device = i == 1;
        const bool allowed = bcs::allow_shared<kernel>();
        printf("%d %d ", (int)allowed, (int)bcs::launch_status());
    }
}
"""


def test_a_refused_call_leaves_no_error_behind(tmp_path):
    """The opt-in to large shared memory, refused by the runtime (a fake here), takes its error with it: the next call asks for the
    last one after its launch."""
    import subprocess
    from paper_2205_10072_b200 import build_ext
    source = tmp_path / "refused.cu"
    source.write_text(FAKE_RUNTIME)
    flags = [f for f in build_ext.NVCC_FLAGS if f != "--shared"]
    subprocess.check_call([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")] + flags +
                          ["-I", os.path.join(os.path.dirname(build_ext.LIB_PATH), "csrc"), "-o", str(tmp_path / "refused"), str(source)])
    assert subprocess.check_output([str(tmp_path / "refused")], text=True) == "0 0 0 0 "


FAKE_LAUNCH = r"""
#include <cuda_runtime.h>
#include <stdio.h>
static int4 split;
template <class... P, class... A>
static cudaError_t fake_launch(const cudaLaunchConfig_t *cfg, void (*)(P...), A &&...)
{
    split = make_int4(cfg->gridDim.x, cfg->gridDim.y, 0, 0);
    return cudaSuccess;
}
#define cudaLaunchKernelEx fake_launch
#include "allgather.cu"
namespace bcs {
bcs_status make_table(uint32_t p, PTable *tab)
{
    tab->p = p;
    for (tab->q = 0; (1ull << tab->q) < p; ++tab->q) {}
    return BCS_OK;
}
}
int main()
{
    alignas(16) static int8_t rows[16];
    alignas(16) static int32_t out[4];
    unsigned p, n;
    int both;
    while (scanf("%u %u %d", &p, &n, &both) == 3) {
        (void)bcs_allgather_tables(p, n, 0, rows, rows, out, both ? out : nullptr, nullptr);
        printf("%d %d\n", split.x, split.y);
    }
}
"""


def test_allgather_grids_that_fit_the_card_are_not_made_smaller(tmp_path):
    """Where CTAs of four rounds each are on the card at once (six per SM with both tables, seven with one), the launch has those; longer
    ones took a tenth more time.  Where they are not, it has fewer CTAs with up to 64 rounds, four per SM or more.  (The launch is a fake.)"""
    import subprocess
    from paper_2205_10072_b200 import build_ext
    source = tmp_path / "split.cu"
    source.write_text(FAKE_LAUNCH)
    flags = [f for f in build_ext.NVCC_FLAGS if f != "--shared"]
    subprocess.check_call([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")] + flags +
                          ["-I", os.path.join(os.path.dirname(build_ext.LIB_PATH), "csrc"), "-o", str(tmp_path / "split"), str(source)])
    sizes = [(p, n, both) for p in (300, 1152, 2000, 5000, 9000, 12000, 20262, 35000, 50000, 70000, 261597)
             for n in (2, 7, 20, 64, 116, 300, 500, 1500, 6000) for both in (0, 1)]
    out = subprocess.run([str(tmp_path / "split")], input="".join("%d %d %d\n" % s for s in sizes), text=True, check=True, capture_output=True)
    whole = 0
    for (p, n, both), line in zip(sizes, out.stdout.splitlines(), strict=True):
        x, y = map(int, line.split())
        rounds, blocks = n - 1 + (p - 1).bit_length(), -(-p // 256)
        finest = -(-rounds // 4)
        assert x == blocks and y <= finest, (p, n, both)
        if x * finest <= 148 * (6 if both else 7):
            assert y == finest, (p, n, both, y)
            whole += 1
        elif y != finest:                                        # the last chunk may be short
            per_cta = -(-rounds // y)
            assert per_cta <= 64 + 3 or x * (-(-rounds // (per_cta - 4))) > 148 * 4, (p, n, both, y)
    assert whole > 60 and len(sizes) - whole > 60
