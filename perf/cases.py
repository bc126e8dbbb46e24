"""What a user has the library do, as cases that can be timed: schedule tables of one processor
count (a few ranks, a range, all ranks, in chunks, rooted anywhere), tables of many counts at once,
and the round tables and allgather index tables made from them.

A program learns its processor count p when it starts, so `p` of a case is the most it may be: the
seed draws the p of the call from the top 64th below it (same q), and the buffers are made for the
largest.  Bytes past the rows of a smaller p stay zero.  All results are whole numbers.
"""
import random

import torch

import paper_2205_10072_b200 as bcs
from paper_2205_10072_b200 import workloads


def listed():
    return [
        # The paper's own use: a node asks for the rows of its own 32 ranks and owns no scratch memory.
        {"name": "own rows 32 of 1M", "kind": "range", "p": 2**20 + 2**14, "ranks": 32, "scratch": False},
        # All ranks of the largest cluster of the paper's experiments (36 nodes x 32): the smallest tables.
        {"name": "table 1152", "kind": "table", "p": 1152},
        # The size up to which the paper's author verified: an ordinary large machine.
        {"name": "table 100003", "kind": "table", "p": 100003},
        # A million ranks, just above a power of two (the benchmark's single p).
        {"name": "table 1M", "kind": "table", "p": 2**20 + 2**14},
        # One of 16 shards of the same job, built where it is needed.
        {"name": "range 64K of 1M", "kind": "range", "p": 2**20 + 2**14, "ranks": 65536 + 17, "scratch": True},
        # A broadcast from a root that is not rank 0, at a count that is no power of two's neighbour.
        {"name": "rooted 1.3M", "kind": "rooted", "p": 1300003},
        # Tables too large to want at once: eight chunks, receive rows as they are built, send rows after.
        {"name": "chunks 256M", "kind": "chunks", "p": 2**28 - 1, "chunks": 8},
        # Exhaustive sweeps over small counts, and a sweep over counts of all sizes.
        {"name": "batch of every p to 1024", "kind": "batch", "small": True, "count": 1023, "lo_exp": 1, "hi_exp": 10},
        {"name": "batch of 1024 p to 1M", "kind": "batch", "small": False, "count": 1024, "lo_exp": 10, "hi_exp": 20},
        # Round tables (send block, receive block, to, from): a short message on a cluster, and 1000
        # blocks on a large machine.
        {"name": "rounds 1152 n=64", "kind": "rounds", "p": 1152, "n": 64},
        {"name": "rounds 100003 n=1000", "kind": "rounds", "p": 100003, "n": 1000},
        # Pack and unpack block numbers of one processor of an irregular allgather.
        {"name": "allgather 100003 n=1000", "kind": "allgather", "p": 100003, "n": 1000},
    ]


def _log_uniform(rng, lo, hi):
    return min(hi, max(lo, round(lo * (hi / lo) ** rng.random())))


def draw(rng):
    kind = rng.choice(["range", "table", "table", "rooted", "chunks", "batch", "batch", "rounds", "allgather"])
    if kind == "table" or kind == "rooted":
        return {"kind": kind, "p": _log_uniform(rng, 256, 2**23)}
    if kind == "range":
        scratch = rng.random() < 0.5
        p = _log_uniform(rng, 2**14, 2**23)
        return {"kind": kind, "p": p, "ranks": _log_uniform(rng, 1024, p // 4) if scratch else _log_uniform(rng, 8, 4096),
                "scratch": scratch}
    if kind == "chunks":
        return {"kind": kind, "p": _log_uniform(rng, 2**22, 2**28 - 1), "chunks": rng.randrange(2, 12)}
    if kind == "batch":
        if rng.random() < 0.3:
            return {"kind": kind, "small": True, "count": _log_uniform(rng, 64, 1023), "lo_exp": 1, "hi_exp": 10}
        lo = rng.randrange(6, 15)
        return {"kind": kind, "small": False, "count": _log_uniform(rng, 16, 700), "lo_exp": lo,
                "hi_exp": rng.randrange(lo + 2, 21)}
    p = _log_uniform(rng, 256, 2**18)
    if kind == "rounds":
        return {"kind": kind, "p": p, "n": _log_uniform(rng, 2, max(4, 2**26 // p))}
    return {"kind": kind, "p": p, "n": _log_uniform(rng, 2, max(4, 2**27 // p))}


def _smallest(p):
    return max(p - p // 64, (1 << (bcs.bcs_q(p) - 1)) + 1)


def _bytes(n):
    return torch.zeros(max(n, 1), dtype=torch.int8, device="cuda")


def _p_list(case):
    if case["small"]:
        return workloads.small_sweep()[-case["count"]:]
    return workloads.batch_p_list(case["count"], workloads.SEED_BATCH, case["lo_exp"], case["hi_exp"])


def prepare(case, seed):
    rng = random.Random(seed)
    s = dict(case)
    if case["kind"] == "batch":
        ps = list(_p_list(case))
        rng.shuffle(ps)
        plan = bcs.bcs_batch_plan(ps)
        s["plan"] = plan.to("cuda")
        s["recv"], s["send"] = _bytes(plan.total_entries), _bytes(plan.total_entries)
        s["ws"] = _bytes(plan.workspace_bytes())
        return s
    most = case["p"]
    s["p"] = p = rng.randint(_smallest(most), most)
    q = bcs.bcs_q(p)
    if case["kind"] == "range":
        s["lo"] = lo = rng.randrange(0, p - case["ranks"] + 1)
        s["hi"] = hi = lo + case["ranks"]
        s["recv"], s["send"] = _bytes(case["ranks"] * q), _bytes(case["ranks"] * q)
        s["ws"] = _bytes(bcs.bcs_build_workspace_bytes(p, lo, hi)) if case["scratch"] else None
        return s
    s["recv"], s["send"] = _bytes(most * q), _bytes(most * q)
    if case["kind"] == "table":
        s["ws"] = _bytes(bcs.bcs_build_workspace_bytes(p, 0, p))
    elif case["kind"] == "rooted":
        s["root"] = root = rng.randrange(1, p)
        s["ws"] = _bytes(bcs.bcs_build_rooted_workspace_bytes(p, root, 0, p))
    elif case["kind"] == "chunks":
        step = (-(-p // case["chunks"]) + 15) // 16 * 16
        s["ranges"] = [(lo, min(lo + step, p)) for lo in range(0, p, step)]
        s["recv_of"] = [s["recv"][lo * q:hi * q] for lo, hi in s["ranges"]]
        s["send_of"] = [s["send"][lo * q:hi * q] for lo, hi in s["ranges"]]
        s["ws"] = _bytes(bcs.bcs_prepare_workspace_bytes(p))
    else:
        # the schedule tables are at hand, built once before
        bcs.bcs_build(p, 0, p, s["recv"], s["send"], _bytes(bcs.bcs_build_workspace_bytes(p, 0, p)))
        rounds = case["n"] - 1 + q
        if case["kind"] == "rounds":
            s["table"] = torch.zeros((most, rounds, 4), dtype=torch.int32, device="cuda")
        else:
            s["rank"] = rng.randrange(p)
            s["pack"] = torch.zeros(rounds * most, dtype=torch.int32, device="cuda")
            s["unpack"] = torch.zeros(rounds * most, dtype=torch.int32, device="cuda")
    return s


def run(s):
    kind = s["kind"]
    if kind == "batch":
        bcs.bcs_build_batch(s["plan"], s["recv"], s["send"], s["ws"])
    elif kind == "range":
        bcs.bcs_build(s["p"], s["lo"], s["hi"], s["recv"], s["send"], s["ws"])
    elif kind == "table":
        bcs.bcs_build(s["p"], 0, s["p"], s["recv"], s["send"], s["ws"])
    elif kind == "rooted":
        bcs.bcs_build_rooted(s["p"], s["root"], 0, s["p"], s["recv"], s["send"], s["ws"])
    elif kind == "chunks":
        p, ws = s["p"], s["ws"]
        bcs.bcs_prepare_codes(p, ws)
        for (lo, hi), out in zip(s["ranges"], s["recv_of"]):
            bcs.bcs_prepare_rows(p, lo, hi, out, ws)
        for (lo, hi), out in zip(s["ranges"], s["send_of"]):
            bcs.bcs_build_prepared(p, lo, hi, None, out, ws)
    elif kind == "rounds":
        bcs.bcs_expand(s["p"], s["n"], 0, s["p"], s["recv"], s["send"], s["table"])
        return s["table"]
    else:
        bcs.bcs_allgather_tables(s["p"], s["n"], s["rank"], s["recv"], s["send"], s["pack"], s["unpack"])
        return s["pack"], s["unpack"]
    return s["recv"], s["send"]


def work(case):
    """Bytes only: rows of both tables written; for the tables made from them, the rows read too."""
    if case["kind"] == "batch":
        return {"bytes": 2 * sum(p * bcs.bcs_q(p) for p in _p_list(case)), "flops": 0}
    p, q = (_smallest(case["p"]) + case["p"]) / 2, bcs.bcs_q(case["p"])
    if case["kind"] == "range":
        return {"bytes": 2 * case["ranks"] * q, "flops": 0}
    rows = 2 * p * q
    if case["kind"] == "rounds":
        return {"bytes": rows + 16 * p * (case["n"] - 1 + q), "flops": 0}
    if case["kind"] == "allgather":
        return {"bytes": rows + 8 * p * (case["n"] - 1 + q), "flops": 0}
    return {"bytes": rows, "flops": 0}


def tolerance(case):
    return "exact"
