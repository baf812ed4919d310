"""Batched calls in graph mode (apo_graph_mode): every call, replayed or not,
gives the offsets and results of the plain call."""
import numpy as np
import pytest

import workloads as W
from test_gpu_parity import apo, tokens_dev  # noqa: F401 (apo: the fixture)

pytestmark = pytest.mark.gpu

ARRAYS = ("sa", "lcp", "cand_len", "cand_id", "cand_start", "sel_start", "sel_len", "sel_trace", "trace_len",
          "trace_start")


def snap(r):
    from paper_2406_18111_gb300 import as_u32
    d = {k: as_u32(getattr(r, k)).copy() for k in ARRAYS}
    d["accepted"] = r.cand_accepted.cpu().numpy().copy()
    for k in ("cand_off", "sel_off", "trace_off"):
        d[k] = getattr(r, k).copy()
    d["rounds"] = r.rounds
    return d


def check(got, want):
    for k, v in want.items():
        assert np.array_equal(got[k], v), k


@pytest.mark.parametrize("n", [700, 20000])
def test_one_window(apo, n):
    """A batch of one window: its offsets come from the counts on a replay."""
    from paper_2406_18111_gb300 import Apo
    t = tokens_dev(W.periodic_window(n, 50, 0.05, 1000, 3), 4)
    off = np.array([0, n], np.uint64)
    want = snap(apo.find_repeats_batched(t, off, 5))
    assert want["cand_off"][1] == len(want["cand_len"]) > 0 and want["trace_off"][1] > 0
    g = Apo(0)
    try:
        g.graph_mode(True)
        for _ in range(4):
            check(snap(g.find_repeats_batched(t, off, 5, reuse=True)), want)
        assert g.graph_stats()["replays"] >= 2
    finally:
        g.close()


def code(kind, n, seed):
    """n tokens: small values, wide u32 values (a dictionary packs more per key), u64 hashes."""
    a = W.periodic_window(max(n, 1), 50, 0.05, 1000, seed)[:n].astype(np.uint64)
    return {"u32": a, "wide": (a * np.uint64(2654435761)) & np.uint64(0xFFFFFFFF),
            "u64": a * np.uint64(0x9E3779B97F4A7C15)}[kind]


@pytest.mark.parametrize("kind", ["u32", "wide", "u64"])
@pytest.mark.parametrize("lens", [(3000,), (8192,), (0, 700, 1, 0, 8192, 2, 4096, 300, 0), (5,) * 900])
def test_small_windows(apo, kind, lens):
    """Windows of at most 8,192 tokens: the same contents (replayed), changed
    ones of the same shape (discarded, recorded again) and back."""
    from paper_2406_18111_gb300 import Apo
    n = sum(lens)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.uint64)
    tb = 8 if kind == "u64" else 4
    first = tokens_dev(code(kind, n, 7), tb)
    other = first.flip(0).contiguous()
    other[n // 3:n // 3 + n // 9] = other[0]  # a run: other candidates, longer matches
    want = [snap(apo.find_repeats_batched(t, off, 2)) for t in (first, other)]
    assert len(want[0]["cand_len"]) != len(want[1]["cand_len"])
    g = Apo(0)
    try:
        g.graph_mode(True)
        buf = first.clone()
        g.profile_reset()
        for k in (0, 0, 0, 1, 1, 0):
            buf.copy_((first, other)[k])
            check(snap(g.find_repeats_batched(buf, off, 2, reuse=True)), want[k])
        st = g.graph_stats()
        assert st["replays"] >= 3 and st["captures"] >= 2 and st["discarded"] >= 1, st
        assert g.profile_read()["small"][0] >= 6
    finally:
        g.close()
