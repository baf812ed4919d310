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
