"""Windows that one block analyses whole (up to 8,192 tokens each) against the
oracle and against the general path: a batch holding one longer window takes
the general path for all of its windows, and a window's results do not depend
on the batch.  Sizes lie at the edges of warps, of the block shapes and of the
path itself; the contents make the doubling count comparisons directly, sort,
or alternate, and leave matches that the LCP finishes by lifting."""
import numpy as np
import pytest

import oracle
import workloads as W
from test_gpu_parity import FIELDS, apo, compare, tokens_dev  # noqa: F401 (apo: the fixture)

pytestmark = pytest.mark.gpu

SIZES = (1, 2, 31, 33, 64, 255, 511, 512, 513, 1024, 2047, 2048, 2049, 4095, 4096, 4097, 8191, 8192)


def window(kind, n, seed):
    j = np.arange(n)
    if kind == "loop":
        return W.periodic_window(n, 50, 0.05, 1000, seed)
    if kind == "run":  # one token, then a short period
        return np.where(j < n // 2, 7, j % 3).astype(np.uint32)
    if kind == "random":
        return (W.splitmix64(seed, n) >> np.uint64(32)).astype(np.uint32)
    if kind == "few":
        return W.uniform_int(seed, n, 0, 2).astype(np.uint32)
    tok = oracle.hash_tasks(W.config2_tasks(max(n, 8), seed=seed))[:n].copy()
    tok[::97] = np.uint64(0xFFFFFFFFFFFFFFFF)
    return tok


@pytest.mark.parametrize("kind,tb", [("loop", 4), ("run", 4), ("random", 8), ("few", 4), ("tasks", 8)])
def test_single_windows(apo, kind, tb):
    for k, n in enumerate(SIZES):
        compare(apo, window(kind, n, 40 + k), 1 if n < 100 else 5, tb=tb, sa_method="doubling")


@pytest.mark.parametrize("tb,hi", [(4, 500), (8, 5000), (4, 8192)])
def test_batches_equal_the_general_path(apo, tb, hi):
    from paper_2406_18111_gb300 import as_u32
    kinds = ("loop", "run", "few") if tb == 4 else ("tasks", "random", "loop")
    lens = np.r_[0, W.log_uniform_int(W.uniform01(hi, 60), 3, hi), hi, 0]
    lens = np.insert(lens, np.arange(1, len(lens), 3), 1)  # one-token windows between the others
    wins = [window(kinds[w % 3], int(n), 900 + w) for w, n in enumerate(lens)]

    def run(ws):
        off = np.zeros(len(ws) + 1, np.uint64)
        off[1:] = np.cumsum([len(x) for x in ws])
        return apo.find_repeats_batched(tokens_dev(np.concatenate([np.asarray(x, np.uint64) for x in ws]), tb), off, 5)

    small, general = run(wins), run(wins + [window("few", 8193, 5)])
    W_ = len(wins)
    assert np.array_equal(small.win_off, general.win_off[:W_ + 1])
    for name in ("cand_off", "sel_off", "trace_off"):
        assert np.array_equal(getattr(small, name), getattr(general, name)[:W_ + 1]), name
    at = {"sa": small.win_off, "lcp": small.win_off, "sel_start": small.sel_off, "sel_len": small.sel_off,
          "sel_trace": small.sel_off, "trace_len": small.trace_off, "trace_start": small.trace_off}
    for f in FIELDS + ("cand_accepted",):
        end = int(at.get(f, small.cand_off)[-1])
        a, b = getattr(small, f), getattr(general, f)
        assert a.shape[0] == end and bool((a == b[:end]).all()), f


def test_capacities_and_missing_outputs(apo):
    """The counts are exact and nothing is written past a capacity."""
    import ctypes
    import torch
    import paper_2406_18111_gb300 as gb
    S = W.config1_window()
    want = oracle.find_repeats(S.astype(np.uint64), 5)
    tok = tokens_dev(S, 4)
    for cap in (0, 3, len(want.sel_start)):
        sel = torch.full((len(want.sel_start) + 1,), -1, dtype=torch.int32, device="cuda")
        counts = np.zeros(4, np.uint64)
        o = gb.apo_repeats_out(None, None, None, None, None, None, 0, sel.data_ptr(), None, None, cap, None, None, 0,
                               counts.ctypes.data, None, None, None)
        code = gb.lib().apo_find_repeats(apo._h, ctypes.byref(gb.apo_window(len(S), tok.data_ptr(), 4)),
                                         ctypes.byref(gb.apo_repeats_params(5, 0)), ctypes.byref(o), None)
        torch.cuda.synchronize()
        assert code == (gb.APO_OK if cap == len(want.sel_start) else gb.APO_ECAPACITY)
        assert counts[:3].tolist() == [len(want.cand_len), len(want.sel_start), len(want.trace_len)]
        got = sel.cpu().numpy().view(np.uint32)
        assert np.array_equal(got[:cap], want.sel_start[:cap]) and (got[cap:] == 0xFFFFFFFF).all()
