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


@pytest.mark.parametrize("tb", [4, 8])
@pytest.mark.parametrize("lens", [(8192,) * 3, (700, 0, 5000, 1, 64), tuple(i % 3 for i in range(6000)), (1,)])
def test_caller_workspace(apo, lens, tb):
    """A caller workspace of exactly the queried size holds the small windows'
    scratch, for many tiny windows as well; a byte less is refused."""
    import torch
    from paper_2406_18111_gb300 import Apo, ApoError
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.uint64)
    t = tokens_dev(window("loop", int(off[-1]), 8).astype(np.uint64) * np.uint64(2654435761 if tb == 4 else 1 << 33), tb)
    want = apo.find_repeats_batched(t, off, 2)
    a = Apo(0)
    need = a.find_repeats_workspace(off)
    buf = torch.empty(need, dtype=torch.uint8, device="cuda")
    a.set_workspace(buf)
    a.profile_reset()
    for _ in range(2):
        got = a.find_repeats_batched(t, off, 2)
        for f in FIELDS + ("cand_accepted",):
            assert bool((getattr(got, f) == getattr(want, f)).all()), f
        for f in ("cand_off", "sel_off", "trace_off"):
            assert np.array_equal(getattr(got, f), getattr(want, f)), f
    assert a.profile_read()["small"][0] == 2
    a.set_workspace(buf[:need - 1])
    with pytest.raises(ApoError, match="APO_ENOMEM"):
        a.find_repeats_batched(t, off, 2)
    a.set_workspace(None)
    a.close()


def rounds_of(S, lcp, windows=1):
    """The doubling rounds reported: the first key holds h0 tokens (as plain
    values, or dense codes where fewer than four of those fit), and round r runs
    iff some LCP is at least h0 * 2^(r-1)."""
    S = np.asarray(S, np.uint64)
    top = int(S.max())
    bits = (windows - 1).bit_length() if windows > 1 else 0
    h0 = (64 - bits) // (top + 1).bit_length() if top < 1 << 32 else 0
    if h0 < 4 and len(S) >= 4096:
        sigma = len(np.unique(S[S != np.uint64(2**64 - 1)]))
        cap = min(1 << (2 * len(S) - 1).bit_length(), 1 << 23)
        if sigma <= cap // 2:
            h0 = max(h0, (64 - bits) // (sigma + 1).bit_length())
    h0 = min(h0, 32) if h0 >= 2 else 1
    r = 0
    while int(lcp.max()) >= h0 << r:
        r += 1
    return r


@pytest.mark.parametrize("kind,tb", [("loop", 4), ("run", 4), ("random", 4), ("random", 8), ("few", 4), ("tasks", 8)])
@pytest.mark.parametrize("n", [1, 64, 1000, 4095, 4096, 8192, 8193, 1 << 15])
def test_rounds_reported(apo, kind, tb, n):
    """The same count from both paths (here and just past 8,192 tokens)."""
    from paper_2406_18111_gb300 import as_u32
    S = window(kind, n, 70 + n)
    r = apo.find_repeats(tokens_dev(S, tb), 5)
    assert r.rounds == rounds_of(S, as_u32(r.lcp))


@pytest.mark.parametrize("tb", [4, 8])
@pytest.mark.parametrize("lens", [(1300000,), ((1 << 21) + (1 << 14),), (700000, 0, 9000, 1, 600000)])
def test_mostly_distinct_windows(apo, lens, tb):
    """Millions of nearly distinct tokens: where a first key would hold two of
    them (the last two shapes) it holds one, with the window in a batch; the
    rounds reported stay those of two."""
    from paper_2406_18111_gb300 import as_u32
    n = sum(lens)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.uint64)
    S = W.splitmix64(11, n) >> np.uint64(34)  # 30-bit values
    S[500:800] = S[100:400]
    S[9500:11000] = S[15000:16500]
    S[n - 3000:n - 2000] = 5  # a run
    r = apo.find_repeats_batched(tokens_dev(S, tb), off, 5)
    assert r.rounds == rounds_of(S, as_u32(r.lcp), len(lens)) > 5
    for w in range(len(lens)):
        a, b = int(off[w]), int(off[w + 1])
        if b - a < 2:
            continue
        o = oracle.find_repeats(S[a:b], 5, sa_method="doubling")
        assert np.array_equal(as_u32(r.sa)[a:b], o.sa) and np.array_equal(as_u32(r.lcp)[a:b], o.lcp)
        s0, s1, t0, t1 = (int(x) for x in (r.sel_off[w], r.sel_off[w + 1], r.trace_off[w], r.trace_off[w + 1]))
        assert np.array_equal(as_u32(r.sel_start)[s0:s1], o.sel_start)
        assert np.array_equal(as_u32(r.trace_len)[t0:t1], o.trace_len)


@pytest.mark.parametrize("windows,n,tb,small", [(10000, 600, 8, False), (50000, 250, 8, False), (20000, 128, 4, False),
                                                (12000, 2, 8, False), (6000, 2, 8, True),
                                                (5000, 600, 8, True), (10000, 64, 8, True), (300, 8192, 4, True)])
def test_many_windows_take_the_faster_path(apo, windows, n, tb, small):
    """Thousands of short windows go the general path where its shared launches
    are the faster ones; the results are those of smaller batches, which go
    window by window."""
    t = tokens_dev(window("few", windows * n, 3), tb)
    off = np.arange(windows + 1, dtype=np.uint64) * np.uint64(n)
    apo.profile_reset()
    r = apo.find_repeats_batched(t, off, 5, stages=False)
    assert ("small" in apo.profile_read()) == small
    at, step = 0, 1250
    for w in range(0, windows, step):
        k = min(step, windows - w)
        apo.profile_reset()
        p = apo.find_repeats_batched(t[w * n:(w + k) * n], off[:k + 1], 5, stages=False)
        assert "small" in apo.profile_read()
        for f, o in (("sel_start", "sel_off"), ("sel_len", "sel_off"), ("sel_trace", "sel_off"),
                     ("trace_len", "trace_off"), ("trace_start", "trace_off")):
            ro, po = getattr(r, o), getattr(p, o)
            assert np.array_equal(ro[w:w + k + 1] - ro[w], po), o
            assert bool((getattr(r, f)[int(ro[w]):int(ro[w + k])] == getattr(p, f)).all()), f


@pytest.mark.parametrize("distinct,loops", [(14 << 20, 2 << 20), (12 << 20, 12 << 20)])
def test_key_length_does_not_depend_on_the_order(apo, distinct, loops):
    """Three times as many distinct tokens as the dictionary takes (2^22), and
    loops before, behind or between them: the same first key, which shows in the
    rounds run."""
    a = W.splitmix64(5, distinct) >> np.uint64(33)
    b = W.periodic_window(loops, 50, 0.05, 1000, 6).astype(np.uint64)
    seen = set()
    for S in (np.r_[a, b], np.r_[b, a], np.r_[a[:distinct // 2], b, a[distinct // 2:]]):
        apo.profile_reset()
        r = apo.find_repeats(tokens_dev(S, 4), 5, stages=False)
        seen.add((apo.profile_read()["minor"][0], r.rounds))
    assert len(seen) == 1, seen
