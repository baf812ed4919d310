"""Matching at its limits: output chains whose flattened length passes 2^32,
chains longer than the stream, outputs with too little room, more matches
than 32 bits hold, matches on few positions, source arrays that are no
permutation."""
import ctypes

import numpy as np
import pytest

import oracle
from test_gpu_parity import apo, tokens_dev  # noqa: F401 (apo: the fixture)

pytestmark = pytest.mark.gpu


def nested(copies, deepest):
    """`copies` one-token patterns 7, then 7^2 .. 7^deepest (CSR)."""
    lens = np.r_[np.ones(copies, np.int64), np.arange(2, deepest + 1)]
    off = np.zeros(len(lens) + 1, np.uint64)
    off[1:] = np.cumsum(lens)
    return np.full(int(off[-1]), 7, np.uint32), off


def test_chain_lengths_past_32_bits(apo):
    """2^20 copies of 7 below 7^2 .. 7^4096: the chains add up to 2^32 and some
    8 million entries, which wrapped to a total that looked short enough to
    flatten.  They are walked instead, with and without matches."""
    from paper_2406_18111_gb300 import as_u32
    copies, deepest = 1 << 20, 4096
    pt, off = nested(copies, deepest)
    wrapped = sum(copies + k - 1 for k in range(1, deepest + 1)) - (1 << 32)
    assert 0 < wrapped < 1 << 28
    pats = tokens_dev(pt, 4)
    apo.profile_reset()
    e, _ = apo.match_candidates(pats, off, tokens_dev([9, 8, 9, 9, 8], 4), cap=16)
    prof = apo.profile_read()
    assert len(e) == 0 and "ac.match_offsets" in prof and "ac.ac_fill" not in prof
    e, i = apo.match_candidates(pats, off, tokens_dev([9, 7, 9, 9, 7, 7, 9], 4), cap=4 * copies)
    one = np.arange(copies, dtype=np.uint32)
    assert np.array_equal(as_u32(i), np.r_[one, one, np.uint32(copies), one])
    assert np.array_equal(as_u32(e), np.repeat(np.array([1, 4, 5], np.uint32), [copies, copies, copies + 1]))


def raw_match(a, pats, off, stream, cap):
    """(status, count, ends, ids) with one more entry than cap in both arrays."""
    import torch
    import paper_2406_18111_gb300 as gb
    end = torch.full((cap + 1,), -1, dtype=torch.int32, device="cuda")
    pid = torch.full((cap + 1,), -1, dtype=torch.int32, device="cuda")
    count = ctypes.c_uint64()
    p = gb.apo_patterns(len(off) - 1, pats.data_ptr(), 4, off.ctypes.data, None, None)
    code = gb.lib().apo_match_candidates(a._h, ctypes.byref(p), stream.data_ptr(), stream.shape[0], end.data_ptr(),
                                         pid.data_ptr(), cap, ctypes.byref(count), None)
    torch.cuda.synchronize()
    return code, int(count.value), end.cpu().numpy().view(np.uint32), pid.cpu().numpy().view(np.uint32)


FLAT = 64 * 64 + 63 * 64 // 2  # entries of nested(64, 64)'s flattened chains


@pytest.mark.parametrize("n", [50, FLAT - 1, FLAT, FLAT + 1, 3 * FLAT])
def test_chains_around_the_stream_length(apo, n):
    """Chains that fit beside the stream are flattened before the matches are
    counted, longer ones after; with exactly the room, one entry less, none."""
    import paper_2406_18111_gb300 as gb
    pt, off = nested(64, 64)
    text = np.full(n, 7, np.uint32)
    text[::101] = 9
    oe, oi = oracle.match(pt, off, text)
    pats, stream = tokens_dev(pt, 4), tokens_dev(text, 4)
    for cap in (len(oe), len(oe) - 1, 1000, 0):
        code, count, e, i = raw_match(apo, pats, off, stream, cap)
        assert count == len(oe) and e[cap] == i[cap] == 0xFFFFFFFF
        assert code == (gb.APO_OK if cap == count else gb.APO_ECAPACITY)
        if cap == count:
            assert np.array_equal(e[:-1], oe) and np.array_equal(i[:-1], oi)


def test_no_memory_for_chains_without_a_match():
    """67.6 million entries of flattened chains (270 MB) and no match, or none
    that fits: the context holds no more than for patterns of the same sizes
    whose chains are short."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2406_18111_gb300 as gb
    a = gb.Apo(0)
    pt, off = nested(1 << 16, 1024)
    flat, nest = tokens_dev(np.arange(len(pt)) + 100, 4), tokens_dev(pt, 4)
    none, some = tokens_dev(np.full(4096, 9), 4), tokens_dev(np.full(4096, 7), 4)
    assert raw_match(a, flat, off, none, 16)[:2] == (gb.APO_OK, 0)
    raw_match(a, flat, off, none, 0)
    free = torch.cuda.mem_get_info()[0]
    assert raw_match(a, nest, off, none, 16)[:2] == (gb.APO_OK, 0)
    assert raw_match(a, nest, off, none, 0)[:2] == (gb.APO_OK, 0)
    want = (1 << 16) * 4096 + sum(min(x, 1023) for x in range(4096))
    assert raw_match(a, nest, off, some, 16)[:2] == (gb.APO_ECAPACITY, want)
    assert raw_match(a, nest, off, some, 0)[:2] == (gb.APO_ECAPACITY, want)
    assert free - torch.cuda.mem_get_info()[0] < 32 << 20
    a.close()


@pytest.mark.parametrize("copies,n", [(1 << 20, 4096), (4097, 1 << 20), (4097, 1 << 22)])
def test_more_matches_than_32_bits(apo, copies, n):
    """The count is exact past 2^32 (it was taken modulo 2^32: 0, 2^20 and 2^22
    here), with the chains flattened after the count and before it."""
    import paper_2406_18111_gb300 as gb
    pt, off = nested(copies, 1)
    assert copies * n >= 1 << 32
    code, count, e, i = raw_match(apo, tokens_dev(pt, 4), off, tokens_dev(np.full(n, 7), 4), 1 << 23)
    assert (code, count) == (gb.APO_ECAPACITY, copies * n)
    assert e[-1] == i[-1] == 0xFFFFFFFF


def test_replay_refuses_more_occurrences_than_31_bits(apo):
    """2^20 tokens and the slices 7 .. 7^4200: 4.4e9 occurrences."""
    from paper_2406_18111_gb300 import ApoError
    n, q = 1 << 20, 4200
    start, length = tokens_dev(np.zeros(q), 4), tokens_dev(np.arange(1, q + 1), 4)
    with pytest.raises(ApoError, match="APO_EINVAL.*occurrences"):
        apo.replay(tokens_dev(np.full(n, 7), 4), start, length, start)


@pytest.mark.parametrize("n,start,k,copies", [(1, 0, 1, 4097), (40, 7, 33, 4096), (5000, 1000, 32, 128),
                                              (5000, 1024, 32, 128), (5000, 1024, 32, 129), (5000, 1010, 32, 300),
                                              (20001, 19993, 8, 9000), ((1 << 22) + 5, 4096, 256, 1000),
                                              ((1 << 22) + 5, (1 << 22) - 90, 95, 500), (3, 1, 1, 20000),
                                              (5000, 1024, 64, 256), (5000, 1024, 64, 257),
                                              ((1 << 22) + 5, 4096, 256, 64), ((1 << 22) + 5, 4096, 256, 65)])
def test_matches_on_few_positions(apo, n, start, k, copies):
    """k positions with `copies` matches each: a warp's rows (64 positions, 256 in
    long streams) at and past 16,384 matches, chains of 4,096 and more, rows cut
    by the stream's end."""
    import paper_2406_18111_gb300 as gb
    pt, off = nested(copies, 1)
    text = np.full(n, 9, np.uint32)
    text[start:start + k] = 7
    m = k * copies
    for cap in (m, m - 1):
        code, count, e, i = raw_match(apo, tokens_dev(pt, 4), off, tokens_dev(text, 4), cap)
        assert (code, count) == (gb.APO_OK if cap == m else gb.APO_ECAPACITY, m)
        assert e[cap] == i[cap] == 0xFFFFFFFF
        if cap == m:
            assert np.array_equal(e[:m], np.repeat(np.arange(start, start + k, dtype=np.uint32), copies))
            assert np.array_equal(i[:m], np.tile(np.arange(copies, dtype=np.uint32), k))


@pytest.mark.parametrize("tb", [4, 8])
def test_source_array_that_is_no_permutation(apo, tb):
    """Entries out of range, listed twice, or all the same: APO_EDEVICE, and the
    context goes on."""
    import torch
    import workloads as W
    from paper_2406_18111_gb300 import ApoError, as_u32
    S = W.periodic_window(20000, 113, 0.03, 1000, seed=41)
    t = tokens_dev(S, tb)
    r = apo.find_repeats(t, 5)

    def match(sa):
        return apo.match_candidates(t, None, t, pat_start=r.trace_start, pat_len=r.trace_len, src_sa=sa, src_lcp=r.lcp)

    want = match(r.sa)
    assert len(want[0]) > 1000
    for at, value in (([0], 20000), ([19999], -1), ([7, 12345], 1 << 30), ([100], int(r.sa[200])),
                      (list(range(5000)), 17), (list(range(20000)), 0), (list(range(20000)), -2)):
        bad = r.sa.clone()
        bad[torch.tensor(at, device="cuda")] = value
        with pytest.raises(ApoError, match="APO_EDEVICE"):
            match(bad)
        got = match(r.sa)
        assert all(np.array_equal(as_u32(x), as_u32(y)) for x, y in zip(got, want))


@pytest.mark.parametrize("start,length", [((1 << 32) - 1, 2), ((1 << 32) - 5, 5), (1, (1 << 32) - 1)])
def test_slice_whose_end_wraps(apo, start, length):
    """A slice that ends past 2^32 is refused (its end, taken modulo 2^32, lies
    inside the tokens)."""
    from paper_2406_18111_gb300 import ApoError
    t = tokens_dev(np.arange(50), 4)
    with pytest.raises(ApoError, match="APO_EINVAL"):
        apo.match_candidates(t, None, t, pat_start=tokens_dev([3, start], 4), pat_len=tokens_dev([4, length], 4))
