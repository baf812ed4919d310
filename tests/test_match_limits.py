"""Matching at its limits: output chains whose flattened length passes 2^32."""
import numpy as np
import pytest

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
