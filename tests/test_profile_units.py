"""The units that the profiler records for sorts which skip digit places."""
import numpy as np
import pytest

from test_gpu_parity import apo, tokens_dev  # noqa: F401 (apo: the fixture)

pytestmark = pytest.mark.gpu


def test_skipped_places_move_nothing(apo):
    """A constant window of n tokens: 16 tokens make the first key, and the
    doubling round at distance h sorts one group of n - h + 1 suffixes by minor
    keys of 0 .. h, above which every digit of its keys is the same.  Each place
    that differs moves the entries once; the others count for nothing."""
    n = 1 << 18
    t = tokens_dev(np.full(n, 7), 4)
    want = sum((n - h + 1) * (1 if h < 1 << 8 else 2 if h < 1 << 16 else 3) for h in (16 << k for k in range(14)))
    apo.sort_tuning(1)  # 8-bit digits
    try:
        apo.profile_reset()
        r = apo.find_repeats(t, 5, stages=False)
        launches, _, units = apo.profile_read()["rs_pass_keys"]
    finally:
        apo.sort_tuning(0)
    assert r.rounds == 14
    assert units == want and launches >= 14 * 4
