"""The optimum where min_len is longer than any window: nothing is chosen."""
import numpy as np
import pytest

from test_gpu_parity import apo, tokens_dev  # noqa: F401 (apo: the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("min_len", [13, 24, 25, 1000, (1 << 31) - 1, 1 << 31, (1 << 32) - 1])
def test_longer_than_the_windows(apo, min_len):
    lens = (24, 0, 1, 16, 24)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.uint64)
    best, _, _, count = apo.optimum_batched(tokens_dev(np.arange(int(off[-1])) % 2, 4), off, min_len)
    assert best.cpu().numpy().tolist() == [[0, 0, 0]] * len(lens)
    assert count.cpu().numpy().tolist() == [0] * len(lens)
