"""Token dictionaries at the size where a thread takes four tokens instead of
one (1,536 per SM in a window, 2,048 in patterns), with repeated, distinct and absent tokens and the all-ones
token, against the oracle."""
import numpy as np
import pytest

import oracle
import workloads as W
from test_gpu_parity import apo, compare, tokens_dev  # noqa: F401 (apo: the fixture)

pytestmark = pytest.mark.gpu


def edge(per_sm):
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count * per_sm


@pytest.mark.parametrize("tb", [4, 8])
@pytest.mark.parametrize("more", [-1, 0, 1, 1025])
def test_window(apo, tb, more):
    n = edge(1536) + more
    S = W.splitmix64(21, n) >> np.uint64(1 if tb == 8 else 33)
    S[n // 3:n // 2] = W.periodic_window(n // 2 - n // 3, 50, 0.05, 1000, 9)
    S[::5003] = np.uint64(2**64 - 1 if tb == 8 else 2**32 - 1)
    compare(apo, S, 5, tb=tb, sa_method="doubling")


@pytest.mark.parametrize("tb", [4, 8])
@pytest.mark.parametrize("more", [-1, 0, 1, 1025])
def test_patterns(apo, tb, more):
    from paper_2406_18111_gb300 import as_u32
    n = edge(2048) + more
    P = 3000
    pt = W.splitmix64(31, n) >> np.uint64(1 if tb == 8 else 33)
    pt[::7] = np.uint64(2**64 - 1 if tb == 8 else 2**32 - 1)
    pt[::3] = W.uniform_int(33, len(pt[::3]), 0, 2)
    off = np.linspace(0, n, P + 1).astype(np.uint64)
    text = W.splitmix64(32, 100000) >> np.uint64(1 if tb == 8 else 33)  # tokens that no pattern has
    for p in range(0, P, 40):  # every 40th pattern occurs
        a, b = int(off[p]), int(off[p + 1])
        text[p * 30:p * 30 + b - a] = pt[a:b]
    e, i = apo.match_candidates(tokens_dev(pt, tb), off, tokens_dev(text, tb))
    oe, oi = oracle.match(pt, off, text)
    assert len(oe) >= P // 40
    assert np.array_equal(as_u32(e), oe) and np.array_equal(as_u32(i), oi)
