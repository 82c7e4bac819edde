"""Loading a graph whose initial peeling weights sit at the edges of 2^63 and
2^64: a row's sum just past 2^63 together with a vertex weight that carries it
past 2^64 is refused, as every weight of 2^63 or more is.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOP = 1 << 63


@pytest.fixture(scope="module")
def dupin():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2504_09311_gb300 import dupin as d

    d.lib()
    return d


def star(dupin, leaves, w, a0):
    """A star whose hub has vertex weight a0 and `leaves` arcs of weight w."""
    n = leaves + 1
    ptr = np.r_[0, leaves + np.arange(n)].astype(np.int64)
    col = np.r_[1 + np.arange(leaves), np.zeros(leaves, int)].astype(np.int32)
    a = np.zeros(n, np.int64)
    a[0] = a0
    return dupin.Graph.load_symmetric(n, ptr, col, np.full(2 * leaves, w, np.int64), a)


# the sum of the arcs' upper halves stays below 2^31, so only the full sum tells;
# 3,000 leaves: the hub's row spans two tiles
@pytest.mark.parametrize("leaves", [3, 5, 7, 2_000, 3_000])
def test_sums_past_the_limit_with_a_vertex_weight(dupin, leaves):
    w = -(-TOP // leaves)  # leaves * w is 2^63 or a little more
    assert TOP <= leaves * w < TOP + (1 << 43) and leaves * (w >> 32) < 1 << 31
    over = leaves * w - TOP
    for a0 in (0, 1, TOP - 1 - over, TOP - 1):
        with pytest.raises(dupin.DupinError) as e:
            star(dupin, leaves, w, a0)
        assert e.value.code == dupin.ERR_OVERFLOW, (leaves, a0)
    below = (TOP - 1) // leaves
    rest = TOP - 1 - leaves * below
    star(dupin, leaves, below, rest).free()  # 2^63 - 1 exactly
    with pytest.raises(dupin.DupinError) as e:
        star(dupin, leaves, below, rest + 1)
    assert e.value.code == dupin.ERR_OVERFLOW
