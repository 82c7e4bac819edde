"""The clique metrics on graphs whose vertices mostly lie outside the adjacency
matrix of the 8,192 highest degrees, so that rows are read (or searched, the
long ones): candidate sets for one warp and for a CTA, rows on both sides of the
reading limit, against the CPU oracle; and bounds on the time of uniform graphs,
where every row is of middling length.
"""
import time

import numpy as np
import pytest

from paper_2504_09311_gb300 import synth

from test_gpu_clique_lists import graph
from test_gpu_kclids import compare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dupin():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2504_09311_gb300 import dupin as d

    d.lib()
    return d


def clusters(n, draws, size, count, hubs, hub_deg, seed):
    """A uniform graph with `count` planted cliques of `size` vertices and `hubs` rows of hub_deg arcs."""
    rng = np.random.default_rng(seed)
    parts = [rng.integers(0, n, (draws, 2))]
    iu, iv = np.triu_indices(size, 1)
    for _ in range(count):
        v = rng.choice(n, size, replace=False)
        parts.append(np.c_[v[iu], v[iv]])
    for h in rng.choice(n, hubs, replace=False):
        parts.append(np.c_[np.full(hub_deg, h), rng.choice(n, hub_deg)])
    return graph(n, np.concatenate(parts))


# degrees of about 12, 40 (one warp), 250 and 500 (a CTA), with cliques among and hubs over them
@pytest.mark.parametrize("n,draws,size,count,hubs,hub_deg", [
    (12_000, 70_000, 9, 300, 0, 0), (12_000, 70_000, 20, 60, 30, 700), (9_500, 190_000, 34, 30, 10, 5_000),
    (9_000, 1_100_000, 40, 8, 3, 6_000), (8_600, 2_200_000, 30, 4, 0, 0)])
@pytest.mark.parametrize("q", [3, 4])
def test_rows_outside_the_matrix(dupin, n, draws, size, count, hubs, hub_deg, q):
    g = clusters(n, draws, size, count, hubs, hub_deg, seed=n + q)
    compare(dupin, g, q, q, (1, 10), 0, (n, draws, q))
    if draws < 100_000:
        compare(dupin, g, q, 2, (1, 10), dupin.LPO, (n, draws, q))


@pytest.mark.parametrize("n,draws,ms", [(1_000_000, 8_000_000, 5.5), (300_000, 18_000_000, 30.0)])
def test_time_on_uniform_graphs(dupin, n, draws, ms):
    """TDS, k = 3: 2.9 and 15 ms (7.8 and 54 ms when every pair of candidates was searched in a row)."""
    import torch

    dg = dupin.Graph.from_synth(synth.random_general(n, draws, seed=3))
    pr = torch.empty(n, dtype=torch.int32, device="cuda")
    p = dupin.make_params("tds", 3, (1, 10))
    best = 1e9
    for _ in range(5):
        torch.cuda.synchronize()
        t = time.perf_counter()
        dupin.peel_device(dg, p, pr)
        best = min(best, (time.perf_counter() - t) * 1e3)
    dg.free()
    assert best < ms, best
