"""The dense tail (the live core as a matrix over a thread-block cluster) against
the CPU oracle, element by element, through the C ABI.

It takes a cluster-sized tail once the live set's matrix fits the tail's arc
buffer: from the start (the whole graph fits), after the grid-wide rounds, or
after the sparse cluster tail.  Sizes put the slice of a CTA below and above one
pair of columns per thread (512 columns at 256 threads), at odd remainders, and
with many vertices tied at the minimum (more than an inbox record takes).
"""
import numpy as np
import pytest

import oracle
from paper_2504_09311_gb300 import synth

from test_gpu_cluster import assert_same, run_both

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dupin():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2504_09311_gb300 import dupin as d

    d.lib()
    return d


def core(n, draws, metric, seed):
    """A dense random graph on n vertices with a sparse fringe, over 2^20 arcs."""
    rng = np.random.default_rng(seed)
    u, v = rng.integers(0, n, draws), rng.integers(0, n, draws)
    fu, fv = rng.integers(0, n, n), n + np.arange(n)
    a, b = np.minimum(np.r_[u, fu], np.r_[v, fv]), np.maximum(np.r_[u, fu], np.r_[v, fv])
    key = np.unique((a.astype(np.int64) << 32) | b)
    a, b = key >> 32, key & 0xFFFFFFFF
    keep = a != b
    g = synth.SynthGraph(2 * n, 0, a[keep].astype(np.int32), b[keep].astype(np.int32))
    return synth.with_weights(g, metric, seed=seed, a_range=(0, 7) if metric == "dw" else None)


@pytest.mark.parametrize("metric", ["dg", "dw", "fd"])
@pytest.mark.parametrize("n,draws", [(1203, 1_200_000), (2501, 1_100_000), (9001, 2_600_000)])
def test_dense_core(dupin, metric, n, draws):
    g = core(n, draws, metric, n)
    assert 2 * g.m > 1 << 20
    for flags in (0, dupin.TAIL_CLUSTER, dupin.TAIL_CLUSTER | dupin.LPO):
        for k in (1, 2):
            out, ref = run_both(dupin, g, metric, k, (1, 10), flags=flags)
            assert_same(out, ref, (metric, n, flags, k))


@pytest.mark.parametrize("metric", ["dg", "fd"])
def test_sparse_cluster_then_dense(dupin, metric):
    """A ring of equal vertices around a dense core: the cluster tail starts with more vertices than the
    matrix takes (the hand-over is forced early) and leaves the core to the dense tail."""
    rng = np.random.default_rng(5)
    c, n = 1500, 60_000
    u, v = rng.integers(0, c, 1_000_000), rng.integers(0, c, 1_000_000)
    ru = np.repeat(np.arange(c, n), 3)
    rv = c + (ru - c + np.tile([1, 2, 3], n - c)) % (n - c)
    a, b = np.minimum(np.r_[u, ru], np.r_[v, rv]), np.maximum(np.r_[u, ru], np.r_[v, rv])
    key = np.unique((a.astype(np.int64) << 32) | b)
    a, b = key >> 32, key & 0xFFFFFFFF
    keep = a != b
    g = synth.SynthGraph(n, 0, a[keep].astype(np.int32), b[keep].astype(np.int32))
    synth.with_weights(g, metric, seed=1)
    for flags in (dupin.TAIL_CLUSTER, dupin.TAIL_CLUSTER | dupin.GPO):
        out, ref = run_both(dupin, g, metric, 1, (0, 1), flags=flags, tail_arc_cap=1 << 26)
        assert_same(out, ref, (metric, flags))
        assert out.tail_ctas in (8, 16)
        assert out.n_min_rule > 0


def test_ties_longer_than_an_inbox_record(dupin):
    """A complete multipartite core: every vertex of a part ties, so minimum-rule rounds take hundreds."""
    parts, size = 8, 190
    n = parts * size
    iu, iv = np.triu_indices(n, 1)
    keep = iu // size != iv // size
    g = synth.SynthGraph(n, 0, iu[keep].astype(np.int32), iv[keep].astype(np.int32))
    g.c = ((2 + (g.eu // size) + (g.ev // size)).astype(np.int64)) << 32
    for metric in ("dg", "dw"):
        out, ref = run_both(dupin, g, metric, 1, (0, 1), flags=dupin.TAIL_CLUSTER)
        assert_same(out, ref, metric)
