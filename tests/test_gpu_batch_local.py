"""Batched peels at the edges of the move into shared memory, against the CPU
oracle: graphs that fit a CTA from the start and ones that fit after some
rounds (by the launch shape's shared memory), rounds of more than 32 vertices on
both sides of the move, rows longer than a warp takes alone, hub rows, sums
beyond 64 bits, and the launch shapes' graph counts.
"""
import numpy as np
import pytest

import oracle
from paper_2504_09311_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dupin():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2504_09311_gb300 import dupin as d

    d.lib()
    return d


def check(dupin, graphs, metric, k, eps=(1, 10), flags=0):
    dgs = [dupin.Graph.from_synth(g) for g in graphs]
    p = dupin.make_params(metric, k, eps, flags=flags)
    of = (oracle.FLAG_GPO if flags & dupin.GPO else 0) | (oracle.FLAG_LPO if flags & dupin.LPO else 0)
    for want_trace in (True, False):
        outs = dupin.peel_batch(dgs, [p] * len(dgs), want_trace=want_trace, want_mask=want_trace)
        for j, (g, o) in enumerate(zip(graphs, outs)):
            og = oracle.Graph.from_synth(g, metric)
            r = oracle.peel_batch(og, k, eps, flags=of)
            og.close()
            ctx = (j, g.n, metric, k, flags)
            assert np.array_equal(o.peel_round, r.peel_round), ctx
            assert (o.n_rounds, o.best_round, o.best_size, o.best_f) == (r.n_rounds, r.best_round, r.best_size, r.best_f), ctx
            assert o.n_min_rule == r.n_min_rule, ctx
            if want_trace:
                assert o.trace_f == r.trace_f, ctx
                assert np.array_equal(np.asarray(o.trace_size), r.trace_size), ctx
                assert np.array_equal(o.best_mask, r.best_mask), ctx
    for d in dgs:
        d.free()


# vertices whose state fits a CTA: about 2,900 at four CTAs per SM, 5,900 at two, 11,800 at one
@pytest.mark.parametrize("threads", [0, 128, 256])
@pytest.mark.parametrize("metric", ["fd", "dg"])
def test_around_the_shared_memory_limit(dupin, threads, metric):
    dupin.batch_threads(threads)
    try:
        graphs = []
        for n in (63, 64, 65, 2_850, 2_950, 5_800, 6_000, 11_700, 12_000, 30_000):
            g = synth.bipartite_zipf(n - n // 3, n // 3, 5 * n, 1.8, 1, 40, 40, 0.6, 5, seed=n)
            graphs.append(synth.with_weights(g, metric))
        for k, flags in ((1, 0), (1, dupin.LPO), (2, 0)):
            check(dupin, graphs, metric, k, flags=flags)
    finally:
        dupin.batch_threads(0)


@pytest.mark.parametrize("count", [153, 305])
def test_launch_shapes_by_graph_count(dupin, count):
    """One CTA per SM up to 152 graphs, two up to 304, four beyond."""
    graphs = []
    for j in range(count):
        g = synth.bipartite_zipf(120 + j, 60 + j // 2, 900 + 7 * j, 1.8, 0, 0, 0, 0.0, 0, seed=j)
        graphs.append(synth.with_weights(g, "fd"))
    check(dupin, graphs, "fd", 1)


def test_long_rows_hubs_and_wide_sums(dupin):
    star = synth.SynthGraph(1500, 0, np.zeros(1499, np.int32), np.arange(1, 1500, dtype=np.int32))
    star.c = (1 + np.arange(1499) % 97).astype(np.int64) << 32
    rmat = synth.rmat_weighted(12, 24, "dw", seed=5)  # hub rows above 1,024 arcs
    wide = synth.random_general(700, 9000, seed=3)  # f beyond 2^62
    wide.c = np.full(wide.m, (1 << 56) + 12345, np.int64) - np.arange(wide.m)
    for k in (1, 2):
        check(dupin, [star, rmat, wide], "dw", k)
        check(dupin, [star, rmat, wide], "dw", k, flags=dupin.GPO)
