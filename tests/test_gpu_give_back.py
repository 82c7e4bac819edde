"""Peels that their cluster tail gives back to the grid-wide rounds, against the
oracle: alone, two in one batched call (their stages side by side on several
streams) and six (one after another).

An R-MAT graph of more than 2^27 arcs, handed over as soon as a tail holds it
(tail_arc_cap = 2^27), still collapses: the cluster's first round takes thousands
of vertices by the threshold, the next would too, and the peel goes back.
"""
import numpy as np
import pytest

import oracle
from paper_2504_09311_gb300 import synth

pytestmark = pytest.mark.gpu

ARCS = 1 << 27      # only graphs of at least this many arcs are given back ...
ROUND = 256         # ... after a round of this many vertices
DENSE = 32_768      # the most vertices that a dense tail takes in place of the cluster


@pytest.fixture(scope="module")
def env():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2504_09311_gb300 import dupin as d

    d.lib()
    g = synth.rmat_weighted(22, 20, "fd", seed=1)
    assert 2 * g.m >= ARCS
    refs = {}
    for m in ("fd", "dg"):
        og = oracle.Graph.from_synth(g, m)
        refs[m] = oracle.peel_batch(og, 1, (1, 10))
        og.close()
    dg = d.Graph.from_synth(g)
    yield torch, d, dg, refs
    dg.free()
    d.trim_cache()


@pytest.mark.parametrize("metrics", [["fd"], ["dg"], ["fd", "dg"], ["dg", "fd"], ["fd", "fd"], ["fd", "dg"] * 3])
def test_given_back_peels_equal_the_oracle(env, metrics):
    torch, dupin, dg, refs = env
    params = [dupin.make_params(m, 1, (1, 10), tail_arc_cap=ARCS) for m in metrics]
    rounds = [torch.empty(dg.n, dtype=torch.int32, device="cuda") for _ in metrics]
    masks = [torch.empty(dg.n, dtype=torch.uint8, device="cuda") for _ in metrics]
    for _ in range(2):
        for x in rounds:
            x.zero_()
        if len(metrics) == 1:
            out = [dupin.peel_device(dg, params[0], rounds[0], masks[0])]
        else:
            out = dupin.peel_batch_device([dg] * len(metrics), params, rounds, masks)
        torch.cuda.synchronize()
        for m, r, pr, mk in zip(metrics, out, rounds, masks):
            ref = refs[m]
            b = r.n_bulk_rounds  # rounds before the first tail: the cluster's, then given back
            assert DENSE < ref.trace_size[b] and list(ref.trace_kind[b + 1:b + 3]) == [0, 0], (m, b)
            assert ref.trace_peeled[b + 1] >= ROUND, (m, b)
            assert r.tail_ctas > 1, m
            assert np.array_equal(pr.cpu().numpy(), ref.peel_round), m
            assert np.array_equal(mk.cpu().numpy(), ref.best_mask), m
            assert (r.n_rounds, r.best_round, r.best_size) == (ref.n_rounds, ref.best_round, ref.best_size), m
            assert (int(r.best_f_hi) << 64) + int(r.best_f_lo) == ref.best_f and r.n_min_rule == ref.n_min_rule, m
