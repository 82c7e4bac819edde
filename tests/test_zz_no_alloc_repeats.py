"""dupin_peel_noalloc on rows that dupin_graph_load would refuse: a neighbour
listed more than once, and rows in any order.  Every arc counts by itself, so
the peel equals the oracle's on the simple graph whose edge weights are the sums
over the repeats.
"""
import numpy as np
import pytest

import oracle
from paper_2504_09311_gb300 import synth

pytestmark = pytest.mark.gpu

Q = 1 << 32


@pytest.fixture(scope="module")
def env():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2504_09311_gb300 import dupin

    dupin.lib()
    return torch, dupin


def multigraph(n, draws, most, order, seed):
    """A random graph with each edge 1 .. most times, as a symmetric CSR with whole weights per repeat,
    and the simple graph of summed weights.  order: "sorted" or "any" (rows shuffled)."""
    rng = np.random.default_rng(seed)
    e = np.sort(rng.integers(0, n, (draws, 2)), 1)
    e = np.unique(e[e[:, 0] != e[:, 1]], axis=0)
    rep = rng.integers(1, most + 1, len(e))
    at = np.repeat(np.arange(len(e)), rep)
    w = rng.integers(1, 10, len(at))
    a = rng.integers(0, 5, n)
    u, v = np.r_[e[at, 0], e[at, 1]], np.r_[e[at, 1], e[at, 0]]
    ww = np.r_[w, w]
    o = np.lexsort((rng.random(len(u)) if order == "any" else v, u))
    u, v, ww = u[o], v[o], ww[o]
    ptr = np.searchsorted(u, np.arange(n + 1))

    def simple(per_arc):
        g = synth.SynthGraph(n, 0, e[:, 0].astype(np.int32).copy(), e[:, 1].astype(np.int32).copy())
        g.c = np.bincount(at, per_arc, len(e)).astype(np.int64) * Q
        return g

    return ptr, v, ww, a, simple(w), simple(np.ones(len(at)))


# rows of about 12, 60 and 110 arcs (one warp's rounds take up to 128), and longer ones
@pytest.mark.parametrize("n,draws,most", [(40, 90, 3), (300, 4_500, 3), (700, 19_000, 3), (500, 20_000, 4), (2_000, 6_000, 9)])
@pytest.mark.parametrize("order", ["sorted", "any"])
def test_repeated_pairs_count_each(env, n, draws, most, order):
    torch, dupin = env
    for seed in (1, 2):
        ptr, idx, w, a, dw, dg = multigraph(n, draws, most, order, seed)
        dw.a = a.astype(np.int64) * Q
        d = lambda x, t: torch.tensor(x, dtype=t, device="cuda")  # noqa: E731
        dptr, didx = d(ptr, torch.int64), d(idx, torch.int32)
        for metric, simple, dwt, da in (("dw", dw, d(w * Q, torch.int64), d(a * Q, torch.int64)), ("dg", dg, None, None)):
            og = oracle.Graph.from_synth(simple, "dw")
            for k, eps, flags, of in ((1, (1, 10), 0, 0), (1, (0, 1), 0, 0), (2, (1, 10), 0, 0),
                                      (1, (1, 10), dupin.LPO, oracle.FLAG_LPO)):
                ref = oracle.peel_batch(og, k, eps, flags=of)
                pr = torch.empty(n, dtype=torch.int32, device="cuda")
                r = dupin.peel_noalloc(n, dptr, didx, dwt, da, dupin.make_params(metric, k, eps, flags=flags), pr)
                ctx = (metric, k, eps, flags, seed)
                assert np.array_equal(pr.cpu().numpy(), ref.peel_round), ctx
                assert (r.n_rounds, r.best_round, r.best_size) == (ref.n_rounds, ref.best_round, ref.best_size), ctx
                assert (int(r.best_f_hi) << 64) + int(r.best_f_lo) == ref.best_f, ctx
            og.close()
