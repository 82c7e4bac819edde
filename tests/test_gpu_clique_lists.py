"""The clique metrics' listing at the edges of its forms, against the CPU oracle:
candidate sets around the warp form's limit (128) and past the shared-memory
matrix (1,216, where the rows are walked), adjacency from the matrix over the
highest degrees and from rows outside it (more than 8,192 vertices), and sets
of 31, 32, 33 and 64 candidates (word boundaries of a matrix row).
"""
import numpy as np
import pytest

from paper_2504_09311_gb300 import synth

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


def graph(n, pairs):
    p = np.unique(np.sort(np.asarray(pairs, np.int64), axis=1), axis=0)
    p = p[p[:, 0] != p[:, 1]]
    return synth.SynthGraph(n, 0, p[:, 0].astype(np.int32), p[:, 1].astype(np.int32))


@pytest.mark.parametrize("n", [32, 33, 34, 65, 129, 130, 131])
def test_complete_graphs_at_word_and_warp_limits(dupin, n):
    """K_n plus a pendant path: the lowest-ranked clique member has n - 1 candidates."""
    iu, iv = np.triu_indices(n, 1)
    pairs = np.r_[np.c_[iu, iv], [[0, n], [n, n + 1]]]
    for q in (3, 4):
        compare(dupin, graph(n + 2, pairs), q, q, (1, 10), 0, (n, q))
        compare(dupin, graph(n + 2, pairs), q, 1, (0, 1), dupin.LPO, (n, q))


@pytest.mark.parametrize("q", [3, 4, 5])
def test_dense_random_past_the_warp_form(dupin, q):
    g = synth.random_general(420 if q < 5 else 300, 44_000 if q < 5 else 20_000, seed=7)
    for k in (1, q):
        compare(dupin, g, q, k, (1, 10), 0, (q, k))


@pytest.mark.parametrize("spokes", [127, 129, 1300])
def test_hub_over_small_cliques(dupin, spokes):
    """A hub joined to one vertex of each of many 6-cliques lies in no 4-clique and leaves first with
    'spokes' surviving candidates; over 8,192 vertices, most of them outside the adjacency matrix."""
    k6 = np.array(np.triu_indices(6, 1)).T
    count = 1400
    pairs = (np.arange(count)[:, None, None] * 6 + k6[None]).reshape(-1, 2)
    hub = np.c_[np.full(spokes, 6 * count), 6 * np.arange(spokes)]
    g = graph(6 * count + 1, np.r_[pairs, hub])
    for q in (3, 4):
        for k, flags in ((q, 0), (1, 0), (q, dupin.LPO)):
            compare(dupin, g, q, k, (0, 1), flags, (spokes, q, k, flags))
