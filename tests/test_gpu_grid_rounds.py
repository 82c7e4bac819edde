"""The initial weights by tiles of arcs and the grid-wide rounds, against the CPU
oracle: arc counts on both sides of a tile's edge (2,048 arcs), rows that span
several tiles, runs of empty rows at the start, in the middle and at the end,
vertex counts on both sides of a 32-vertex rank word, and peels that stay in the
grid-wide kernel to the end, through many compactions, by threshold and by
minimum-rule rounds.
"""
import numpy as np
import pytest

from paper_2504_09311_gb300 import synth

from test_gpu_parity import assert_same, run_both

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dupin():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2504_09311_gb300 import dupin as d

    d.lib()
    return d


def exact(n, m, hub, gaps, seed):
    """m edges on n vertices: a hub row of `hub` arcs, the rest at random, none in the id ranges of `gaps`."""
    rng = np.random.default_rng(seed)
    ids = np.setdiff1d(np.arange(n), np.concatenate([np.arange(a, b) for a, b in gaps] or [np.zeros(0, int)]))
    h = ids[len(ids) // 3]
    others = ids[ids != h]
    keys = set()
    for v in rng.permutation(others)[:hub]:
        keys.add((min(h, v), max(h, v)))
    while len(keys) < m:
        a, b = rng.choice(others, 2, replace=False)
        keys.add((min(a, b), max(a, b)))
    e = np.array(sorted(keys), np.int32)
    assert len(e) == m
    return synth.SynthGraph(n, 0, e[:, 0].copy(), e[:, 1].copy())


CASES = [
    # n, m, hub, gaps
    (33, 1, 1, []),
    (64, 512, 63, []),
    (95, 1023, 90, [(0, 2)]),
    (97, 1024, 90, [(93, 97)]),
    (128, 1025, 90, [(40, 72)]),
    (2_050, 2_047, 2_000, []),  # the hub's row ends a tile or spans two
    (2_111, 3_072, 1_024, [(0, 70), (900, 1_300), (2_000, 2_111)]),
    (7_000, 12_289, 6_500, [(1, 300), (6_900, 7_000)]),  # a row over four tiles
]


@pytest.mark.parametrize("metric", ["dg", "dw", "fd"])
@pytest.mark.parametrize("n,m,hub,gaps", CASES)
def test_tiles_and_grid_wide_rounds(dupin, metric, n, m, hub, gaps):
    g = synth.with_weights(exact(n, m, hub, gaps, n), metric, seed=n, a_range=(0, 5) if metric == "dw" else None)
    for k, eps in ((1, (1, 10)), (2, (1, 10)), (1, (0, 1))):
        for flags in (0, dupin.LPO):
            out, ref = run_both(dupin, g, metric, k, eps, flags=flags, tail_cap=1)
            assert_same(out, ref, (metric, n, m, k, eps, flags))


@pytest.mark.parametrize("k", [1, 2])
def test_wide_weights_by_tiles(dupin, k):
    """Sums that need all 63 bits of a weight and 128 bits of f."""
    g = exact(1_201, 6_145, 1_100, [(500, 600)], 7)
    g.c = (1 << 50) + np.arange(g.m, dtype=np.int64) * 977
    g.a = np.arange(g.n, dtype=np.int64) << 40
    out, ref = run_both(dupin, g, "dw", k, (1, 10), tail_cap=1)
    assert_same(out, ref, k)


def load(dupin, n, ptr, col, w):
    return dupin.Graph.load_symmetric(n, ptr, col, w)


@pytest.mark.parametrize("at", [1, 8, 2_047, 2_048, 2_049, 6_143, 6_144, 6_145, 8_192, -1])
def test_load_checks_at_tile_edges(dupin, at):
    """One fault at an arc beside a tile's edge (or a thread's, or the last arc): refused, with its code;
    the graph without it loads."""
    n = 7_000
    g = synth.with_weights(exact(n, 12_289, 6_500, [(1, 300), (6_900, 7_000)], 5), "dw", seed=5)
    ptr, col, w = g.symmetric_csr()
    load(dupin, n, ptr, col, w).free()
    row = np.repeat(np.arange(n), np.diff(ptr))
    x = at if at >= 0 else len(col) - 1
    while row[x] != row[x - 1] and at not in (2_048, 6_144, 8_192):  # two arcs of one row
        x += 1 if at >= 0 else -1
    faults = {"swap": (dupin.ERR_INVALID_ARG, "strictly"), "repeat": (dupin.ERR_INVALID_ARG, "strictly"),
              "loop": (dupin.ERR_OVERFLOW, "self-loop"), "id": (dupin.ERR_OVERFLOW, "out of range"),
              "sign": (dupin.ERR_INVALID_ARG, "out of range"), "weight": (dupin.ERR_INVALID_ARG, "symmetric")}
    for what, (code, text) in faults.items():
        c, v = col.copy(), w.copy()
        if what in ("swap", "repeat") and row[x] != row[x - 1]:
            continue
        if what == "swap":
            c[x - 1], c[x] = col[x], col[x - 1]
            v[x - 1], v[x] = w[x], w[x - 1]
        elif what == "repeat":
            c[x] = col[x - 1]
        elif what == "loop":
            c[x] = row[x]
        elif what == "id":
            c[x] = n
        elif what == "sign":
            v[x] = -1
        else:
            v[x] += 1
        with pytest.raises(dupin.DupinError) as e:
            load(dupin, n, ptr, c, v)
        assert e.value.code == code and text in str(e.value), (what, x, str(e.value))


@pytest.mark.parametrize("leaves,below", [(4_096, (1 << 51) - 1), (1_000, ((1 << 63) - 1) // 1_000), (1, (1 << 63) - 1),
                                          (6_000, ((1 << 63) - 1) // 6_000)])
def test_load_weight_sums(dupin, leaves, below):
    """A star whose hub's weight is just below 2^63 loads; one more per arc, and sums that wrap 64 bits, do not."""
    n = leaves + 1
    ptr = np.r_[0, leaves + np.arange(n)].astype(np.int64)
    col = np.r_[1 + np.arange(leaves), np.zeros(leaves, int)].astype(np.int32)
    load(dupin, n, ptr, col, np.full(2 * leaves, below, np.int64)).free()
    if leaves > 1:
        for c in (below + 1, 2 * below + 2, min(4 * below + 4, (1 << 63) - 1), (1 << 62)):
            with pytest.raises(dupin.DupinError) as e:
                load(dupin, n, ptr, col, np.full(2 * leaves, c, np.int64))
            assert e.value.code == dupin.ERR_OVERFLOW, c
