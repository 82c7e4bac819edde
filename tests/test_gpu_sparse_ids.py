"""Graphs with far more vertices than arcs (ids that were never compacted): the
initial weights and the load's checks walk tiles of arcs, and the empty rows
between two arcs must cost next to nothing.  Peels against the oracle, faults
beside the gaps, and a bound on the time.
"""
import time

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


def sparse(n, ids, draws, seed, hub=0):
    """draws random edges among the vertices `ids` of n (and a hub row), with weights 1 .. 97."""
    rng = np.random.default_rng(seed)
    e = rng.choice(ids, (draws, 2))
    if hub:
        e = np.r_[e, np.c_[np.full(hub, ids[len(ids) // 2]), rng.choice(ids, hub)]]
    e = np.sort(e, 1)
    e = np.unique(e[e[:, 0] != e[:, 1]], axis=0)
    g = synth.SynthGraph(n, 0, e[:, 0].astype(np.int32).copy(), e[:, 1].astype(np.int32).copy())
    g.c = (1 + (e.sum(1) * 31) % 97).astype(np.int64) << 32
    return g


N = 300_000  # 8,192 rows are walked before the arcs are searched


def ends(k):
    return np.r_[np.arange(k), np.arange(N - k, N)]


CASES = {
    "ends": (ends(400), 3_000, 0),
    "one block of ids": (np.arange(8_000, 9_000), 5_000, 0),
    "every 100th": (np.arange(0, N, 100), 6_000, 1_500),
    "every 3rd": (np.arange(1, N, 3), 40_000, 0),
    "just past the walk": (np.r_[0, 8_191, 8_192, 8_193, 16_384, N - 1], 40, 0),
    "last": (np.arange(N - 50, N), 300, 0),
}


@pytest.mark.parametrize("name", list(CASES))
def test_peels_equal_the_oracle(dupin, name):
    ids, draws, hub = CASES[name]
    g = sparse(N, ids, draws, 3, hub)
    g.a = (np.arange(N, dtype=np.int64) % 5) << 32
    for k, flags in ((1, 0), (2, 0), (2, dupin.LPO)):
        out, ref = run_both(dupin, g, "dw", k, (1, 10), flags=flags)
        assert_same(out, ref, (name, k, flags))
    g.c[::7] += 1 << 52  # tiles whose sums are formed in two halves
    out, ref = run_both(dupin, g, "dw", 2, (1, 10))
    assert_same(out, ref, name)


@pytest.mark.parametrize("name", list(CASES))
def test_load_checks_beside_gaps(dupin, name):
    ids, draws, hub = CASES[name]
    ptr, col, w = sparse(N, ids, draws, 4, hub).symmetric_csr()
    dupin.Graph.load_symmetric(N, ptr, col, w).free()
    row = np.repeat(np.arange(N), np.diff(ptr))
    for x in (0, len(col) // 2, len(col) - 1):
        for what, code in (("loop", dupin.ERR_OVERFLOW), ("weight", dupin.ERR_INVALID_ARG)):
            c, v = col.copy(), w.copy()
            if what == "loop":
                c[x] = row[x]
            else:
                v[x] += 1
            with pytest.raises(dupin.DupinError) as e:
                dupin.Graph.load_symmetric(N, ptr, c, v)
            assert e.value.code == code, (what, x)


@pytest.mark.parametrize("arcs", [1_000, 60_000])
def test_time_with_few_arcs(dupin, arcs):
    """15 million vertices: the initial weights alone (a pass over the vertices, and a few hundred or
    thousand arcs) within 1.5 ms, a load within 10 ms; a walk over all rows takes 58 ms (1,000 arcs at the
    ends of the ids) and 2 ms (60,000 over all of them)."""
    import torch

    n = 15_000_000
    if arcs == 1_000:
        g = sparse(n, np.r_[np.arange(300), np.arange(n - 300, n)], arcs // 2, 5)
    else:
        g = sparse(n, np.random.default_rng(6).choice(n, arcs, replace=False), arcs // 2, 5)
    ptr, col, w = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in g.symmetric_csr())
    load, init = [], []
    p = dupin.make_params("dw", 2, (1, 10), flags=dupin.TIMING)
    for _ in range(5):
        torch.cuda.synchronize()
        t = time.perf_counter()
        dg = dupin.Graph.load_symmetric(n, ptr, col, w, device_ptrs=True)
        load.append(time.perf_counter() - t)
        init.append(dupin.peel_device(dg, p).phase_ms[0])
        dg.free()
    assert min(init) < 1.5, init
    assert min(load) < 0.010, load
