"""A peel that max_rounds stops: NO_PROGRESS, with the rounds it ran and how many
of them took the minimum rule, in whichever stage it stops (the grid-wide rounds
before and after any number of compactions, the tails).
"""
import ctypes

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


@pytest.mark.parametrize("scale,tail", [(12, 1), (14, 1), (16, 1), (14, 0), (14, 300)])
def test_stopped_peels_report_their_rounds(dupin, scale, tail):
    g = synth.rmat_weighted(scale, 16, "fd", seed=1)
    dg = dupin.Graph.from_synth(g)
    og = oracle.Graph.from_synth(g, "fd")
    ref = oracle.peel_batch(og, 1, (1, 10))
    og.close()
    assert ref.n_rounds > 59
    for stop in list(range(1, 25)) + [40, 59]:
        p = dupin.make_params("fd", 1, (1, 10), max_rounds=stop, tail_cap=tail)
        r = dupin.Result()
        rc = dupin.lib().dupin_peel(dg.handle, ctypes.byref(p), ctypes.byref(r), None)
        assert rc == dupin.ERR_NO_PROGRESS, stop
        assert r.n_rounds == stop
        assert r.n_min_rule == int((ref.trace_kind[1:stop + 1] == 1).sum()), stop
    out = dupin.peel(dg, "fd", 1, (1, 10), tail_cap=tail)  # and to the end afterwards
    assert np.array_equal(out.peel_round, ref.peel_round)
    dg.free()
