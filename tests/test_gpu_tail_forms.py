"""The one-CTA tail's two forms of a round (one warp alone, the whole block):
peels whose rows and segment counts lie on both sides of where the warp form
runs, against the oracle, and a bound on what trying it may cost where it
cannot run.
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


# vertices: 63 .. 65 segments of 64, the warp form's limit; rows around its 128 arcs
@pytest.mark.parametrize("n,deg", [(63 * 64, 20), (64 * 64, 20), (64 * 64 + 1, 20), (65 * 64, 20), (700, 124), (700, 132)])
def test_rounds_on_both_sides_of_the_warp_form(dupin, n, deg):
    g = synth.random_general(n, n * deg // 2, seed=n + deg)
    synth.with_weights(g, "dw", seed=n, a_range=(0, 5))
    for k, eps, flags in ((1, (1, 10), 0), (1, (0, 1), 0), (1, (1, 10), dupin.LPO)):
        out, ref = run_both(dupin, g, "dw", k, eps, flags=flags | dupin.TAIL_ONE_CTA)
        assert_same(out, ref, (n, deg, k, eps, flags))


def test_rows_too_long_for_the_warp_cost_little(dupin):
    """A transaction graph whose 5,000-vertex core has rows of 160 arcs: its 3,100 one-vertex rounds by
    one CTA take 1.8 times as long as on the dense tail (2.2 times with a try of the warp form every
    second round)."""
    g = synth.fd_camouflage(seed=2, nU=330_000, nI=165_000, m_bg=6_600_000)
    dg = dupin.Graph.from_synth(g)
    ms = {}
    for flags in (dupin.TAIL_ONE_CTA, dupin.TAIL_CLUSTER):
        p = dupin.make_params("fd", 1, (1, 10), flags=flags | dupin.TIMING)
        runs = [dupin.peel_device(dg, p) for _ in range(8)]
        ms[flags] = min(r.phase_ms[3] for r in runs)
        assert (runs[0].tail_ctas == 1) == (flags == dupin.TAIL_ONE_CTA)
    dg.free()
    assert ms[dupin.TAIL_ONE_CTA] < 2.0 * ms[dupin.TAIL_CLUSTER], ms
