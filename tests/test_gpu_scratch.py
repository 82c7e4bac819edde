"""What a call leaves on the device: the state of a batch or of a clique peel goes
back when the stream is next waited for, all but DUPIN_SCRATCH_KEEP bytes, and
dupin_trim_cache releases those too.
"""
import gc

import pytest

from paper_2504_09311_gb300 import synth

pytestmark = pytest.mark.gpu

KEEP = 1 << 30


@pytest.fixture(scope="module")
def env():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2504_09311_gb300 import dupin as d

    d.lib()
    return torch, d


def free(torch):
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_a_large_batch_leaves_at_most_the_kept_part(env):
    torch, dupin = env
    gc.collect()
    torch.cuda.empty_cache()
    dupin.trim_cache()
    g = dupin.Graph.from_synth(synth.random_general(100_000, 150_000, seed=1))
    p = dupin.make_params("dg", 1, (1, 10))
    graphs = [g] * 1_500  # 16 bytes a vertex: 2.4 GB of state
    bufs = dupin.BatchBuffers.for_graphs(graphs, want_rounds=False)
    dupin.peel_batch(graphs[:2], [p] * 2, want_rounds=False)  # one-time set-up
    before = free(torch)
    for _ in range(3):
        dupin.peel_batch(graphs, [p] * len(graphs), buffers=bufs)
    assert before - free(torch) <= KEEP + (64 << 20)
    dupin.trim_cache()
    assert before - free(torch) <= 64 << 20
    g.free()


def test_clique_state_is_released(env):
    torch, dupin = env
    n = 30_000_000  # 49 bytes a vertex: 1.5 GB of state
    g = synth.random_general(1_000, 20_000, seed=2)
    g.n_left = n  # the other vertices have no arcs
    dg = dupin.Graph.from_synth(g)
    torch.cuda.synchronize()
    dupin.trim_cache()
    before = free(torch)
    pr = torch.empty(n, dtype=torch.int32, device="cuda")
    held = before - free(torch)
    for _ in range(2):
        dupin.peel_device(dg, dupin.make_params("tds", 3, (1, 10)), pr)
    assert before - held - free(torch) <= KEEP + (64 << 20)
    dupin.trim_cache()
    assert before - held - free(torch) <= 64 << 20
    dg.free()
