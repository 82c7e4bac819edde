"""Where a batch's peel rounds go on the host: touching slices of one page-locked
block (copied together), touching page-locked ranges registered one by one,
touching pageable slices, page-locked next to pageable, and buffers out of order.
"""
import mmap

import numpy as np
import pytest

from paper_2504_09311_gb300 import synth

pytestmark = pytest.mark.gpu

PAGE = mmap.PAGESIZE


@pytest.fixture(scope="module")
def env():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2504_09311_gb300 import dupin as d

    d.lib()
    n = PAGE // 4  # a graph's rounds fill a page
    graphs = [d.Graph.from_synth(synth.random_general(n, 5 * n, seed=s)) for s in range(6)]
    refs = [d.peel(g, "dg", 1, (1, 10)).peel_round for g in graphs]
    yield torch, d, graphs, refs
    for g in graphs:
        g.free()


# pages registered together, in order of the graphs' buffers
@pytest.mark.parametrize("ranges", [[(0, 6)], [(0, 1), (1, 1), (2, 1), (3, 1), (4, 1), (5, 1)], [(0, 2), (2, 3)],
                                    [(1, 2), (4, 2)], []])
@pytest.mark.parametrize("order", [[0, 1, 2, 3, 4, 5], [5, 4, 3, 2, 1, 0], [0, 1, 3, 2, 4, 5]])
def test_touching_buffers(env, ranges, order):
    torch, dupin, graphs, refs = env
    host = mmap.mmap(-1, 6 * PAGE)
    block = np.frombuffer(host, np.int32)
    rt = torch.cuda.cudart()
    n = graphs[0].n
    bufs = [(block[p * n:(p + 1) * n], None, None) for p in order]
    params = [dupin.make_params("dg", 1, (1, 10))] * 6
    try:
        for first, pages in ranges:
            assert int(rt.cudaHostRegister(block.ctypes.data + first * PAGE, pages * PAGE, 0)) == 0
        for _ in range(2):
            block[:] = -1
            outs = dupin.peel_batch(graphs, params, buffers=bufs)
            for o, r in zip(outs, refs):
                assert np.array_equal(o.peel_round, r)
    finally:
        for first, _ in ranges:
            rt.cudaHostUnregister(block.ctypes.data + first * PAGE)
