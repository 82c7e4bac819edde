"""A small peel runs beside a kernel that holds most of every SM's shared memory: it
asks for its own state and arcs, not for a whole SM's.
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle
from paper_2504_09311_gb300 import synth

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def env(tmp_path_factory):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    so = str(tmp_path_factory.mktemp("hold") / "libhold.so")
    subprocess.check_call([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-shared", "-Xcompiler", "-fPIC",
                           "-o", so, os.path.join(HERE, "hold_shared.cu")])
    hold = ctypes.CDLL(so).hold_shared
    hold.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_void_p]
    from paper_2504_09311_gb300 import dupin as d

    d.lib()
    return torch, d, hold


@pytest.mark.parametrize("call", ["noalloc", "peel"])
def test_small_peel_beside_a_kernel_that_holds_shared_memory(env, call):
    torch, dupin, hold = env
    g = synth.random_general(150, 1_000, seed=1)
    synth.with_weights(g, "dw", seed=1)
    ptr, idx, w = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in g.symmetric_csr())
    dg = dupin.Graph.from_synth(g)
    pr = torch.empty(g.n, dtype=torch.int32, device="cuda")
    p = dupin.make_params("dw", 1, (1, 10))
    side, own = torch.cuda.Stream(), torch.cuda.Stream()

    def peel():
        if call == "noalloc":
            dupin.peel_noalloc(g.n, ptr, idx, w, None, p, pr, stream=own)
        else:
            dupin.peel_device(dg, dupin.make_params("dw", 1, (1, 10), flags=dupin.TAIL_ONE_CTA), pr, stream=own)

    peel()  # one-time set-up
    torch.cuda.synchronize()
    # 150 KB held for 0.3 s leave 78 KB an SM: the checks' 33 KB fit, and a peel of 150 vertices
    assert hold(150 << 10, 300, side.cuda_stream) == 0
    done = torch.cuda.Event()
    done.record(side)
    peel()
    ran_beside = not done.query()
    torch.cuda.synchronize()
    assert ran_beside
    og = oracle.Graph.from_synth(g, "dw")
    assert np.array_equal(pr.cpu().numpy(), oracle.peel_batch(og, 1, (1, 10)).peel_round)
    og.close()
    dg.free()
