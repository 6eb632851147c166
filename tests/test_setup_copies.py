"""Set-up copies are over when a builder returns (no GPU), and the first step of
a batch on a stream of its own is the step on the default stream (GPU)."""
import os
import shutil
import subprocess

import pytest

from paper_1912_12453_gb300 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1912_12453_gb300", "csrc")


def test_no_copy_is_on_its_way(tmp_path):
    inc = "/usr/local/cuda/include"
    if shutil.which("g++") is None or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("g++ or the CUDA headers are missing")
    exe = str(tmp_path / "setup_copies")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-pthread", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                           "-I", inc, os.path.join(CSRC, "mesh.cpp"),
                           os.path.join(ROOT, "tests", "host", "setup_copies_main.cpp"), "-o", exe])
    out = subprocess.check_output([exe], text=True).split("\n")
    assert out[:4] == ["mesh 0", "mesh 0", "union 0", "bounds 1"]


@pytest.mark.gpu
def test_first_batch_step_on_a_side_stream():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1912_12453_gb300 import build, chns
    build.build()
    wls = [wl for wl in W.batched_workloads(12) if wl.params.dim == 2][:4]
    assert len(wls) >= 2
    states, meshes = [], []
    for wl in wls:
        m = chns.Mesh(wl.leaves)
        U = torch.from_numpy(W.initial_state(m.coords, wl).reshape(-1)).cuda()
        chns.init_mu(m, wl.params, U)
        meshes.append(m)
        states.append(U)
    opts = chns.SolverOpts.make(precision="fp32", newton_rtol=1e-9)
    res = []
    for st in (None, torch.cuda.Stream()):
        torch.cuda.synchronize()
        b = chns.Batch(meshes, [wl.params for wl in wls])
        outs = [torch.empty_like(U) for U in states]
        b.step(states, outs, opts, stream=st)
        torch.cuda.synchronize()
        res.append(outs)
    for a, c in zip(*res):
        assert torch.equal(a, c)
