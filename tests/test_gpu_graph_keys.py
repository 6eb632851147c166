"""Captured Arnoldi steps are not kept past a rebuild that changes the V-cycle,
in whatever order builds in the two precisions come (own process: the numbers
that tell the builds apart count from its start), nor past another coarse space."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = """
import sys
import torch
from paper_1912_12453_gb300 import build, chns, workloads as W
build.build()
wl = W.workload("droplet2d_l5")
U0 = None

def new_mesh():
    global U0
    m = chns.Mesh(wl.leaves)
    if U0 is None:
        U0 = torch.from_numpy(W.initial_state(m.coords, wl).reshape(-1)).cuda()
        chns.init_mu(m, wl.params, U0)
    return m

def step(m, precision, sweeps):
    out = torch.empty_like(U0)
    st = chns.step(m, wl.params, U0, out, chns.SolverOpts.make(
        precision=precision, newton_rtol=1e-6, preconditioner="multigrid", mg_smooth=sweeps, use_graph=True))
    return out, st["krylov_its_total"]

m = new_mesh()
for precision, sweeps in ORDER:
    got = step(m, precision, sweeps)
want = step(new_mesh(), *ORDER[-1])
print(got[1], want[1], int(torch.equal(got[0], want[0])))
"""

ORDERS = [[("fp64", 1), ("fp32", 1), ("fp64", 2), ("fp32", 1), ("fp32", 2)],
          [("fp64", 2), ("fp32", 2), ("fp64", 1), ("fp32", 2), ("fp32", 1)],
          [("fp32", 1), ("fp64", 1), ("fp32", 2), ("fp64", 1), ("fp64", 2)],
          [("fp32", 1), ("fp32", 2), ("fp32", 1), ("fp64", 1), ("fp32", 2)]]


@pytest.mark.parametrize("order", ORDERS, ids=lambda o: "-".join(f"{p}x{s}" for p, s in o))
def test_a_step_does_not_depend_on_the_builds_before_it(order):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    r = subprocess.run([sys.executable, "-c", SCRIPT.replace("ORDER", repr(order))], cwd=ROOT, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    got, want, same = (int(x) for x in r.stdout.split()[-3:])
    assert got == want and same == 1


def test_coarse_level_there_and_back():
    """The coarse space of a captured step is released and set up again in between
    by steps that capture nothing."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1912_12453_gb300 import build, chns, workloads as W
    build.build()
    wl = W.workload("droplet2d_l5")
    meshes = [chns.Mesh(wl.leaves) for _ in range(2)]
    U0 = torch.from_numpy(W.initial_state(meshes[0].coords, wl).reshape(-1)).cuda()
    chns.init_mu(meshes[0], wl.params, U0)

    def step(m, level, graph):
        out = torch.empty_like(U0)
        st = chns.step(m, wl.params, U0, out, chns.SolverOpts.make(newton_rtol=1e-6, coarse_level=level,
                                                                   use_graph=graph))
        return out, st["krylov_its_total"]

    for level, graph in ((2, True), (3, False), (2, True)):
        got = step(meshes[0], level, graph)
    want = step(meshes[1], 2, True)
    assert got[1] == want[1] and torch.equal(got[0], want[0])
    for m in meshes:
        m.close()
