"""The mu projection in one cooperative kernel: meshes of one block, of part of
a warp and of the whole device, and two threads at once on two streams."""
import threading

import pytest

from paper_1912_12453_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def setup(dim, base, top):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1912_12453_gb300 import build, chns
    build.build()
    g = (0.0, -1.0, 0.0) if dim == 2 else (0.0, 0.0, -1.0)
    prm = W.Params(dim, 1e-3, 0.1, 10.0, 5.0, 10.0, 1.0, 0.3, 0.5, gravity=g)
    sph = [W.Sphere((0.45, 0.5, 0.55)[:dim], 0.25)]
    leaves = W.uniform_leaves(dim, top) if base == top else W.band_leaves(dim, base, top, sph, 0.04)
    mesh = chns.Mesh(leaves)
    wl = W.Workload("t", leaves, prm, sph, False)
    U = torch.from_numpy(W.initial_state(mesh.coords, wl).reshape(-1)).cuda()
    return torch, chns, mesh, prm, U


@pytest.mark.parametrize("dim,base,top", [(2, 1, 1), (2, 3, 3), (2, 3, 6), (3, 1, 1), (3, 2, 4), (3, 4, 7), (3, 6, 6)])
def test_mu_row_vanishes(dim, base, top):
    torch, chns, mesh, prm, U = setup(dim, base, top)
    F0 = chns.residual(mesh, prm, U, U).view(-1, dim + 3)[:, -1].clone()
    out = []
    for _ in range(2):
        V = U.clone()
        chns.init_mu(mesh, prm, V)
        out.append(V)
    assert torch.equal(*out)
    assert torch.equal(out[0].view(-1, dim + 3)[:, :-1], U.view(-1, dim + 3)[:, :-1])
    # the iteration stops at 1e-13 of the first residual; a row sums at most 64
    # terms of about its own size, rounded at 1e-16 each
    F = chns.residual(mesh, prm, out[0], out[0]).view(-1, dim + 3)[:, -1]
    assert float(F.norm()) <= 1e-12 * float(F0.norm()) + 1e-18
    mesh.close()


def test_two_threads_two_streams():
    runs = [setup(3, 4, 7), setup(3, 4, 4)]
    want = []
    for torch, chns, mesh, prm, U in runs:
        V = U.clone()
        chns.init_mu(mesh, prm, V)
        want.append(V)
    torch.cuda.synchronize()
    bad = []

    def work(k):
        torch, chns, mesh, prm, U = runs[k]
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            for _ in range(20):
                V = U.clone()
                chns.init_mu(mesh, prm, V, stream=st)
                if not torch.equal(V, want[k]):
                    bad.append(k)

    ts = [threading.Thread(target=work, args=(k,)) for k in (0, 1)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad
    for r in runs:
        r[2].close()
