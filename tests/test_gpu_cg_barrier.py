"""A grid barrier of the mu projection that never fills: the kernel gives it up
after a bounded number of polls (milliseconds here), the call returns an error
and leaves the state alone, and the next call is as good as any."""
import pytest

from paper_1912_12453_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,level", [(2, 2), (2, 6), (3, 5)])  # one block, four, all SMs
def test_given_up_barrier(monkeypatch, dim, level):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1912_12453_gb300 import build, chns
    build.build()
    prm = W.Params(dim, 1e-3, 0.1, 10.0, 5.0, 10.0, 1.0, 0.3, 0.5, gravity=(0.0, -1.0, 0.0))
    leaves = W.uniform_leaves(dim, level)
    mesh = chns.Mesh(leaves)
    wl = W.Workload("t", leaves, prm, [W.Sphere((0.45, 0.5, 0.55)[:dim], 0.25)], False)
    U = torch.from_numpy(W.initial_state(mesh.coords, wl).reshape(-1)).cuda()
    want = U.clone()
    chns.init_mu(mesh, prm, want)
    V = U.clone()
    monkeypatch.setenv("CHNS_INJECT", "barrier")
    with pytest.raises(chns.ChnsError) as ei:
        chns.init_mu(mesh, prm, V)
    monkeypatch.delenv("CHNS_INJECT")
    assert ei.value.status == 6 and "barrier" in str(ei.value)
    assert torch.equal(V, U)
    chns.init_mu(mesh, prm, V)
    assert torch.equal(V, want)
    mesh.close()
