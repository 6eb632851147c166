"""Residual on meshes with hanging corners: the time derivative sees the increments
of the states, not the difference of two interpolated states.

With v = 0 and mu = 0 the Cahn-Hilliard row is the mass matrix times (phi_new -
phi_old) / dt.  The increments d are exact, so the row from phi_old + d is the one
from 0 + d to the roundings of a row's few dozen terms; the rounding of a mean of
states, 1e-16, would be 1e-9 of d."""
import pytest

from paper_1912_12453_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,base,top", [(2, 3, 6), (3, 2, 4)])
def test_phi_row_of_small_increments(dim, base, top):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1912_12453_gb300 import build, chns
    build.build()
    prm = W.Params(dim, 1e-3, 0.1, 10.0, 5.0, 10.0, 1.0, 0.3, 0.5)
    mesh = chns.Mesh(W.band_leaves(dim, base, top, [W.Sphere((0.45, 0.5, 0.55)[:dim], 0.25)], 0.04))
    assert mesh.n_hanging > 0
    n, nf = mesh.n_nodes, dim + 3
    gen = torch.Generator().manual_seed(1)
    old = torch.zeros(n, nf, dtype=torch.float64)
    d = torch.zeros(n, nf, dtype=torch.float64)
    # odd last bits: the mean of two or four such values in [1/2, 1) is not a double
    old[:, dim + 1] = torch.randint(2 ** 52, 2 ** 53, (n,), generator=gen).double() / 2.0 ** 53
    d[:, dim + 1] = torch.randint(-2 ** 29, 2 ** 29, (n,), generator=gen).double() * 2.0 ** -53
    new = old + d
    d = new - old
    rows = [chns.residual(mesh, prm, a.reshape(-1).cuda(), b.reshape(-1).cuda()).view(n, nf)[:, dim + 1]
            for a, b in ((new, old), (d, torch.zeros_like(d)))]
    assert float((rows[0] - rows[1]).norm()) <= 64 * 2.0 ** -53 * float(rows[1].norm())
    mesh.close()
