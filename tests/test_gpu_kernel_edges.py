"""Edges of single kernels: the rounding of the prepared state, the energy
kernel's comparisons on the bits and its launches under stream capture, and the
two-level restriction with lists of several pieces."""
import ctypes

import pytest

from paper_1912_12453_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1912_12453_gb300 import build, chns
    build.build()
    return torch, chns


def params(dim):
    g = (0.0, -1.0, 0.0) if dim == 2 else (0.0, 0.0, -1.0)
    return W.Params(dim, 1e-3, 0.1, 10.0, 5.0, 10.0, 1.0, 0.3, 0.5, gravity=g)


@pytest.mark.parametrize("dim,base,top", [(2, 3, 3), (2, 2, 4), (3, 2, 2), (3, 2, 4)])
def test_prepared_state_rounds_like_a_conversion(lib, dim, base, top):
    """States whose sum and difference are floats already give the same J.w, bit
    by bit, as the states whose sum and difference round to those floats."""
    torch, chns = lib
    leaves = W.uniform_leaves(dim, top) if base == top else W.band_leaves(
        dim, base, top, [W.Sphere((0.45, 0.5, 0.55)[:dim], 0.25)], 0.05)
    mesh = chns.Mesh(leaves)
    n = mesh.coords.shape[0] * (dim + 3)
    gen = torch.Generator().manual_seed(5)
    s = 2 * torch.rand(n, generator=gen, dtype=torch.float64) - 1
    d = s.roll(1)
    s[0::7] = 0.25 + 2.0 ** -26 * torch.arange(s[0::7].numel(), dtype=torch.float64)  # half floats: ties at the odd ones
    s[1::7] = -(0.5 - 2.0 ** -40)  # a carry into the exponent
    for k in (0, 1):               # so that a + b below is s exactly
        d[k::7] = (d[k::7] * 2 ** 20).round() / 2 ** 20
    s[2::7] = 1e-40 * s[2::7]      # not normal in float
    d[2::7] = s[2::7] / 2
    s[3::7] = 0.0
    a, b = (s + d) / 2, (s - d) / 2
    S, D = (a + b).float().double(), (a - b).float().double()
    a1, b1 = (S + D) / 2, (S - D) / 2
    keep = ((a1 + b1 == S) & (a1 - b1 == D))  # exact in double; elsewhere both sides use the rounded pair
    a, b = torch.where(keep, a, a1), torch.where(keep, b, b1)
    assert int(keep.sum()) > n // 2
    w = (2 * torch.rand(n, generator=gen) - 1).cuda()
    y = [chns.jacvec(mesh, params(dim), p.cuda(), q.cuda(), w, precision="fp32") for p, q in ((a, b), (a1, b1))]
    assert bool(torch.isfinite(y[0]).all()) and torch.equal(*y)
    mesh.close()


@pytest.mark.parametrize("dim", [2, 3])
def test_energy_bits_and_capture(lib, dim):
    torch, chns = lib
    mesh = chns.Mesh(W.band_leaves(dim, 2, 4, [W.Sphere((0.45, 0.5, 0.55)[:dim], 0.25)], 0.05))
    prm = chns.Params.of(params(dim))
    L = chns.lib()
    U = torch.zeros(mesh.n_dof, dtype=torch.float64, device="cuda")
    phi = U.view(-1, dim + 3)[:, dim + 1]
    out = torch.zeros(3, dtype=torch.float64, device="cuda")

    def call(stream):
        assert L.chns_energy_mass_noalloc(mesh.handle, ctypes.byref(prm), U.data_ptr(), out.data_ptr(), stream) == 0

    call(None)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call(torch.cuda.current_stream().cuda_stream)
    # volume with phi < 0 of a constant phi: the box or nothing (a sum of at most
    # 2^15 weights, each rounded once)
    for value, volume in [(-1.0, 1.0), (1.0, 0.0), (0.0, 0.0), (-0.0, 0.0), (-1e-300, 1.0), (-1e300, 1.0),
                          (float("-inf"), None), (float("nan"), 0.0)]:
        phi.fill_(value)
        graph.replay()
        torch.cuda.synchronize()
        got = out.clone()
        e, m, v = ctypes.c_double(), ctypes.c_double(), ctypes.c_double()
        assert L.chns_energy_mass(mesh.handle, ctypes.byref(prm), U.data_ptr(), ctypes.byref(e), ctypes.byref(m),
                                  ctypes.byref(v), None) == 0
        ref = torch.tensor([e.value, m.value, v.value], dtype=torch.float64)
        assert torch.allclose(got.cpu(), ref, rtol=1e-12, atol=0.0, equal_nan=True)
        if volume is not None:
            assert abs(v.value - volume) <= 1e-12
        assert (e.value != e.value) == (value != value or value == float("-inf"))
        assert (abs(e.value) == float("inf")) == (value == -1e300)
    mesh.close()


@pytest.mark.parametrize("dim,level,coarse", [(2, 6, 1), (2, 7, 1), (3, 4, 1), (3, 5, 1)])
def test_two_level_lists_of_several_pieces(lib, dim, level, coarse):
    """Coarse cells of more than 1,024 list entries.  The coarse space can only
    be of use if R = P^T over all pieces; repeated steps give the same bits."""
    torch, chns = lib
    prm = params(dim)
    wl = W.Workload("t", W.uniform_leaves(dim, level), prm, [W.Sphere((0.45, 0.5, 0.55)[:dim], 0.25)], False)
    mesh = chns.Mesh(wl.leaves)
    U0 = torch.from_numpy(W.initial_state(mesh.coords, wl).reshape(-1)).cuda()
    chns.init_mu(mesh, prm, U0)
    outs = []
    for _ in range(2):
        out = torch.empty_like(U0)
        chns.step(mesh, prm, U0, out, chns.SolverOpts.make(
            precision="fp64", newton_rtol=1e-8, newton_atol=1e-16, krylov_rtol=1e-4, newton_max_it=12,
            krylov_max_it=4000, reuse_preconditioner=0, preconditioner="two_level", coarse_level=coarse))
        outs.append(out)
    assert torch.equal(*outs)
    F, F0 = chns.residual(mesh, prm, outs[0], U0), chns.residual(mesh, prm, U0, U0)
    assert float(F.norm()) <= 1e-8 * float(F0.norm()) + 1e-16
    mesh.close()
