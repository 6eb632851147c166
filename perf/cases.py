"""Timed cases of the CHNS operator library: operator applies, diagnostics,
the mu projection and whole CN steps, through the Python entry points.

A case is a plain dict: what is called (``call``), the mesh (a band of fine
leaves around one sphere between octree levels ``base`` and ``top``; uniform
when both are equal) and the nondimensional parameters.  Meshes and parameters
are those of the repository's workloads or of the same kind.

The second half of the file is the same discretisation in plain torch double
precision (``exact``): node numbering, hanging constraints, weak form,
directional derivative by forward-mode differentiation, and dense Newton for
the smallest steps.
"""
import functools
import math

import numpy as np
import torch

from paper_1912_12453_gb300 import chns
from paper_1912_12453_gb300 import workloads as W

DEV = "cuda"

DROPLET2D = dict(dim=2, dt=1e-3, Cn=0.04, Re=35.0, We=125.0, Pe=25.0, Fr=1.0, rho=0.1, eta=0.1,
                 cx=0.5, cy=0.3, cz=0.5, R=0.15, bubble=False)
DROPLET3D = dict(dim=3, dt=5e-4, Cn=0.02, Re=100.0, We=50.0, Pe=50.0, Fr=1.0, rho=1e-2, eta=1e-2,
                 cx=0.5, cy=0.5, cz=0.3, R=0.15, bubble=False)
BUBBLE3D = dict(dim=3, dt=2.5e-4, Cn=0.01, Re=35.0, We=1.0, Pe=100.0, Fr=1.0, rho=1e-3, eta=1e-2,
                cx=0.5, cy=0.5, cz=0.25, R=0.125, bubble=True)


def listed():
    return [
        # one Krylov operator apply of the small 2D droplet (1,024 leaves):
        # launch latency and the host call count here
        dict(DROPLET2D, name="jacvec_2d_l5_fp32", call="jacvec", precision="fp32", base=5, top=5),
        # the headline workload's apply: uniform level-6 octree, 262,144 leaves
        dict(DROPLET3D, name="jacvec_3d_l6_fp32", call="jacvec", precision="fp32", base=6, top=6),
        # the adaptive rising bubble's apply: 1.4M leaves, levels 5-9, hanging nodes
        dict(BUBBLE3D, name="jacvec_3d_l5_9_fp32", call="jacvec", precision="fp32", base=5, top=9),
        # the apply of the double-precision finish on an adaptive mesh (78k leaves)
        dict(DROPLET3D, name="jacvec_3d_l4_7_fp64", call="jacvec", precision="fp64", base=4, top=7),
        # the residual with a nodal source and prescribed boundary values, as a
        # manufactured-solution study evaluates it
        dict(DROPLET2D, name="residual_2d_l5_forced", call="residual", forced=True, base=5, top=5),
        # the Newton residual of the headline workload (262,144 leaves)
        dict(DROPLET3D, name="residual_3d_l6", call="residual", forced=False, base=6, top=6),
        # energy, mass and light-phase volume of an adaptive state, the
        # diagnostics printed every step
        dict(BUBBLE3D, name="energy_3d_l5_8", call="energy", base=5, top=8, Cn=0.02, Pe=50.0),
        # mu projected on the mesh after a remesh or at the start (78k leaves)
        dict(DROPLET3D, name="init_mu_3d_l4_7", call="init_mu", base=4, top=7),
        # one CN step of the 2D droplet with the library's default options
        # (double precision, two-level preconditioner)
        dict(DROPLET2D, name="step_2d_l5_fp64", call="step", precision="fp64", pc="two_level", rtol=1e-10,
             krylov_rtol=1e-4, base=5, top=5),
        # one CN step of the 3D droplet, mixed precision with multigrid: the
        # production configuration on a mesh of 32,768 leaves
        dict(DROPLET3D, name="step_3d_l5_mg_fp32", call="step", precision="fp32", pc="multigrid", rtol=1e-12,
             krylov_rtol=1e-3, base=5, top=5, Cn=0.04, Pe=25.0),
        # eight independent 2D droplets of uneven size advanced as one batch
        dict(DROPLET2D, name="batch_2d_8_mg_fp32", call="batch", precision="fp32", pc="multigrid", rtol=1e-12,
             krylov_rtol=1e-3, base=4, top=6, count=8, Cn=0.02, Pe=50.0, dt=5e-4, We=10.0),
    ]


def draw(rng):
    """One more case of the same ranges: random sphere, interface width and
    levels, so leaf and node counts are ragged."""
    call, prec, dim, hi, lo = rng.choice([
        ("jacvec", "fp32", 2, 10, 4), ("jacvec", "fp32", 3, 8, 3), ("jacvec", "fp32", 3, 8, 4),
        ("jacvec", "fp64", 2, 9, 4), ("jacvec", "fp64", 3, 7, 3), ("residual", "fp64", 2, 9, 4),
        ("residual", "fp64", 3, 7, 3), ("energy", "fp64", 3, 8, 4), ("energy", "fp64", 2, 9, 5),
        ("init_mu", "fp64", 3, 6, 4), ("init_mu", "fp64", 2, 8, 5), ("step", "fp64", 2, 6, 5),
        ("step", "fp32", 3, 5, 4)])
    top = rng.randint(lo, hi)
    base = max(3 if dim == 3 else 4, top - rng.randint(0, 3))
    base = min(base, top)
    if dim == 3:  # at most as many leaves as the largest listed mesh
        base = min(base, 6)
    Cn = min(0.08, 2.0 ** (rng.uniform(0.3, 2.3) - top))
    c = dict(call=call, precision=prec, dim=dim, base=base, top=top, Cn=Cn, Pe=1.0 / Cn,
             dt=10.0 ** rng.uniform(-3.6, -3.0), Re=10.0 ** rng.uniform(1.3, 2.0), We=10.0 ** rng.uniform(0.0, 2.0),
             Fr=1.0, rho=10.0 ** rng.uniform(-3.0, 0.0), eta=10.0 ** rng.uniform(-2.0, 0.0),
             cx=rng.uniform(0.35, 0.65), cy=rng.uniform(0.35, 0.65), cz=rng.uniform(0.35, 0.65),
             R=rng.uniform(0.1, 0.25), bubble=rng.random() < 0.5)
    if call == "residual":
        c["forced"] = rng.random() < 0.5
    if call == "step":
        c.update(rho=10.0 ** rng.uniform(-2.0, 0.0), krylov_rtol=1e-4 if prec == "fp64" else 1e-3,
                 pc="two_level" if prec == "fp64" else "multigrid", rtol=1e-10 if prec == "fp64" else 1e-12)
        if dim == 2:
            c["base"] = max(base, 4)
    return c


# --------------------------------------------------------------------------
# meshes and inputs
# --------------------------------------------------------------------------

@functools.lru_cache(maxsize=32)
def _leaves(dim, base, top, center, R, Cn):
    """The leaf list a user's mesh generator hands over (host arrays)."""
    if base == top:
        return W.uniform_leaves(dim, top)
    return W.band_leaves(dim, base, top, [W.Sphere(center[:dim], R)], Cn)


def _instance(case, k):
    """Parameters of the k-th problem of a case (a batch has several)."""
    if case["call"] != "batch":
        return case
    r = np.random.default_rng(1000 + k)
    return dict(case, cx=float(r.uniform(0.35, 0.65)), cy=float(r.uniform(0.35, 0.65)), R=float(r.uniform(0.1, 0.25)),
                rho=float(10 ** r.uniform(-2, 0)), eta=float(10 ** r.uniform(-2, 0)), bubble=bool(r.random() < 0.5),
                base=case["top"] - int(r.integers(0, 3)))


def _case_leaves(c):
    return _leaves(c["dim"], c["base"], c["top"], (c["cx"], c["cy"], c["cz"]), c["R"], c["Cn"])


def _params(c):
    g = (0.0, -1.0, 0.0) if c["dim"] == 2 else (0.0, 0.0, -1.0)
    return W.Params(c["dim"], c["dt"], c["Cn"], c["Re"], c["We"], c["Pe"], c["Fr"], c["rho"], c["eta"], gravity=g)


def _rand(seed, k, *shape):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 64 + k)
    return torch.rand(shape, generator=g, device=DEV, dtype=torch.float64) * 2.0 - 1.0


def _start_state(c, x, seed, k=0):
    """U_n at the node coordinates x [n, dim]: a solenoidal velocity that
    vanishes on the walls, p = 0, the tanh interface of a slightly moved
    sphere, mu = 0."""
    dim = c["dim"]
    a = _rand(seed, 8 + k, 8)
    s, co = torch.sin(math.pi * x), torch.cos(math.pi * x)
    U = torch.zeros(x.shape[0], dim + 3, dtype=torch.float64, device=DEV)
    q = 0.05 * (1.0 + 0.5 * a[0]) * (s[:, 2] * (1.0 + 0.5 * a[1] * co[:, 2]) if dim == 3 else 1.0)
    U[:, 0] = q * s[:, 0] ** 2 * s[:, 1] * co[:, 1]
    U[:, 1] = -q * s[:, 0] * co[:, 0] * s[:, 1] ** 2
    wall = ((x <= 0.0) | (x >= 1.0)).any(1)
    U[wall, :dim] = 0.0
    cen = torch.tensor([c["cx"], c["cy"], c["cz"]][:dim], dtype=torch.float64, device=DEV)
    cen = cen + 0.2 * c["Cn"] * a[2:2 + dim]
    d = ((x - cen) ** 2).sum(1).sqrt() - c["R"] * (1.0 + 0.01 * a[5])
    phi = torch.tanh(d / (math.sqrt(2.0) * c["Cn"]))
    U[:, dim + 1] = phi if c["bubble"] else -phi
    return U


def _free_rows(x, nf):
    """1 in the unconstrained rows, 0 in the wall velocities and the pinned
    pressure: an iterate satisfies the boundary rows, and Krylov vectors
    vanish there."""
    m = torch.ones(x.shape[0], nf, dtype=torch.float64, device=DEV)
    m[((x <= 0.0) | (x >= 1.0)).any(1), :nf - 3] = 0.0
    m[(x == 0.0).all(1), nf - 3] = 0.0
    return m


def _newton_pair(c, x, seed):
    """(U_new, U_old) as an operator apply inside a Newton iteration sees
    them: an evolved state and an iterate near it."""
    dim, n = c["dim"], x.shape[0]
    U = _start_state(c, x, seed)
    a = _rand(seed, 1, 6)
    wv = torch.sin(math.pi * (x * torch.arange(1, dim + 1, device=DEV)).sum(1) + a[0]) - torch.sin(a[0])
    U[:, dim] = c["We"] / c["Fr"] * x[:, dim - 1] * 0.5 * (1.0 + c["rho"]) * (1.0 + 0.1 * a[1]) + 0.1 * wv
    phi = U[:, dim + 1]
    U[:, dim + 2] = 0.5 * (phi ** 3 - phi) + 0.05 * wv
    U_new = U + 1e-2 * _rand(seed, 2, n, dim + 3) * _free_rows(x, dim + 3)
    return U_new.reshape(-1).contiguous(), U.reshape(-1).contiguous()


def _source(c, x, seed, U_new):
    """A nodal source and boundary values close to the iterate's."""
    f = _rand(seed, 4, U_new.numel())
    bc = U_new + 1e-6 * _rand(seed, 5, U_new.numel())
    return f, bc


def prepare(case, seed):
    call = case["call"]
    prec = case.get("precision", "fp64")
    parts = []
    for k in range(case.get("count", 1)):
        c = _instance(case, k)
        mesh = chns.Mesh(_case_leaves(c))
        x = torch.from_numpy(mesh.coords).to(DEV)
        prm = _params(c)
        if call in ("step", "batch", "init_mu"):
            U = _start_state(c, x, seed, k).reshape(-1).contiguous()
            if call == "init_mu":
                parts.append((mesh, prm, torch.empty_like(U), U))
            else:
                chns.init_mu(mesh, prm, U)
                parts.append((mesh, prm, U, torch.empty_like(U)))
        else:
            U_new, U_old = _newton_pair(c, x, seed)
            parts.append((mesh, prm, U_new, U_old, torch.empty_like(U_new)))
    s = {"call": call, "precision": prec, "parts": parts}
    mesh = parts[0][0]
    if call == "jacvec":
        dt = torch.float64 if prec == "fp64" else torch.float32
        s["w"] = (_rand(seed, 3, mesh.n_dof) * _free_rows(x, mesh.nf).reshape(-1)).to(dt)
        s["y"] = torch.empty_like(s["w"])
    if call == "residual":
        s["f"], s["bc"] = _source(c, x, seed, U_new) if case["forced"] else (None, None)
    if call in ("step", "batch"):
        s["opts"] = chns.SolverOpts.make(precision=prec, newton_rtol=case["rtol"], krylov_rtol=case["krylov_rtol"],
                                         preconditioner=case["pc"], newton_max_it=30)
    if call == "batch":
        s["batch"] = chns.Batch([p[0] for p in parts], [p[1] for p in parts])
    return s


def run(state):
    call, p = state["call"], state["parts"][0]
    if call == "jacvec":
        return chns.jacvec(p[0], p[1], p[2], p[3], state["w"], out=state["y"], precision=state["precision"])
    if call == "residual":
        return chns.residual(p[0], p[1], p[2], p[3], state["f"], state["bc"], out=p[4])
    if call == "energy":
        e, m, b = chns.energy_mass(p[0], p[1], p[2])
        return {"energy": e, "mass": m, "light_volume": b}
    if call == "init_mu":
        return chns.init_mu(p[0], p[1], p[2].copy_(p[3]))  # in place: every pass starts from mu = 0
    if call == "step":
        st = chns.step(p[0], p[1], p[2], p[3], state["opts"])
        return {"U": p[3], "energy": st["energy_new"], "mass": st["mass_new"]}
    if call == "batch":
        st = state["batch"].step([q[2] for q in state["parts"]], [q[3] for q in state["parts"]], state["opts"])
        return {"U": [q[3] for q in state["parts"]], "mass": [t["mass_new"] for t in st]}
    raise ValueError(call)


# Operations of the weak form per Gauss point that any evaluation needs
# (interpolation by sum factorisation, the Gauss-point coefficients, the
# contraction), counted from the formulas with shared factors taken out.
RESIDUAL_FLOPS = {2: 230, 3: 480}
JACVEC_FLOPS = {2: 470, 3: 980}
ENERGY_FLOPS = {2: 60, 3: 90}


def work(case):
    """Bytes and operations of one pass; nodes are counted as leaves.  A solve
    is counted with the fewest iterations such a solve takes: 3 Newton
    iterations of 8 Krylov iterations, 20 CG iterations of the mu row."""
    total_b = total_f = 0.0
    for k in range(case.get("count", 1)):
        c = _instance(case, k)
        n, dim = _case_leaves(c).n, c["dim"]
        nf, gp = dim + 3, n << dim
        mesh_b = n * (4 * (1 << dim) + 1)
        vec = 8 * nf * n
        call = c["call"]
        if call == "jacvec":
            wb = 2 * nf * n * (8 if c["precision"] == "fp64" else 4)
            b, f = 2 * vec + wb + mesh_b, gp * JACVEC_FLOPS[dim]
        elif call == "residual":
            b, f = (5 if c["forced"] else 3) * vec + mesh_b, gp * RESIDUAL_FLOPS[dim]
        elif call == "energy":
            b, f = vec + mesh_b, gp * ENERGY_FLOPS[dim]
        elif call == "init_mu":
            b, f = 2 * vec + mesh_b, gp * 20 * 40
        else:
            b = 2 * vec + mesh_b
            f = gp * (4 * RESIDUAL_FLOPS[dim] + 24 * JACVEC_FLOPS[dim])
        total_b += b
        total_f += f
    return {"bytes": total_b, "flops": total_f}


# --------------------------------------------------------------------------
# the same results in plain torch, double precision
# --------------------------------------------------------------------------

class _Grid:
    """Nodes, hanging constraints and element geometry of a leaf list: nodes
    are the leaves' corners numbered at their first appearance (leaf by leaf,
    x fastest), hanging ones left out."""

    def __init__(self, leaves):
        dim, top = leaves.dim, 1 << leaves.max_level
        self.dim, nc = dim, 1 << leaves.dim
        lev = torch.from_numpy(leaves.level.astype(np.int64)).to(DEV)
        anc = torch.from_numpy(leaves.anchor.astype(np.int64)).to(DEV)
        size = (1 << (leaves.max_level - lev))
        bits = torch.tensor([[(c >> a) & 1 for a in range(dim)] for c in range(nc)], device=DEV)
        mul = torch.tensor([(2 * top + 1) ** a for a in range(dim)], device=DEV)
        corner = anc[:, None, :] + bits[None] * size[:, None, None]
        keys = (corner * mul).sum(-1).reshape(-1)
        uk, inv = torch.unique(keys, return_inverse=True)
        first = torch.full((uk.shape[0],), keys.shape[0], device=DEV)
        first.scatter_reduce_(0, inv, torch.arange(keys.shape[0], device=DEV), "amin")
        n_all = uk.shape[0]
        # hanging: midpoints of edges and faces of leaves, with their corners
        par = torch.full((n_all, 4), -1, device=DEV)

        def find(k):
            i = torch.searchsorted(uk, k).clamp_(max=n_all - 1)
            return torch.where(uk[i] == k, i, -1)

        for pat in range(3 ** dim):
            ch = [(pat // 3 ** a) % 3 for a in range(dim)]
            half = [a for a in range(dim) if ch[a] == 1]
            if not half or len(half) == dim:
                continue
            sel = size > 1
            base, s = anc[sel], size[sel]
            x = base + torch.stack([ch[a] * s // 2 for a in range(dim)], -1)
            ids = find((x * mul).sum(-1))
            ok = ids >= 0
            base, s, ids = base[ok], s[ok], ids[ok]
            for b in range(1 << len(half)):
                y = torch.stack([base[:, a] + (((b >> half.index(a)) & 1) * s if a in half else (ch[a] // 2) * s)
                                 for a in range(dim)], -1)
                par[ids, b] = find((y * mul).sum(-1))
        hanging = par[:, 0] >= 0
        order = torch.argsort(torch.where(hanging, keys.shape[0] + first, first))
        n = int((~hanging).sum())
        num = torch.full((n_all,), -1, device=DEV)
        num[order[:n]] = torch.arange(n, device=DEV)
        self.n = n
        xi = torch.empty(n_all, dim, dtype=torch.int64, device=DEV)
        xi[inv] = corner.reshape(-1, dim)
        self.x = xi[order[:n]].double() / top
        # corner value = sum of w over up to four nodes
        npar = (par >= 0).sum(1).clamp(min=1)
        idx = torch.where(hanging[:, None], torch.where(par >= 0, num[par.clamp(min=0)], 0),
                          torch.where(torch.arange(4, device=DEV) == 0, num.clamp(min=0)[:, None], 0))
        w = torch.where(hanging[:, None], (par >= 0) / npar[:, None].double(),
                        (torch.arange(4, device=DEV) == 0).double())
        self.idx, self.wt = idx[inv].reshape(-1, nc, 4), w[inv].reshape(-1, nc, 4)
        if not bool(hanging.any()):
            self.idx, self.wt = self.idx[..., :1].contiguous(), self.wt[..., :1].contiguous()
        self.h = size.double() / top
        xin = xi[order[:n]]
        self.wall = ((xin == 0) | (xin == top)).any(1)
        self.origin = int(torch.nonzero((xin == 0).all(1))[0])
        g = 1.0 / math.sqrt(3.0)
        self.gp = []
        for q in range(nc):
            xq = [(g if (q >> a) & 1 else -g) for a in range(dim)]
            N = torch.ones(nc, dtype=torch.float64, device=DEV)
            dN = torch.ones(nc, dim, dtype=torch.float64, device=DEV)
            ddN = torch.ones(nc, dim, dim, dtype=torch.float64, device=DEV)
            for c in range(nc):
                for a in range(dim):
                    sg = 1.0 if (c >> a) & 1 else -1.0
                    v, d = 0.5 * (1.0 + sg * xq[a]), sg  # d/dx of the hat is +-1/h
                    N[c] *= v
                    for i in range(dim):
                        dN[c, i] *= d if i == a else v
                        for j in range(dim):
                            ddN[c, i, j] *= 0.0 if i == j else (d if a in (i, j) else v)
            self.gp.append((xq, N, dN, ddN))

    def gather(self, U):
        return (U[self.idx] * self.wt[..., None]).sum(2)

    def scatter(self, R):
        out = torch.zeros(self.n, R.shape[-1], dtype=R.dtype, device=R.device)
        v = (R[:, :, None, :] * self.wt[..., None]).reshape(-1, R.shape[-1])
        return out.index_add(0, self.idx.reshape(-1), v)


def _residual(G, p, Un, Uo, f=None, bc=None):
    """F(U_new; U_old), [n, dim + 3]."""
    d = G.dim
    un, uo = G.gather(Un), G.gather(Uo)
    ut, dl = 0.5 * (un + uo), un - uo
    ff = G.gather(f) if f is not None else None
    h = G.h[:, None]
    gv = torch.tensor(p.gravity[:d], dtype=torch.float64, device=DEV)
    Gm, inv_trG = 4.0 / h ** 2, h ** 2 / (4.0 * d)
    al, be = 0.5 * (1 - p.rho_ratio), 0.5 * (1 + p.rho_ratio)
    ga, xi = 0.5 * (1 - p.eta_ratio), 0.5 * (1 + p.eta_ratio)
    R = torch.zeros_like(un)
    for xq, N, dN, ddN in G.gp:
        val = torch.einsum("ecf,c->ef", ut, N)
        grad = torch.einsum("ecf,ca->efa", ut, dN) / h[..., None]
        inc = torch.einsum("ecf,c->ef", dl, N)
        v, dv = val[:, :d], grad[:, :d]
        phi, dphi, mu, dmu = val[:, d + 1:d + 2], grad[:, d + 1], val[:, d + 2:d + 3], grad[:, d + 2]
        hphi = torch.einsum("ec,cij->eij", ut[..., d + 1], ddN) / h[..., None] ** 2
        pn = phi + 0.5 * inc[:, d + 1:d + 2]
        dpn = dphi + 0.5 * torch.einsum("ec,ca->ea", dl[..., d + 1], dN) / h
        fq = torch.einsum("ecf,c->ef", ff, N) if ff is not None else torch.zeros_like(val)
        inside = pn.abs() <= 1
        ps = torch.where(inside, pn, torch.sign(pn).detach())
        rho, eta = al * ps + be, ga * ps + xi
        deta = torch.where(inside, ga * dpn, torch.zeros_like(dpn))
        J = 0.5 * (p.rho_ratio - 1) * dmu
        rad = (4 / p.dt ** 2 + Gm * (v * v).sum(1, True) + Gm * (v * J).sum(1, True) / (rho * p.Pe)
               + p.C_I * (eta / (rho * p.Re)) ** 2 * (d * Gm ** 2))
        rad = torch.where(rad < 4 / p.dt ** 2, torch.full_like(rad, 4 / p.dt ** 2), rad)
        tau = rad ** -0.5
        tau_c = inv_trG / tau
        dot = lambda a: torch.einsum("eij,ej->ei", dv, a)  # noqa: E731
        mom = rho * (inc[:, :d] / p.dt + dot(v)) + dot(J) / p.Pe - rho * gv / p.Fr - fq[:, :d]
        Rm = mom + p.Cn / p.We * torch.einsum("eij,ej->ei", hphi, dphi) + grad[:, d] / p.We - dot(deta) / p.Re
        divv = torch.diagonal(dv, dim1=1, dim2=2).sum(1, True)
        Rc = divv - fq[:, d:d + 1]
        t = tau * Rm
        S = torch.cat([mom - dot(t), Rc, inc[:, d + 1:d + 2] / p.dt - fq[:, d + 1:d + 2],
                       phi ** 3 - phi - mu - fq[:, d + 2:]], 1)
        V = (t[:, :, None] * (v + (J / p.Pe - t) / rho)[:, None, :]
             - p.Cn / p.We * dphi[:, :, None] * dphi[:, None, :] + (eta / p.Re)[..., None] * dv)
        V = V + torch.eye(d, dtype=V.dtype, device=V.device) * ((rho * tau_c * Rc - val[:, d:d + 1]) / p.We)[..., None]
        V = torch.cat([V, (t / rho)[:, None], (dmu / (p.Pe * p.Cn) - v * phi)[:, None],
                       (p.Cn ** 2 * dphi)[:, None]], 1)
        Wq = (h / 2) ** d
        R = R + N[:, None] * (Wq * S)[:, None, :] + torch.einsum("efa,ca->ecf", V * (Wq / h)[..., None], dN)
    F = G.scatter(R)
    g = bc if bc is not None else torch.zeros_like(Un)
    con = torch.zeros_like(Un, dtype=torch.bool)
    con[:, :d] = G.wall[:, None]
    con[G.origin, d] = True
    return torch.where(con, Un - g, F)


def _energy(G, p, U):
    d = G.dim
    u = G.gather(U)
    z0 = torch.tensor(p.gravity[:d], dtype=torch.float64, device=DEV)
    # the lowest corner of each leaf; it is never interpolated when the leaf
    # touches it as an own node, so interpolate the coordinates instead
    xc = G.gather(torch.cat([G.x, torch.zeros(G.n, 3, dtype=torch.float64, device=DEV)], 1))[..., :d]
    E = M = L = 0.0
    for xq, N, dN, _ in G.gp:
        val = torch.einsum("ecf,c->ef", u, N)
        dphi = torch.einsum("ec,ca->ea", u[..., d + 1], dN) / G.h[:, None]
        x = torch.einsum("eca,c->ea", xc, N)
        phi = val[:, d + 1]
        rho = 0.5 * (1 - p.rho_ratio) * phi.clamp(-1, 1) + 0.5 * (1 + p.rho_ratio)
        e = (0.5 * rho * (val[:, :d] ** 2).sum(1) + (0.25 * (phi ** 2 - 1) ** 2 / p.Cn + 0.5 * p.Cn * (dphi ** 2).sum(1)) / p.We
             - rho * (x * z0).sum(1) / p.Fr)
        Wq = (G.h / 2) ** d
        E, M, L = E + (Wq * e).sum(), M + (Wq * phi).sum(), L + (Wq * (phi < 0)).sum()
    return {"energy": float(E), "mass": float(M), "light_volume": float(L)}


def _project_mu(G, p, U):
    """M mu = (N, phi^3 - phi) + Cn^2 (grad N, grad phi) by conjugate gradients."""
    d = G.dim

    def row(a, grad_of=None, cubic=False):
        ua = G.gather(a[:, None])[..., 0]
        R = torch.zeros_like(ua)
        for xq, N, dN, _ in G.gp:
            Wq = (G.h / 2) ** d
            v = ua @ N
            s = v ** 3 - v if cubic else v
            R = R + (Wq * s)[:, None] * N
            if grad_of is not None:
                R = R + grad_of * (Wq / G.h ** 2)[:, None] * ((ua @ dN) @ dN.T)
        return G.scatter(R[..., None])[:, 0]

    phi = U[:, d + 1]
    b = row(phi, p.Cn ** 2, cubic=True)
    D = row(torch.ones_like(phi))
    x = b / D
    r = b - row(x)
    z = r / D
    q, rz, stop = z.clone(), (r * z).sum(), 1e-32 * (b * b / D).sum()
    for _ in range(400):
        if rz <= stop:
            break
        Aq = row(q)
        a = rz / (q * Aq).sum()
        x, r = x + a * q, r - a * Aq
        z = r / D
        rz, old = (r * z).sum(), rz
        q = z + rz / old * q
    out = U.clone()
    out[:, d + 2] = x
    return out


def _newton(G, p, Un):
    """The root of F(.; U_n) by Newton's method with a dense Jacobian."""
    n = Un.numel()
    U = Un.clone()
    eye = torch.eye(n, dtype=torch.float64, device=DEV)
    best = math.inf
    for _ in range(12):
        F = _residual(G, p, U, Un).reshape(-1)
        nrm = float(F.norm())
        if not nrm < 0.5 * best:
            break
        best, keep = nrm, U
        fn = lambda w: torch.func.jvp(lambda X: _residual(G, p, X, Un), (U,), (w.reshape(U.shape),))[1].reshape(-1)  # noqa: E731
        Jt = torch.cat([torch.func.vmap(fn)(eye[k:k + 363]) for k in range(0, n, 363)])
        U = U - torch.linalg.solve(Jt.T, F).reshape(U.shape)
    return keep


def exact(case, seed):
    call = case["call"]
    if call == "batch" or (call == "step" and (case["dim"] == 3 or case["top"] > 5)):
        return None  # the direct solve of a larger Jacobian takes too long
    G, p = _Grid(_case_leaves(case)), _params(case)
    nf = G.dim + 3
    if call in ("init_mu", "step"):
        U = _project_mu(G, p, _start_state(case, G.x, seed))
        if call == "init_mu":
            return U.reshape(-1)
        U = _newton(G, p, U)
        e = _energy(G, p, U)
        return {"U": U.reshape(-1), "energy": e["energy"], "mass": e["mass"]}
    Un, Uo = (u.reshape(-1, nf) for u in _newton_pair(case, G.x, seed))
    if call == "energy":
        return _energy(G, p, Un)
    if call == "residual":
        f = bc = None
        if case["forced"]:
            f, bc = (u.reshape(-1, nf) for u in _source(case, G.x, seed, Un.reshape(-1)))
        return _residual(G, p, Un, Uo, f, bc).reshape(-1)
    dt = torch.float64 if case["precision"] == "fp64" else torch.float32
    w = (_rand(seed, 3, G.n * nf) * _free_rows(G.x, nf).reshape(-1)).to(dt).double().reshape(-1, nf)
    return torch.func.jvp(lambda X: _residual(G, p, X, Uo), (Un,), (w,))[1].reshape(-1)
