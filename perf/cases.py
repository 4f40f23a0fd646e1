"""Timed workloads of the immersed-boundary coupling framework.

Every case is one call (or the few calls) that a simulation, an inverse
problem or a parameter sweep repeats, through the public entry points of
paper_2503_22695_gb300.ibfe:

  step      ib_step, one explicit time step: nodal force, spreading, fluid
            solve, interpolation, position update (the state advances in place)
  fluid     ib_fluid_step alone, the projection step on the MAC grid
  forward   ib_forward, the coupling step: force, spreading, interpolation
  backward  ib_backward, the fused vector-Jacobian product of ib_forward
  grad      the autograd module IBCoupling, forward and backward of a loss
  transfer  ib_spread and ib_interp as separate calls
  batch     a parameter sweep of independent shells: Batch.forward, .adjoint
            and .gparams

Structures are the repository's synthetic ones (paper_2503_22695_gb300.inputs):
the elastic block, the ventricle-like shell, the shell with two leaflet
sheets; as trilinear hexahedra, P1 or P2 tetrahedra.  exact() evaluates the
same definitions in 64-bit torch, with derivatives by autograd.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2503_22695_gb300 import ibfe
from paper_2503_22695_gb300 import inputs as I

RHO, MU = 1.0, 0.01           # fluid density and viscosity
DT_FLUID = 1e-4               # time step of the fluid alone
CFL = 0.004                   # time step of the explicit IB step, in units of h (elastic waves of speed ~20)
NODES = {"hex": 8, "tet4": 4, "tet10": 10}


def listed():
    return [
        # smallest time step: a block of 128 elements on a 32^3 grid; launches and latency
        dict(name="step_block_32", kind="step", body="block", elem="hex", prec="f32", quad="gauss",
             n=32, dims="8x8x2"),
        # contracting ventricle-like shell (active fibre tension) on the 128^3 grid
        dict(name="step_shell_128", kind="step", body="shell", elem="hex", prec="f32",
             quad="gauss", n=128, dims="60x40x6", active=20.0),
        # the largest time step: shell and leaflet sheets, 1.4 M Gauss points, 256^3 grid
        dict(name="step_sheets_256", kind="step", body="sheets", elem="hex", prec="f32",
             quad="gauss", n=256, dims="160x100x10"),
        # the fluid alone on a grid that is not a power of two
        dict(name="fluid_192", kind="fluid", n0=192, n1=192, n2=192),
        # plain FP64 coupling of the small block
        dict(name="forward_block_32_f64", kind="forward", body="block", elem="hex", prec="f64",
             quad="gauss", n=32, dims="8x8x2"),
        # the coupling step inside someone else's fluid solver: medium and large
        dict(name="forward_shell_128", kind="forward", body="shell", elem="hex", prec="f32",
             quad="gauss", n=128, dims="60x40x6"),
        dict(name="forward_sheets_256", kind="forward", body="sheets", elem="hex", prec="f32",
             quad="gauss", n=256, dims="160x100x10"),
        # valve leaflets are tetrahedral meshes: ragged sizes, an odd number of grid tiles
        dict(name="forward_tet4_104", kind="forward", body="shell", elem="tet4", prec="f32",
             quad="gauss", n=104, dims="37x23x5"),
        # parameter and shape estimation: loss and gradients through autograd
        dict(name="grad_shell_128", kind="grad", body="shell", elem="hex", prec="f32",
             quad="gauss", n=128, dims="60x40x6"),
        # the backward of the large coupling step
        dict(name="backward_sheets_256", kind="backward", body="sheets", elem="hex", prec="f32",
             quad="gauss", n=256, dims="160x100x10"),
        # the paper's nodal quadrature, spreading and interpolation on their own
        dict(name="transfer_nodal_176", kind="transfer", body="shell", elem="hex", prec="f32",
             quad="nodal", n=176, dims="121x83x9"),
        # parameter sweep: shells of uneven sizes on grids of 32^3 .. 128^3
        dict(name="batch_16", kind="batch", count=16, first=5000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "fluid", "forward", "forward", "backward", "grad",
                       "transfer", "batch"])
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(4, 20), first=rng.randrange(6000, 9000))
    # grids the fluid's multigrid halves down to 8 cells or fewer
    fluid_n = [32, 48, 64, 96, 128, 192, 256]
    if kind == "fluid":
        n = rng.choice(fluid_n)
        other = [m for m in fluid_n if m in (n, 2 * n) or 2 * m == n]
        return dict(kind=kind, n0=n, n1=rng.choice(other), n2=rng.choice([n, n, rng.choice(other)]))
    quad = rng.choice(["gauss", "gauss", "gauss", "nodal"])
    elem = rng.choice(["hex", "hex", "hex", "tet4", "tet10"])
    prec = "f32"
    if kind == "step":
        n = rng.choice(fluid_n[:6])
    else:
        n = 8 * _log_int(rng, 4, 30)
        if kind in ("forward", "transfer") and n <= 96 and rng.random() < 0.3:
            prec = "f64"
    if kind == "transfer":
        elem = "hex"
    # element counts that follow the grid, odd ones among them
    scale = n / 128.0 * rng.uniform(0.8, 1.25) * (0.6 if elem != "hex" else 1.0)
    dims = (max(7, int(60 * scale)), max(5, int(40 * scale)), max(2, int(6 * scale)))
    c = dict(kind=kind, body="shell", elem=elem, prec=prec, quad=quad, n=n,
             dims="%dx%dx%d" % dims)
    if rng.random() < 0.3:
        c["active"] = float(rng.choice([5, 20, 60]))
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _rng(seed, salt):
    return np.random.Generator(np.random.PCG64([seed, salt]))


def _structure(case, seed):
    """An inputs.Problem without a velocity field."""
    rng = _rng(seed, 1)
    n = case["n"]
    fp64 = case["prec"] == "f64"
    grid = I.Grid((n, n, n), 1.0 / n)
    dims = tuple(int(v) for v in case["dims"].split("x"))
    active = float(case.get("active", 0.0))
    if case["body"] == "block":
        conn, X = I.box_block(*dims, edge=grid.h, centre=(0.5, 0.5, 0.5))
        fib = np.zeros((6, conn.shape[1]))
        fib[0] = fib[4] = 1.0
        mats = [I.Material(I.NEO_HOOKEAN, (0.5, 100.0), active)]
        mat_id = np.zeros(conn.shape[1])
    else:
        conn, X, fib = I.ellipsoid_shell(*dims)
        mat_id = np.zeros(conn.shape[1])
        # tetrahedral shells take the valve law, hexahedral ones the ventricle's
        mats = [I.Material(I.HO, I.HO_DEFAULT, active) if case["elem"] == "hex"
                else I.Material(I.FIBRE2, I.FIBRE2_AV, active)]
        if case["body"] == "sheets":
            for facing, y in ((-1.0, 0.66), (1.0, 0.34)):
                c2, X2, f2 = I.cylinder_sheet(80, 40, 2, axis_point=(0.5, y, 0.62), facing=facing)
                conn = np.concatenate([conn, c2 + X.shape[1]], axis=1)
                X = np.concatenate([X, X2], axis=1)
                fib = np.concatenate([fib, f2], axis=1)
                mat_id = np.concatenate([mat_id, np.ones(c2.shape[1])])
            mats.append(I.Material(I.FIBRE1, I.FIBRE1_LEAFLET, 0.0))
    # a block in a time loop is nearer rest than the one of the single coupling step
    return _problem(grid, conn, X, fib, mat_id, mats, fp64, case["body"], case["elem"], rng,
                    noise=0.1 if case["kind"] == "step" else 0.2)


def _problem(grid, conn, X, fib, mat_id, mats, fp64, body, elem, rng, noise=0.2):
    ft = np.float64 if fp64 else np.float32
    X = X.astype(ft).astype(np.float64)
    if body == "block":
        x = X + rng.uniform(-noise * grid.h, noise * grid.h, size=X.shape)
    else:
        x = I.smooth_deformation(X, rng)
    cell, off = I.to_split(x, grid)
    p = I.Problem(body, grid, np.ascontiguousarray(conn.astype(np.int32)), X.astype(ft),
                  np.ascontiguousarray(fib.astype(ft)), mat_id.astype(np.int32), mats, x, cell,
                  off, None, fp64)
    if elem == "tet4":
        p = I.tet_problem(p)
    elif elem == "tet10":
        p = I.tet10_problem(p, seed=int(rng.integers(1 << 30)))
    return p


def _batch_problems(case, seed):
    """The sweep's shells: sizes from the case, deformations from the seed."""
    out = []
    for i in range(case["count"]):
        size = np.random.Generator(np.random.PCG64(case["first"] + i))
        n = int(size.choice((32, 64, 96, 128)))
        nt = int(size.integers(2, 7))
        target = size.uniform(2000, 20000)
        nl = max(4, int(round(math.sqrt(target / nt / 1.5))))
        nc = max(6, int(round(target / nt / nl)))
        rng = _rng(seed, 100 + i)
        ho = np.array(I.HO_DEFAULT)
        ho[:4] *= rng.uniform(0.7, 1.3, size=4)
        conn, X, fib = I.ellipsoid_shell(nc, nl, nt)
        out.append(_problem(I.Grid((n, n, n), 1.0 / n), conn, X, fib, np.zeros(conn.shape[1]),
                            [I.Material(I.HO, tuple(ho))], False, "shell", "hex", rng))
    return out


def _modes(n, rng, solenoidal, count=12, kmax=4):
    """A smooth periodic MAC field [3][n2][n1][n0] (float64, rms 0.5): `count`
    Fourier modes, discretely divergence-free if asked."""
    L = 1.0                      # cubes of unit edge; other boxes keep h = 1 / n0
    h = L / n[0]
    k = rng.integers(-kmax, kmax + 1, size=(count, 3))
    k[(k == 0).all(axis=1)] = 1
    a = rng.normal(size=(count, 3)) + 1j * rng.normal(size=(count, 3))
    if solenoidal:
        kt = 2.0 * np.sin(math.pi * k / np.array(n)) / h
        kt /= np.linalg.norm(kt, axis=1, keepdims=True)
        a -= (a * kt).sum(axis=1, keepdims=True) * kt
    dev = "cuda"
    out = torch.empty((3, n[2], n[1], n[0]), dtype=torch.float64, device=dev)
    for c in range(3):
        e = []
        for d in range(3):
            s = 0.0 if d == c else 0.5
            th = 2 * math.pi * np.outer(k[:, d], (np.arange(n[d]) + s) / n[d])
            e.append(torch.from_numpy(np.exp(1j * th)).to(dev))
        B = torch.einsum("m,mz,my->zym", torch.from_numpy(a[:, c]).to(dev), e[2], e[1])
        # real part of B @ E0, plane by plane
        out[c] = B.real @ e[0].real - B.imag @ e[0].imag
    return out * (0.5 / out.square().mean().sqrt())


def _velocity(n, seed, dtype, kind=""):
    """The velocity on the grid; slower and smoother for a time loop, which
    carries its structure along for thousands of steps."""
    u = _modes(n, _rng(seed, 2), True, kmax=2 if kind == "step" else 4)
    return (u * (0.2 if kind == "step" else 1.0)).to(dtype).contiguous()


def _body_force(n, seed, dtype):
    """A force density like a spread one: smooth modes of magnitude 50 within
    a shell of the box."""
    f = _modes(n, _rng(seed, 3), False, count=8) * 100.0
    r2 = 0.0
    for d, ax in ((0, 3), (1, 2), (2, 1)):
        t = (torch.arange(n[d], device="cuda", dtype=torch.float64) + 0.5) / n[d] - 0.5
        shape = [1, 1, 1, 1]
        shape[ax] = n[d]
        r2 = r2 + t.reshape(shape) ** 2
    return (f * torch.exp(-((r2.sqrt() - 0.25) / 0.06) ** 2)).to(dtype).contiguous()


def _dtype(case):
    return torch.float64 if case.get("prec") == "f64" else torch.float32


def _cotangents(p, seed, dtype):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 7919 + 5)
    n0, n1, n2 = p.grid.n
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda", dtype=torch.float64).to(dtype)
    return dict(gG=rnd(3, p.n_nodes), gU=rnd(3, p.n_nodes), gf=rnd(3, n2, n1, n0) * 1e-3)


def _mats(p):
    return [ibfe.Material(m.model, m.params, m.active) for m in p.materials]


def _to_dev(p, dtype):
    dev = "cuda"
    t = lambda a, d=None: torch.from_numpy(np.ascontiguousarray(a)).to(dev, d)
    d = dict(conn=t(p.conn), X=t(p.X, dtype), fibres=t(p.fibres, dtype), mat_id=t(p.mat_id))
    if p.fp64:
        d["x64"] = t(p.x)
        d["pos"] = ibfe.Pos(x64=d["x64"])
    else:
        d["cell"], d["off"] = t(p.cell), t(p.off)
        d["pos"] = ibfe.Pos(cell=d["cell"], off=d["off"])
    return d


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = case
    if case["kind"] == "fluid":
        n = (case["n0"], case["n1"], case["n2"])
        s.fluid = ibfe.Fluid(n, 1.0 / n[0], RHO, MU, DT_FLUID)
        s.u, s.f = _velocity(n, seed, torch.float32), _body_force(n, seed, torch.float32)
        s.un = torch.empty_like(s.u)
        s.p = torch.empty(n[::-1], device="cuda")
        return s
    if case["kind"] == "batch":
        s.inst = []
        for i, p in enumerate(_batch_problems(case, seed)):
            d = _to_dev(p, torch.float32)
            d.update(n=p.grid.n, h=p.grid.h, mats=_mats(p))
            d.update(_cotangents(p, seed + i, torch.float32))
            d["u"] = _velocity(p.grid.n, seed + i, torch.float32)
            for k in ("G", "U", "gx"):
                d[k] = torch.empty((3, p.n_nodes), device="cuda")
            for k in ("f", "gu"):
                d[k] = torch.empty_like(d["u"])
            s.inst.append(d)
        s.batch = ibfe.Batch(s.inst)
        return s
    p = _structure(case, seed)
    dtype = _dtype(case)
    s.d = _to_dev(p, dtype)
    s.pos, s.mats = s.d["pos"], _mats(p)
    s.plan = ibfe.Plan(s.d["conn"], s.d["X"], p.grid.n, p.grid.h, fibres=s.d["fibres"],
                       mat_id=s.d["mat_id"],
                       precision=ibfe.IB_FP64 if p.fp64 else ibfe.IB_FP32_SPLIT,
                       quad=ibfe.IB_QUAD_NODAL if case["quad"] == "nodal" else ibfe.IB_QUAD_GAUSS2)
    s.u = _velocity(p.grid.n, seed, dtype, case["kind"])
    s.G = torch.empty((3, p.n_nodes), device="cuda", dtype=dtype)
    s.U = torch.empty_like(s.G)
    s.f = torch.empty_like(s.u)
    if case["kind"] == "step":
        s.fluid = ibfe.Fluid(p.grid.n, p.grid.h, RHO, MU, CFL * p.grid.h)
        s.p = torch.empty(s.u.shape[1:], device="cuda", dtype=dtype)
    elif case["kind"] == "backward":
        ibfe.ib_forward(s.plan, s.mats, s.pos, s.u, s.G, s.f, s.U)
        s.cot = _cotangents(p, seed, dtype)
        s.gx, s.gu = torch.empty_like(s.G), torch.empty_like(s.u)
    elif case["kind"] == "transfer":
        # nodal forces of the structure, as the spreading meets them
        ibfe.ib_fe_force(s.plan, s.mats, s.pos, s.G)
    elif case["kind"] == "grad":
        s.net = ibfe.IBCoupling(s.plan, [m.model for m in p.materials])
        s.params = _theta(p.materials).requires_grad_()
        s.off = s.d["off"].clone().requires_grad_()
        s.u.requires_grad_()
    return s


def run(s):
    k = s.case["kind"]
    if k == "fluid":
        u, p, _ = ibfe.ib_fluid_step(s.fluid, s.u, s.f, s.un, s.p)
        return dict(u=u, p=p)
    if k == "batch":
        s.batch.forward()
        s.batch.adjoint()
        gp = s.batch.gparams().float()   # sums of FP32 terms
        out = dict(gparams=gp)
        for i, d in enumerate(s.inst[:10]):
            out["i%d" % i] = [d[v] for v in ("G", "f", "U", "gu", "gx")]
        return out
    if k == "step":
        G, f, U, p = ibfe.ib_step(s.plan, s.fluid, s.mats, s.pos, s.u, s.G, s.f, s.U, s.p)
        x = (s.d["cell"] + s.d["off"]) * s.plan.h   # positions for the caller's output
        return dict(G=G, f=f, U=U, p=p, u=s.u, x=x)
    if k == "forward":
        G, f, U = ibfe.ib_forward(s.plan, s.mats, s.pos, s.u, s.G, s.f, s.U)
        return dict(G=G, f=f, U=U)
    if k == "transfer":
        f = ibfe.ib_spread(s.plan, s.pos, s.G, s.f)
        U = ibfe.ib_interp(s.plan, s.pos, s.u, s.U)
        return dict(f=f, U=U)
    if k == "backward":
        gx, gu, gp = ibfe.ib_backward(s.plan, s.mats, s.pos, s.u, s.G, s.cot["gG"], s.cot["gf"],
                                      s.cot["gU"], s.gx, s.gu)
        return dict(gx=gx, gu=gu, gparams=gp.float())
    G, f, U = s.net(s.d["cell"], s.off, s.params, s.u)
    loss = U.square().sum() + s.plan.h ** 1.5 * f.norm()
    g = torch.autograd.grad(loss, [s.off, s.params, s.u])
    return dict(loss=loss.detach(), G=G.detach(), f=f.detach(), U=U.detach(), goff=g[0],
                gparams=g[1].float(), gu=g[2])


def work(case):
    """Compulsory bytes and operations of one pass."""
    k = case["kind"]
    if k == "fluid":
        cells = case["n0"] * case["n1"] * case["n2"]
        return dict(bytes=40.0 * cells, flops=100.0 * cells)   # u, f in; u, p out
    if k == "batch":
        b = fl = 0.0
        for i in range(case["count"]):
            size = np.random.Generator(np.random.PCG64(case["first"] + i))
            n = int(size.choice((32, 64, 96, 128)))
            nt = int(size.integers(2, 7))
            E = size.uniform(2000, 20000)
            N = E * (nt + 1) / nt
            b += 12.0 * n ** 3 * 3 + 60.0 * E * 2 + 150.0 * N   # f, gf, gu dense; u on its support
            fl += 8 * E * 4 * 1800.0
        return dict(bytes=b, flops=fl)
    nc, nl, nt = (int(v) for v in case["dims"].split("x"))
    rs = 8 if case["prec"] == "f64" else 4
    block = case["body"] == "block"
    E = nc * nl * nt
    N = (nc + 1) * (nl + 1) * (nt + 1) if block else nc * (nl + 1) * (nt + 1)
    if case["body"] == "sheets":
        E, N = E + 12800, N + 2 * 81 * 41 * 3
    if case["elem"] == "tet10":
        N = 7.4 * N
    if case["elem"] != "hex":
        E *= 6
    Q = N if case["quad"] == "nodal" else E * (8 if case["elem"] == "hex" else 4)
    cells = case["n"] ** 3
    support = rs * 3 * min(cells, 2.5 * N)       # velocity faces the stencils reach
    mesh = E * (4 * NODES[case["elem"]] + 6 * rs + 4) + N * 9 * rs
    dense = 3 * rs * cells
    force, transfer = 1000.0 * E * (8 if case["elem"] == "hex" else 1), 800.0 * Q
    if k == "transfer":
        return dict(bytes=dense + support + N * 12 * rs, flops=transfer)
    if k == "forward":
        return dict(bytes=dense + support + mesh, flops=force + transfer)
    if k == "step":
        return dict(bytes=dense + 28.0 * cells + mesh + 12 * rs * N,
                    flops=force + transfer + 100.0 * cells)
    if k == "backward":
        return dict(bytes=dense + 2 * support + mesh, flops=2 * force + 3 * transfer)
    return dict(bytes=2 * dense + 3 * support + 2 * mesh, flops=3 * force + 4 * transfer)


# ---------------------------------------------------------------------------
# the same definitions in 64-bit torch
# ---------------------------------------------------------------------------

def _theta(materials):
    """[n_mats][10] float64: the law's parameters, zeros, T_a."""
    t = torch.zeros(len(materials), 10, dtype=torch.float64)
    for i, m in enumerate(materials):
        t[i, :len(m.params)] = torch.tensor(m.params, dtype=torch.float64)
        t[i, 9] = m.active
    return t


def _rule(elem):
    """N [C][Q], dN/dxi [C][Q][3] and the weight of the element's point rule."""
    if elem == "hex":
        c = I.HEX_CORNERS.astype(float)
        pts = np.array([[(2 * ((q >> d) & 1) - 1) / math.sqrt(3.0) for d in range(3)]
                        for q in range(8)])
        fac = 0.5 * (1.0 + c[:, None, :] * pts[None])            # [C][Q][3]
        dN = np.stack([0.5 * c[:, None, d] * np.prod(np.delete(fac, d, axis=2), axis=2)
                       for d in range(3)], axis=2)
        return fac.prod(axis=2), dN, 1.0
    a, b = (5 + 3 * math.sqrt(5)) / 20, (5 - math.sqrt(5)) / 20
    Lq = np.full((4, 4), b) + np.eye(4) * (a - b)                # [L_i][q]
    dL = np.concatenate([-np.ones((1, 3)), np.eye(3)])
    if elem == "tet4":
        return Lq, np.repeat(dL[:, None, :], 4, axis=1), 1.0 / 24.0
    N = np.empty((10, 4))
    dN = np.empty((10, 4, 3))
    for i in range(4):
        N[i] = Lq[i] * (2 * Lq[i] - 1)
        dN[i] = (4 * Lq[i] - 1)[:, None] * dL[i]
    for e, (i, j) in enumerate(I.TET10_EDGES):
        N[4 + e] = 4 * Lq[i] * Lq[j]
        dN[4 + e] = 4 * (Lq[i][:, None] * dL[j] + Lq[j][:, None] * dL[i])
    return N, dN, 1.0 / 24.0


def _psi(model, t, F, ef, es):
    """Strain energy at the points of F [Q][E][3][3]; t: one row of _theta."""
    np_ = I.N_PARAMS[model]
    lnJ = torch.log(torch.linalg.det(F))
    I1b = torch.exp(-2.0 / 3.0 * lnJ) * F.square().sum((-1, -2))
    psi = 0.5 * t[np_ - 1] * lnJ ** 2
    Ff = (F * ef[:, None, :]).sum(-1)
    I4 = Ff.square().sum(-1)

    def fibre(i4, a, b, clamp=True):
        d = torch.where(i4 > 1.0, i4 - 1.0, torch.zeros_like(i4)) if clamp else i4 - 1.0
        return a / (2.0 * b) * torch.expm1(b * d ** 2)

    if model == I.NEO_HOOKEAN:
        psi = psi + t[0] * (I1b - 3.0)
    elif model == I.FIBRE1:
        psi = psi + t[0] * (I1b - 3.0) + fibre(I4, t[1], t[2])
    elif model == I.FIBRE2:
        psi = psi + t[0] * torch.expm1(t[1] * (I1b - 3.0)) + fibre(I4, t[2], t[3], False)
    else:
        Fs = (F * es[:, None, :]).sum(-1)
        I8 = (Ff * Fs).sum(-1)
        psi = (psi + t[0] / (2.0 * t[1]) * torch.expm1(t[1] * (I1b - 3.0))
               + fibre(I4, t[2], t[3]) + fibre(Fs.square().sum(-1), t[4], t[5])
               + t[6] / (2.0 * t[7]) * torch.expm1(t[7] * I8 ** 2))
    return psi + 0.5 * t[9] * (-3.9 * (I4 - 1.0) + 4.9 * 2.0 / 3.0 * (I4 ** 1.5 - 1.0))


class _Exact:
    """Force, spreading and interpolation of one structure, differentiable."""

    def __init__(self, p, elem, quad):
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
        N, dN, w = _rule(elem)
        self.N, self.dN = t(N), t(dN)
        self.conn = t(p.conn.astype(np.int64))
        self.X = t(p.X.astype(np.float64))
        self.n, self.h, self.nodes = p.grid.n, p.grid.h, p.n_nodes
        self.nodal = quad == "nodal"
        fib = t(p.fibres.astype(np.float64))
        self.ef, self.es = fib[:3].T, fib[3:].T
        self.mat = t(p.mat_id.astype(np.int64))
        self.models = [m.model for m in p.materials]
        J0 = torch.einsum("iae,aqd->qeid", self.X[:, self.conn], self.dN)
        self.J0inv = torch.linalg.inv(J0)
        self.wj0 = w * torch.linalg.det(J0)                      # [Q][E]
        if elem == "tet10":
            d = torch.einsum("aq,qe->ae", self.N ** 2, self.wj0)
            d = d * (self.wj0.sum(0) / d.sum(0))
        else:
            d = torch.einsum("aq,qe->ae", self.N, self.wj0)
        self.m = self._assemble(d[None])[0]

    def _assemble(self, elem):                                   # [k][C][E] -> [k][N]
        k = elem.shape[0]
        out = torch.zeros(k, self.nodes, dtype=torch.float64, device="cuda")
        return out.index_add(1, self.conn.reshape(-1), elem.reshape(k, -1))

    def force(self, x, theta, create_graph=False):
        x = x if x.requires_grad else x.detach().requires_grad_()
        with torch.enable_grad():
            F = torch.einsum("iae,aqd->qeid", x[:, self.conn], self.dN) @ self.J0inv
            E = 0.0
            for k, model in enumerate(self.models):
                sel = (self.mat == k).nonzero()[:, 0]
                psi = _psi(model, theta[k], F[:, sel], self.ef[sel], self.es[sel])
                E = E + (psi * self.wj0[:, sel]).sum()
            return -torch.autograd.grad(E, x, create_graph=create_graph)[0]

    def _stencils(self, x):
        """Per component: flat face indices and weights [64][points], with the
        coupling points at chi."""
        if self.nodal:
            chi = x
        else:
            chi = torch.einsum("iae,aq->iqe", x[:, self.conn], self.N).reshape(3, -1)
        for c in range(3):
            idx, w = [], []
            for d in range(3):
                r = chi[d] / self.h - (0.0 if d == c else 0.5)
                i0 = torch.floor(r.detach())
                th = r - i0
                q = torch.sqrt(1.0 + 4.0 * th * (1.0 - th))
                w.append(torch.stack([(3 - 2 * th - q) / 8, (3 - 2 * th + q) / 8,
                                      (1 + 2 * th + q) / 8, (1 + 2 * th - q) / 8]))
                i = i0.long()[None] + torch.arange(-1, 3, device="cuda")[:, None]
                idx.append(i % self.n[d])
            n0, n1, _ = self.n
            flat = ((idx[2][:, None, None] * n1 + idx[1][None, :, None]) * n0
                    + idx[0][None, None, :])
            wt = w[2][:, None, None] * w[1][None, :, None] * w[0][None, None, :]
            yield flat.reshape(64, -1), wt.reshape(64, -1)

    def spread(self, x, G):
        if self.nodal:
            V = G
        else:
            Vn = (G / self.m)[:, self.conn]
            V = (torch.einsum("iae,aq->iqe", Vn, self.N) * self.wj0).reshape(3, -1)
        cells = self.n[0] * self.n[1] * self.n[2]
        out = []
        for c, (flat, w) in enumerate(self._stencils(x)):
            z = torch.zeros(cells, dtype=torch.float64, device="cuda")
            out.append(z.index_add(0, flat.reshape(-1), (w * V[c]).reshape(-1)))
        return torch.stack(out).reshape(3, self.n[2], self.n[1], self.n[0]) / self.h ** 3

    def interp(self, x, u):
        vals = [(u[c].reshape(-1)[flat] * w).sum(0)
                for c, (flat, w) in enumerate(self._stencils(x))]
        U = torch.stack(vals)
        if self.nodal:
            return U
        U = U.reshape(3, *self.wj0.shape) * self.wj0
        return self._assemble(torch.einsum("iqe,aq->iae", U, self.N)) / self.m


def _exact_fluid(u, f, h, dt):
    """The discrete projection step, diagonalised by the FFT."""
    n2, n1, n0 = u.shape[1:]
    k = [torch.exp(2j * math.pi * torch.arange(n, device="cuda", dtype=torch.float64) / n)
         for n in (n2, n1, n0)]
    sh = [k[0].reshape(-1, 1, 1), k[1].reshape(1, -1, 1), k[2].reshape(1, 1, -1)[..., :n0 // 2 + 1]]
    div = [(s - 1.0) / h for s in (sh[2], sh[1], sh[0])]          # forward differences
    lam = -sum(d.abs() ** 2 for d in div)
    a = RHO / dt
    us = [torch.fft.rfftn(a * u[c] + f[c]) / (a - MU * lam) for c in range(3)]
    lam0 = lam.clone()
    lam0[0, 0, 0] = 1.0
    p = sum(d * v for d, v in zip(div, us)) / dt / lam0
    p[0, 0, 0] = 0.0
    # (grad p)^c = (p(i) - p(i - e_c)) / h, the negative adjoint of div
    un = torch.stack([torch.fft.irfftn(v + dt * d.conj() * p, s=(n2, n1, n0))
                      for d, v in zip(div, us)])
    return un, torch.fft.irfftn(p, s=(n2, n1, n0))


def _exact_x(p):
    x = p.x if p.fp64 else I.from_split(p.cell, p.off, p.grid)
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def exact(case, seed):
    k = case["kind"]
    if k == "fluid":
        n = (case["n0"], case["n1"], case["n2"])
        u, p = _exact_fluid(_velocity(n, seed, torch.float32).double(),
                            _body_force(n, seed, torch.float32).double(), 1.0 / n[0], DT_FLUID)
        return dict(u=u, p=p)
    if k == "batch":
        probs = _batch_problems(case, seed)
        gp = torch.zeros(len(probs), ibfe.IB_MAX_MATERIALS, 10, dtype=torch.float64)
        out = dict(gparams=gp)
        for i, p in enumerate(probs):
            u = _velocity(p.grid.n, seed + i, torch.float32).double()
            r = _exact_vjp(p, "hex", "gauss", u, _cotangents(p, seed + i, torch.float32))
            gp[i, :1] = r["gparams"]
            if i < 10:
                out["i%d" % i] = [r[v] for v in ("G", "f", "U", "gu", "gx")]
        return out
    p = _structure(case, seed)
    u = _velocity(p.grid.n, seed, _dtype(case), k).double()
    if k == "grad":
        return _exact_grad(p, case, u)
    if k == "backward":
        r = _exact_vjp(p, case["elem"], case["quad"], u, _cotangents(p, seed, _dtype(case)))
        return dict(gx=r["gx"], gu=r["gu"], gparams=r["gparams"])
    ex = _Exact(p, case["elem"], case["quad"])
    x, theta = _exact_x(p), _theta(p.materials).cuda()
    G = ex.force(x, theta)
    if k == "transfer":
        # the nodal forces as given, in the path's own type
        G = G.to(_dtype(case)).double()
        return dict(f=ex.spread(x, G), U=ex.interp(x, u))
    f = ex.spread(x, G)
    if k == "forward":
        return dict(G=G, f=f, U=ex.interp(x, u))
    dt = CFL * p.grid.h
    un, pr = _exact_fluid(u, f, p.grid.h, dt)
    U = ex.interp(x, un)
    return dict(G=G, f=f, U=U, p=pr, u=un, x=x + dt * U)


def _exact_vjp(p, elem, quad, u, cot):
    ex = _Exact(p, elem, quad)
    x = _exact_x(p).requires_grad_()
    theta = _theta(p.materials).cuda().requires_grad_()
    u = u.requires_grad_()
    G = ex.force(x, theta, create_graph=True)
    f = ex.spread(x, G)
    U = ex.interp(x, u)
    loss = sum((cot[g].double() * v).sum() for g, v in (("gG", G), ("gf", f), ("gU", U)))
    gx, gp, gu = torch.autograd.grad(loss, [x, theta, u])
    return dict(G=G.detach(), f=f.detach(), U=U.detach(), gx=gx, gu=gu, gparams=gp)


def _exact_grad(p, case, u):
    ex = _Exact(p, case["elem"], case["quad"])
    x = _exact_x(p).requires_grad_()
    theta = _theta(p.materials).cuda().requires_grad_()
    u = u.requires_grad_()
    G = ex.force(x, theta, create_graph=True)
    f = ex.spread(x, G)
    U = ex.interp(x, u)
    loss = U.square().sum() + p.grid.h ** 1.5 * f.norm()
    gx, gp, gu = torch.autograd.grad(loss, [x, theta, u])
    return dict(loss=loss.detach(), G=G.detach(), f=f.detach(), U=U.detach(),
                goff=gx * p.grid.h, gparams=gp, gu=gu)
