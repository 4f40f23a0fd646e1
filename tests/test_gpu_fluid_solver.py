"""The fluid solver object: which of the two solvers serves it, its first step
on any stream."""
import numpy as np
import pytest

from oracle import fluid as OF
from paper_2503_22695_gb300 import inputs as I

from helpers import np_, rel_l2

pytestmark = pytest.mark.gpu

RHO, MU, DT = 1.0, 0.02, 2e-4


def _fields(n, seed):
    """As test_gpu_fluid's: solenoidal modes and white noise, a white force."""
    g = I.Grid(tuple(n), 1.0 / n[0])
    rng = np.random.Generator(np.random.PCG64(seed))
    u = I.fourier_velocity(g, 6, rng, dtype=np.float64)
    u = (u + 0.1 * rng.normal(size=u.shape)).astype(np.float32)
    f = (50.0 * rng.normal(size=u.shape)).astype(np.float32)
    return g, u, f


@pytest.mark.parametrize("n", [(16, 16, 16), (1024, 8, 8), (48, 40, 360)])
def test_first_step_on_another_stream(n):
    """A solver created and used at once on a stream that does not wait for the
    default one has its tables: the bits of a solver used later."""
    import torch
    from paper_2503_22695_gb300 import ibfe
    g, u, f = _fields(n, 1)
    ud, fd = torch.from_numpy(u).cuda(), torch.from_numpy(f).cuda()
    ref = ibfe.Fluid(g.n, g.h, RHO, MU, DT)
    torch.cuda.synchronize()
    a, pa, _ = ibfe.ib_fluid_step(ref, ud, fd)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    for _ in range(20):
        with torch.cuda.stream(side):
            fl = ibfe.Fluid(g.n, g.h, RHO, MU, DT)
            b, pb, _ = ibfe.ib_fluid_step(fl, ud, fd)
        side.synchronize()
        assert torch.equal(a, b) and torch.equal(pa, pb)


def test_solver_of_a_lattice():
    from paper_2503_22695_gb300 import ibfe
    for n, fp64, direct in [((32, 32, 32), False, True), ((90, 36, 20), False, True),
                            ((4, 4, 900), False, True), ((56, 8, 8), False, False),
                            ((8, 22, 8), False, False), ((4, 4, 1024), False, False),
                            ((32, 32, 32), True, False)]:
        fl = ibfe.Fluid(n, 1.0 / n[0], RHO, MU, DT,
                        precision=ibfe.IB_FP64 if fp64 else ibfe.IB_FP32_SPLIT)
        which = {True: ibfe.IB_SOLVER_DIRECT, False: ibfe.IB_SOLVER_CYCLES}
        assert fl.solver() == which[direct], n
        default = fl.cycles()
        fl.set_cycles(default[0], default[1] + 1)
        assert fl.solver() == ibfe.IB_SOLVER_CYCLES
        fl.set_cycles(*default)
        assert fl.solver() == which[direct], n


def test_only_a_refused_workspace_leaves_the_cycles(monkeypatch):
    """No room for the direct solve's modes: the V-cycles serve the solver, at the
    tolerances that test_gpu_fluid states for them.  Any other error is the call's."""
    import torch
    from paper_2503_22695_gb300 import ibfe
    g, u, f = _fields((64, 32, 32), 2)
    monkeypatch.setenv("IBFE_FAULT", "modes:%d" % ibfe.IB_ERR_CAPACITY)
    fl = ibfe.Fluid(g.n, g.h, RHO, MU, DT)
    monkeypatch.setenv("IBFE_FAULT", "modes")
    with pytest.raises(ibfe.IBError) as e:
        ibfe.Fluid(g.n, g.h, RHO, MU, DT)
    assert e.value.code == ibfe.IB_ERR_CUDA
    monkeypatch.delenv("IBFE_FAULT")
    assert fl.solver() == ibfe.IB_SOLVER_CYCLES
    un, p, _ = ibfe.ib_fluid_step(fl, torch.from_numpy(u).cuda(), torch.from_numpy(f).cuda())
    _, po, uo = OF.fluid_step(u.astype(np.float64), f.astype(np.float64), RHO, MU, DT, g.h)
    assert rel_l2(np_(un), uo) <= 1e-5
    assert rel_l2(np_(p), po) <= 2e-5


@pytest.mark.parametrize("n", [(32, 32, 32), (64, 64, 64), (32, 16, 48), (96, 96, 96)])
def test_cycles_at_the_default_counts(n):
    """V-cycles asked for on lattices that have the direct solve, at the
    tolerances that test_gpu_fluid states for them."""
    import torch
    from paper_2503_22695_gb300 import ibfe
    g, u, f = _fields(n, 100 + n[0] + n[2])
    ud, fd = torch.from_numpy(u).cuda(), torch.from_numpy(f).cuda()
    fl = ibfe.Fluid(g.n, g.h, RHO, MU, DT)
    d, pd, _ = ibfe.ib_fluid_step(fl, ud, fd)
    fl.set_solver(ibfe.IB_SOLVER_CYCLES)
    assert fl.solver() == ibfe.IB_SOLVER_CYCLES and fl.cycles() == [2, 6]
    un, p, res = ibfe.ib_fluid_step(fl, ud, fd, residuals=True)
    _, po, uo = OF.fluid_step(u.astype(np.float64), f.astype(np.float64), RHO, MU, DT, g.h)
    assert rel_l2(np_(un), uo) <= 1e-5 and rel_l2(np_(p), po) <= 2e-5
    assert max(res) <= 1e-5
    assert not torch.equal(p, pd)
    fl.set_solver(ibfe.IB_SOLVER_DIRECT)
    e, pe, _ = ibfe.ib_fluid_step(fl, ud, fd)
    assert fl.solver() == ibfe.IB_SOLVER_DIRECT and torch.equal(e, d) and torch.equal(pe, pd)


def test_solver_choice_is_checked():
    from paper_2503_22695_gb300 import ibfe
    for n, prec in (((56, 8, 8), ibfe.IB_FP32_SPLIT), ((16, 16, 16), ibfe.IB_FP64)):
        fl = ibfe.Fluid(n, 1.0 / n[0], RHO, MU, DT, precision=prec)
        fl.set_solver(ibfe.IB_SOLVER_CYCLES)
        with pytest.raises(ibfe.IBError) as e:
            fl.set_solver(ibfe.IB_SOLVER_DIRECT)
        assert e.value.code == ibfe.IB_ERR_UNSUPPORTED
        with pytest.raises(ibfe.IBError) as e:
            fl.set_solver(2)
        assert e.value.code == ibfe.IB_ERR_INVALID_ARG


@pytest.mark.parametrize("n", [(56, 8, 8), (8, 22, 8), (56, 56, 56), (28, 56, 56), (104, 104, 104)])
def test_fp32_cycles_match_the_same_cycles_in_fp64(n):
    """Lattices that only the V-cycles take, at the default counts: the iterate
    that FP64 gives at the same counts, to the FP32 rounding floor of
    test_gpu_fluid's tolerances (the cycles contract errors of the iterate)."""
    import torch
    from paper_2503_22695_gb300 import ibfe
    g, u, f = _fields(n, sum(n))
    ud, fd = torch.from_numpy(u).cuda(), torch.from_numpy(f).cuda()
    fl = ibfe.Fluid(g.n, g.h, RHO, MU, DT)
    assert fl.solver() == ibfe.IB_SOLVER_CYCLES and fl.cycles() == [2, 6]
    un, p, _ = ibfe.ib_fluid_step(fl, ud, fd)
    fl64 = ibfe.Fluid(g.n, g.h, RHO, MU, DT, precision=ibfe.IB_FP64)
    fl64.set_cycles(2, 6)
    u64, p64, _ = ibfe.ib_fluid_step(fl64, ud.double(), fd.double())
    assert rel_l2(np_(un), np_(u64)) <= 1e-5
    assert rel_l2(np_(p), np_(p64)) <= 2e-5


@pytest.mark.parametrize("n", [(56, 56, 56), (64, 32, 32)])
def test_cycles_replayed_and_launched_directly(n):
    """A step's V-cycles as a graph replay, recaptured for other arrays, in place
    and as direct launches (with residuals): the same bits."""
    import torch
    from paper_2503_22695_gb300 import ibfe
    g, u, f = _fields(n, 5)
    ud, fd = torch.from_numpy(u).cuda(), torch.from_numpy(f).cuda()
    fl = ibfe.Fluid(g.n, g.h, RHO, MU, DT)
    fl.set_solver(ibfe.IB_SOLVER_CYCLES)
    a, pa = torch.empty_like(ud), torch.empty_like(ud[0])
    ibfe.ib_fluid_step(fl, ud, fd, a, pa)
    ref, pref = a.clone(), pa.clone()
    a.fill_(float("nan"))
    pa.fill_(float("nan"))
    ibfe.ib_fluid_step(fl, ud, fd, a, pa)                    # the graph again
    assert torch.equal(a, ref) and torch.equal(pa, pref)
    b, pb, _ = ibfe.ib_fluid_step(fl, ud.clone(), fd.clone())  # other arrays
    assert torch.equal(b, ref) and torch.equal(pb, pref)
    uin = ud.clone()
    c, pc, _ = ibfe.ib_fluid_step(fl, uin, fd, u_next=uin)
    assert torch.equal(c, ref) and torch.equal(pc, pref)
    d, pd, res = ibfe.ib_fluid_step(fl, ud, fd, residuals=True)
    assert torch.equal(d, ref) and torch.equal(pd, pref) and np.isfinite(res).all()


@pytest.mark.parametrize("n", [(8, 6, 12), (48, 24, 40), (30, 128, 16), (64, 64, 64)])
def test_direct_solve_without_viscosity(n):
    """mu = 0: the stencils' own branch, within the direct solve's bounds."""
    import torch
    from paper_2503_22695_gb300 import ibfe
    import test_gpu_spectral as S
    g, u, f = S._fields(n, sum(n))
    fl = ibfe.Fluid(g.n, g.h, S.RHO, 0.0, S.DT)
    assert fl.solver() == ibfe.IB_SOLVER_DIRECT
    ud, fd = torch.from_numpy(u).cuda(), torch.from_numpy(f).cuda()
    us, po, uo = OF.fluid_step(u, f, S.RHO, 0.0, S.DT, g.h)
    tu, tp = S._bounds(u, us, uo, g.h)
    un, p, _ = ibfe.ib_fluid_step(fl, ud, fd)
    assert S._rms(np_(un) - uo) <= tu
    assert S._rms(np_(p) - po) <= tp


@pytest.mark.parametrize("n", [(16, 18, 20), (64, 32, 32)])
def test_residuals_when_the_step_overwrites_an_input(n):
    """u_next in u's array, in f's and in its own: the same fields and residuals,
    by either solver."""
    import torch
    from paper_2503_22695_gb300 import ibfe
    g, u, f = _fields(n, 7)
    ud, fd = torch.from_numpy(u).cuda(), torch.from_numpy(f).cuda()
    fl = ibfe.Fluid(g.n, g.h, RHO, MU, DT)
    for solver in (ibfe.IB_SOLVER_DIRECT, ibfe.IB_SOLVER_CYCLES):
        fl.set_solver(solver)
        ref, pref, res = ibfe.ib_fluid_step(fl, ud, fd, residuals=True)
        assert res[0] <= 1e-5 and res[1] <= 1e-5
        for name in ("u", "f", "both"):
            a, b = ud.clone(), fd.clone()
            if name == "both":
                b = a
                ref, pref, res = ibfe.ib_fluid_step(fl, ud, ud, residuals=True)
            un, p, r = ibfe.ib_fluid_step(fl, a, b, u_next=a if name == "u" else b, residuals=True)
            assert torch.equal(un, ref) and torch.equal(p, pref), (solver, name)
            assert list(r) == list(res), (solver, name)
