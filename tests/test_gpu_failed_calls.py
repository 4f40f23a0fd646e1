"""Calls that fail half-way (host-side injection, nothing faults) leave the
plan usable: the calls after them give the bits of an undisturbed plan."""
import numpy as np
import pytest

from paper_2503_22695_gb300 import inputs as I

from helpers import Case

pytestmark = pytest.mark.gpu


def _case(fp64, quad=0):
    c = Case(I.block_problem(fp64=fp64), quad=quad)
    rng = np.random.default_rng(3)
    c.G = c.to_dev(rng.normal(size=(3, c.prob.n_nodes)))
    c.gU = c.to_dev(rng.normal(size=(3, c.prob.n_nodes)))
    return c


def _equal(a, b):
    import torch
    return all(torch.equal(s, t) for s, t in zip(a, b))


@pytest.mark.parametrize("quad", [0, 1])
@pytest.mark.parametrize("fp64", [False, True])
def test_points_counted_by_a_failed_call_are_forgotten(fp64, quad, monkeypatch):
    """A call that stops between counting the points of each tile and binning
    them: its counts would double the next binning's, which would write past
    the plan's arrays."""
    c = _case(fp64, quad)
    ibfe = c.ibfe

    def ops():
        return (ibfe.ib_spread(c.plan, c.pos, c.G), ibfe.ib_interp(c.plan, c.pos, c.u),
                *ibfe.ib_interp_adj(c.plan, c.pos, c.u, c.gU))

    ref = ops()
    for op in (lambda: ibfe.ib_spread(c.plan, c.pos, c.G),
               lambda: ibfe.ib_interp(c.plan, c.pos, c.u),
               lambda: ibfe.ib_interp_adj(c.plan, c.pos, c.u, c.gU)):
        monkeypatch.setenv("IBFE_FAULT", "points")
        for _ in range(2):
            with pytest.raises(ibfe.IBError) as e:
                op()
            assert e.value.code == ibfe.IB_ERR_CUDA
        monkeypatch.delenv("IBFE_FAULT")
        assert _equal(ops(), ref)
    assert ibfe.ib_plan_sync_status(c.plan) == ibfe.IB_OK


@pytest.mark.parametrize("stage", ["points", "gather"])
@pytest.mark.parametrize("fp64", [False, True])
def test_failed_calls_rejoin_the_plans_streams(fp64, stage, monkeypatch):
    """The fused operators fork to streams of the plan.  One that fails there
    lets the caller's stream wait for them: the next call on that stream finds
    the workspaces and counters unused, and a capture of the stream can end."""
    import torch
    c = _case(fp64)
    ibfe = c.ibfe
    gf = c.to_dev(np.random.default_rng(4).normal(size=c.prob.u.shape) * 1e-3)
    G, f, U = ibfe.ib_forward(c.plan, c.mats, c.pos, c.u)
    out = [torch.empty_like(t) for t in (G, f, U, G, f)]

    def forward():
        return ibfe.ib_forward(c.plan, c.mats, c.pos, c.u, *out[:3])

    def backward():
        return ibfe.ib_backward(c.plan, c.mats, c.pos, c.u, G, c.gU, gf, c.gU, *out[3:])

    def direct():
        return (ibfe.ib_fe_force(c.plan, c.mats, c.pos), ibfe.ib_spread(c.plan, c.pos, c.G),
                *ibfe.ib_fe_force_adj(c.plan, c.mats, c.pos, c.gU))

    refs = [[t.clone() for t in op()] for op in (direct, forward, backward)]
    side = torch.cuda.Stream()
    for op in (forward, backward):
        monkeypatch.setenv("IBFE_FAULT", stage)
        with pytest.raises(ibfe.IBError):
            op()
        monkeypatch.delenv("IBFE_FAULT")
        assert _equal(direct(), refs[0])
        # captured: the graph holds what was queued before the failure
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            monkeypatch.setenv("IBFE_FAULT", stage)
            with pytest.raises(ibfe.IBError):
                op()
            monkeypatch.delenv("IBFE_FAULT")
        graph.replay()
        for fn, ref in zip((direct, forward, backward), refs):
            assert _equal(fn(), ref)
    assert ibfe.ib_plan_sync_status(c.plan) == ibfe.IB_OK


@pytest.mark.parametrize("fp64", [False, True])
def test_an_earlier_error_is_not_the_next_calls(fp64, monkeypatch):
    """An error that another call left with the runtime (a refused allocation)
    neither fails a call nor ends it half-way."""
    import torch
    c = _case(fp64)
    ibfe = c.ibfe
    gf = c.to_dev(np.random.default_rng(4).normal(size=c.prob.u.shape) * 1e-3)
    prec = ibfe.IB_FP64 if fp64 else ibfe.IB_FP32_SPLIT
    g = c.prob.grid

    def ops():
        out = [ibfe.ib_fe_force(c.plan, c.mats, c.pos), ibfe.ib_spread(c.plan, c.pos, c.G),
               ibfe.ib_interp(c.plan, c.pos, c.u)]
        out += ibfe.ib_forward(c.plan, c.mats, c.pos, c.u)
        out += ibfe.ib_backward(c.plan, c.mats, c.pos, c.u, out[3], c.gU, gf, c.gU)
        out += ibfe.ib_spread_adj(c.plan, c.pos, c.G, gf)
        out += ibfe.ib_interp_adj(c.plan, c.pos, c.u, c.gU)
        out += ibfe.ib_fe_force_adj(c.plan, c.mats, c.pos, c.gU)
        fl = ibfe.Fluid(g.n, g.h, 1.0, 0.02, 2e-4, precision=prec)
        out += ibfe.ib_fluid_step(fl, c.u, out[4])[:2]
        if fp64:
            pos = ibfe.Pos(x64=c.pos.x64.clone())
        else:
            pos = ibfe.Pos(cell=c.pos.cell.clone(), off=c.pos.off.clone())
        out += ibfe.ib_step(c.plan, fl, c.mats, pos, c.u.clone())
        if not fp64:
            inst = []
            for _ in range(2):
                d = dict(conn=c.conn, X=c.X, fibres=c.fib, mat_id=c.mat_id, n=g.n, h=g.h,
                         mats=c.mats, cell=c.cell, off=c.off, u=c.u, gU=c.gU, gf=gf)
                d.update({k: torch.empty_like(c.G) for k in ("G", "U", "gx")})
                d.update({k: torch.empty_like(c.u) for k in ("f", "gu")})
                inst.append(d)
            b = ibfe.Batch(inst)
            b.forward()
            b.adjoint()
            out += [d[k] for d in inst for k in ("G", "U", "gx", "f", "gu")] + [b.gparams()]
            e = torch.empty(1, device="cuda", dtype=torch.float64)
            out += [ibfe.ib_fe_energy_noalloc(c.conn, c.X, c.mats, c.pos, g.h, e, fibres=c.fib,
                                              mat_id=c.mat_id)]
        return out

    ref = ops()
    monkeypatch.setenv("IBFE_FAULT", "earlier_error")
    again = ops()
    monkeypatch.delenv("IBFE_FAULT")
    assert _equal(again, ref)
    assert ibfe.ib_plan_sync_status(c.plan) == ibfe.IB_OK


@pytest.mark.parametrize("fp64", [False, True])
def test_objects_released_during_a_capture(fp64):
    """Plans, fluid solvers and sweeps that are collected while an unrelated
    stream is captured do not invalidate the capture."""
    import torch
    c = _case(fp64)
    ibfe = c.ibfe
    g = c.prob.grid
    ref = ibfe.ib_spread(c.plan, c.pos, c.G)
    f = torch.empty_like(ref)
    other = [_case(fp64)]
    ibfe.ib_spread(other[0].plan, other[0].pos, other[0].G)
    fl = ibfe.Fluid(g.n, g.h, 1.0, 0.02, 2e-4,
                    precision=ibfe.IB_FP64 if fp64 else ibfe.IB_FP32_SPLIT)
    un = ibfe.ib_fluid_step(fl, c.u)[0]
    other.append(fl)
    if not fp64:
        inst = [dict(conn=c.conn, X=c.X, fibres=c.fib, mat_id=c.mat_id, n=g.n, h=g.h, mats=c.mats,
                     cell=c.cell, off=c.off, u=c.u, G=torch.empty_like(c.G),
                     U=torch.empty_like(c.G), f=torch.empty_like(c.u)) for _ in range(2)]
        other.append(ibfe.Batch(inst))
        other[-1].forward()
    del fl
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ibfe.ib_spread(c.plan, c.pos, c.G, f)
        while other:
            other.pop()
        ibfe.ib_interp(c.plan, c.pos, c.u)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(f, ref) and bool(torch.isfinite(un).all())
