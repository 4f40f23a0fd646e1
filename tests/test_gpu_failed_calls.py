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
