"""The direct (Fourier) solve of the FP32 fluid step at the lattices where its
transforms can go wrong: the smallest lengths, every radix and number of
passes, plane row counts that leave a CTA's last row pairs empty, lengths whose
modes fill no whole tile, velocities off 8-byte alignment; and the lattices it
does not take (a prime factor above 5), which keep the V-cycles.

Tolerances: the transformed fields carry white rounding noise of relative
size e = 2^-24 log2(cells) (stencils and transforms), and the algebra per mode
(spectral.cu) takes it to the results: q = (d + D delta) / S amplifies the
noise of d = h div u^n by 1/S and that of the increment delta = u* - u^n by
|D|/S = S^-1/2, w = delta - conj(D) q by S^-1/2 and 1.  With A_k the root mean
square of S^-k over the nonzero modes, the errors' root mean squares are
bounded by
  p:  (h / dt) e (A_1 |d| + 3 A_1/2 |delta|),
  u:  2^-24 |u| + e (A_1/2 |d| + 4 |delta|),
all norms root mean squares of the exact fields."""
import numpy as np
import pytest

from oracle import fluid as OF
from paper_2503_22695_gb300 import inputs as I

from helpers import np_, rel_l2

pytestmark = pytest.mark.gpu

RHO, MU, DT = 1.0, 0.02, 2e-4


def _rms(a):
    return float(np.sqrt(np.mean(np.square(np.asarray(a, dtype=np.float64)))))


def _bounds(u, ustar, uo, h):
    """(tolerance of u, tolerance of p), root mean squares."""
    S = -OF.symbol(u.shape[1:], 1.0).ravel()[1:]
    amp = lambda k: _rms(S ** -k)
    e = 2.0 ** -24 * np.log2(S.size + 1)
    d = _rms(h * OF.divergence(u.astype(np.float64), h))
    dl = _rms(ustar - u)
    return (2.0 ** -24 * _rms(uo) + e * (amp(0.5) * d + 4 * dl),
            h / DT * e * (amp(1.0) * d + 3 * amp(0.5) * dl))


def _fields(n, seed):
    g = I.Grid(tuple(n), 1.0 / n[0])
    rng = np.random.Generator(np.random.PCG64(seed))
    u = I.fourier_velocity(g, 4, rng, kmax=1, dtype=np.float64)
    u = (u + 0.1 * rng.normal(size=u.shape)).astype(np.float32)
    f = (50.0 * rng.normal(size=u.shape)).astype(np.float32)
    return g, u, f


@pytest.mark.parametrize("n", [(4, 4, 4), (6, 10, 4), (8, 6, 12), (16, 18, 20), (10, 30, 50),
                               (48, 24, 40), (80, 60, 36), (128, 64, 32), (64, 8, 90),
                               (256, 16, 8), (30, 128, 16), (12, 20, 256), (320, 4, 6),
                               (4, 512, 6), (6, 4, 640), (1024, 4, 4), (4, 1024, 4)])
def test_direct_solve_matches_oracle(n):
    import torch
    from paper_2503_22695_gb300 import ibfe
    g, u, f = _fields(n, sum(n))
    fl = ibfe.Fluid(g.n, g.h, RHO, MU, DT)
    ud, fd = torch.from_numpy(u).cuda(), torch.from_numpy(f).cuda()
    un, p, res = ibfe.ib_fluid_step(fl, ud, fd, residuals=True)
    us, po, uo = OF.fluid_step(u, f, RHO, MU, DT, g.h)
    tu, tp = _bounds(u, us, uo, g.h)
    assert _rms(np_(un) - uo) <= tu
    assert _rms(np_(p) - po) <= tp
    assert np.isfinite(res).all()
    # the same bits without residuals, in place, and from arrays that are only
    # 4-byte aligned
    pad = torch.zeros(u.size + 1, device="cuda")
    um = pad[1:].view(u.shape)
    um.copy_(ud)
    for uin in (ud.clone(), um):
        b, pb, _ = ibfe.ib_fluid_step(fl, uin, fd, u_next=uin)
        assert torch.equal(b, un) and torch.equal(pb, p)


@pytest.mark.parametrize("L", [32, 40, 48, 64, 80, 96, 128, 160, 192, 256, 320, 384, 512])
def test_compile_time_lengths_match_oracle(L):
    """Each length with transforms of its own, along each dimension."""
    import torch
    from paper_2503_22695_gb300 import ibfe
    for n in ((L, 4, 6), (6, L, 4), (4, 6, L)):
        g, u, f = _fields(n, sum(n))
        fl = ibfe.Fluid(g.n, g.h, RHO, MU, DT)
        un, p, _ = ibfe.ib_fluid_step(fl, torch.from_numpy(u).cuda(), torch.from_numpy(f).cuda())
        us, po, uo = OF.fluid_step(u, f, RHO, MU, DT, g.h)
        tu, tp = _bounds(u, us, uo, g.h)
        assert _rms(np_(un) - uo) <= tu, n
        assert _rms(np_(p) - po) <= tp, n


def test_modes_larger_than_l2_match_oracle():
    """172 MB of modes: the y transforms ask for later planes ahead."""
    import torch
    from paper_2503_22695_gb300 import ibfe
    n = (320, 256, 128)
    g, u, f = _fields(n, 11)
    fl = ibfe.Fluid(g.n, g.h, RHO, MU, DT)
    un, p, _ = ibfe.ib_fluid_step(fl, torch.from_numpy(u).cuda(), torch.from_numpy(f).cuda())
    us, po, uo = OF.fluid_step(u, f, RHO, MU, DT, g.h)
    tu, tp = _bounds(u, us, uo, g.h)
    assert _rms(np_(un) - uo) <= tu
    assert _rms(np_(p) - po) <= tp


@pytest.mark.parametrize("n", [(56, 8, 8), (8, 22, 8), (8, 8, 28), (4, 4, 1024)])
def test_other_lattices_keep_the_cycles(n):
    import torch
    from paper_2503_22695_gb300 import ibfe
    g, u, f = _fields(n, sum(n))
    a = ibfe.Fluid(g.n, g.h, RHO, MU, DT)
    ud, fd = torch.from_numpy(u).cuda(), torch.from_numpy(f).cuda()
    _, p2, r2 = ibfe.ib_fluid_step(a, ud, fd, residuals=True)
    a.set_cycles(2, 5)   # one Poisson cycle fewer: the iterate before the last
    _, p1, r1 = ibfe.ib_fluid_step(a, ud, fd, residuals=True)
    assert not torch.equal(p1, p2) and r2[1] <= r1[1]


def test_chosen_cycle_counts_run_v_cycles():
    import torch
    from paper_2503_22695_gb300 import ibfe
    g, u, f = _fields((32, 32, 32), 3)
    fl = ibfe.Fluid(g.n, g.h, RHO, MU, DT)
    ud, fd = torch.from_numpy(u).cuda(), torch.from_numpy(f).cuda()
    d, pd, rd = ibfe.ib_fluid_step(fl, ud, fd, residuals=True)
    fl.set_cycles(1, 1)
    _, p1, r1 = ibfe.ib_fluid_step(fl, ud, fd, residuals=True)
    assert r1[1] > 100 * rd[1]             # one cycle leaves a residual
    fl.set_cycles(3, 12)
    c, pc, _ = ibfe.ib_fluid_step(fl, ud, fd)
    assert rel_l2(np_(c), np_(d)) <= 1e-6 and rel_l2(np_(pc), np_(pd)) <= 2e-5
    fl.set_cycles(2, 6)                    # the defaults again
    e, pe, _ = ibfe.ib_fluid_step(fl, ud, fd)
    assert torch.equal(e, d) and torch.equal(pe, pd)
