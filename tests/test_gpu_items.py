"""Spreading and interpolation at the edges of the work items: all coupling
points in one tile (or in two), their number around the item sizes a small
plan uses (128 points, at most eight small items per tile, 1024 points), FP32
and FP64.  Nodal rule, one element and loose nodes, against the sums written
out in FP64.  Tolerances as the parity tests' (relative L2 1e-5 of the spread
force, 1e-6 of the interpolated velocity; FP64 1e-12)."""
import numpy as np
import pytest

from paper_2503_22695_gb300 import inputs as I

from helpers import np_, rel_l2

pytestmark = pytest.mark.gpu


def _phi(th):
    q = np.sqrt(1 + 4 * th * (1 - th))
    return np.stack([3 - 2 * th - q, 3 - 2 * th + q, 1 + 2 * th + q, 1 + 2 * th - q]) / 8


def _stencil(x, c, n):
    idx, w = [], []
    for d in range(3):
        t = x[d] - (0.0 if d == c else 0.5)
        i = np.floor(t)
        w.append(_phi(t - i))
        idx.append((i.astype(np.int64)[None] + np.arange(-1, 3)[:, None]) % n)
    flat = (idx[2][:, None, None] * n + idx[1][None, :, None]) * n + idx[0][None, None, :]
    wt = w[2][:, None, None] * w[1][None, :, None] * w[0][None, None, :]
    return flat.reshape(64, -1), wt.reshape(64, -1)


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("tiles", [1, 2])
@pytest.mark.parametrize("N", [8, 31, 33, 127, 128, 129, 257, 1023, 1024, 1025, 1152, 2049, 8193,
                               9000])
def test_item_edges(N, tiles, fp64):
    import torch
    from paper_2503_22695_gb300 import ibfe
    n, h = 32, 1.0 / 32
    rng = np.random.default_rng(N)
    dt = np.float64 if fp64 else np.float32
    # cube corners (the element) and loose nodes, in cell units
    t = np.concatenate([I.HEX_CORNERS.T * 0.25 + 12.0,
                        8.0 + 8.0 * rng.uniform(0.001, 0.999, size=(3, N - 8))], axis=1)
    if tiles == 2:
        t[0, 8::2] += 16.0          # the other tile, across the periodic seam's neighbour
    g = I.Grid((n, n, n), h)
    cell, off = I.to_split(t * h, g)
    x = t * h if fp64 else I.from_split(cell, off, g)
    conn = torch.arange(8, dtype=torch.int32, device="cuda").reshape(8, 1)
    X = torch.from_numpy((t * h).astype(dt)).cuda()
    plan = ibfe.Plan(conn, X, g.n, h, quad=ibfe.IB_QUAD_NODAL,
                     precision=ibfe.IB_FP64 if fp64 else ibfe.IB_FP32_SPLIT)
    pos = (ibfe.Pos(x64=torch.from_numpy(x).cuda()) if fp64 else
           ibfe.Pos(cell=torch.from_numpy(cell).cuda(), off=torch.from_numpy(off).cuda()))
    G = rng.normal(size=(3, N)).astype(dt)
    u = rng.normal(size=(3, n, n, n)).astype(dt)
    f = ibfe.ib_spread(plan, pos, torch.from_numpy(G).cuda())
    U = ibfe.ib_interp(plan, pos, torch.from_numpy(u).cuda())
    assert ibfe.ib_plan_sync_status(plan) == ibfe.IB_OK
    fo, Uo = np.zeros((3, n ** 3)), np.zeros((3, N))
    for c in range(3):
        flat, w = _stencil(x / h, c, n)
        np.add.at(fo[c], flat.ravel(), (w * G[c].astype(np.float64)).ravel() / h ** 3)
        Uo[c] = (u[c].astype(np.float64).ravel()[flat] * w).sum(0)
    tf, tU = (1e-12, 1e-12) if fp64 else (1e-5, 1e-6)
    assert rel_l2(np_(f).reshape(3, -1), fo) <= tf
    assert rel_l2(np_(U), Uo) <= tU


@pytest.mark.parametrize("fp64", [False, True])
def test_full_items(fp64):
    """Enough points for full items on every SM: the kernels of large plans."""
    import torch
    from paper_2503_22695_gb300 import ibfe
    n, h, N = 32, 1.0 / 32, 650_000
    rng = np.random.default_rng(7)
    dt = np.float64 if fp64 else np.float32
    t = np.concatenate([I.HEX_CORNERS.T * 0.25 + 12.0,
                        n * rng.uniform(0.001, 0.999, size=(3, N - 8))], axis=1)
    g = I.Grid((n, n, n), h)
    cell, off = I.to_split(t * h, g)
    x = t * h if fp64 else I.from_split(cell, off, g)
    conn = torch.arange(8, dtype=torch.int32, device="cuda").reshape(8, 1)
    plan = ibfe.Plan(conn, torch.from_numpy((t * h).astype(dt)).cuda(), g.n, h,
                     quad=ibfe.IB_QUAD_NODAL,
                     precision=ibfe.IB_FP64 if fp64 else ibfe.IB_FP32_SPLIT)
    pos = (ibfe.Pos(x64=torch.from_numpy(x).cuda()) if fp64 else
           ibfe.Pos(cell=torch.from_numpy(cell).cuda(), off=torch.from_numpy(off).cuda()))
    G = rng.normal(size=(3, N)).astype(dt)
    u = rng.normal(size=(3, n, n, n)).astype(dt)
    f = ibfe.ib_spread(plan, pos, torch.from_numpy(G).cuda())
    U = ibfe.ib_interp(plan, pos, torch.from_numpy(u).cuda())
    fo, Uo = np.zeros((3, n ** 3)), np.zeros((3, N))
    for c in range(3):
        flat, w = _stencil(x / h, c, n)
        fo[c] = np.bincount(flat.ravel(), (w * G[c].astype(np.float64)).ravel(), n ** 3) / h ** 3
        Uo[c] = (u[c].astype(np.float64).ravel()[flat] * w).sum(0)
    tf, tU = (1e-12, 1e-12) if fp64 else (1e-5, 1e-6)
    assert rel_l2(np_(f).reshape(3, -1), fo) <= tf
    assert rel_l2(np_(U), Uo) <= tU


@pytest.mark.parametrize("N", [513, 16385, 65536, 65537])
def test_fp64_point_order(N):
    """FP64 points in every one of 512 tiles, up to and beyond the number that
    is ordered tile by tile; twice, the same bits."""
    import torch
    from paper_2503_22695_gb300 import ibfe
    n, h = 64, 1.0 / 64
    rng = np.random.default_rng(N)
    t = np.concatenate([I.HEX_CORNERS.T * 0.25 + 12.0,
                        n * rng.uniform(0.001, 0.999, size=(3, N - 8))], axis=1)
    g = I.Grid((n, n, n), h)
    conn = torch.arange(8, dtype=torch.int32, device="cuda").reshape(8, 1)
    plan = ibfe.Plan(conn, torch.from_numpy(t * h).cuda(), g.n, h, quad=ibfe.IB_QUAD_NODAL,
                     precision=ibfe.IB_FP64)
    pos = ibfe.Pos(x64=torch.from_numpy(t * h).cuda())
    G, u = rng.normal(size=(3, N)), rng.normal(size=(3, n, n, n))
    f = ibfe.ib_spread(plan, pos, torch.from_numpy(G).cuda())
    assert torch.equal(f, ibfe.ib_spread(plan, pos, torch.from_numpy(G).cuda()))
    U = ibfe.ib_interp(plan, pos, torch.from_numpy(u).cuda())
    fo, Uo = np.zeros((3, n ** 3)), np.zeros((3, N))
    for c in range(3):
        flat, w = _stencil(t, c, n)
        fo[c] = np.bincount(flat.ravel(), (w * G[c]).ravel(), n ** 3) / h ** 3
        Uo[c] = (u[c].ravel()[flat] * w).sum(0)
    assert rel_l2(np_(f).reshape(3, -1), fo) <= 1e-12
    assert rel_l2(np_(U), Uo) <= 1e-12
