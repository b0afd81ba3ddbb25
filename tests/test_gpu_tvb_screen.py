"""The 2D TVB indicator's FP32 screen on the GPU against the oracle's FP64 decision, on data made of
ties: edge values equal to a mean difference or to M h^2 up to a part in 2^10 .. 2^52, in either
direction, over the mean's whole range of size against the differences.  The flags are the
oracle's on every cell, and every cell that it reports near a threshold is reported."""
import numpy as np
import pytest

import oracle
import paper_1904_11147_gb300 as dgl

pytestmark = pytest.mark.gpu


def _data(pde, N, nx, ny, bc, hx, hy, M, scale, seed):
    rng = np.random.default_rng(seed)
    nv, NP = (4 if pde else 1), (N + 1) * (N + 2) // 2
    n = nx * ny
    u = np.zeros((n, nv, NP))
    step = 10.0 ** rng.uniform(-15, -0.5, (n, nv)) * rng.choice([-1, 1], (n, nv))
    u[:, :, 0] = scale * (1.0 + np.cumsum(step, axis=0) * 0.02)
    mean = 0.5 * u[:, :, 0].reshape(ny, nx, nv)
    pad = np.pad(mean, ((1, 1), (1, 1), (0, 0)), mode="wrap" if bc == 0 else "edge")
    diff = [pad[1:-1, 2:] - mean, mean - pad[1:-1, :-2], pad[2:, 1:-1] - mean, mean - pad[:-2, 1:-1]]
    t = np.sqrt(0.75)  # psi_1(1) psi_0
    kind = rng.integers(0, 8, (n, nv))
    delta = rng.choice([-1, 0, 1], (n, nv)) * 2.0 ** -rng.uniform(10, 52, (n, nv))
    for k in range(4):  # mode (1, 0) or (0, 1) from a mean difference
        w = kind == k
        u[:, :, 1 if k < 2 else 2][w] = ((diff[k].reshape(n, nv) / t) * (1 + delta))[w]
    for k, h in ((4, hx), (5, hy)):  # from M h^2
        w = kind == k
        s = rng.choice([-1, 1], (n, nv))
        u[:, :, 1 if k == 4 else 2][w] = (M * h * h / t * (1 + delta) * s)[w]
    w = kind == 6  # all modes, of the differences' size
    u[:, :, 1:][w] = (step[:, :, None] * scale * 0.02 * rng.uniform(-1, 1, (n, nv, NP - 1)))[w]
    return u


@pytest.mark.parametrize("pde,N", [(0, 1), (0, 2), (0, 3), (1, 2), (1, 3)])
@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("scale,m", [(1.0, 0.0), (1.0, 1e-12), (1.0, 1e-4), (1e-12, 1e-6), (1e12, 1e-8), (-3.0, 1e-2)])
def test_ties(pde, N, bc, scale, m):
    nx, ny, box = 97, 131, (0.0, 1.7, 0.0, 0.8)
    hx, hy = 1.7 / nx, 0.8 / ny
    M = m * abs(scale) / (hx * hy)  # M h^2 = some m |scale|
    u = _data(pde, N, nx, ny, bc, hx, hy, M, scale, 17 * N + pde)
    g = dgl.Mesh(2, pde, N, [nx], [ny], [box], bc=bc)
    o = oracle.Mesh(2, pde, N, nx, ny, box=box, bc=bc)
    g.set_modes(u)
    fl, nf, nn, near = g.flag_cells(dgl.IND_TVB, M, near_cells=True)
    fo, nfo, nno, near_o = o.flag_tvb(u, M, near_cells=True)
    assert 0 < nf < nx * ny or pde == 1 and nf > 0
    assert nno > 100
    assert np.array_equal(fl, fo)
    assert not (near_o & ~near & 1).any()
