"""A negative TVB constant, which dg_step and dg_harvest accept: no |a| is within M h^2, so the
minmod test decides every cell; an edge value equal to the mean (a = 0) is never kept.  The
2D indicator's FP32 screen must leave an a inside its margins to FP64."""
import numpy as np
import pytest

import paper_1904_11147_gb300 as dgl
from paper_1904_11147_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _flags(pde, N, nx, ny, u, M):
    import torch
    m = dgl.Mesh(2, pde, N, [nx], [ny], [(0.0, 1.0, 0.0, 1.0)], bc=1)
    m.set_modes(u)
    X = torch.empty(nx * ny, dgl.n_features(2, pde, N), dtype=torch.float32, device="cuda")
    fl = torch.empty(nx * ny, dtype=torch.uint8, device="cuda")
    ch = torch.empty(nx * ny, dtype=torch.float32, device="cuda")
    m.harvest(X, fl, ch, M)
    return fl.cpu().numpy()


@pytest.mark.parametrize("pde,N", [(0, 1), (0, 3), (1, 2)])
@pytest.mark.parametrize("modes", [0.0, 1e-20])
def test_values_inside_the_margin(pde, N, modes):
    """Cell means on slopes of either sign, higher modes zero or lost beside the mean."""
    nx, ny = 37, 19
    u = W.random_modes(2, pde, N, nx * ny, np.random.default_rng(3), smooth=0.02)
    u[:, :, 1:] *= 0.0 if modes == 0.0 else modes
    y, x = np.mgrid[:ny, :nx]
    for k, s in enumerate(((1, 1), (-1, 1), (-1, -1))):
        slope = 1.0 + 1e-2 * (s[0] * x + s[1] * y) / nx
        v = u.copy()
        v[:, :, 0] = u[0, :, 0] * slope.reshape(-1, 1)
        assert _flags(pde, N, nx, ny, v, -1.0 - k).all()


@pytest.mark.parametrize("pde,N", [(0, 2), (1, 1), (1, 3)])
def test_values_outside_the_margin(pde, N):
    """Nowhere a = 0: the same flags as with M = 0."""
    nx, ny = 61, 23
    u = W.random_modes(2, pde, N, nx * ny, np.random.default_rng(4), smooth=0.02)
    f0, f1 = _flags(pde, N, nx, ny, u, 0.0), _flags(pde, N, nx, ny, u, -3.0)
    assert 0 < f0.sum() and np.array_equal(f0, f1)
