"""The 2D limiters where their reconstruction changes its form: data so large that products
of the smoothness denominators would overflow (the scaled reciprocals take over), data far
below the weights' epsilon, lists that end inside a warp, and states that are not finite.

Tolerance: both sides are FP64 evaluations of the same formulas; a limited mode takes about
300 rounded operations on averages of the variable's scale, so 300 x 1.1e-16 x (condition
of the reconstruction, below 100) < 1e-11 of that scale, the bound of the parity tests.
"""
import numpy as np
import pytest

import oracle
import paper_1904_11147_gb300 as dgl
from parity_cases import rel, rel_hi
from paper_1904_11147_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _scaled(pde, N, nx, ny, scale, seed):
    u = W.random_modes(2, pde, N, nx * ny, np.random.default_rng(seed), smooth=0.15 if pde == 0 else 0.02)
    if pde == 0:
        return u * scale
    u[:, 1:3] *= scale  # velocities by `scale`, pressure and energy by its square
    u[:, 3] *= scale * scale
    return u


def _limited(pde, N, nx, ny, bc, parent, u):
    box = (0.0, 1.3, 0.0, 0.9)
    g = dgl.Mesh(2, pde, N, [nx], [ny], [box], bc=bc)
    o = oracle.Mesh(2, pde, N, nx, ny, box=box, bc=bc)
    g.set_modes(u)
    fl, nf, _ = g.flag_cells(dgl.IND_TVB, 0.0, want=True)
    if parent:
        g.parent_wenolimit()
        return g.get_modes(), o.parent_limit(u, fl), fl, nf
    g.cswenolimit()
    return g.get_modes(), o.limit(u, fl), fl, nf


@pytest.mark.parametrize("pde,N", [(p, n) for p in (0, 1) for n in (1, 2, 3)])
@pytest.mark.parametrize("parent", [False, True])
@pytest.mark.parametrize("nx,ny,bc,scale", [(7, 5, 1, 1.0), (41, 23, 0, 1e-12), (9, 4, 0, 1e7), (33, 9, 1, 1e14)])
def test_limiters_over_magnitudes(pde, N, parent, nx, ny, bc, scale):
    u = _scaled(pde, N, nx, ny, scale, 40 + N)
    got, ref, fl, nf = _limited(pde, N, nx, ny, bc, parent, u)
    assert nf > 0 and np.isfinite(ref).all()
    assert np.array_equal(got[:, :, 0], u[:, :, 0])
    assert np.array_equal(got[fl == 0], u[fl == 0])
    assert rel(got, ref) <= 1e-11 and rel_hi(got, ref) <= 1e-11


@pytest.mark.parametrize("pde,N", [(0, 2), (1, 2), (0, 3), (1, 3), (1, 1)])
@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_non_finite_modes_stay_non_finite(pde, N, value):
    """Whichever mode holds it, also one whose average over every subcell is zero."""
    nx, ny = 12, 9
    for m in range(1, (N + 1) * (N + 2) // 2):
        u = _scaled(pde, N, nx, ny, 1.0, 60 + N)
        u[4 * nx + 5, 0, m] = value
        got, ref, fl, nf = _limited(pde, N, nx, ny, 1, False, u)
        assert nf > 0
        assert np.array_equal(np.isnan(got[fl == 1]), np.isnan(ref[fl == 1]))
