"""The limiters on states far below 1: every smoothness indicator is lost beside the weights'
epsilon, so the limiters are linear there and a state times a power of two has its limited modes
times that power.  The reference is the same state at 2^-500.

Tolerance: partial sums leave the normal range; each is then off by 2^-1074, which is 2^-69 of a state
at 2^-1005.  Some 300 of them with factors below 8: 2^-58."""
import numpy as np
import pytest

import paper_1904_11147_gb300 as dgl
from paper_1904_11147_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _limited(dim, pde, N, nx, ny, bc, parent, u, k):
    m = dgl.Mesh(dim, pde, N, [nx], [ny] if dim == 2 else None, [(0.0, 1.3, 0.0, 0.9)], bc=bc)
    m.set_modes(u * 2.0 ** -k)
    fl, nf, _ = m.flag_cells(dgl.IND_TVB, 0.0, want=True)
    (m.parent_wenolimit if parent else m.cswenolimit)()
    return m.get_modes() * 2.0 ** 500 * 2.0 ** (k - 500), fl, nf


@pytest.mark.parametrize("dim,pde,N,parent", [(d, p, n, w) for d in (1, 2) for p in (0, 1) for n in (1, 2, 3)
                                              for w in (False, True) if d == 2 or not w])
@pytest.mark.parametrize("k", [958, 965, 1005])
def test_linear_in_small_states(dim, pde, N, parent, k):
    nx, ny, bc = (37, 11, k % 2) if dim == 2 else (300, 1, k % 2)
    u = W.random_modes(dim, pde, N, nx * ny, np.random.default_rng(k + 10 * N), smooth=0.02)
    u = u.astype(np.float32).astype(np.float64)
    u[np.abs(u) < 2.0 ** -17] = 0.0  # exact at every scale
    ref, fl0, nf = _limited(dim, pde, N, nx, ny, bc, parent, u, 500)
    got, fl, _ = _limited(dim, pde, N, nx, ny, bc, parent, u, k)
    assert nf > 10 and np.array_equal(fl, fl0)
    scale = np.abs(ref).max(axis=(0, 2), keepdims=True)
    assert (np.abs(got - ref) <= 2.0 ** -58 * scale).all()
