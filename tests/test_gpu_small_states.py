"""States far below 1: the scheme is homogeneous in an Euler state, so the traces and a stage of a
state times 2^-k are those of the state times 2^-k -- bit for bit for the traces; for a stage to
rounding, since partial sums may leave the normal range (2^-1074 against 2^-1000 here)."""
import numpy as np
import pytest

import paper_1904_11147_gb300 as dgl
from paper_1904_11147_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _traces(N, u):
    import torch
    out = torch.empty((N + 1) * u.shape[1], dtype=torch.float64, device="cuda")
    dgl.refined_arith(5 + N, torch.from_numpy(np.ascontiguousarray(u)).cuda(), out)
    return out.cpu().numpy().reshape(N + 1, -1)


@pytest.mark.parametrize("N", [1, 2, 3])
@pytest.mark.parametrize("k", [950, 957, 958, 959, 960, 990])
def test_traces(N, k):
    rng = np.random.default_rng(k)
    u = rng.uniform(-1, 1, ((N + 1) * (N + 2) // 2, 500)) * rng.choice([1, 2.0 ** -12], 500)
    u[rng.random(u.shape) < 0.1] = 0.0
    u = np.where(np.abs(u) < 2.0 ** -31, 0.0, u.astype(np.float32).astype(np.float64))
    v = _traces(N, u)
    v[np.abs(v) < 2.0 ** -31] = 0.0  # below the normal range at 2^-990
    w = _traces(N, u * 2.0 ** -k) * 2.0 ** 500 * 2.0 ** (k - 500)
    w[np.abs(w) < 2.0 ** -31] = 0.0
    assert np.array_equal(v, w)


@pytest.mark.parametrize("N", [1, 2, 3])
@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("k", [900, 960, 980])
def test_stage(N, bc, k):
    nx, ny = 19, 11
    u = W.random_modes(2, 1, N, nx * ny, np.random.default_rng(k + N), smooth=0.02)
    out = []
    for s in (0, k):
        m = dgl.Mesh(2, 1, N, [nx], [ny], [(0.0, 1.0, 0.0, 1.0)], bc=bc)
        m.set_modes(u * 2.0 ** -s)
        for stage in (1, 2, 3):
            m.rk_stage(stage, 1e-3)
        out.append(m.get_modes() * 2.0 ** (s // 2) * 2.0 ** (s - s // 2))
    scale = np.abs(out[0]).max(axis=(0, 2), keepdims=True)
    assert (np.abs(out[1] - out[0]) <= 2.0 ** -60 * scale).all()
