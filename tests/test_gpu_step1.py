"""The one-kernel 1D step (dg_step with the TVB indicator and CSWENO) against the stage,
indicator and limiter calls it replaces: the same formulas in the same order, so bit for bit,
at the edges of its tiles (116 cells and 6 more on each side), for instances shorter than a
tile's halo, with other kinds of steps in between and inside a caller's stream capture."""
import numpy as np
import pytest

import paper_1904_11147_gb300 as dgl
from paper_1904_11147_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _mesh(pde, N, nx, bc, stream=0):
    return dgl.Mesh(1, pde, N, nx, None, [(0.0, 1.0, 0.0, 1.0)] * len(nx), bc=bc, stream=stream)


def _data(pde, N, cells, seed):
    return W.random_modes(1, pde, N, cells, np.random.default_rng(seed), smooth=0.05 if pde == 0 else 0.02)


def _by_stages(m, dt, n=1):
    flagged = 0
    for _ in range(n):
        for s in (1, 2, 3):
            m.rk_stage(s, dt)
            _, nf, _ = m.flag_cells(dgl.IND_TVB, 0.01, want=True)
            flagged += nf
            m.cswenolimit()
    return flagged


@pytest.mark.parametrize("pde,N", [(p, n) for p in (0, 1) for n in (1, 2, 3)])
@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("nx", [[1], [2], [3, 1, 5], [7], [115], [116, 117], [233, 12, 800]])
def test_step_equals_stage_calls(pde, N, bc, nx):
    u = _data(pde, N, sum(nx), 3 * N + pde)
    dt = 0.02 / max(max(nx), 20)
    a, b = _mesh(pde, N, nx, bc), _mesh(pde, N, nx, bc)
    a.set_modes(u)
    b.set_modes(u)
    a.flag_statistics(reset=True)
    for _ in range(3):
        a.step(dt)
    flagged = _by_stages(b, dt, 3)
    assert np.isfinite(b.get_modes()).all()
    assert np.array_equal(a.get_modes(), b.get_modes())
    assert a.flag_statistics() == (flagged, flagged, 9)


def test_other_steps_in_between():
    import torch
    st = torch.cuda.Stream()
    nx, dt = [130, 40], 1e-4
    u = _data(1, 2, sum(nx), 5)
    a, b = _mesh(1, 2, nx, 1, st.cuda_stream), _mesh(1, 2, nx, 1)
    a.set_modes(u)
    b.set_modes(u)
    for k in range(4):
        a.step(dt)
        _by_stages(b, dt)
        a.step(dt, dgl.IND_KXRCF)
        for s in (1, 2, 3):
            b.rk_stage(s, dt)
            b.flag_cells(dgl.IND_KXRCF, 0.01)
            b.cswenolimit()
        if k % 2:  # twice in a row: the buffers change places an odd number of times
            a.step(dt)
            _by_stages(b, dt)
    assert np.array_equal(a.get_modes(), b.get_modes())


def test_step_inside_a_stream_capture():
    import torch
    st = torch.cuda.Stream()
    nx, dt = [150], 1e-4
    u = _data(1, 3, sum(nx), 6)
    a, b = _mesh(1, 3, nx, 0, st.cuda_stream), _mesh(1, 3, nx, 0)
    a.set_modes(u)
    b.set_modes(u)
    a.step(dt)
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=st):
        a.step(dt)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    _by_stages(b, dt, 4)
    assert np.array_equal(a.get_modes(), b.get_modes())
