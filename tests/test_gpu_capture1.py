"""Work on a 1D mesh that a caller captured into a CUDA graph, replayed with direct steps,
set_modes and steps of other kinds in between: every replay continues from the mesh's
current state and leaves its result there, bit for bit what the plain calls give."""
import numpy as np
import pytest

import paper_1904_11147_gb300 as dgl
from paper_1904_11147_gb300 import workloads as W

pytestmark = pytest.mark.gpu

NX, DT = [150, 33], 1e-4


def _pair(pde, N):
    import torch
    st = torch.cuda.Stream()
    u = W.random_modes(1, pde, N, sum(NX), np.random.default_rng(7 * N + pde), smooth=0.05 if pde == 0 else 0.02)
    box = [(0.0, 1.0, 0.0, 1.0)] * len(NX)
    a = dgl.Mesh(1, pde, N, NX, None, box, bc=1, stream=st.cuda_stream)
    b = dgl.Mesh(1, pde, N, NX, None, box, bc=1)
    a.set_modes(u)
    b.set_modes(u)
    a.set_dt(DT)
    b.set_dt(DT)
    return st, a, b, u


def _stages(m, ind=dgl.IND_TVB):
    for s in (1, 2, 3):
        m.rk_stage(s, 0.0)
        m.flag_cells(ind, 0.01)
        m.cswenolimit()


def _capture(st, fn):
    import torch
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=st):
        fn()
    return g


@pytest.mark.parametrize("pde,N", [(0, 2), (1, 3)])
@pytest.mark.parametrize("what", ["step", "stages"])
@pytest.mark.parametrize("before", [0, 1])
def test_replays_between_direct_steps(pde, N, what, before):
    import torch
    st, a, b, u = _pair(pde, N)
    a.rk_stage(1, 0.0)  # (kernels loaded before the capture)
    a.flag_cells(dgl.IND_TVB, 0.01)
    a.cswenolimit()
    a.set_modes(u)
    for _ in range(before):
        a.step(0.0)
        _stages(b)
    g = _capture(st, (lambda: a.step(0.0)) if what == "step" else (lambda: _stages(a)))

    def replay():
        with torch.cuda.stream(st):
            g.replay()
        _stages(b)

    def direct(ind=dgl.IND_TVB):
        a.step(0.0, ind)
        _stages(b, ind)

    def same():
        st.synchronize()
        assert np.array_equal(a.get_modes(), b.get_modes())

    replay()
    same()
    direct()
    same()
    replay()
    same()
    for _ in range(2):
        direct()
    direct(dgl.IND_KXRCF)
    replay()
    direct()
    same()
    v = 0.5 * (u + u[::-1])
    a.set_modes(v)
    b.set_modes(v)
    replay()
    direct()
    replay()
    same()
