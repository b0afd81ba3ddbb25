"""What is timed: the work users of this framework have it do, through its public calls.

A case is one of five kinds of work (``op``):

  step     a time loop's body: the state goes in, ``steps`` SSP-RK3 steps (stage, indicator,
           limiter, optionally the positivity scaling) advance it, the state comes out
  stage    one Runge-Kutta stage without limiting, as a caller with a limiter of its own uses it
  limit    the troubled-cell flags and the CSWENO limiter of one state
  noalloc  the same in one call that allocates nothing, on planes of one variable's mode each
  grad     loss and gradients of the indicator network on a training batch

Sizes, orders and boundary conditions are those of ``workloads.py``, the benchmark and the
tests.  States stand for developed flows: fronts a cell or two wide, smooth waves, and short
ripples over a part of the domain (the waves behind shocks that the TVB indicator flags),
so that the limiter has the 10 to 50 % of the cells to work on that it has in long runs.
``exact`` restates the method in plain torch, 64 bits.
"""
import ctypes
import math

import numpy as np
import torch

import paper_1904_11147_gb300 as dgl

GAMMA = 1.4
TVB_M = 0.01
PDE = {"burgers": dgl.BURGERS, "euler": dgl.EULER}
BC = {"periodic": dgl.BC_PERIODIC, "outflow": dgl.BC_OUTFLOW, "dmr": dgl.BC_DMR}
IND = {"tvb": dgl.IND_TVB, "kxrcf": dgl.IND_KXRCF, "learned": dgl.IND_MLP}


def listed():
    return [
        # Example 1: one small 1D Burgers run; the smallest call, bound by launches
        dict(name="burgers1d_p2", op="step", dim=1, pde="burgers", order=2, count=1, nx=160, ny=1, bc="periodic",
             indicator="tvb", limiter="cswenolimit", positivity=False, steps=20),
        # the batch of random shock tubes, P3
        dict(name="tubes1d_p3", op="step", dim=1, pde="euler", order=3, count=64, nx=800, ny=1, bc="outflow",
             indicator="tvb", limiter="cswenolimit", positivity=False, steps=4),
        # the four-quadrant problem on the full mesh, the plain method: the headline workload
        dict(name="quadrant_p2", op="step", dim=2, pde="euler", order=2, count=1, nx=1024, ny=1024, bc="outflow",
             indicator="tvb", limiter="cswenolimit", positivity=False, steps=1),
        # the same method with the learned indicator, at the size its network is judged on
        dict(name="learned_p2", op="step", dim=2, pde="euler", order=2, count=1, nx=512, ny=512, bc="outflow",
             indicator="learned", limiter="cswenolimit", positivity=False, steps=2),
        # the batch of uneven P3 problems with the positivity scaling and a time step per instance
        dict(name="batch_p3", op="step", dim=2, pde="euler", order=3, count=8, nx=128, ny=512, bc="outflow",
             indicator="tvb", limiter="cswenolimit", positivity=True, steps=1),
        # the batch of uneven 2D Burgers problems
        dict(name="batch_burgers_p2", op="step", dim=2, pde="burgers", order=2, count=16, nx=64, ny=512,
             bc="periodic", indicator="tvb", limiter="cswenolimit", positivity=False, steps=2),
        # the paper's own indicator with the parent limiter it is compared with
        dict(name="kxrcf_parent_p2", op="step", dim=2, pde="euler", order=2, count=1, nx=400, ny=300, bc="periodic",
             indicator="kxrcf", limiter="parent_wenolimit", positivity=False, steps=2),
        # double Mach reflection (Example 11)
        dict(name="double_mach_p2", op="step", dim=2, pde="euler", order=2, count=1, nx=960, ny=240, bc="dmr",
             indicator="tvb", limiter="cswenolimit", positivity=True, steps=1),
        # one stage of a smooth P1 run on an odd mesh
        dict(name="stage_p1", op="stage", dim=2, pde="euler", order=1, count=1, nx=1537, ny=1021, bc="periodic"),
        # flags and limiter alone, P3, on an odd mesh
        dict(name="limit_p3", op="limit", dim=2, pde="euler", order=3, count=1, nx=301, ny=257, bc="outflow"),
        # the limiter of an application that may not allocate, at that call's size
        dict(name="noalloc_p2", op="noalloc", dim=2, pde="euler", order=2, count=1, nx=128, ny=113, bc="outflow"),
        # a training batch of the learned indicator (2D Euler P2 features)
        dict(name="grad_p2", op="grad", dim=2, pde="euler", order=2, batch=8192),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["step", "step", "step", "stage", "limit", "noalloc", "grad"])
    order = rng.choice([1, 2, 3])
    if op == "grad":
        return dict(op="grad", dim=rng.choice([1, 2]), pde="euler", order=order, batch=_log_int(rng, 257, 16384))
    dim = rng.choice([1, 2, 2])
    pde = rng.choice(["burgers", "euler", "euler"])
    c = dict(op=op, dim=dim, pde=pde, order=order, count=1, bc=rng.choice(["periodic", "outflow"]))
    cells = {1: 1 << 17, 2: 1 << 19, 3: 1 << 18}[order] if dim == 2 else 1 << 16
    if op == "noalloc":
        cells = 16384
    if dim == 1:
        c.update(nx=_log_int(rng, 40, min(cells, 16000)), ny=1)
    else:
        nx = _log_int(rng, 24, 900 if op != "noalloc" else 128)
        c.update(nx=nx, ny=_log_int(rng, 24, max(25, min(900, cells // nx))))
    if op == "step":
        many = rng.random() < 0.4
        if many and dim == 2:
            c.update(count=rng.choice([2, 3, 5, 8]), nx=32, ny=rng.randint(100, 250))
        elif many:
            c.update(count=rng.choice([3, 7, 16]), nx=rng.randint(100, 1000))
        kind = rng.choice(["tvb", "tvb", "kxrcf"])
        c.update(indicator=kind, limiter="parent_wenolimit" if kind == "kxrcf" else "cswenolimit",
                 positivity=pde == "euler" and rng.random() < 0.3, steps=rng.choice([1, 2, 3]))
    return c


# ------------------------------------------------------------------------------ the basis


def psi(n, x):
    """Orthonormal Legendre polynomial n on [-1, 1]."""
    return np.sqrt(n + 0.5) * np.polynomial.legendre.Legendre.basis(n)(np.asarray(x, dtype=np.float64))


def dpsi(n, x):
    return np.sqrt(n + 0.5) * np.polynomial.legendre.Legendre.basis(n).deriv()(np.asarray(x, dtype=np.float64))


def modes_of(dim, N):
    """(a, b) of every mode: psi_a(r) psi_b(s), by total degree, then b."""
    if dim == 1:
        return [(a, 0) for a in range(N + 1)]
    return [(d - b, b) for d in range(N + 1) for b in range(d + 1)]


def sizes_of(case):
    """(nx, ny) of every instance."""
    if case["count"] == 1 or case["dim"] == 1:
        return [(case["nx"], case["ny"])] * case["count"]
    r = np.random.RandomState(1904)
    lo, hi = math.log(case["nx"]), math.log(case["ny"])
    sides = [int(round(math.exp(r.uniform(lo, hi)))) for _ in range(case["count"])]
    return [(n, n) for n in sides]


def box_of(case):
    if case["bc"] == "dmr":
        return (0.0, 4.0, 0.0, 1.0)
    return (-2.0, 2.0, -2.0, 2.0) if case["pde"] == "burgers" else (0.0, 1.0, 0.0, 1.0)


def spacing(case, nx, ny):
    xl, xr, yl, yr = box_of(case)
    return (xr - xl) / nx, (yr - yl) / ny


# ------------------------------------------------------------------------------ the states


def _field(r, X, Y, wx, wy, amp, dim):
    """Fronts, smooth waves and ripples over a part of the unit square; wx, wy: cell widths."""
    f = torch.zeros_like(X + Y)
    for _ in range(3):  # smooth waves
        k = r.randint(1, 3, 2)
        f = f + 0.2 * amp * r.uniform(0.3, 1.0) * torch.sin(
            2 * math.pi * (float(k[0]) * X + (float(k[1]) * Y if dim == 2 else 0.0)) + r.uniform(0, 2 * math.pi))
    for _ in range(4):  # fronts, 1.5 cells wide
        th = r.uniform(0, 2 * math.pi) if dim == 2 else 0.0
        x0, y0 = r.uniform(0.1, 0.9, 2)
        bend = 0.06 * torch.sin(2 * math.pi * r.randint(1, 3) * (Y if dim == 2 else 0.0 * X) + r.uniform(0, 6.28))
        s = math.cos(th) * (X - x0) + (math.sin(th) * (Y - y0) if dim == 2 else 0.0) + bend
        w = 0.75 * max(wx, wy if dim == 2 else 0.0)
        f = f + 0.3 * amp * r.uniform(-1, 1) * torch.tanh(s / w)
    mask = torch.sin(2 * math.pi * X + r.uniform(0, 6.28)) + (
        torch.sin(2 * math.pi * Y + r.uniform(0, 6.28)) if dim == 2 else 0.0)
    mask = torch.sigmoid((mask - 0.85) / 0.05)
    for _ in range(3):  # ripples, 10 to 18 cells long
        th, cells = r.uniform(0, 2 * math.pi), r.uniform(10, 18)
        s = math.cos(th) * X / wx + (math.sin(th) * Y / wy if dim == 2 else 0.0)
        f = f + 0.02 * amp * mask * torch.sin(2 * math.pi * s / cells + r.uniform(0, 6.28))
    return f


def _state(case, seed, nx, ny, k):
    """Modes [ny, nx, V, NP] of instance k."""
    dim, N, dev = case["dim"], case["order"], "cuda"
    r = np.random.RandomState((seed * 1009 + 31 * k + 7) % (1 << 31))
    nvar = 1 if case["pde"] == "burgers" else dim + 2
    state = r.get_state()
    q, w = np.polynomial.legendre.leggauss(N + 2)
    ab = modes_of(dim, N)
    U = torch.zeros(ny, nx, nvar, len(ab), dtype=torch.float64, device=dev)
    wx, wy = 1.0 / nx, 1.0 / ny
    cx = (torch.arange(nx, device=dev, dtype=torch.float64) + 0.5)[None, :] * wx
    cy = (torch.arange(ny, device=dev, dtype=torch.float64) + 0.5)[:, None] * wy
    for j in range(N + 2 if dim == 2 else 1):
        for i in range(N + 2):
            r.set_state(state)  # the same fields at every point
            X = cx + 0.5 * wx * q[i] + 0.0 * cy
            Y = cy + (0.5 * wy * q[j] if dim == 2 else 0.0) + 0.0 * cx
            if nvar == 1:
                u = [0.5 + _field(r, X, Y, wx, wy, 1.0, dim)]
            elif case["bc"] == "dmr":
                # the shock of Example 11 and what it leaves behind: short waves on the post-shock side
                s = (X * 4.0 - 1.0 / 6.0 - Y / math.sqrt(3.0)) * math.sqrt(3.0) / 2.0
                pre = 0.5 * (1.0 + torch.tanh(s / (0.75 * max(4.0 * wx, wy))))
                rip = _field(r, X, Y, wx, wy, 0.15, dim)
                rho = 8.0 * torch.exp(rip) * (1 - pre) + 1.4 * pre
                p = 116.5 * torch.exp(1.4 * rip) * (1 - pre) + pre
                vel = [8.25 * math.sqrt(0.75) * (1 - pre), -8.25 * 0.5 * (1 - pre)]
                u = _conserved(rho, vel, p)
            else:
                rho = torch.exp(_field(r, X, Y, wx, wy, 0.8, dim))
                p = torch.exp(_field(r, X, Y, wx, wy, 0.8, dim))
                vel = [_field(r, X, Y, wx, wy, 0.8, dim) for _ in range(dim)]
                u = _conserved(rho, vel, p)
            for m, (a, b) in enumerate(ab):
                c = w[i] * float(psi(a, q[i])) * (w[j] * float(psi(b, q[j])) if dim == 2 else 1.0)
                for v in range(nvar):
                    U[:, :, v, m] += c * u[v]
    return U


def _conserved(rho, vel, p):
    return [rho] + [rho * x for x in vel] + [p / (GAMMA - 1) + 0.5 * rho * sum(x * x for x in vel)]


def inputs(case, seed):
    """Modes of the whole batch, [cell, var, mode]."""
    parts = [_state(case, seed, nx, ny, k).flatten(0, 1) for k, (nx, ny) in enumerate(sizes_of(case))]
    return torch.cat(parts).contiguous()


def _dt(case, x):
    """CFL 0.1 from the cell means, one step for the whole batch."""
    c = 0.5 if case["dim"] == 2 else math.sqrt(0.5)
    m = x[:, :, 0] * c
    if case["pde"] == "burgers":
        s = [m[:, 0].abs()] * case["dim"]
    else:
        vel = [m[:, 1 + d] / m[:, 0] for d in range(case["dim"])]
        p = (GAMMA - 1) * (m[:, -1] - 0.5 * m[:, 0] * sum(v * v for v in vel))
        snd = torch.sqrt(GAMMA * p / m[:, 0])
        s = [v.abs() + snd for v in vel]
    hs = [spacing(case, nx, ny) for nx, ny in sizes_of(case)]
    h = [min(v[d] for v in hs) for d in range(2)]
    return 0.1 / sum(float(v.max()) / h[d] for d, v in enumerate(s))


# ------------------------------------------------------------------------------ prepare, run


def prepare(case, seed):
    if case["op"] == "grad":
        F = dgl.n_features(case["dim"], PDE[case["pde"]], case["order"])
        g = torch.Generator(device="cuda").manual_seed(seed)
        # features are differences and modes over the cell's scale: mostly small, in [-1, 1]
        X = torch.randn(case["batch"], F, device="cuda", generator=g).tanh_().mul_(0.5)
        X[:, ::3] *= 0.1
        y = (torch.rand(case["batch"], device="cuda", generator=g) < 0.12).to(torch.uint8)
        st = torch.cuda.Stream()
        return dict(case=case, st=st, X=X, y=y, net=dgl.MLP(F, seed=11, stream=st.cuda_stream))
    x = inputs(case, seed)
    s = dict(case=case)
    if case["op"] == "noalloc":
        s["planes"] = x.permute(1, 2, 0).reshape(-1, x.shape[0]).contiguous()
        s["out"] = torch.empty_like(s["planes"])
        s["box"] = np.array(box_of(case))
        return s
    sizes = sizes_of(case)
    st = torch.cuda.Stream()
    mesh = dgl.Mesh(case["dim"], PDE[case["pde"]], case["order"], [a for a, _ in sizes], [b for _, b in sizes],
                    [box_of(case)] * len(sizes), bc=BC[case["bc"]], gamma=GAMMA, stream=st.cuda_stream)
    s.update(x=x, out=torch.empty_like(x), mesh=mesh, st=st)
    if case["op"] != "limit":
        s["dt"] = _dt(case, x)
    if case["op"] == "step":
        if case["positivity"]:
            mesh.set_positivity(True)
        if case["limiter"] == "parent_wenolimit":
            mesh.set_limiter(dgl.LIM_PARENT)
        if case["indicator"] == "learned":
            # a network with fixed weights and the threshold that keeps some 15 % of the flags
            net = dgl.MLP(dgl.n_features(case["dim"], PDE[case["pde"]], case["order"]), seed=11, stream=st.cuda_stream)
            mesh.set_indicator(net, -0.06)
            s["net"] = net
        if case["bc"] == "dmr":
            s3 = math.sqrt(3.0)
            mesh.set_boundary_data([8.0, 8.25 * s3 / 2.0, -8.25 / 2.0, 116.5, 1.4, 0.0, 0.0, 1.0, 1.0 / 6.0,
                                    1.0 / s3, 20.0 / s3])
    return s


def run(s):
    case = s["case"]
    if case["op"] == "grad":
        g, loss = s["net"].grad(s["X"], s["y"], pos_weight=4.0)
        return {"grad": g, "loss": loss}
    if case["op"] == "noalloc":
        st = dgl.lib().dg_cswenolimit_noalloc(
            case["dim"], PDE[case["pde"]], case["order"], case["nx"], case["ny"],
            s["box"].ctypes.data_as(ctypes.POINTER(ctypes.c_double)), BC[case["bc"]], ctypes.c_double(GAMMA),
            ctypes.c_double(TVB_M), ctypes.c_void_p(s["planes"].data_ptr()), ctypes.c_void_p(s["out"].data_ptr()),
            None, None, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))  # calls in order: one scratch array
        if st:
            raise RuntimeError(dgl.lib().dg_last_error().decode())
        return {"modes": s["out"]}
    mesh = s["mesh"]
    if case["op"] == "step" and case["bc"] == "dmr":
        mesh.set_time(0.0)
    mesh.set_modes(s["x"])
    if case["op"] == "stage":
        mesh.rk_stage(1, s["dt"])
        return {"modes": mesh.get_modes(s["out"])}
    if case["op"] == "limit":
        flags, n, near = mesh.flag_cells(dgl.IND_TVB, TVB_M, want=True)
        mesh.cswenolimit()
        return {"flags": flags, "n": n, "near": near, "modes": mesh.get_modes(s["out"])}
    if case["positivity"] and case["bc"] != "dmr" and case["dim"] == 2:
        # every step's time step per instance from the wave speeds at the check points
        h = np.array([spacing(case, nx, ny) for nx, ny in sizes_of(case)])
        for _ in range(case["steps"]):
            mesh.set_dt(0.1 / (mesh.max_wavespeed(points=True) / h).sum(axis=1))
            mesh.step(0.0, IND[case["indicator"]], TVB_M)
    else:
        for _ in range(case["steps"]):
            mesh.step(s["dt"], IND[case["indicator"]], TVB_M)
    return {"modes": mesh.get_modes(s["out"])}


def work(case):
    """Bytes: inputs and outputs once.  Flops: the counts of the method's own formulas (flux
    quadrature, traces, reconstruction of a quarter of the cells), per cell."""
    if case["op"] == "grad":
        F = (4 + 5 * ((case["order"] + 1) * (case["order"] + 2) // 2 - 1)) * 4 if case["dim"] == 2 \
            else 3 * (2 + 3 * case["order"])
        P = 32 * F + 1121
        return {"bytes": case["batch"] * (4.0 * F + 1) + 8.0 * P, "flops": 6.0 * case["batch"] * P}
    N, dim = case["order"], case["dim"]
    euler = case["pde"] == "euler"
    V, NP = (dim + 2 if euler else 1), len(modes_of(dim, N))
    cells = sum(a * b for a, b in sizes_of(case))
    if dim == 2:
        stage = {(1, 1): 640, (1, 2): 1434, (1, 3): 2928, (0, 1): 130, (0, 2): 318, (0, 3): 650}[(int(euler), N)]
        indicator = V * (6 * NP + 12)
        limiter = V * {1: 400, 2: 2300, 3: 5200}[N]
    else:
        stage = {1: 190, 2: 300, 3: 430}[N] if euler else {1: 40, 2: 65, 3: 95}[N]
        indicator = V * (4 * NP + 4)
        limiter = V * {1: 60, 2: 200, 3: 380}[N]
    per = {"stage": stage, "limit": indicator + 0.25 * limiter, "noalloc": indicator + 0.25 * limiter,
           "step": 3 * case.get("steps", 0) * (stage + indicator + 0.25 * limiter)}[case["op"]]
    return {"bytes": 16.0 * cells * V * NP, "flops": float(cells * per)}


# ------------------------------------------------------------------------------ 64-bit values


def exact(case, seed):
    if case["op"] == "grad":
        return _exact_grad(case, seed)
    if case.get("indicator") in ("learned", "kxrcf") or case["bc"] == "dmr":
        return None
    if case.get("positivity") and (case["dim"] == 1 or case["pde"] != "euler"):
        return None
    x = inputs(case, seed)
    dt = None if case["op"] in ("limit", "noalloc") else _dt(case, x)
    outs, at = [], 0
    for nx, ny in sizes_of(case):
        M = _Method(case, nx, ny)
        u = x[at:at + nx * ny].reshape(ny, nx, *x.shape[1:])
        at += nx * ny
        if case["op"] == "stage":
            u = u + dt * M.rhs(u)
        elif case["op"] == "step":
            for _ in range(case["steps"]):
                if case["positivity"]:  # no check point of these states is near zero: the scaling is the identity
                    h = spacing(case, nx, ny)
                    sp = M.point_speeds(u)
                    dt = 0.1 / (sp[0] / h[0] + sp[1] / h[1])
                u1 = M.limit(u + dt * M.rhs(u))
                u2 = M.limit(0.75 * u + 0.25 * (u1 + dt * M.rhs(u1)))
                u = M.limit(u / 3 + 2 / 3 * (u2 + dt * M.rhs(u2)))
        else:
            u = M.limit(u)
        outs.append(u.reshape(nx * ny, *x.shape[1:]))
    u = torch.cat(outs)
    if case["op"] == "noalloc":
        return {"modes": u.permute(1, 2, 0).reshape(-1, u.shape[0]).contiguous()}
    return {"modes": u} if case["op"] != "limit" else {"flags": None, "n": None, "near": None, "modes": u}


def _exact_grad(case, seed):
    s = prepare(case, seed)
    p = torch.from_numpy(s["net"].get_params()).double().cuda()
    F = s["X"].shape[1]
    sizes = [(32, F), (32,), (32, 32), (32,), (32,), (1,)]
    parts = [t.reshape(z).requires_grad_(True) for t, z in zip(p.split([int(np.prod(z)) for z in sizes]), sizes)]
    W1, b1, W2, b2, w3, b3 = parts
    X, y = s["X"].double(), s["y"].double()
    z = torch.relu(torch.relu(X @ W1.T + b1) @ W2.T + b2) @ w3 + b3
    loss = -(4.0 * y * torch.nn.functional.logsigmoid(z) + (1 - y) * torch.nn.functional.logsigmoid(-z)).mean()
    loss.backward()
    return {"grad": torch.cat([t.grad.reshape(-1) for t in parts]), "loss": float(loss)}


class _Method:
    """The method on one instance, state [ny, nx, V, NP] (1D: ny = 1)."""

    def __init__(self, case, nx, ny):
        self.dim, self.N, self.euler = case["dim"], case["order"], case["pde"] == "euler"
        self.periodic = case["bc"] == "periodic"
        self.h = spacing(case, nx, ny)
        N = self.N
        self.ab = modes_of(self.dim, N)
        self.q, self.w = np.polynomial.legendre.leggauss(N + 1)
        dev = "cuda"
        t = lambda v: torch.tensor(np.array(v, dtype=np.float64), device=dev)  # noqa: E731
        one = np.ones(1)
        # faces: [side][point][mode], transverse Gauss points
        s = self.q if self.dim == 2 else np.zeros(1)
        tr = (lambda b, z: psi(b, z)) if self.dim == 2 else (lambda b, z: one)
        self.face = [[t([[float(psi(ab[d], e)) * float(tr(ab[1 - d], z).reshape(-1)[0]) for ab in self.ab]
                         for z in s]) for e in (-1.0, 1.0)] for d in range(self.dim)]
        self.fw = t(self.w if self.dim == 2 else one)
        # volume points and the weighted derivatives
        pts = [(x, y, a * b) for y, b in zip(self.q, self.w) for x, a in zip(self.q, self.w)] if self.dim == 2 \
            else [(x, 0.0, a) for x, a in zip(self.q, self.w)]
        two = self.dim == 2
        self.vol = t([[float(psi(a, x)) * (float(psi(b, y)) if two else 1.0) for a, b in self.ab] for x, y, _ in pts])
        self.dx = t([[c * float(dpsi(a, x)) * (float(psi(b, y)) if two else 1.0) for a, b in self.ab]
                     for x, y, c in pts])
        self.dy = t([[c * float(psi(a, x)) * float(dpsi(b, y)) for a, b in self.ab] for x, y, c in pts]) if two else None
        # face midpoints for the indicator
        self.mid = [[t([float(psi(ab[d], e)) * (float(psi(ab[1 - d], 0.0)) if two else 1.0) for ab in self.ab])
                     for e in (-1.0, 1.0)] for d in range(self.dim)]
        self.c0 = 0.5 if two else math.sqrt(0.5)
        self._weno_tables(t)

    # -- states beyond the boundary
    def pad(self, u):
        sx = torch.tensor([(-1.0) ** a for a, _ in self.ab], dtype=torch.float64, device=u.device)
        lo, hi = (u[:, -1:], u[:, :1]) if self.periodic else (u[:, :1] * sx, u[:, -1:] * sx)
        u = torch.cat([lo, u, hi], 1)
        if self.dim == 1:
            return u
        sy = torch.tensor([(-1.0) ** b for _, b in self.ab], dtype=torch.float64, device=u.device)
        lo, hi = (u[-1:], u[:1]) if self.periodic else (u[:1] * sy, u[-1:] * sy)
        return torch.cat([lo, u, hi], 0)

    # -- the discretisation (Eq. (5), local Lax-Friedrichs)
    def flux(self, u, d):
        """u [V, ...] -> flux, spectral radius."""
        if not self.euler:
            return 0.5 * u * u, u[0].abs()
        r = u[0]
        v = [m / r for m in u[1:-1]]
        p = (GAMMA - 1) * (u[-1] - 0.5 * r * sum(x * x for x in v))
        f = [u[1 + d]] + [u[1 + k] * v[d] + (p if k == d else 0.0) for k in range(len(v))] + [(u[-1] + p) * v[d]]
        return torch.stack(f), v[d].abs() + torch.sqrt(GAMMA * p / r)

    def rhs(self, u):
        P = self.pad(u)
        V = u.shape[2]
        at = lambda U, B: torch.einsum("yxvm,qm->vqyx", U, B)  # noqa: E731
        out = torch.zeros_like(u)
        for d in range(self.dim):
            cut = (P[1:-1] if self.dim == 2 else P) if d == 0 else P[:, 1:-1]
            n = cut.shape[1 - d] - 1
            L, R = at(cut.narrow(1 - d, 0, n), self.face[d][1]), at(cut.narrow(1 - d, 1, n), self.face[d][0])
            (fL, aL), (fR, aR) = self.flux(L, d), self.flux(R, d)
            f = 0.5 * (fL + fR - torch.maximum(aL, aR) * (R - L))
            ax = 3 - d
            k = f.shape[ax] - 1
            for e, g in ((1, f.narrow(ax, 1, k)), (0, f.narrow(ax, 0, k))):
                sgn = -1.0 if e else 1.0
                out += sgn * 2.0 / self.h[d] * torch.einsum("vqyx,qm->yxvm", g * self.fw[None, :, None, None],
                                                            self.face[d][e])
            fv, _ = self.flux(at(u, self.vol), d)
            out += 2.0 / self.h[d] * torch.einsum("vqyx,qm->yxvm", fv, self.dx if d == 0 else self.dy)
        return out

    # -- TVB indicator
    def flags(self, u):
        m = self.pad(u)[..., 0] * self.c0
        c = m[1:-1, 1:-1] if self.dim == 2 else m[:, 1:-1]
        bad = torch.zeros(u.shape[:2], dtype=torch.bool, device=u.device)
        for d in range(self.dim):
            cut = (m[1:-1] if self.dim == 2 else m) if d == 0 else m[:, 1:-1]
            n = cut.shape[1 - d] - 2
            dm, dp = c - cut.narrow(1 - d, 0, n), cut.narrow(1 - d, 2, n) - c
            for e in (1, 0):
                a = (u @ self.mid[d][e] - c) * (1.0 if e else -1.0)
                same = ((a > 0) & (dp > 0) & (dm > 0)) | ((a < 0) & (dp < 0) & (dm < 0))
                keep = (a.abs() <= TVB_M * self.h[d] ** 2) | (
                    same & (a.abs() <= dp.abs()) & (a.abs() <= dm.abs()))
                bad |= ~keep.all(dim=2)
        return bad

    # -- CSWENO (Sec. 3): tables by solving for the polynomial of given cell averages
    def _weno_tables(self, t):
        N = self.N
        e = [-1.5 + k / N for k in range(N + 1)] + [0.5 + k / N for k in range(N + 1)]
        if N == 2:
            x, w = np.array([-1, -math.sqrt(0.2), math.sqrt(0.2), 1]), np.array([1, 5, 5, 1]) / 6.0
        else:
            x, w = np.polynomial.legendre.leggauss(2 if N == 1 else 4)
        mono = np.polynomial.polynomial

        def inverse(edges):  # averages -> monomial coefficients
            n = len(edges) - 1
            A = [[(edges[k + 1] ** (j + 1) - edges[k] ** (j + 1)) / (j + 1) / (edges[k + 1] - edges[k])
                  for j in range(n)] for k in range(n)]
            return np.linalg.inv(np.array(A))

        V = lambda z, n: np.vander(np.atleast_1d(z), n, increasing=True)  # noqa: E731
        big = V(x / 2, 2 * N + 1) @ inverse(e)
        C, B = [], []
        gq, gw = np.polynomial.legendre.leggauss(6)
        for i in range(N + 1):
            inv = inverse(e[i:i + N + 2])
            C.append(V(x / 2, N + 1) @ inv)
            b = np.zeros((N + 1, N + 1))
            for l in range(1, N + 1):
                D = np.stack([mono.polyval(gq / 2, mono.polyder(inv[:, k], l)) * np.ones(6) for k in range(N + 1)], 1)
                b += D.T @ (0.5 * gw[:, None] * D)
            B.append(b)
        gam = np.zeros((len(x), N + 1))
        for g in range(len(x)):
            A = np.zeros((2 * N + 1, N + 1))
            for i in range(N + 1):
                A[i:i + N + 1, i] = C[i][g]
            gam[g] = np.linalg.lstsq(A, big[g], rcond=None)[0]
        neg = gam.min(axis=1) < 0
        gp = 0.5 * (gam + 3 * np.abs(gam))  # the split of Shi, Hu and Shu
        gp[~neg] = gam[~neg]
        gn = gp - gam
        self.sp, self.sn = t(gp.sum(1)), t(gn.sum(1))
        self.gp = t(gp / gp.sum(1, keepdims=True))
        self.gn = t(gn / np.maximum(gn.sum(1, keepdims=True), 1e-300))
        self.C, self.B = t(C), t(B)
        part = lambda k: [0.0, 1.0 / N * k, 1.0 / N * (k + 1)]  # noqa: E731
        sub = []
        for k in range(2 * N + 1):
            _, a, b = part(k) if k < N else ([0.0, 0.0, 1.0] if k == N else part(k - N - 1))
            z = -1 + a + b + (b - a) * gq
            sub.append([float((gw * psi(n, z)).sum() / 2) if not (k == N and n) else 0.0 for n in range(N + 1)])
        self.sub = t(sub)
        self.proj = t([[w[g] * float(psi(n, x[g])) for n in range(N + 1)] for g in range(len(x))])

    def weno(self, a):
        """Averages [..., 2N+1] -> values at the Step 1 points [..., G]."""
        N = self.N
        c = a[..., N:N + 1]
        w = (a - c).unfold(-1, N + 1, 1)  # [..., stencil, cell]
        beta = torch.einsum("...ik,ikl,...il->...i", w, self.B, w)
        iv = 1.0 / (1e-6 + beta) ** 2
        p = torch.einsum("igk,...ik->...gi", self.C, w)
        out = []
        for g in (self.gp, self.gn):
            ww = g * iv[..., None, :]
            s = ww.sum(-1)
            out.append((ww * p).sum(-1) / torch.where(s > 0, s, torch.ones_like(s)))
        return c + self.sp * out[0] - self.sn * out[1]

    def eig(self, m, d):
        """Right and left eigenvectors of the flux Jacobian at the states m [n, V]."""
        r, E = m[:, 0], m[:, -1]
        v = [m[:, 1 + k] / r for k in range(self.dim)]
        q2 = sum(x * x for x in v)
        p = (GAMMA - 1) * (E - 0.5 * r * q2)
        c, H, n = torch.sqrt(GAMMA * p / r), (E + p) / r, v[d]
        o, z = torch.ones_like(r), torch.zeros_like(r)
        col = lambda a, mom, e: torch.stack([a, *mom, e], 1)  # noqa: E731
        cols = []
        for s in (-1.0, 0.0, 1.0):
            mom = [v[k] + (s * c if k == d else 0.0) for k in range(self.dim)]
            cols.append(col(o, mom, H + s * n * c if s else 0.5 * q2))
        if self.dim == 2:
            cols.insert(2, col(z, [o if k != d else z for k in range(2)], v[1 - d]))
        R = torch.stack(cols, 2)
        return R, torch.linalg.inv(R)

    def sweep(self, a, m, d):
        """a [n, V, lines, 2N+1] averages -> [n, V, lines, G]."""
        if not self.euler:
            return self.weno(a)
        R, L = self.eig(m, d)
        return torch.einsum("nvf,nflg->nvlg", R, self.weno(torch.einsum("nfv,nvlk->nflk", L, a)))

    def limit(self, u):
        bad = self.flags(u).nonzero()
        out = u.clone()
        for part in bad.split(1 << 17):
            out[part[:, 0], part[:, 1]] = self._limit(u, part)
        return out

    def _limit(self, u, at):
        P, N, V = self.pad(u), self.N, u.shape[2]
        own = [0] * N + [1] + [2] * N  # which neighbour a subcell lies in
        y, x = at[:, 0], at[:, 1]
        m = u[y, x][:, :, 0] * self.c0
        a = torch.tensor([k for k, _ in self.ab], device=u.device)
        b = torch.tensor([k for _, k in self.ab], device=u.device)
        if self.dim == 1:
            avg = torch.stack([P[y, x + own[k]] @ self.sub[k] for k in range(2 * N + 1)], -1)
            val = self.sweep(avg[:, :, None, :], m, 0)[:, :, 0]
            new = val @ self.proj
        else:
            rows = []
            for ky in range(2 * N + 1):
                rows.append(torch.stack([P[y + own[ky], x + own[kx]] @ (self.sub[kx][a] * self.sub[ky][b])
                                         for kx in range(2 * N + 1)], -1))
            avg = torch.stack(rows, 2)  # [n, V, ky, kx]
            val = self.sweep(avg, m, 0).transpose(2, 3)  # [n, V, gx, ky]
            val = self.sweep(val, m, 1)  # [n, V, gx, gy]
            full = torch.einsum("nvxy,xa,yb->nvab", val, self.proj, self.proj)
            new = full[:, :, a, b]
        new[:, :, 0] = u[y, x][:, :, 0]
        return new

    def point_speeds(self, u):
        """Largest |v_d| + c, both over a cell's check points, over the cells."""
        gl = [-1.0, 1.0] if self.N == 1 else [-1.0, 0.0, 1.0]
        pts = [(x, y) for x in self.q for y in gl] + [(x, y) for x in gl for y in self.q]
        B = torch.tensor([[float(psi(a, x) * psi(b, y)) for a, b in self.ab] for x, y in pts], dtype=torch.float64,
                         device=u.device)
        w = torch.einsum("yxvm,qm->vqyx", u, B)
        v = w[1:-1] / w[0]
        c = torch.sqrt(GAMMA * (GAMMA - 1) * (w[-1] - 0.5 * w[0] * (v * v).sum(0)) / w[0]).amax(0)
        return [float((v[d].abs().amax(0) + c).max()) for d in range(2)]
