"""The split 2D stage's fixed-point traces against exact values.

Tolerance: half a unit in the last place of the result, and the fixed-point sum's own error.
Its unit is at most 2^-59, 2^-58, 2^-57 of the largest mode (N = 1, 2, 3).  Half a unit per product
and one per mode taken without a product, carried to the result with |KQ| <= 1, 1.35, 1.5, make
at most 3.5, 7.1 and 12.3 units: below 2^-57, 2^-55, 2^-53 of the largest mode.
Mean error: the final rounding leaves some 5e-17 of the largest mode (rms), so a mean over 16,000
samples without bias lies within 5 x 5e-17 / 126 = 2e-18."""
import decimal
import math

import numpy as np
import pytest

import paper_1904_11147_gb300 as dgl

pytestmark = pytest.mark.gpu

SH = 700  # integers in units of 2^-SH


def _traces(N, u):
    import torch
    n = u.shape[1]
    x = torch.from_numpy(np.ascontiguousarray(u)).cuda()
    out = torch.empty((N + 1) * n, dtype=torch.float64, device="cuda")
    dgl.refined_arith(5 + N, x, out)
    torch.cuda.synchronize()
    return out.cpu().numpy().reshape(N + 1, n)


def _int(v):
    m, e = math.frexp(float(v))
    return int(m * 2 ** 53) << (e - 53 + SH)


def _coef(N):
    """2^200 times: twice psi_0 psi_n(1) psi_t(x_q) over psi_0^2, modes by degree, then t"""
    D = decimal.Decimal
    with decimal.localcontext() as c:
        c.prec = 90
        r = {1: [-1 / D(3).sqrt()], 2: [-(D(3) / 5).sqrt(), D(0)],
             3: [-(D(3) / 7 + D(2) / 7 * (D(6) / 5).sqrt()).sqrt(), -(D(3) / 7 - D(2) / 7 * (D(6) / 5).sqrt()).sqrt()]}[N]
        x = r + [-v for v in reversed(r) if v != 0]
        P = [lambda z: D(1), lambda z: z, lambda z: (3 * z * z - 1) / 2, lambda z: (5 * z * z * z - 3 * z) / 2]
        k = [D(2 * n + 1).sqrt() for n in range(N + 1)]
        return [[int((k[d - t] * k[t] * P[t](z) * 2 ** 200).to_integral_value()) for d in range(N + 1) for t in range(d + 1)]
                for z in x]


def _errors(N, u):
    """(error, |value|) of the computed traces over the largest mode, [q][i]"""
    got, coef = _traces(N, u), _coef(N)
    err, val = np.empty(got.shape), np.empty(got.shape)
    for i in range(u.shape[1]):
        m = [_int(v) for v in u[:, i]]
        top = max(abs(v) for v in m) << 200
        for q in range(N + 1):
            w = sum(c * v for c, v in zip(coef[q], m))
            err[q, i] = ((_int(got[q, i]) << 200) - w) / top
            val[q, i] = abs(w) / top
    return err, val


def _modes(N, n, seed, spread):
    rng = np.random.default_rng(seed)
    NP = (N + 1) * (N + 2) // 2
    u = rng.uniform(-1, 1, (NP, n)) * 10.0 ** rng.uniform(-spread, 0, (NP, n)) * 0.02
    u[0] = rng.uniform(1, 2, n) * rng.choice([-1, 1], n)
    return u


@pytest.mark.parametrize("N", [1, 2, 3])
def test_accuracy(N):
    u = _modes(N, 4000, 70 + N, 8)
    u[:, :1000] = np.random.default_rng(80 + N).uniform(-1, 1, (u.shape[0], 1000))
    u *= 10.0 ** np.random.default_rng(90 + N).uniform(-100, 100, 4000)
    err, val = _errors(N, u)
    assert (np.abs(err) <= 2.0 ** -53 * val + {1: 2.0 ** -57, 2: 2.0 ** -55, 3: 2.0 ** -53}[N]).all()


@pytest.mark.parametrize("N", [1, 2, 3])
def test_no_bias(N):
    u = _modes(N, 16000, 100 + N, 0)
    u[0] = np.abs(u[0])  # the rounding of the sum does not depend on the sign, a floor does
    err, _ = _errors(N, u)
    print("mean", err.mean(axis=1), "rms", np.sqrt((err ** 2).mean()))
    assert (np.abs(err.mean(axis=1)) <= 2e-18).all()


@pytest.mark.parametrize("N", [1, 2, 3])
def test_odd_in_the_modes(N):
    """The mirror image of a state has the mirrored traces, bit for bit."""
    u = _modes(N, 20000, 110 + N, 3)
    u[:, ::7] = np.ldexp(np.sign(u[:, ::7]), np.random.default_rng(5).integers(-20, 1, u[:, ::7].shape))
    u[0, ::5] = 0.0
    assert np.array_equal(_traces(N, -u), -_traces(N, u))
