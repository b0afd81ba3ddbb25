"""The arithmetic that the default kernels run, against IEEE operations and exact integers: the split
stage's and 1D's reciprocal and root, the 2D limiters' integer quotient, the rounding of
fixed-point sums and the fixed-point traces.

Tolerances.  Reciprocal and root: two units in the last place (relative 2^-51); special values as
IEEE.  Quotient: half a unit (relative 2^-53) and the 2^-60 before rounding.  Rounding of an
integer: half a unit, exactly; results below the normal range are 0."""
from fractions import Fraction

import numpy as np
import pytest

import paper_1904_11147_gb300 as dgl
from test_gpu_arith import SPECIAL, _same

pytestmark = pytest.mark.gpu


def _run(op, x, planes=1):
    import torch
    t = torch.from_numpy(np.ascontiguousarray(x)).cuda()
    out = torch.empty(planes * (t.shape[-1] if t.dim() > 1 else t.numel()), dtype=torch.float64, device="cuda")
    dgl.refined_arith(op, t, out)
    torch.cuda.synchronize()
    return out.cpu().numpy()


@pytest.mark.parametrize("op", [2, 3])
def test_reciprocal_and_root(op):
    rng = np.random.default_rng(50 + op)
    x = np.exp(rng.uniform(np.log(2.3e-308), np.log(1.7e308), 500_000))
    x = np.concatenate([SPECIAL, x * rng.choice([-1.0, 1.0], x.size) if op == 2 else x])
    with np.errstate(divide="ignore", invalid="ignore", over="ignore"):
        want = 1.0 / x if op == 2 else np.sqrt(x)
    got = _run(op, x)
    ax = np.abs(x)
    ieee = ~np.isfinite(x) | (ax < 2.0 ** -1022) | ((ax >= 2.0 ** 1022) if op == 2 else (x < 0))
    assert np.all(_same(got[ieee], want[ieee])), (x[ieee], got[ieee])
    assert (np.abs(got[~ieee] - want[~ieee]) / np.abs(want[~ieee])).max() <= 2.0 ** -51


def _ints(rng, n, bits):
    """random integers of 1..bits bits, runs of ones and single bits among them"""
    w = rng.integers(1, bits + 1, n)
    v = [int(a) << 32 | int(b) for a, b in rng.integers(0, 2 ** 32, (n, 2))]
    out = []
    for k in range(n):
        m = (1 << int(w[k])) - 1
        out.append(m if k % 11 == 0 else (1 << int(w[k]) - 1) if k % 11 == 1 else max(1, v[k] & m))
    return out


def _planes(*rows):
    return np.array([[(v + 2 ** 63) % 2 ** 64 - 2 ** 63 for v in r] for r in rows], dtype=np.int64)


def test_quotient():
    rng = np.random.default_rng(60)
    n = 20000
    t = [v * int(s) for v, s in zip(_ints(rng, n, 63), rng.choice([-1, 1], n))]
    s, q = _ints(rng, n, 64), [int(v) for v in rng.integers(-900, 900, n)]
    got = _run(4, _planes(t, s, q))
    half, slack = Fraction(1, 2 ** 53), Fraction(1, 2 ** 60)
    for k in range(n):
        want = Fraction(t[k], s[k]) * Fraction(2) ** q[k]
        assert abs(Fraction(float(got[k])) - want) <= (half + slack) * abs(want), (t[k], s[k], q[k], got[k])


def test_quotient_and_rounding_at_the_ends_of_the_range():
    one, big = 1 << 62, (1 << 63) - 1
    t = [0, 0, one, -one, one, -one, big, big, -big]
    s = [1, one, one, one, one, one, 1 << 63, 1 << 63, 1 << 63]
    q = [5, -3000, -1021, -1023, 1023, 1024, 1023, 1024, 8000]
    with np.errstate(over="ignore"):
        want = np.array([0.0, 0.0, 2.0 ** -1021, -0.0, 2.0 ** 1023, -np.inf, 2.0 ** 1023, np.inf, -np.inf])
    assert np.all(_same(_run(4, _planes(t, s, q)), want))  # 2^63 - 1 over 2^63 rounds up to 1
    q = [0, 7, -1084, -1085, 961, 962, 960, 961, 962]
    want = np.array([0.0, 0.0, 2.0 ** -1022, -0.0, 2.0 ** 1023, -np.inf, 2.0 ** 1023, np.inf, -np.inf])
    assert np.all(_same(_run(5, _planes(t, q)), want))


def test_rounding():
    rng = np.random.default_rng(61)
    n = 20000
    t = [v * int(s) for v, s in zip(_ints(rng, n, 63), rng.choice([-1, 1], n))]
    for k in range(0, n, 3):  # ties and their neighbours: one bit below the 53
        t[k] = (int(rng.integers(2 ** 52, 2 ** 53)) * 2 + 1) * 2 ** int(rng.integers(0, 9)) + int(rng.integers(-1, 2))
    q = [int(v) for v in rng.integers(-900, 900, n)]
    got = _run(5, _planes(t, q))
    for k in range(n):
        want = Fraction(t[k]) * Fraction(2) ** q[k]
        ulp = Fraction(2) ** (max(abs(t[k]).bit_length() - 53, 0) + q[k])
        assert abs(Fraction(float(got[k])) - want) <= ulp / 2, (t[k], q[k], got[k])


@pytest.mark.parametrize("N", [1, 2, 3])
def test_traces_of_special_modes(N):
    NP = (N + 1) * (N + 2) // 2
    assert not _run(5 + N, np.zeros((NP, 4)), N + 1).any()
    u = np.zeros((NP, 3))
    u[0] = [1.0, -0.3, 1e300]  # a constant: exactly twice its value times psi_0
    assert np.array_equal(_run(5 + N, u, N + 1).reshape(N + 1, 3), np.tile(u[0], (N + 1, 1)))
    for bad in (np.nan, np.inf, -np.inf):
        u = np.ones((NP, NP))
        u[np.arange(NP), np.arange(NP)] = bad  # in each mode in turn
        assert not np.isfinite(_run(5 + N, u, N + 1)).any()
