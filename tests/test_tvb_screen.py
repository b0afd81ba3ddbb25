"""The FP32 screen of the 2D TVB indicator (csrc/dg_kernels2d.cu) on the CPU: an emulation of
its arithmetic, operation by operation, against the FP64 decision on bit patterns.  Where the
screen decides, FP64 must decide the same and must not be near a threshold; adversarial
triples sit ulps away from every tie.  Planted mistakes in the margins are caught."""
import numpy as np
import pytest

f32, f64 = np.float32, np.float64


def trunc32(x):
    """trunc_f"""
    b = np.asarray(x, f64).view(np.uint64)
    hi, lo = (b >> np.uint64(32)).astype(np.int64), (b & np.uint64(0xffffffff)).astype(np.int64)
    e = np.clip((hi & 0x7fffffff) - (896 << 20), 0, 255 << 20)
    r = ((e << 3) | (lo >> 29)) & 0xffffffff | (hi & 0x80000000)
    return r.astype(np.uint32).view(f32)


def split(x):
    b = np.asarray(x, f64).view(np.uint64)
    e = ((b >> np.uint64(52)) & np.uint64(0x7ff)).astype(np.int64) - 1023
    low = (b & np.uint64(0x1fffffff)).astype(np.uint32).astype(f32)
    sc = (np.clip(e - 52 + 127, 1, 254).astype(np.uint32) << np.uint32(23)).view(f32)
    l = np.where(np.signbit(x), -(low * sc), low * sc).astype(f32)
    out = (e < -60) | (e > 120)
    l = np.where(out, np.where(np.asarray(x) == 0, f32(0), f32(np.nan)), l).astype(f32)
    return trunc32(x), l


def diff(a, b):
    (ah, al), (bh, bl) = a, b
    return ((ah - bh) + (al - bl)).astype(f32)


def fp64_test(a1, a2, a3, mh2):
    """tvb_changes_bits: (changes, near) per element."""
    k = np.int64(0x7fffffffffffffff)
    i1, i2, i3 = (np.asarray(v, f64).view(np.int64) for v in (a1, a2, a3))
    b1, b2, b3, m = i1 & k, i2 & k, i3 & k, np.asarray(mh2, f64).view(np.int64)
    near = np.abs(b1 - m) <= 32768
    small = b1 <= m
    s = np.maximum(np.maximum(b1, b2), b3)
    thr = np.where(s >= (np.int64(40) << np.int64(52)), s - (np.int64(39) << np.int64(52)), 0)
    near |= ~small & ((b2 <= thr) | (b3 <= thr))
    pos, neg = (i1 > 0) & (i2 > 0) & (i3 > 0), (a1 < 0) & (a2 < 0) & (a3 < 0)
    m23 = np.minimum(b2, b3)
    near |= ~small & (pos | neg) & (np.abs(b1 - m23) <= 32768)
    return ~small & (~(pos | neg) | ~((b1 <= b2) & (b1 <= b3))), near


def screen(a, ma, dp, dm, md, mlo, mhi, margin=1.0):
    fa = np.abs(a)
    lo, hi = fa - ma * f32(margin), fa + ma * f32(margin)
    p, q = np.abs(dp), np.abs(dm)
    mp, mq = (p * f32(2.0 ** -21) + md) * f32(margin), (q * f32(2.0 ** -21) + md) * f32(margin)
    plo, qlo = p - mp, q - mq
    top = np.maximum(hi, np.maximum(p + mp, q + mq)) * f32(2.0 ** -38)
    r = np.full(a.shape, 2)
    ok = (lo > mhi) & (plo > top) & (qlo > top)
    same = ((a > 0) == (dp > 0)) & ((a > 0) == (dm > 0))
    r[ok & same & (hi < np.minimum(plo, qlo) * f32(1 - 2.0 ** -20))] = 0
    r[ok & same & (lo > np.minimum(p + mp, q + mq) * f32(1 + 2.0 ** -20))] = 1
    r[ok & ~same] = 1
    r[hi < mlo] = 0
    return r


def data(n, rng, M):
    """U [n, 3] (U_00 of the cell, of its two neighbours), modes [n, k] and their table values."""
    U = rng.uniform(-2, 2, (n, 1)) * 10.0 ** rng.uniform(-12, 12, (n, 1))
    d = 10.0 ** rng.uniform(-17, 0, (n, 2)) * rng.choice([-1, 1, 1, 1], (n, 2)) * np.abs(U)
    modes = rng.uniform(-1, 1, (n, 5)) * 10.0 ** rng.uniform(-17, 0, (n, 1)) * np.abs(U)
    t = np.array([1.2247, 1.5811, 1.8708, 0.7905, 0.4330]) * 0.7071
    nb = np.concatenate([U + d[:, :1], U - d[:, 1:]], 1)
    # a third of the cells: the edge value tied with a mean difference, up to a few parts in 2^10..2^50
    k = rng.integers(0, n, n // 3)
    tie = (nb[k, 0] - U[k, 0]) * 0.5 * (1 + rng.choice([-1, 0, 1], k.size) * 2.0 ** -rng.uniform(10, 52, k.size))
    modes[k] = 0
    modes[k, 0] = tie / t[0]
    # and some tied with M h^2
    k = rng.integers(0, n, n // 6)
    modes[k] = 0
    modes[k, 0] = M * (1 + rng.choice([-1, 0, 1], k.size) * 2.0 ** -rng.uniform(10, 52, k.size)) / t[0]
    return U[:, 0], nb, modes, t


def decide(U, nb, modes, t, M, margin=1.0):
    c = 0.5000000000000001
    mean, mE, mW = U * c, nb[:, 0] * c, nb[:, 1] * c
    uE = mean.copy()
    for j in range(modes.shape[1]):
        uE = uE + modes[:, j] * t[j]
    want, near = fp64_test(uE - mean, mE - mean, mean - mW, np.full(U.shape, M))
    tf = t.astype(f32)
    a, s = np.zeros(U.shape, f32), np.zeros(U.shape, f32)
    for j in range(modes.shape[1]):
        x = trunc32(modes[:, j]) * tf[j]
        a, s = a + x, s + np.abs(x)
    cf, me = f32(c), split(U)
    dp, dm = cf * diff(split(nb[:, 0]), me), cf * diff(me, split(nb[:, 1]))
    am = np.abs(me[0]) * cf
    big = np.maximum(am, cf * np.maximum(np.abs(trunc32(nb[:, 0])), np.abs(trunc32(nb[:, 1]))))
    md = big * f32(2.0 ** -44) + f32(2.0 ** -100)
    ma = s * f32(2.0 ** -19) + (am * f32(2.0 ** -46) + f32(2.0 ** -100))
    m = trunc32(np.full(U.shape, M))
    got = screen(a, ma, dp, dm, md, m * f32(1 - 2.0 ** -20), m * f32(1 + 2.0 ** -20) + f32(2.0 ** -100), margin)
    return got, want, near


@pytest.mark.parametrize("M", [0.0, 1e-12, 1e-8, 1e-3])
def test_screen_never_decides_otherwise(M):
    rng = np.random.default_rng(12)
    with np.errstate(all="ignore"):
        got, want, near = decide(*data(300000, rng, M), M)
    dec = got < 2
    assert dec.mean() > 0.3
    assert np.array_equal(got[dec] == 1, want[dec]) and not near[dec].any()


def test_margins_are_needed():
    rng = np.random.default_rng(13)
    with np.errstate(all="ignore"):
        got, want, near = decide(*data(300000, rng, 1e-8), 1e-8, margin=0.0)
    dec = got < 2
    assert not (np.array_equal(got[dec] == 1, want[dec]) and not near[dec].any())


def test_non_finite_and_extreme_values_are_left_to_fp64():
    with np.errstate(all="ignore"):
        for bad in (np.nan, np.inf, -np.inf, 1e300):
            U, nb, modes, t = data(64, np.random.default_rng(14), 1e-8)
            for where in range(3):
                u, b, m = U.copy(), nb.copy(), modes.copy()
                if where == 0:
                    u[:] = bad
                elif where == 1:
                    b[:, 0] = bad
                else:
                    m[:, 2] = bad
                got, want, near = decide(u, b, m, t, 1e-8)
                dec = got < 2
                assert np.array_equal(got[dec] == 1, want[dec]) and not near[dec].any()
