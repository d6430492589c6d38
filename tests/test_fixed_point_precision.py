"""The fixed-point FP64 map and adjoint against the same formulas in FP64 arithmetic: both are compared with extended
precision, and the fixed-point side may not be further off -- where values are small, too: below threshold m^3 h and the
Jacobian entries made of it are 1e-4 and less, deep in a spike the gate h falls to 1e-4.  The allowances are a quarter of
FP64's own error (two sides of one rounding differ by less over thousands of states) and, for Jacobian entries, half an
ulp (2^-54 of the entry, one rounding)."""
import ctypes

import numpy as np
import pytest

from .test_fixed_point import NOMINAL, L, _call_map, lib  # noqa: F401 (lib: the fixture)

N = 6000


def _steady(V):
    a = (-(V + 40) / 10 / np.expm1(-(V + 40) / 10), 0.07 * np.exp(-(V + 65) / 20), -(V + 55) / 100 / np.expm1(-(V + 55) / 10))
    b = (4 * np.exp(-(V + 65) / 18), 1 / (1 + np.exp(-(V + 35) / 10)), 0.125 * np.exp(-(V + 65) / 80))
    return np.stack([x / (x + y) for x, y in zip(a, b)])


def _psi(u):
    small = np.abs(u) < 1e-6
    v = np.where(small, 1, u)
    return np.where(small, 1 + u / 2 + u * u / 12, -v / np.expm1(-v))


def _rhs(x, q, I):  # in the arithmetic of x
    V, m, h, n = x
    a = (_psi((V + 40) / 10), 7 * np.exp(-(V + 65) / 20) / 100, _psi((V + 55) / 10) / 10)
    b = (4 * np.exp(-(V + 65) / 18), 1 / (1 + np.exp(-(V + 35) / 10)), np.exp(-(V + 65) / 80) / 8)
    dV = (I - q[0] * m ** 3 * h * (V - q[3]) - q[1] * n ** 4 * (V - q[4]) - q[2] * (V - q[5])) / q[6]
    return np.stack([dV] + [a[g] * (1 - x[1 + g]) - b[g] * x[1 + g] for g in range(3)])


def _map(x, q, I, dt):
    k1 = _rhs(x, q, I)
    k2 = _rhs(x + dt / 2 * k1, q, I)
    k3 = _rhs(x + dt / 2 * k2, q, I)
    k4 = _rhs(x + dt * k3, q, I)
    return x + dt / 6 * (k1 + 2 * k2 + 2 * k3 + k4)


def _states(kind):
    rng = np.random.default_rng(3)
    q = NOMINAL[:, None] * rng.uniform(0.8, 1.2, (7, N))
    V = rng.uniform(*{"rest": (-68, -62), "spike": (-20, 40), "wide": (-78, 45), "small": (-78, 45)}[kind], N)
    g = _steady(V)
    if kind == "small":
        g = 10.0 ** rng.uniform(-4, -2, (3, N))
    elif kind == "spike":
        g = g * rng.uniform(0.5, 1.0, (3, N))
    elif kind == "wide":
        g = np.minimum(g * rng.uniform(0.7, 1.3, (3, N)), 1.0)
    x = np.concatenate([V[None], g])
    I = rng.uniform(-5, 20, N)
    if kind == "rest":  # net currents of 0.1
        I = -_rhs(x, q, 0.0)[0] * q[6] + rng.uniform(-0.1, 0.1, N)
    return x, q, I


def _rms(v):
    return float(np.sqrt(np.mean(np.square(v.astype(np.float64)))))


@pytest.mark.parametrize("dt", [0.01, 0.02, 0.04])
@pytest.mark.parametrize("kind", ["rest", "spike", "wide", "small"])
def test_map_is_as_exact_as_fp64(lib, kind, dt):  # noqa: F811
    x, q, I = _states(kind)
    f, ok = _call_map(lib, dt, q, x, I)
    ref = _map(x.astype(L), q.astype(L), I.astype(L), L(dt))
    fp64 = _map(x, q, I, dt)
    assert ok.mean() > 0.7  # wide states at dt = 0.04 leave the formats' range
    e, e64 = (f - ref)[:, ok], (fp64 - ref)[:, ok]
    assert _rms(e[0]) <= 1.25 * _rms(e64[0])
    binade = np.floor(np.log2(np.abs(fp64[:, ok])))
    seen = 0
    for g in (1, 2, 3):
        for k in range(-13, 1):
            at = binade[g] == k
            if at.sum() >= 200:
                assert _rms(e[g, at]) <= 1.25 * _rms(e64[g, at]), (g, k)
                seen += 1
    assert seen >= 3


@pytest.mark.parametrize("dt", [0.01, 0.02, 0.04])
@pytest.mark.parametrize("kind", ["rest", "spike", "wide", "small"])
def test_adjoint_is_as_exact_as_fp64(lib, kind, dt):  # noqa: F811
    """Every entry of the Jacobian (unit cotangents) against complex steps, in extended precision and in FP64."""
    x, q, I = _states(kind)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    qa, xa = np.ascontiguousarray(np.concatenate([q, 1.0 / q[6:7]]).T), np.ascontiguousarray(x.T)
    ok, got = np.zeros(N, dtype=np.uint8), np.zeros((4, 11, N))
    for a in range(4):
        w = np.zeros((N, 4))
        w[:, a] = 1.0
        f, gx, gp = np.zeros((N, 4)), np.zeros((N, 4)), np.zeros((N, 7))
        lib.adjoint(ctypes.c_double(dt), p(qa), p(xa), p(np.ascontiguousarray(I)), p(w), ctypes.c_long(N), p(f), p(gx),
                    p(gp), p(ok))
        got[a, :4], got[a, 4:] = gx.T, gp.T
    at = ok.astype(bool)
    assert at.mean() > 0.7
    for k in range(11):
        col = []
        for T, C in ((L, np.clongdouble), (np.float64, np.complex128)):
            d = np.zeros((11, N), dtype=C)
            d[k] = 1j * T(1e-30)
            y = _map(x.astype(T) + d[:4], q.astype(T) + d[4:], I.astype(T), T(dt))
            col.append(y.imag / T(1e-30))
        for a in range(4):
            ref = col[0][a, at]
            scale = _rms(ref)
            if scale > 0:
                assert _rms(got[a, k, at] - ref) <= 1.25 * _rms(col[1][a, at] - ref) + 2.0 ** -54 * scale, (a, k)


@pytest.mark.parametrize("where", ["anywhere", "u near 1", "next to a zero of the sine or cosine", "both"])
def test_draws_are_as_exact_as_fp64(lib, where):  # noqa: F811
    """Normals and -log u relative to their own size, beside the FP64 formulas (the angle reduced exactly to its distance
    from the nearest zero, as sincospi does); one rounding (2^-53 at most) is allowed for."""
    rng = np.random.default_rng(17)
    n = 20000
    w = rng.integers(0, 1 << 32, (n, 4), dtype=np.uint64).astype(np.uint32)
    bits = rng.integers(4, 25, n)
    if where in ("u near 1", "both"):  # ones at the top of u1
        w[:, 0] |= ((np.uint64(0xFFFFFFFF) << (32 - bits).astype(np.uint64)) & np.uint64(0xFFFFFFFF)).astype(np.uint32)
    if where in ("next to a zero of the sine or cosine", "both"):  # zeros or ones below u2's quadrant bits
        mask = (np.uint64(0x3FFFFFFF) & ~(np.uint64(0x3FFFFFFF) >> bits.astype(np.uint64))).astype(np.uint32)
        w[:, 2] = np.where(rng.random(n) < 0.5, w[:, 2] | mask, w[:, 2] & ~mask)
    z, e = np.zeros((n, 2)), np.zeros(n)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    lib.draws(p(np.ascontiguousarray(w)), ctypes.c_long(n), p(z), p(e))
    k = [((w[:, a] >> 6).astype(np.uint64) << np.uint64(26)) | (w[:, a + 1] >> 6) for a in (0, 2)]
    got, ref = (z[:, 0], z[:, 1], e), {}
    for T in (L, np.float64):
        pi = 4 * np.arctan(T(1))
        u1 = (k[0].astype(T) + T(0.5)) / T(2) ** 52
        quad = (k[1] >> np.uint64(50)).astype(np.int64)
        fr = ((k[1] & np.uint64((1 << 50) - 1)).astype(T) + T(0.5)) / T(2) ** 50
        s, c = np.where(fr < 0.5, np.sin(pi / 2 * fr), np.cos(pi / 2 * (1 - fr))), \
            np.where(fr < 0.5, np.cos(pi / 2 * fr), np.sin(pi / 2 * (1 - fr)))
        cs = np.choose(quad, [c, -s, -c, s])
        sn = np.choose(quad, [s, c, -s, -c])
        E = -np.where(u1 > 0.5, np.log1p(-(T(1) - u1)), np.log(u1))
        r = np.sqrt(2 * E)
        ref[T] = (r * cs, r * sn, E)
    for g, x, y in zip(got, ref[L], ref[np.float64]):
        err, err64 = (g - x) / x, (y - x) / x
        assert _rms(err) <= 1.25 * _rms(err64)
        assert np.abs(err).max() <= np.abs(err64).max() + 2.0 ** -53


@pytest.mark.parametrize("tiny", [0.0, 5e-324, 1e-300, -1e-150, 1e-80, -1e-40, 1e-19])
def test_adjoint_at_vanishing_gates(lib, tiny):  # noqa: F811
    """Gates of no size to speak of (and a drive of none): their Jacobian is that of gates at zero, to 2^-50 of a unit
    entry, the gates' own scale."""
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    out = []
    for v in (tiny, 0.0):
        for which in range(4):
            x = np.array([[-65.0, 0.05, 0.6, 0.32]])
            x[0, 1 + which % 3 if which < 3 else slice(1, 4)] = v
            q, I, w = np.append(NOMINAL, 1.0)[None].copy(), np.array([v]), np.array([[1.0, 2.0, -1.0, 0.5]])
            f, gx, gp, ok = np.zeros((1, 4)), np.zeros((1, 4)), np.zeros((1, 7)), np.zeros(1, dtype=np.uint8)
            lib.adjoint(ctypes.c_double(0.02), p(q), p(x), p(I), p(w), ctypes.c_long(1), p(f), p(gx), p(gp), p(ok))
            assert ok[0]
            out.append(np.concatenate([f[0], gx[0], gp[0]]))
    a, b = np.array(out[:4]), np.array(out[4:])
    assert np.all(np.abs(a - b) <= 2.0 ** -50 * np.maximum(1.0, np.abs(b)))
