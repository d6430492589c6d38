"""The fixed-point FP64 map and draws (csrc/fixed.cuh: integer arithmetic, the same on the host) against extended
precision.  Tolerances: half an ulp of the rounded result plus the formats' truncations -- V: currents in format 45 and
increments in format 50, below 2^-46 together; gates: increments in format 59 and rates to 2^-58, below 2^-56, and a
stage's error in V (2^-47) times dt |dF/dV|, F' being below 2 per ms and mV over the range; -log u:
four units of its format (57, 62 for u >= 1/2, 70 for u >= 255/256); normals: that error through r = sqrt(-2 log u), and
the radius, sine and product in formats 59, 62 and 57."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1103_4887_gb300", "csrc")
L = np.longdouble

SHIM = r'''
#include "%s/fixed.cuh"
using namespace pimc;
extern "C" int map(double dt, const double* q, const double* x, const double* I, long n, double* f, unsigned char* ok)
{
    const HhFixed c = hh_fixed_of(dt);
    for (long i = 0; i < n; ++i) {
        const HhFixedParams p = hh_fixed_params(c, q + 8 * i, dt);
        ok[i] = hh_map_fixed(c, p, x + 4 * i, I[i], f + 4 * i);
    }
    return c.ok;
}
extern "C" void adjoint(double dt, const double* q, const double* x, const double* I, const double* w, long n, double* f,
                        double* gx, double* gp, unsigned char* ok)
{
    const HhFixed c = hh_fixed_of(dt);
    for (long i = 0; i < n; ++i) {
        double J[4 * kJlen];
        const HhFixedParams p = hh_fixed_params(c, q + 8 * i, dt);
        ok[i] = hh_map_fixed_adj(c, p, x + 4 * i, I[i], f + 4 * i, J, 1);
        if (ok[i]) hh_reverse(J, 1, dt * q[8 * i + 7] * q[8 * i + 2], q[8 * i + 7], w + 4 * i, gx + 4 * i, gp + 7 * i);
    }
}
extern "C" void draws(const unsigned* w, long n, double* z, double* e)
{
    for (long i = 0; i < n; ++i) {
        fx_box_muller(w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3], z[2 * i], z[2 * i + 1]);
        e[i] = fx_neglog_uniform(w[4 * i], w[4 * i + 1]);
    }
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if np.finfo(L).eps > 2e-19:
        pytest.skip("no extended precision")
    d = tmp_path_factory.mktemp("fx")
    src, so = d / "fx.cpp", d / "libfx.so"
    src.write_text(SHIM % CSRC)
    subprocess.check_call(["g++", "-O1", "-shared", "-fPIC", "-ffp-contract=off", str(src), "-o", str(so)])
    return ctypes.CDLL(str(so))


def _psi(u):
    small = np.abs(u) < L(1e-6)
    v = np.where(small, L(1), u)
    return np.where(small, 1 + u / 2 + u * u / 12, -v / np.expm1(-v))


def _rhs(x, q, I):
    V, m, h, n = x
    a = (_psi((V + 40) / 10), L(7) / 100 * np.exp(-(V + 65) / 20), _psi((V + 55) / 10) / 10)
    b = (4 * np.exp(-(V + 65) / 18), 1 / (1 + np.exp(-(V + 35) / 10)), np.exp(-(V + 65) / 80) / 8)
    dV = (I - q[0] * m ** 3 * h * (V - q[3]) - q[1] * n ** 4 * (V - q[4]) - q[2] * (V - q[5])) / q[6]
    return np.stack([dV] + [a[g] * (1 - x[1 + g]) - b[g] * x[1 + g] for g in range(3)])


def _map(x, q, I, dt):
    k1 = _rhs(x, q, I)
    k2 = _rhs(x + dt / 2 * k1, q, I)
    k3 = _rhs(x + dt / 2 * k2, q, I)
    k4 = _rhs(x + dt * k3, q, I)
    return x + dt / 6 * (k1 + 2 * k2 + 2 * k3 + k4)


def _call_map(lib, dt, q, x, I):
    n = x.shape[1]
    qa = np.ascontiguousarray(np.concatenate([q, 1.0 / q[6:7]]).T)
    xa, f, ok = np.ascontiguousarray(x.T), np.full((n, 4), np.nan), np.zeros(n, dtype=np.uint8)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    lib.map(ctypes.c_double(dt), p(qa), p(xa), p(np.ascontiguousarray(I)), ctypes.c_long(n), p(f), p(ok))
    return f.T, ok.astype(bool)


NOMINAL = np.array([120.0, 36.0, 0.3, 50.0, -77.0, -54.4, 1.0])


@pytest.mark.parametrize("dt", [0.01, 0.02, 0.04])
@pytest.mark.parametrize("around", [None, -40.0, -55.0, 0.0, -41.0 + 0.375, 99.9, -99.9])
def test_map(lib, dt, around):
    """States over the whole range and at the removable singularities, their series cuts, V = 0 and the range's ends."""
    rng = np.random.default_rng(7)
    n = 4000
    V = rng.uniform(-90, 60, n) if around is None else around + rng.choice([-1, 1], n) * 10.0 ** rng.uniform(-18, 0, n)
    x = np.stack([V, rng.uniform(-0.02, 1.02, n), rng.uniform(-0.02, 0.7, n), rng.uniform(0, 0.9, n)])
    x[1, ::7], x[2, ::7] = rng.uniform(1.0, 1.37, x[1, ::7].size), 0.3 * x[2, ::7]
    q = NOMINAL[:, None] * rng.uniform(0.5, 1.5, (7, n))
    I = rng.uniform(-20, 40, n)
    f, ok = _call_map(lib, dt, q, x, I)
    ref = _map(x.astype(L), q.astype(L), I.astype(L), L(dt))
    assert ok.any() and np.all(np.isnan(f[:, ~ok]))
    if around is None and dt <= 0.02:
        assert ok.mean() > 0.9
    err, half = np.abs(f - ref), np.spacing(np.abs(ref.astype(np.float64))) / 2
    assert np.all(err[0, ok] <= half[0, ok] + 2.0 ** -46)
    assert np.all(err[1:, ok] <= half[1:, ok] + 2.0 ** -56 + 2 * dt * 2.0 ** -47)


@pytest.mark.parametrize("dt", [0.02, 0.04])
@pytest.mark.parametrize("around", [None, -40.0, -55.0, -41.0 + 0.375, 95.0, -95.0])
def test_adjoint(lib, dt, around):
    """w^T J_x f and w^T J_p f against central differences in extended precision (h = 1e-5 of a scale: truncation below
    1e-9 of the largest entry, rounding below 1e-12), and the forward half against the map, bit for bit."""
    rng = np.random.default_rng(5)
    n = 600
    V = rng.uniform(-90, 60, n) if around is None else around + rng.choice([-1, 1], n) * 10.0 ** rng.uniform(-18, 0, n)
    x = np.stack([V, rng.uniform(0, 1, n), rng.uniform(0, 0.5, n), rng.uniform(0, 0.8, n)])
    q = NOMINAL[:, None] * rng.uniform(0.7, 1.3, (7, n))
    I, w = rng.uniform(-20, 40, n), rng.standard_normal((4, n)) * np.array([[10.0], [100.0], [100.0], [100.0]])
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    qa = np.ascontiguousarray(np.concatenate([q, 1.0 / q[6:7]]).T)
    xa, wa = np.ascontiguousarray(x.T), np.ascontiguousarray(w.T)
    f, gx, gp, ok = np.full((n, 4), np.nan), np.zeros((n, 4)), np.zeros((n, 7)), np.zeros(n, dtype=np.uint8)
    lib.adjoint(ctypes.c_double(dt), p(qa), p(xa), p(np.ascontiguousarray(I)), p(wa), ctypes.c_long(n), p(f), p(gx), p(gp),
                p(ok))
    fm, okm = _call_map(lib, dt, q, x, I)
    ok = ok.astype(bool)
    assert not np.any(ok & ~okm) and ok.mean() > 0.5 and np.array_equal(f.T[:, ok], fm[:, ok])
    xl, ql, Il, wl = (a.astype(L) for a in (x, q, I, w))
    for k in range(11):
        scale = L(1) if k < 4 else np.abs(ql[k - 4])
        h = scale * L(1e-5)
        d = np.zeros((11, n), dtype=L)
        d[k] = h
        up, dn = _map(xl + d[:4], ql + d[4:], Il, L(dt)), _map(xl - d[:4], ql - d[4:], Il, L(dt))
        ref = ((wl * (up - dn)).sum(0) / (2 * h))[ok]
        got = (gx[:, k] if k < 4 else gp[:, k - 4])[ok]
        assert np.all(np.abs(got - ref) <= 1e-8 * np.abs(ref).max())


@pytest.mark.parametrize("index,value", [(0, 100.0), (0, -1e300), (0, np.nan), (1, 1.4), (2, -np.inf), (3, np.nan)])
def test_out_of_range_is_refused(lib, index, value):
    x = np.array([[-65.0], [0.05], [0.6], [0.32]])
    x[index] = value
    assert not _call_map(lib, 0.02, NOMINAL[:, None].copy(), x, np.zeros(1))[1].any()


@pytest.mark.parametrize("k,value", [(0, 300.0), (1, 64.0), (2, 8.0), (3, 151.0), (6, 0.1), (6, 0.0), (0, np.nan)])
def test_parameters_out_of_range_are_refused(lib, k, value):
    q = NOMINAL[:, None].copy()
    q[k] = value
    x = np.array([[-65.0], [0.05], [0.6], [0.32]])
    with np.errstate(divide="ignore"):
        assert not _call_map(lib, 0.02, q, x, np.zeros(1))[1].any()
    for dt in (0.005, 0.05, np.nan):
        assert not _call_map(lib, dt, NOMINAL[:, None].copy(), x, np.zeros(1))[1].any()


@pytest.mark.parametrize("mode", range(7))
def test_draws(lib, mode):
    """Random words, and the corners: u near 0 and 1, the ends of the quadrants and of the tables' intervals."""
    rng = np.random.default_rng(11 + mode)
    n = 20000
    w = rng.integers(0, 1 << 32, (n, 4), dtype=np.uint64).astype(np.uint32)
    if mode == 1:
        w[:, 0] = 0xFFFFFFFF
    if mode == 2:
        w[:, 0], w[:, 1] = 0, w[:, 1] & 0xFFF
    if mode == 3:
        w[:, 0] = (w[:, 0] & 0xFF000000) | rng.choice([0, 0xFFFFFF], n).astype(np.uint32)
    if mode == 4:
        w[:, 2] = (w[:, 2] & 0xC0000000) | rng.choice([0, 0x3FFFFFFF], n).astype(np.uint32)
    if mode == 5:
        w[:, 2] = (w[:, 2] & 0xFC000000) | rng.choice([0, 0x3FFFFFF], n).astype(np.uint32)
    if mode == 6:
        w[:2], w[2:4] = 0, 0xFFFFFFFF
    z, e = np.zeros((n, 2)), np.zeros(n)
    lib.draws(np.ascontiguousarray(w).ctypes.data_as(ctypes.c_void_p), ctypes.c_long(n),
              z.ctypes.data_as(ctypes.c_void_p), e.ctypes.data_as(ctypes.c_void_p))
    u = lambda a, b: (((w[:, a] >> 6).astype(np.uint64) << 26 | (w[:, b] >> 6)).astype(L) + L(0.5)) / L(2) ** 52  # noqa: E731
    u1, u2 = u(0, 1), u(2, 3)
    r, t = np.sqrt(-2 * np.log(u1)), 2 * (4 * np.arctan(L(1))) * u2
    dL = np.where(u1 < 0.5, 2.0 ** -55, np.where(u1 < 1 - 2.0 ** -8, 2.0 ** -60, 2.0 ** -68))
    for got, want, tol in ((z[:, 0], r * np.cos(t), dL / r + 2.0 ** -55), (z[:, 1], r * np.sin(t), dL / r + 2.0 ** -55),
                           (e, -np.log(u1), dL)):
        assert np.all(np.abs(got - want) <= np.spacing(np.abs(got)) / 2 + tol)
    assert np.all(e > 0)
