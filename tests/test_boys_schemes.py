"""The FP64 and double-float Boys evaluations of the kernels, restated on the CPU from the definition of
their tables (Taylor coefficients about a grid, exp(-T), downward recursion; the asymptote and upward
recursion above the grid), against the oracle.  Bounds: FP64, about ten rounded operations and 2L of
the recursion, 5e-15; double-float, whose operations are good to 2^-46, 1e-13."""
import math

import numpy as np

F = np.float32


def _taylor_f64(T, L, boys):
    k = int(np.rint(32.0 * T))
    c, e, x = boys(L + 6, k / 32.0), math.exp(-k / 32.0), k / 32.0 - T
    s = 0.0
    for j in range(6, -1, -1):
        s = c[L + j] / math.factorial(j) + x * s
    ex = 1.0
    for j in range(6, 0, -1):
        ex = 1.0 + x * ex / j
    out = [s]
    for m in range(L, 0, -1):
        out.append((2.0 * T * out[-1] + e * ex) / (2 * m - 1))
    return out[::-1]


def _asymptote_f64(T, L):
    out, e = [0.886226925452758014 / math.sqrt(T)], float(np.exp(F(-T)))
    for m in range(L):
        out.append(((2 * m + 1) * out[-1] - e) * 0.5 / T)
    return out


def _split(v):
    return F(v), F(v - float(F(v)))


def _two_sum(a, b):
    s = F(a + b)
    t = F(s - a)
    return s, F(F(a - F(s - t)) + F(b - t))


def _add(a, b):
    s, e = _two_sum(a[0], b[0])
    return _two_sum(s, F(e + F(a[1] + b[1])))


def _mul(a, b):
    p = F(a[0] * b[0])
    e = F(float(a[0]) * float(b[0]) - float(p))
    e = F(float(a[0]) * float(b[1]) + float(e))
    e = F(float(a[1]) * float(b[0]) + float(e))
    return _two_sum(p, e)


def _taylor_df(T, L, boys):
    T2 = _split(T)
    k = int(np.rint(64.0 * float(T2[0])))
    Tk = k / 64.0
    c = [v / math.factorial(j) for j, v in enumerate(boys(L + 5, Tk)[L:])]
    xh = F(Tk - float(T2[0]))
    assert float(xh) == Tk - float(T2[0])            # exact, as the kernel assumes
    x = _two_sum(xh, F(-T2[1]))
    s = _two_sum(_split(c[3])[0], F(F(x[0] * F(F(c[4]) + x[0] * F(c[5]))) + _split(c[3])[1]))
    for j in (2, 1, 0):
        s = _add(_split(c[j]), _mul(x, s))
    x2 = _mul(x, x)
    u = _mul(_split(1.0 / 6), x)
    u = _two_sum(u[0], F(u[1] + F(x2[0] * F(F(1.0 / 24) + x[0] * F(1.0 / 120)))))
    u = _add((F(0.5 * x2[0]), F(0.5 * x2[1])), _mul(x2, u))
    e = _mul(_split(math.exp(-Tk)), _add((F(1), F(0)), _add(x, u)))
    out, t2 = [s], (F(2 * T2[0]), F(2 * T2[1]))
    for m in range(L, 0, -1):
        out.append(_mul(_add(_mul(t2, out[-1]), e), _split(1.0 / (2 * m - 1))))
    return float(T2[0]) + float(T2[1]), [float(v[0]) + float(v[1]) for v in out[::-1]]


def test_fp64_scheme(oracle_mod):
    rng = np.random.default_rng(3)
    for T in np.concatenate([[0.0, 1e-9, 1.0 / 64, 47.999], rng.uniform(0, 48, 150), rng.uniform(0, 1, 50)]):
        for L in (0, 1, 4, 8):
            ref = oracle_mod.boys(L, T)
            assert np.abs(np.array(_taylor_f64(T, L, oracle_mod.boys)) / ref - 1).max() <= 5e-15, (T, L)
    for T in (48.0, 48.7, 60.0, 200.0, 1e4):
        for L in (0, 1, 4, 8):
            assert np.abs(np.array(_asymptote_f64(T, L)) / oracle_mod.boys(L, T) - 1).max() <= 5e-15, (T, L)


def test_double_float_scheme(oracle_mod):
    rng = np.random.default_rng(4)
    for T in np.concatenate([[0.0, 1e-9, 1.0 / 128, 35.99], rng.uniform(0, 36, 100), rng.uniform(0, 1, 40)]):
        for L in (0, 1, 4, 8):
            Ts, got = _taylor_df(T, L, oracle_mod.boys)
            assert np.abs(np.array(got) / oracle_mod.boys(L, Ts) - 1).max() <= 1e-13, (T, L)


def _scheme_f32(T, L, boys):
    """The FP32 scheme: second-order expansion about k / 128 (third order about k / 32 for L = 0) and downward recursion
    below 36, the asymptote without exp(-T) above."""
    T = F(T)
    rt = F(1.0 / math.sqrt(float(T))) if T > 0 else F(0)
    if T >= F(36.0):
        h, out = F(F(0.5) * rt * rt), [F(F(0.886226925) * rt)]
        for m in range(L):
            out.append(F(out[-1] * F(F(2 * m + 1) * h)))
        return float(T), [float(v) for v in out]
    fma = lambda a, b, c: F(float(a) * float(b) + float(c))
    step = 128.0 if L else 32.0
    k = int(np.rint(step * float(T)))
    c, x = boys(L + 3, k / step), F(k / step - float(T))
    assert float(x) == k / step - float(T)
    d = fma(x, fma(x, F(0.5 * c[L + 2]) if L else fma(x, F(c[3] / 6), F(0.5 * c[2])), F(c[L + 1])), F(c[L]))
    e = F(F(math.exp(-k / step)) * fma(x, fma(x, fma(x, F(1 / 6), F(0.5)), F(1)), F(1)))
    out = [d]
    for m in range(L, 0, -1):
        d = F(fma(F(2) * T, d, e) * F(1.0 / (2 * m - 1)))
        out.append(d)
    return float(T), [float(v) for v in out[::-1]]


def test_fp32_scheme(oracle_mod):
    """Each order within its roundings (u = 2^-24): two of the table and expansion (and 8e-9 left out), 3 more per
    step of the recursion; above the grid the root's and three per order.  The highest order drifts to
    no side: every FP32 integral would inherit that."""
    rng = np.random.default_rng(6)
    u = 2.0 ** -24
    near = np.concatenate([[0.0, 1e-9, 1.0 / 256, 35.999], rng.uniform(0, 36, 600), rng.uniform(0, 1, 100)])
    for L in (0, 1, 2, 4, 8):
        drift = []
        for T in near:
            Ts, got = _scheme_f32(T, L, oracle_mod.boys)
            rel = np.array(got) / oracle_mod.boys(L, Ts) - 1
            for m in range(L + 1):
                assert abs(rel[m]) <= (3 + 3 * (L - m)) * u + 8e-9, (T, L, m, rel[m])
            drift.append(rel[L])
        assert abs(np.mean(drift)) < 6e-9, (L, np.mean(drift))
        for T in (36.0, 36.5, 40.0, 90.0, 1e3, 1e4):
            Ts, got = _scheme_f32(T, L, oracle_mod.boys)
            rel = np.array(got) / oracle_mod.boys(L, Ts) - 1
            for m in range(L + 1):
                assert abs(rel[m]) <= (3 + 5 * m) * u + 1e-8, (T, L, m, rel[m])
