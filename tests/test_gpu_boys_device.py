"""The FP64 and FP32 Boys functions as compiled into the kernels, with the tables they read, against the oracle: every order, either side
of every grid's end, on and between the rows.

Bounds, u the unit roundoff of the arithmetic (2^-53, 2^-24):
  FP64            5e-15: the expansion's ten rounded operations and two per step of the recursion.
  FP32            two roundings of table and expansion and 3 per step of the downward recursion, 8e-9 left out by
                  the expansion; above the grid the reciprocal root's 2^-22.9 enters F_m (2m + 1)-fold beside three
                  roundings per order, and 1e-8 is left out with exp(-T).
  FP32, mean      a quarter of u over 4000 arguments below the end, for every order (the roundings, 1.7 u at most, average to
                  0.03 u): each FP32 integral inherits a one-signed error, and J and K sum it up.
  FP32 by FP64    one rounding below the end, as FP32 above."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
U = {0: 2.0 ** -53, 1: 2.0 ** -24, 2: 2.0 ** -24}
FP64, BY_FP64, FP32 = 0, 1, 2


@pytest.fixture(scope="module")
def boys_device(mess, tmp_path_factory):
    from paper_2406_03121_gb300 import build
    out = str(tmp_path_factory.mktemp("host") / "boys_device.so")
    subprocess.run([build._nvcc()] + build.NVCC_FLAGS + ["-shared", os.path.join(HERE, "host", "boys_device.cu"), "-o", out],
                   check=True)
    fn = ctypes.CDLL(out).boys_device
    dp = ctypes.POINTER(ctypes.c_double)
    fn.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_int, dp, dp]

    def call(mode, L, T):
        T = np.ascontiguousarray(T)
        F = np.zeros((len(T), L + 1))
        assert fn(mode, L, len(T), T.ctypes.data_as(dp), F.ctypes.data_as(dp)) == 0
        return F
    return call


def _end(mode, L):
    return {FP64: 48.0, BY_FP64: 36.0, FP32: 30.0 if L <= 5 else 36.0}[mode]


def _arguments(mode, L, rng):
    """Arguments as the arithmetic holds them."""
    e = _end(mode, L)
    T = np.concatenate([[0.0, 1e-12, 1e-6, 1.0 / 256, 1.0 / 128, 1.0 / 64, 1.0 / 32, e], np.arange(0.25, 60.0, 0.25),
                        rng.uniform(0.0, e, 200), rng.uniform(0.0, 1.0, 50), rng.uniform(e, 3 * e, 50), [1e2, 1e3, 1e5]])
    if mode in (BY_FP64, FP32):
        return np.concatenate([T.astype(np.float32), [np.nextafter(np.float32(e), np.float32(0))]]).astype(np.float64)
    return np.append(T, np.nextafter(e, 0.0))


@pytest.mark.parametrize("L", range(9))
@pytest.mark.parametrize("mode", [FP64, BY_FP64, FP32], ids=["fp64", "fp32-by-fp64", "fp32"])
def test_every_order(boys_device, oracle_mod, mode, L):
    T = _arguments(mode, L, np.random.default_rng(100 * mode + L))
    rel = boys_device(mode, L, T) / np.array([oracle_mod.boys(L, t) for t in T]) - 1.0
    m, u = np.arange(L + 1), U[mode]
    near = T < _end(mode, L)
    far32 = (4 + 8 * m) * u + 1e-8
    below, above = {FP64: (5e-15 + 0 * m, 5e-15 + 0 * m), BY_FP64: (u + 5e-15 + 0 * m, far32),
                    FP32: ((3 + 3 * (L - m)) * u + 8e-9, far32)}[mode]
    for sel, bound in ((near, below), (~near, above)):
        worst = np.abs(rel[sel]).max(axis=0)
        assert (worst <= bound).all(), (worst / u, bound / u)


@pytest.mark.parametrize("L", range(9))
def test_fp32_drifts_to_no_side(boys_device, oracle_mod, L):
    rng = np.random.default_rng(L)
    T = rng.uniform(0.0, _end(FP32, L), 4000).astype(np.float32).astype(np.float64)
    rel = boys_device(FP32, L, T) / np.array([oracle_mod.boys(L, t) for t in T]) - 1.0
    assert (np.abs(rel.mean(axis=0)) <= 0.25 * U[FP32]).all(), rel.mean(axis=0) / U[FP32]
