"""The fixed-point Box--Muller pair of FP64 paths (csrc/normal64.cuh), compiled for the host, against
extended precision (numpy longdouble: 64-bit mantissa or more).

Bounds, from the reductions' units: the angle's table entries carry 2^-63 each, the first-order
remainder's 32-bit factors 2^-58 and 2^-59.6: |d cos|, |d sin| < 2^-57 + 2^-62 < 2^-56.5.  The radius
is formed from L/2 = -ln u in units of 2^-59 with an error of at most two units, so d rho <=
2^-57 / rho + 2^-60; next to u = 1 (1 - u < 2^-10, rho < 2^-4.5) L/2 has twelve more bits, and the
smallest rho outside it is 2^-4.5: d rho < 2^-52.5 there and < 2^-56 from rho = 1/2 on.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1505_00965_gb300", "csrc")
SHIM = """
#include "normal64.cuh"
using namespace mlmcgb;
extern "C" void pairs(const uint32_t *y, long n, uint64_t *rho, uint64_t *c, uint64_t *s, uint32_t *q)
{
    for (long i = 0; i < n; ++i) {
        const uint32_t w = fx_word(y[i], false);
        rho[i] = fx_radius(w, kFxTables);
        fx_circle(w, kFxTables, c[i], s[i]);
        const bool minus_c = fx_cos_sign(w) != 0, minus_s = fx_sin_sign(w) != 0;
        q[i] = fx_swapped(w) ? (minus_c ? 1 : 3) : (minus_c ? 2 : 0);  // and minus_s from quadrant 2 on
        if (minus_s != (q[i] >= 2)) q[i] = 9;
    }
}
extern "C" void doubles(const uint64_t *x, long n, int unit, uint64_t *d)
{
    for (long i = 0; i < n; ++i) d[i] = fx_double_bits<true>(x[i], unit);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("normal64")
    src, so = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", f"-I{CSRC}", str(src), "-o", str(so)], check=True)
    return ctypes.CDLL(str(so))


def _ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _words(kind):
    rng = np.random.default_rng(7)
    d = np.arange(-300, 300, dtype=np.int64)
    if kind == "random":
        return rng.integers(0, 1 << 32, 200_000)
    if kind == "ends":  # powers of two from both ends: exponents of u and of 1 - u
        e = (np.int64(1) << np.arange(33))[:, None] + d[None, :]
        return np.concatenate([e.ravel(), ~e.ravel()])
    if kind == "angles":  # the table's angles and the quadrants
        return (np.arange(2048, dtype=np.int64)[:, None] * (1 << 21) + d[None, ::6]).ravel()
    # the switch from one reciprocal k / 512 to the next, in every binade
    m = (2.0 ** 41 / (np.arange(512, 1025) + 0.5)).astype(np.int64)
    return ((m[:, None] >> np.arange(32)[None, :])[:, :, None] + d[None, None, ::30]).ravel()


@pytest.mark.parametrize("kind", ["random", "ends", "angles", "reciprocals"])
def test_pair_against_extended_precision(lib, kind):
    y = (_words(kind) & 0xFFFFFFFF).astype(np.uint32)
    n = len(y)
    rho, c, s, q = (np.zeros(n, np.uint64), np.zeros(n, np.uint64), np.zeros(n, np.uint64), np.zeros(n, np.uint32))
    lib.pairs(_ptr(y), ctypes.c_long(n), _ptr(rho), _ptr(c), _ptr(s), _ptr(q))
    L = np.longdouble
    u = (y.astype(L) + 1) * L(2) ** -32
    # ln u from 1 - u where u is close to 1 (both exact)
    ln = np.where(u > 0.5, np.log1p(-(1 - u)), np.log(u))
    ref = np.sqrt(-2 * ln)
    err = np.abs(rho.astype(L) * L(2) ** -60 - ref)
    assert np.all(err <= np.where(ref >= 0.5, L(2) ** -56, L(2) ** L(-52.5)))
    assert rho[y == 0xFFFFFFFF].sum() == 0
    pi = L("3.14159265358979323846264338327950288")
    t = (y.astype(np.uint64) + 1) & np.uint64(0x3FFFFFFF)  # the angle in its quadrant
    assert np.array_equal(q, (((y.astype(np.uint64) + 1) & np.uint64(0xFFFFFFFF)) >> np.uint64(30)).astype(np.uint32))
    half = t > (1 << 29)  # the smaller of the angle and its complement
    th = np.where(half, (1 << 30) - t.astype(np.int64), t.astype(np.int64)).astype(L) * (2 * pi * L(2) ** -32)
    cr, sr = np.where(half, np.sin(th), np.cos(th)), np.where(half, np.cos(th), np.sin(th))
    for got, want in ((c, cr), (s, sr)):
        assert np.all(got.astype(np.int64) >= 0)
        assert np.abs(got.astype(L) * L(2) ** -62 - want).max() <= L(2) ** L(-56.5)


def test_conversion_to_double(lib):
    rng = np.random.default_rng(3)
    a = rng.integers(0, 1 << 63, 20_000) >> rng.integers(0, 60, 20_000)
    x = np.concatenate([a.astype(np.uint64), np.uint64(1) << np.arange(64, dtype=np.uint64),
                        ~(np.uint64(1) << np.arange(64, dtype=np.uint64)), np.array([0, 1, 2 ** 64 - 1], np.uint64)])
    d = np.zeros(len(x), np.uint64)
    lib.doubles(_ptr(x), ctypes.c_long(len(x)), 60, _ptr(d))
    got = d.view(np.float64)
    want = np.array([float(int(v)) for v in x]) * 2.0 ** -60
    assert np.all(np.abs(got - want) <= np.abs(want) * 2.0 ** -52)
    small = x < (1 << 53)
    assert np.array_equal(got[small], want[small])
