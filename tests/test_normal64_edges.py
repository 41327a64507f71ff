"""The fixed-point normals of FP64 paths (csrc/normal64.cuh) at the edges of their reductions, compiled
for the host: every table entry and angle, both streams' uniforms, the radius.

Bounds.  cos, sin: the three shears drop at most 2 units of 2^-62 each and the angle's series 2^-61:
below 2^-58.  The radius from rho = 1/2 on: F is two units of 2^-59 off at most, d rho = dF / rho
< 2^-57, the root and its unit 2^-59 more: below 2^-56.6.
"""
import ctypes
import os
import re
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1505_00965_gb300", "csrc")
SHIM = """
#include "normal64.cuh"
using namespace mlmcgb;
extern "C" void radius(const uint32_t *w, long n, uint64_t *rho)
{
    for (long i = 0; i < n; ++i) rho[i] = fx_radius(w[i], kFxTables);
}
extern "C" void circle(const uint32_t *t, long n, uint64_t *c, uint64_t *s)
{
    for (long i = 0; i < n; ++i) fx_circle(t[i], kFxTables, c[i], s[i]);
}
extern "C" void words(const uint32_t *x, long n, int u23, uint32_t *w)
{
    for (long i = 0; i < n; ++i) w[i] = fx_word(x[i], u23 != 0);
}
extern "C" void doubles(const uint64_t *x, long n, int unit, uint64_t *d)
{
    for (long i = 0; i < n; ++i) d[i] = fx_double_bits<true>(x[i], unit);
}
"""
L = np.longdouble


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("normal64_edges")
    src, so = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", f"-I{CSRC}", str(src), "-o", str(so)], check=True)
    return ctypes.CDLL(str(so))


def _call(f, x, dtypes, *args):
    x = np.ascontiguousarray(x, np.uint32)
    out = [np.zeros(len(x), t) for t in dtypes]
    f(x.ctypes.data_as(ctypes.c_void_p), ctypes.c_long(len(x)), *args,
      *[o.ctypes.data_as(ctypes.c_void_p) for o in out])
    return out


def _rho(w):
    u = w.astype(L) * L(2) ** -32
    return np.sqrt(-2 * np.where(u > 0.5, np.log1p(-(1 - u)), np.log(u)))


def test_radius_bound(lib):
    w = np.random.default_rng(3).integers(1, 1 << 32, 400_000).astype(np.uint32)
    ref = _rho(w)
    err = np.abs(_call(lib.radius, w, [np.uint64])[0].astype(L) * L(2) ** -60 - ref)
    assert err[ref >= 0.5].max() <= L(2) ** L(-56.6)


def test_every_table_angle(lib):
    t = (np.arange(16384, dtype=np.int64)[:, None] * (1 << 18) + np.array([-2, -1, 0, 1, 2, 1 << 17])).ravel()
    t = (t & 0xFFFFFFFF).astype(np.uint32)
    c, s = _call(lib.circle, t, [np.uint64, np.uint64])
    q = (t & 0x3FFFFFFF).astype(np.int64)  # the angle in its quadrant
    half = q > (1 << 29)
    pi = L("3.14159265358979323846264338327950288")
    th = np.where(half, (1 << 30) - q, q).astype(L) * (2 * pi * L(2) ** -32)
    for got, want in ((c, np.where(half, np.sin(th), np.cos(th))), (s, np.where(half, np.cos(th), np.sin(th)))):
        assert np.abs(got.astype(L) * L(2) ** -62 - want).max() <= L(2) ** -58


def test_uniforms_of_both_streams(lib):
    x = np.concatenate([np.random.default_rng(4).integers(0, 1 << 32, 10_000), [0, 1, 0x7FFFFF, 0x800000, 0xFFFFFFFF]])
    x = x.astype(np.uint32)
    y = x.astype(np.int64)
    for u23, want in ((0, y + 1), (1, ((1 << 23) - (y & 0x7FFFFF)) << 9)):
        assert np.array_equal(_call(lib.words, x, [np.uint32], ctypes.c_int(u23))[0], (want & 0xFFFFFFFF).astype(np.uint32))


def test_table_entries():
    mp = pytest.importorskip("mpmath")
    text = open(os.path.join(CSRC, "normal64_tables.h")).read()
    have = [int(v, 16) for v in re.findall(r"0x[0-9A-F]{16}", text[text.index("kFxTables[kFxWords] = {"):])]
    with mp.workdps(40):
        lnc = [int(mp.nint(mp.log(mp.mpf(k) / 512) * 2 ** 59)) for k in range(512, 1025)]
        ln2 = [-lnc[-1] % 2 ** 64] + [int(mp.nint(n * mp.log(2) * 2 ** 59)) for n in range(32)]
        cos = [int(mp.nint(mp.cos(i * mp.pi / 8192) * 2 ** 62)) for i in range(4097)]
        assert have == ln2 + lnc + cos + [0]
        two_pi = re.search(r"kFxTwoPi60 = 0x([0-9A-F]+)", text).group(1)
        assert int(two_pi, 16) == int(mp.nint(2 * mp.pi * 2 ** 60))


def test_conversion_rounds_to_nearest(lib):
    rng = np.random.default_rng(6)
    x = (rng.integers(1, 1 << 63, 50_000) >> rng.integers(0, 60, 50_000)).astype(np.uint64)
    d = np.zeros(len(x), np.uint64)
    lib.doubles(x.ctypes.data_as(ctypes.c_void_p), ctypes.c_long(len(x)), 60, d.ctypes.data_as(ctypes.c_void_p))
    want = x.astype(L) * L(2) ** -60  # 64-bit mantissa: exact
    assert np.all(np.abs(d.view(np.float64).astype(L) - want) <= want * L(2) ** -53)
