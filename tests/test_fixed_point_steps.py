"""The fixed-point steps of FP64 paths (csrc/normal64.cuh, csrc/fx_drift.h), compiled for the host, against
the same steps in long double (64 bits of mantissa or more).

Units are 2^-u of an increment.  Bounds:
- the drift of a lane's run of Philox calls is within one unit a step of one group (256 steps) of the exact
  one, below half a unit a step on a run shorter than that, plus 2^-30 units per call for the fraction's
  own 32 bits;
- whole paths of 2^20 steps: FP64 steps round four times a call, each by up to 2^-53 S, so their error walks
  to 2^-53 sqrt(n / 3) of S.  The fixed-point path's error is held to that: one rounding of S a call (half
  the walk), the integer products' half units (2^-64 sqrt(n), below 2^-53) and the normals' 2^-58 (the
  same normals enter both paths here);
- the mean error of an increment: 0.05 units, the Milstein square's 2^8 c2 units of 2^-63 (or coarser) (z and z^2 are cut
  by up to two units of 2^-58 each, E |z| < 1), and four standard errors of increments that err by up to a
  unit and 2^-58 a;
- fx_mul64s: within 2 units, mean 0.05; running products: their own product's error and those before,
  carried through factors below 2: 2^(64 - u) (2 + 4 + 8) units;
- Milstein P_f - P_c on levels of up to 1024 steps: its rms error no larger than that of FP64 steps, its mean
  within three standard errors of 0."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1505_00965_gb300", "csrc")
SHIM = r"""
#include "normal64.cuh"
#include "fx_drift.h"
#include <cmath>
using namespace mlmcgb;
typedef long double L;

// drift of calls [j0, j1) in units of 2^-u less the exact one
extern "C" double drift_error(double drift, int u, int j0, int j1)
{
    const FxDrift f = fx_drift(drift, u);
    uint32_t sum = fx_drift_sum(f.rest, j0 / kDriftCalls<false>);
    int64_t more = 0;  // beyond rh
    for (int g = j0; g < j1; g += kDriftCalls<false>) {
        const int64_t rh = fx_drift_next(f.rh, f.rest, sum);
        more += 4 * (rh - f.rh) * ((g + kDriftCalls<false> < j1 ? g + kDriftCalls<false> : j1) - g);
    }
    return (double)((L)more - ((L)std::ldexp(drift, u) - (L)f.rh) * 4 * (L)(j1 - j0));
}

// Relative error of S after `calls` calls, fixed point and FP64 steps, against long double steps on the
// fixed-point normals.
extern "C" void path_errors(const uint32_t *words, long calls, double a, double drift, int u, double *err)
{
    const FxDrift f = fx_drift(drift, u);
    const uint64_t A = (uint64_t)std::nearbyint(std::ldexp(a, u + 6));
    uint32_t sum = fx_drift_sum(f.rest, 0);
    int64_t rh = 0;
    double S = 1.0, S64 = 1.0;
    L ref = 1.0L;
    const double a58 = std::ldexp(a, -58);
    for (long j = 0; j < calls; ++j) {
        const uint32_t *x = words + 4 * j;
        int64_t d[4], z[4], D2, D3, D4;
        if (j % kDriftCalls<false> == 0) rh = fx_drift_next(f.rh, f.rest, sum);
        fx_increment_pair(x[0], x[1], false, kFxTables, A, rh, d[0], d[1]);
        fx_increment_pair(x[2], x[3], false, kFxTables, A, rh, d[2], d[3]);
        fx_pair(x[0], x[1], false, kFxTables, z[0], z[1]);
        fx_pair(x[2], x[3], false, kFxTables, z[2], z[3]);
        fx_products(d[0], d[1], d[2], d[3], 64 - u, D2, D3, D4);
        S = std::fma(S, std::ldexp((double)D4, -u), S);
        for (int k = 0; k < 4; ++k) {
            S64 = std::fma(S64, std::fma(a58, (double)z[k], drift), S64);
            ref += ref * ((L)a58 * (L)z[k] + (L)drift);
        }
    }
    err[0] = (double)(((L)S - ref) / ref);
    err[1] = (double)(((L)S64 - ref) / ref);
}

// Mean error, in units of 2^-u, of the increments of `calls` consecutive calls against long double.
template <bool MIL> double increment_mean(const uint32_t *words, long calls, double a, double c2, double drift, int u)
{
    const uint64_t A = (uint64_t)std::nearbyint(std::ldexp(a, u + 6)), C2 = (uint64_t)std::nearbyint(std::ldexp(c2, u + 6));
    const FxDrift f = fx_drift(drift, u, MIL ? fx_dropped_mean(C2) : 0.0);
    const L pi = 3.14159265358979323846264338327950288L, scale = std::ldexp((L)1, u);
    uint32_t sum = fx_drift_sum(f.rest, 0);
    int64_t rh = 0;
    L total = 0;
    for (long j = 0; j < calls; ++j) {
        if (j % kDriftCalls<MIL> == 0) rh = fx_drift_next(f.rh, f.rest, sum);
        for (int k = 0; k < 4; k += 2) {
            const uint32_t xa = words[4 * j + k], xb = words[4 * j + k + 1];
            int64_t d[2], z[2];
            if (MIL) {
                fx_pair(xa, xb, false, kFxTables, z[0], z[1]);
                for (int i = 0; i < 2; ++i) d[i] = fx_increment_milstein(z[i], A, C2, rh);
            } else {
                fx_increment_pair(xa, xb, false, kFxTables, A, rh, d[0], d[1]);
            }
            const L rho = std::sqrt(-2 * std::log(((L)xa + 1) * 0x1p-32L)), t = 2 * pi * ((L)xb + 1) * 0x1p-32L;
            const L n[2] = {rho * std::cos(t), rho * std::sin(t)};
            for (int i = 0; i < 2; ++i)
                total += (L)d[i] - scale * ((L)drift + (L)a * n[i] + (MIL ? (L)c2 * n[i] * n[i] : 0));
        }
    }
    return (double)(total / (4 * calls));
}
extern "C" double mean_em(const uint32_t *w, long calls, double a, double c2, double drift, int u)
{
    return increment_mean<false>(w, calls, a, c2, drift, u);
}
extern "C" double mean_milstein(const uint32_t *w, long calls, double a, double c2, double drift, int u)
{
    return increment_mean<true>(w, calls, a, c2, drift, u);
}

// Mean and largest error of fx_mul64s, and the largest of fx_products in units of their result.
extern "C" void products(const int64_t *d, long n, int u, double *out)
{
    L mean = 0, most = 0, worst = 0;
    for (long i = 0; i + 3 < n; i += 4) {
        const L e = (L)fx_mul64s(d[i], d[i + 1]) - (L)d[i] * (L)d[i + 1] * 0x1p-64L;
        mean += e;
        most = std::fmax(most, std::fabs(e));
        int64_t D2, D3, D4;
        fx_products(d[i], d[i + 1], d[i + 2], d[i + 3], 64 - u, D2, D3, D4);
        const L s = std::ldexp((L)1, -u);
        const L x0 = s * d[i], x1 = s * d[i + 1], x2 = s * d[i + 2], x3 = s * d[i + 3];
        const L y2 = x0 + x1 + x0 * x1, y3 = y2 + x2 + y2 * x2, y4 = y3 + x3 + y3 * x3;
        worst = std::fmax(worst, std::fmax(std::fabs((L)D2 - y2 / s), std::fmax(std::fabs((L)D3 - y3 / s), std::fabs((L)D4 - y4 / s))));
    }
    out[0] = (double)(mean / (n / 4));
    out[1] = (double)most;
    out[2] = (double)worst;
}

// Milstein P_f - P_c (relative to S0, M = 4) of `calls` calls: fixed-point fine steps and FP64 coarse ones,
// all FP64, each less long double.
extern "C" void milstein_errors(const uint32_t *words, long calls, double a, double c2, double rh, int u, double *err)
{
    const double drift = rh - c2, H = 4 * (rh - c2), a58 = std::ldexp(a, -58), c58 = std::ldexp(c2, -116);
    const uint64_t A = (uint64_t)std::nearbyint(std::ldexp(a, u + 6)), C2 = (uint64_t)std::nearbyint(std::ldexp(c2, u + 6));
    const FxDrift f = fx_drift(drift, u, fx_dropped_mean(C2));
    uint32_t sum = fx_drift_sum(f.rest, 0);
    double S = 1, S64 = 1, C = 1;
    L ref = 1, refc = 1;
    for (long j = 0; j < calls; ++j) {
        const uint32_t *x = words + 4 * j;
        const int64_t r = fx_drift_next(f.rh, f.rest, sum);
        int64_t z[4], d[4], D2, D3, D4;
        fx_pair(x[0], x[1], false, kFxTables, z[0], z[1]);
        fx_pair(x[2], x[3], false, kFxTables, z[2], z[3]);
        for (int k = 0; k < 4; ++k) d[k] = fx_increment_milstein(z[k], A, C2, r);
        fx_products(d[0], d[1], d[2], d[3], 64 - u, D2, D3, D4);
        S = std::fma(S, std::ldexp((double)D4, -u), S);
        for (int k = 0; k < 4; ++k) {
            S64 = std::fma(S64, std::fma(std::fma(c58, (double)z[k], a58), (double)z[k], drift), S64);
            ref += ref * (((L)c58 * z[k] + (L)a58) * z[k] + (L)drift);
        }
        const int64_t zs = z[0] + z[1] + z[2] + z[3];
        const double zc = (double)zs;
        C = std::fma(C, std::fma(std::fma(c58, zc, a58), zc, H), C);
        refc += refc * (((L)c58 * zs + (L)a58) * zs + (L)H);
    }
    err[0] = (double)((S - C) - (ref - refc));
    err[1] = (double)((S64 - C) - (ref - refc));
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed_point")
    src, so = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", f"-I{CSRC}", str(src), "-o",
                    str(so)], check=True)
    lib = ctypes.CDLL(str(so))
    for name in ("drift_error", "mean_em", "mean_milstein"):
        getattr(lib, name).restype = ctypes.c_double
    return lib


def _f(x):
    return ctypes.c_double(x)


def _ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _unit(level, sigma):
    """The unit's exponent of r = 0.05, T = 1, M = 4 (the rule of csrc/api.cu, Milstein's dmax)."""
    h = 4.0 ** -level
    dmax = 0.05 * h + 7 * sigma * math.sqrt(h) + 49 * 0.5 * sigma * sigma * h
    return 63 - max(0, math.ceil(math.log2(max((1 + dmax) ** 4 - 1, 4 * dmax) / 0.999)))


@pytest.mark.parametrize("level", range(1, 13))
@pytest.mark.parametrize("r", [0.05, 0.03, -0.02, 0.0])
def test_drift_of_a_path(lib, r, level):
    calls = 4 ** (level - 1)
    for u in (63, 62, 60):
        for lanes in (1, 8):
            if calls % lanes:
                continue
            n = calls // lanes
            for i in range(lanes):
                err = lib.drift_error(_f(r / 4 ** level), u, i * n, (i + 1) * n)
                assert abs(err) <= min(256.0, 2.0 * n if lanes == 1 else 4.0 * n) + calls * 2.0 ** -30


@pytest.mark.parametrize("r,sigma", [(0.05, 0.2), (0.03, 0.1), (-0.04, 0.3)])
def test_long_paths_round_no_more_than_fp64_steps(lib, r, sigma):
    n = 1 << 20
    rng = np.random.default_rng(12)
    err = np.zeros((6, 2))
    for i in range(len(err)):
        w = rng.integers(0, 1 << 32, n, dtype=np.uint32)
        lib.path_errors(_ptr(w), ctypes.c_long(n // 4), _f(sigma / math.sqrt(n)), _f(r / n), 63, _ptr(err[i]))
    rms = np.sqrt((err ** 2).mean(axis=0))
    walk = 2.0 ** -53 * math.sqrt(n / 3)
    assert np.abs(err[:, 0]).max() <= 3 * walk / 2  # three standard deviations of one rounding a call
    assert rms[0] <= rms[1]
    assert abs(err[:, 0].mean()) <= 3 * (walk / 2) / math.sqrt(len(err))


@pytest.mark.parametrize("scheme", ["em", "milstein"])
@pytest.mark.parametrize("sigma", [0.05, 0.2, 0.5])
@pytest.mark.parametrize("level", range(4, 13))
def test_mean_error_of_an_increment(lib, level, sigma, scheme):
    calls, h = 1 << 18, 4.0 ** -level
    u = _unit(level, sigma)
    w = np.random.default_rng(level).integers(0, 1 << 32, 4 * calls, dtype=np.uint32)
    a, c2 = sigma * math.sqrt(h), 0.5 * sigma * sigma * h
    drift = 0.05 * h - (c2 if scheme == "milstein" else 0.0)
    mean = getattr(lib, "mean_" + scheme)(_ptr(w), ctypes.c_long(calls), _f(a), _f(c2), _f(drift), u)
    assert abs(mean) <= 0.05 + 2.0 ** 8 * c2 + 4 * (1 + 2.0 ** 5 * a) / math.sqrt(4 * calls)


@pytest.mark.parametrize("u", [63, 62, 61, 60])
def test_products(lib, u):
    # |d| as large as the rule for the unit allows: (1 + d)^4 - 1 < 2^(63 - u)
    dmax = (1.0 + 2.0 ** (63 - u)) ** 0.25 - 1.0
    d = (np.random.default_rng(u).uniform(-dmax, dmax, 400_000) * 2.0 ** u).astype(np.int64)
    out = np.zeros(3)
    lib.products(_ptr(d), ctypes.c_long(len(d)), u, _ptr(out))
    assert abs(out[0]) <= 0.05
    assert out[1] <= 2.0
    assert out[2] <= 2.0 ** (64 - u) * 14


@pytest.mark.parametrize("level", [2, 3, 4, 5])
@pytest.mark.parametrize("sigma", [0.1, 0.2, 0.4])
def test_milstein_differences(lib, level, sigma):
    n, paths, u = 4 ** level, 2000, _unit(level, sigma)
    h = 1.0 / n
    if u < 60:
        pytest.skip("FP64 steps")
    err = np.zeros((paths, 2))
    rng = np.random.default_rng(level)
    for i in range(paths):
        w = rng.integers(0, 1 << 32, n, dtype=np.uint32)
        lib.milstein_errors(_ptr(w), ctypes.c_long(n // 4), _f(sigma * math.sqrt(h)), _f(0.5 * sigma * sigma * h),
                            _f(0.05 * h), u, _ptr(err[i]))
    rms = np.sqrt((err ** 2).mean(axis=0))
    assert rms[0] <= rms[1]
    assert abs(err[:, 0].mean()) <= 3 * err[:, 0].std() / math.sqrt(paths)
