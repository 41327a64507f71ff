"""The fixed-point steps of FP64 paths (csrc/normal64.cuh, csrc/fx_drift.h), compiled for the host, against
the same steps in long double (64 bits of mantissa or more).

Units are 2^-u of an increment.  Bounds:
- the drift of a lane's run of Philox calls is within one unit a step of one group (256 steps) of the exact
  one, below half a unit a step on a run shorter than that, plus 2^-30 units per call for the fraction's
  own 32 bits;
- whole paths of 2^20 steps: FP64 steps round four times a call, each by up to 2^-53 S, so their error walks
  to 2^-53 sqrt(n / 3) of S.  The fixed-point path's error is held to that: one rounding of S a call (half
  the walk), the integer products' half units (2^-64 sqrt(n), below 2^-53) and the normals' 2^-58 (the
  same normals enter both paths here)."""
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
    uint32_t sum = fx_drift_sum(f.rest, j0 / kDriftCalls);
    int64_t more = 0;  // beyond rh
    for (int g = j0; g < j1; g += kDriftCalls) {
        const int64_t rh = fx_drift_next(f.rh, f.rest, sum);
        more += 4 * (rh - f.rh) * ((g + kDriftCalls < j1 ? g + kDriftCalls : j1) - g);
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
        if (j % kDriftCalls == 0) rh = fx_drift_next(f.rh, f.rest, sum);
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
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed_point")
    src, so = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", f"-I{CSRC}", str(src), "-o",
                    str(so)], check=True)
    lib = ctypes.CDLL(str(so))
    lib.drift_error.restype = ctypes.c_double
    return lib


def _f(x):
    return ctypes.c_double(x)


def _ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


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
