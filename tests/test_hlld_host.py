"""The FP64 HLLD of csrc/physics.cuh, compiled for the host without contraction:
the parity form equals the oracle's solver bit for bit, on admissible states
and on states with a density or pressure that is zero or negative (which the
status word reports, and whose fluxes keep the oracle's pattern of finite and
undefined values); the reciprocal form of the contracted build stays within its
rounding of it and is finite nowhere that the parity form is not."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
N = 4000

SRC = r"""
#include <cmath>
#define __device__
#define __forceinline__ inline
static inline float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float rsqrtf(float a) { return 1.0f / std::sqrt(a); }
using std::fabs;
#include "physics.cuh"
namespace mhd { namespace i64 {
static float rcp(float f) { return (float)(1.0 / f); }
static float rsq(float f) { return (float)(1.0 / std::sqrt((double)f)); }
float (*seed_rcp)(float) = rcp;
float (*seed_rsqrt)(float) = rsq;
} }
extern "C" void run(long n, int fr, const double* L, const double* R, const double* bn, double* f, double* up) {
  const double g = 5.0 / 3.0;
  for (long i = 0; i < n; ++i, L += 8, R += 8, f += 8)
    if (fr) mhd::hlld_side<double, true>(L, R, bn[i], g, 1.0 / (g - 1.0), 1e-10, true, f, up + i);
    else mhd::hlld_side<double, false>(L, R, bn[i], g, 1.0 / (g - 1.0), 1e-10, true, f, up + i);
}
"""


@pytest.fixture(scope="module")
def solver(tmp_path_factory):
    d = tmp_path_factory.mktemp("hlld")
    (d / "h.cpp").write_text(SRC)
    so = str(d / "h.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC",
                    "-I" + os.path.join(ROOT, "paper_1112_1710_gb300", "csrc"), str(d / "h.cpp"), "-o", so], check=True)
    lib = C.CDLL(so)

    def run(L, R, bn, fr):
        f, up = np.zeros((len(bn), 8)), np.zeros(len(bn))
        lib.run(C.c_long(len(bn)), C.c_int(fr), *[C.c_void_p(a.ctypes.data) for a in (L, R, bn, f, up)])
        f[:, 5] = 0.0  # the normal-B slot holds the upwind side instead
        return f, up
    return run


def _states(kind):
    rng = np.random.default_rng(8)
    w = [np.concatenate([rng.uniform(0.1, 2.0, (N, 1)), rng.normal(0, 1, (N, 3)), rng.uniform(0.1, 2.0, (N, 1)),
                         rng.normal(0, 0.7, (N, 3))], axis=1) for _ in range(2)]
    bn = rng.normal(0, 0.7, N)
    L, R = w
    if kind == "no normal field":
        bn[:] = 0.0
    elif kind == "equal":
        R[:] = L
    elif kind == "weak jump":
        R[:] = L * (1.0 + 1e-9 * rng.normal(size=L.shape))
    elif kind == "at rest":
        L[:, 1] = R[:, 1] = 0.0
    elif kind == "zero":
        m = rng.integers(0, 4, N)
        L[m == 0, 0] = L[m == 2, 4] = R[m == 1, 0] = R[m == 3, 4] = 0.0
    elif kind != "plain":
        q = 0 if "rho" in kind else 4
        for s, x in (("L", L), ("R", R)):
            if s in kind:
                x[:, q] *= -1.0
    return L, R, bn


@pytest.mark.parametrize("kind", ["plain", "no normal field", "equal", "weak jump", "at rest", "zero", "rho L", "rho R",
                                  "rho LR", "p L", "p R", "p LR"])
def test_hlld_fp64_equals_oracle(orc, solver, kind):
    L, R, bn = _states(kind)
    want, side = np.zeros((N, 8)), np.zeros(N)
    with np.errstate(all="ignore"):
        for i in range(N):
            want[i], side[i] = orc.hlld(0, L[i], R[i], bn[i], eps_up=1e-10, with_upwind=True)
    want[:, 5] = 0.0
    f, up = solver(L, R, bn, 0)
    assert np.array_equal(f, want, equal_nan=True) and np.array_equal(up, side)
    c, up = solver(L, R, bn, 1)
    assert np.array_equal(up, side)
    bad = ~np.isfinite(want)
    assert not np.any(np.isfinite(c[bad]))
    if kind in ("plain", "no normal field", "equal", "weak jump", "at rest"):
        # the fan's cancellations amplify a rounding of 1.1e-16 by at most 1 / (relative
        # distance of two of its waves), above 1e-4 in these draws
        assert np.abs(c - want).max() <= 1e-12 * np.abs(want).max()
