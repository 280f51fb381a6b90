"""The compensated dot product of FP32 pairs behind the ChEES statistics
(pairs.cuh), compiled for the host and held against exact rational arithmetic."""
import ctypes as C
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include <cmath>
#define __device__
#define __forceinline__ inline
static float __fadd_rn(float a, float b) { return a + b; }
static float __fsub_rn(float a, float b) { return a - b; }
static float __fmul_rn(float a, float b) { return a * b; }
static float __fmaf_rn(float a, float b, float c) { return fmaf(a, b, c); }
static float __double2float_rn(double a) { return (float)a; }
#include "pairs.cuh"
// the terms of the sum as pairs [D][2], as k_chees_finish adds them up
extern "C" double dot(int D, const float* x, const float* y) {
    smc::f2dot s{0.0f, 0.0f, 0.0f};
    for (int d = 0; d < D; ++d) f2_dot(s, smc::f2sum{x[2 * d], x[2 * d + 1]}, smc::f2sum{y[2 * d], y[2 * d + 1]});
    return f2_to_double(s);
}
"""


@pytest.fixture(scope="module")
def dot(tmp_path_factory):
    d = tmp_path_factory.mktemp("pairs")
    (d / "dot.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-Wno-unused-function",
                    "-I" + os.path.join(ROOT, "paper_2504_02627_gb300", "csrc"), "-o", str(d / "dot.so"),
                    str(d / "dot.cpp")], check=True)
    f = C.CDLL(str(d / "dot.so")).dot
    f.restype, f.argtypes = C.c_double, [C.c_int, C.c_void_p, C.c_void_p]
    return f


def _pairs(v):
    hi = v.astype(np.float32)
    return np.ascontiguousarray(np.stack([hi, (v - hi).astype(np.float32)], axis=1))


@pytest.mark.parametrize("D", [1, 2, 7, 10, 52, 128, 256])
def test_pair_dot_error_bound(dot, D):
    """u = 2^-24.  A term's error: its two small products are added in FP32 to the
    exact error of the large one (2 u + 3 u of u |x y|), the product of the low
    parts is dropped (1): 6 u^2 |x y|.  Three levels of running sums: the first
    two are exact, the third adds 2 D terms of at most (D + 3) u^2 S, S = sum
    |x y|, in FP32.  The conversion rounds in FP64."""
    rng = np.random.default_rng(D)
    u = 2.0 ** -24
    bound = 6 * u ** 2 + 4 * D ** 2 * (D + 3) * u ** 3 + 2.0 ** -52
    for k in range(100):
        x = _pairs(rng.standard_normal(D) + (0.0, 0.3)[k % 2])
        # squared distances, and projections on FP32 momenta
        y = x if k % 4 < 2 else np.ascontiguousarray(np.stack([rng.standard_normal(D).astype(np.float32),
                                                                np.zeros(D, np.float32)], axis=1))
        exact = [sum(map(Fraction, map(float, a))) * sum(map(Fraction, map(float, b))) for a, b in zip(x, y)]
        err = abs(Fraction(dot(D, x.ctypes.data, y.ctypes.data)) - sum(exact))
        assert err <= Fraction(bound) * sum(map(abs, exact))
