"""Positions of the back-projection (split_axis, spg_grid.cu), compiled for the
host from the kernel's source with its rounding intrinsics: the point and the
remainder equal exact arithmetic's from grid points to positions far outside
the box, and beyond the integers an int holds the Gaussian weight is zero."""
import ctypes
import os
import re
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_1905_13408_gb300 import build

SHIM = r"""
#include <cmath>
#include <climits>
#define __device__
#define __forceinline__ inline
#define __noinline__
#define __fmul_rn(a, b) ((float)(a) * (float)(b))
#define __fadd_rn(a, b) ((float)(a) + (float)(b))
#define __fsub_rn(a, b) ((float)(a) - (float)(b))
#define __fmaf_rn std::fmaf
#define __dadd_rn(a, b) ((double)(a) + (double)(b))
#define __dmul_rn(a, b) ((double)(a) * (double)(b))
static int __double2int_rn(double v)
{
    v = std::nearbyint(v);
    return v != v ? 0 : v >= 2147483647.0 ? INT_MAX : v <= -2147483648.0 ? INT_MIN : (int)v;
}
using std::floor;
namespace spg { namespace ff { struct FF { float hi, lo; };
"""


@pytest.fixture(scope="module")
def split(tmp_path_factory):
    ff = open(os.path.join(build.CSRC, "spg_ff.cuh")).read()
    grid = open(os.path.join(build.CSRC, "spg_grid.cu")).read()
    two_sum = re.search(r"__device__ __forceinline__ FF two_sum.*?\n\}", ff, re.S).group(0)
    axis = grid[grid.index("struct AxisPos"):grid.index("__device__ __forceinline__ void make_sample")]
    code = SHIM + two_sum + "\n}}\n" + axis + """
extern "C" void split(int m, const float *r0, const float *r1, const int *kx, const int *ky, int kernel, int *b, float *f)
{
    for (int i = 0; i < m; i++)
        if (!split_axis(r0[i], r1[i], kx[i], ky[i], kernel, b[i], f[i])) {
            const AxisPos a = split_axis_wide(r0[i], r1[i], kx[i], ky[i], kernel);
            b[i] = a.b;
            f[i] = a.f;
        }
}
"""
    d = tmp_path_factory.mktemp("split")
    (d / "s.cpp").write_text(code)
    subprocess.run(["g++", "-O1", "-ffp-contract=off", "-shared", "-fPIC", "-o", str(d / "s.so"), str(d / "s.cpp")],
                   check=True)
    lib = ctypes.CDLL(str(d / "s.so"))

    def run(r0, r1, kx, ky, kernel):
        m = len(r0)
        b, f = np.zeros(m, np.int32), np.zeros(m, np.float32)
        args = [np.ascontiguousarray(r0, np.float32), np.ascontiguousarray(r1, np.float32),
                np.ascontiguousarray(kx, np.int32), np.ascontiguousarray(ky, np.int32)]
        lib.split(m, *[a.ctypes.data_as(ctypes.c_void_p) for a in args], kernel,
                  b.ctypes.data_as(ctypes.c_void_p), f.ctypes.data_as(ctypes.c_void_p))
        return args, b, f
    return run


@pytest.mark.parametrize("kernel", [0, 1])
@pytest.mark.parametrize("scale", [1.0, 300.0, 1e4, 2.0 ** 15, 1e5, 3e6])
def test_positions(split, scale, kernel):
    """Positions up to 600 x scale (below 2^31): exact in rationals, the remainder
    to a float32 rounding or two of at most 1."""
    rng = np.random.default_rng(int(scale))
    m = 4000
    r = scale * rng.uniform(-1, 1, (2, m))
    r[:, ::4] = np.round(r[:, ::4] * 4) / 4  # some on quarters: half-way positions
    (r0, r1, kx, ky), b, f = split(r[0], r[1], rng.integers(-300, 300, m), rng.integers(0, 300, m), kernel)
    for i in range(m):
        p = Fraction(float(r0[i])) * int(kx[i]) + Fraction(float(r1[i])) * int(ky[i])
        want = round(p) if kernel == 0 else p.__floor__()
        assert b[i] == want
        assert abs(float(f[i]) - float(p - want)) <= 2.0 ** -23


def test_beyond_int(split):
    _, b, f = split([1e10, -1e10, 1e38, 3e9], [0, 0, 1e38, 0], [1, 1, 300, 1], [5, 5, 300, 0], 0)
    assert (np.abs(f) > 8e8).all()  # the weight exp(-f^2 / h) is zero
    assert (np.sign(b) == [1, -1, 1, 1]).all()
