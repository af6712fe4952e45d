"""The tile number of a particle is computed by several kernels that must agree
to the bit (a block places as many particles into a tile as it counted).  The
function's roundings are its own: compiled with and without contraction of
products and sums it gives the same cells, also far outside the grid where
the periods are no longer exact."""
import ctypes
import os
import platform
import re
import subprocess

import numpy as np
import pytest

from paper_1409_5574_gb300 import build

SHIM = r"""
#include <algorithm>
#include <cmath>
#define __device__
#define __forceinline__ inline
struct int2 { int x, y; };
static int2 make_int2(int x, int y) { return int2{x, y}; }
using std::floor;
using std::fmin;
using std::fmax;
#define RN static __attribute__((noinline))
RN float __fsub_rn(float a, float b) { volatile float r = a - b; return r; }
RN float __fmul_rn(float a, float b) { volatile float r = a * b; return r; }
RN float __fdiv_rn(float a, float b) { volatile float r = a / b; return r; }
RN float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
RN double __dsub_rn(double a, double b) { volatile double r = a - b; return r; }
RN double __dmul_rn(double a, double b) { volatile double r = a * b; return r; }
RN double __ddiv_rn(double a, double b) { volatile double r = a / b; return r; }
RN double __fma_rn(double a, double b, double c) { return std::fma(a, b, c); }
"""
ENTRY = r"""
#define ENTRY(R, NAME)                                                                   \
  extern "C" void NAME(const R* x, const R* y, int n, int nx, int ny, R x0, R y0, R ix, R iy, \
                       int* out) {                                                       \
    for (int i = 0; i < n; ++i) {                                                        \
      const int2 c = cell_xy<R>(x[i], y[i], nx, ny, x0, y0, ix, iy);                     \
      out[2 * i] = c.x;                                                                  \
      out[2 * i + 1] = c.y;                                                              \
    }                                                                                    \
  }
ENTRY(float, cells32)
ENTRY(double, cells64)
"""


def _fma_flags():
    if platform.machine() != "x86_64":
        return []  # (part of the base instruction set)
    with open("/proc/cpuinfo") as f:
        if not re.search(r"^flags.*\bfma\b", f.read(), re.M):
            pytest.skip("no fused multiply-add on this host")
    return ["-mfma"]


@pytest.fixture(scope="module")
def libs(tmp_path_factory):
    with open(os.path.join(build.CSRC, "tile_sort.cu")) as f:
        text = f.read()
    body = text.split("namespace {", 1)[1].split(
        "template <typename R>\n__device__ __forceinline__ int tile_of", 1)[0]
    d = tmp_path_factory.mktemp("cells")
    src = d / "cells.cpp"
    src.write_text(SHIM + body + ENTRY)
    out = []
    for mode in ("off", "fast"):
        so = d / ("cells_%s.so" % mode)
        subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=" + mode, *_fma_flags(), "-fPIC",
                        "-shared", "-o", str(so), str(src)], check=True)
        out.append(ctypes.CDLL(str(so)))
    return out


@pytest.mark.parametrize("dtype,name,c", [(np.float32, "cells32", ctypes.c_float),
                                          (np.float64, "cells64", ctypes.c_double)])
@pytest.mark.parametrize("nx,ny", [(130, 100), (4129, 4100)])
@pytest.mark.parametrize("far", [0.5, 3e3, 3e6, 3e15])
def test_cells_do_not_depend_on_contraction(libs, dtype, name, c, nx, ny, far):
    rng = np.random.default_rng(nx)
    dx, n = 2 * np.pi / 32, 40_000
    # cell edges and points between them, over `far` periods to either side
    k = rng.uniform(-far, far, (2, n)) * np.array([[nx], [ny]])
    k[:, ::2] = np.rint(k[:, ::2])
    x, y = np.ascontiguousarray((k * dx).astype(dtype))
    x[:3] = np.nan, np.inf, -np.inf
    got = []
    for lib in libs:
        out = np.zeros((n, 2), np.int32)
        p = ctypes.c_void_p
        getattr(lib, name)(p(x.ctypes.data), p(y.ctypes.data), n, nx, ny, c(0.25 * dx), c(-dx),
                           c(1.0 / dx), c(1.0 / dx), p(out.ctypes.data))
        got.append(out)
    assert (got[0] >= 0).all() and (got[0] < [nx, ny]).all()
    np.testing.assert_array_equal(got[0], got[1])
    if far < 1.0:  # (within a period the cell is the position's, up to an edge)
        want = np.floor((x[3:].astype(np.float64) - 0.25 * dx) / dx) % nx
        off = np.abs(got[0][3:, 0] - want)
        assert np.minimum(off, nx - off).max() <= 1
