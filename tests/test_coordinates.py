"""The device code's box wrap, compiled for the host from its own source (each
operation is one IEEE operation there as on the device). CPU only."""
import ctypes
import os
import re
import subprocess

import numpy as np
import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1303_4523_gb300", "csrc",
                   "enuf_kernels.cuh")

PRELUDE = """
#include <cmath>
#define __device__
#define __forceinline__ static inline
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fdiv_rn(float a, float b) { return a / b; }
static inline float __fmaf_rn(float a, float b, float c) { return fmaf(a, b, c); }
static inline double __dmul_rn(double a, double b) { return a * b; }
static inline double __dsub_rn(double a, double b) { return a - b; }
static inline float __double2float_rn(double a) { return (float)a; }
static inline int max(int a, int b) { return a > b ? a : b; }
static inline unsigned min(unsigned a, unsigned b) { return a < b ? a : b; }
"""

DRIVER = """
extern "C" void wrap32(int n, const float* x, double L, float xmaxf, float Lhi, float Llo, float* w, double* w64) {
    for (int i = 0; i < n; ++i) {
        w[i] = wrap_r(x[i], L, xmaxf, Lhi, Llo);
        w64[i] = wrap_pos((double)x[i], L);
    }
}
extern "C" void grid64(int n, double* x, double ratio, int ng, int* base, double* frac) {
    for (int i = 0; i < n; ++i) grid_coord(x[i], ratio, ng, base[i], frac[i]);
}
extern "C" void cells(int n, const double* x, double rinv, int ncd, int* c64, int* c32) {
    for (int i = 0; i < n; ++i) {
        c64[i] = cell_of(x[i], rinv, ncd);
        c32[i] = cell_of((float)x[i], (float)rinv, ncd);
    }
}
"""


def _functions(names):
    src = open(SRC).read()
    out = []
    for name in names:
        found = re.findall(r"^(?:template <typename R>\n)?__device__ __forceinline__ \w+ " + name + r"\([^;{]*\{(?:[^\n]*\}$|.*?^\})", src, re.M | re.S)
        assert found, name
        out += found
    return "\n".join(out)


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    d = tmp_path_factory.mktemp("coords")
    (d / "c.cpp").write_text(PRELUDE + _functions(["wrap_pos", "wrap_diff", "wrap_r", "grid_coord", "cell_of"]) + DRIVER)
    so = str(d / "c.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-shared", "-fPIC", "-o", so, str(d / "c.cpp")],
                   check=True)
    return ctypes.CDLL(so)


def _ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _consts(L):
    Lhi = np.float32(L)
    xmax = Lhi if float(Lhi) < L else np.nextafter(Lhi, np.float32(0))   # the largest float below L
    return [ctypes.c_float(float(v)) for v in (xmax, Lhi, np.float32(L - float(Lhi)))], xmax


@pytest.mark.parametrize("L", [5.0, 8.1, 14.449686898305517, 25.543647746451768, 30.0, 49.999999999999986,
                               55.90911419702041, 99.99999999999997, 100.00000000000001, 160.0 / 3.0])
def test_float_wrap_is_the_double_wrap_rounded(host, L):
    """wrap_r of floats up to 2^19 boxes away, uniform and within 100 floats of
    multiples of L: the FP64 wrap rounded to float, up to 1/32 unit beyond the
    rounding itself (a result nearer than that to a tie may round either way); what
    rounds to L or above is 0; results lie in [0, L)."""
    rng = np.random.default_rng(int(1000 * L))
    k = np.concatenate([rng.integers(-4, 5, 40000), rng.integers(-(1 << 19), 1 << 19, 40000)]).astype(np.float64)
    uniform = ((k + rng.uniform(0, 1, k.size)) * L).astype(np.float32)
    near = (k * L).astype(np.float32)
    near = near + np.spacing(near) * rng.integers(-100, 101, k.size).astype(np.float32)
    tiny = -np.exp(rng.uniform(np.log(1e-12), np.log(1.0), 2000)).astype(np.float32)
    x = np.ascontiguousarray(np.concatenate([uniform, near, tiny]), np.float32)
    w, w64 = np.empty_like(x), np.empty(x.size)
    c, xmax = _consts(L)
    host.wrap32(x.size, _ptr(x), ctypes.c_double(L), c[0], c[1], c[2], _ptr(w), _ptr(w64))
    assert np.all((w >= 0) & (w <= xmax))
    top = w64.astype(np.float32) > xmax
    assert np.all(w[top] == 0.0)
    err = np.abs(w[~top] - w64[~top])
    bound = np.spacing(w[~top]).astype(np.float64) * (0.5 + 1.0 / 32)
    assert not np.any(err > bound)


def test_cells_lie_in_the_list(host):
    """The cell of every coordinate, numbers or not, is one of the list's."""
    x = np.array([0.0, 4.999999999999999, 5.0, 30.0, np.nextafter(30.0, 0.0), np.nan, np.inf, -np.inf, -1e-300, 1e300])
    c64, c32 = np.empty(x.size, np.int32), np.empty(x.size, np.int32)
    host.cells(x.size, _ptr(x), ctypes.c_double(29.0 / 30.0), 29, _ptr(c64), _ptr(c32))
    for c in (c64, c32):
        assert np.all((c >= 0) & (c < 29)) and list(c[[0, 3]]) == [0, 28]


def test_grid_base_lies_in_the_grid(host):
    """FP64 grid base and fraction: inside the grid for every wrapped coordinate and for
    what is not a number (whose fraction is none either); a coordinate whose product
    with n/L rounds to n is stored as 0 with base 0."""
    L, n = 30.0, 96
    x = np.array([0.0, 1.0, np.nextafter(L, 0.0), np.nan, 29.9, 1e-300])
    assert x[2] * (n / L) >= n
    base, frac = np.empty(x.size, np.int32), np.empty(x.size)
    host.grid64(x.size, _ptr(x), ctypes.c_double(n / L), n, _ptr(base), _ptr(frac))
    assert list(base) == [0, 3, 0, 0, 95, 0] and x[2] == 0.0 and frac[2] == 0.0
    assert np.isnan(x[3]) and np.isnan(frac[3]) and np.all((frac[[0, 1, 4, 5]] >= 0) & (frac[[0, 1, 4, 5]] < 1))
