"""The FP64 logarithm of the small-lattice kernels (csrc/log64.cuh), compiled for the host and
compared with the logarithm in extended precision: the stated 1.2 units in the last place over the
exponent range, at both ends of every table interval, around 1 and where the exponent changes,
and log()'s own answers where the table does not apply."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0704_3444_gb300", "csrc")

SHIM = r"""
#include <cmath>
#include <cstring>
#include <cstdint>
#define __device__
#define __forceinline__ inline
struct Index { int x; };
static Index threadIdx{0}, blockDim{1};
static inline uint64_t bits_of(double x) { uint64_t b; std::memcpy(&b, &x, 8); return b; }
static inline int __double2hiint(double x) { return (int)(bits_of(x) >> 32); }
static inline int __double2loint(double x) { return (int)(uint32_t)bits_of(x); }
static inline double __hiloint2double(int hi, int lo)
{
    const uint64_t b = ((uint64_t)(uint32_t)hi << 32) | (uint32_t)lo;
    double x;
    std::memcpy(&x, &b, 8);
    return x;
}
static inline double __ldg(const double* p) { return *p; }
using std::fma;
using std::log;
#include "log64.cuh"
extern "C" void log64_of(const double* x, double* y, long n)
{
    static mclb::Log64Row tab[mclb::LOG64_ROWS];
    mclb::log64_load(tab);
    for (long k = 0; k < n; ++k) y[k] = mclb::log64(x[k], tab);
}
"""


@pytest.fixture(scope="module")
def log64(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx or np.finfo(np.longdouble).nmant < 63:
        pytest.skip("needs g++ and an extended precision")
    d = tmp_path_factory.mktemp("log64")
    (d / "cuda_runtime.h").write_text("")      # the header includes it for the device only
    (d / "shim.cpp").write_text(SHIM)
    lib = d / "log64.so"
    subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", str(d), "-I", CSRC,
                    str(d / "shim.cpp"), "-o", str(lib)], check=True)
    fn = ctypes.CDLL(str(lib)).log64_of
    dp = ctypes.POINTER(ctypes.c_double)

    def call(x):
        x = np.ascontiguousarray(x, dtype=np.float64)
        y = np.empty_like(x)
        fn(x.ctypes.data_as(dp), y.ctypes.data_as(dp), ctypes.c_long(x.size))
        return y

    return call


def _ulps(y, x):
    want = np.log(x.astype(np.longdouble))
    return np.abs((y.astype(np.longdouble) - want) / np.spacing(np.abs(want.astype(np.float64))))


def _ends():
    """Both ends of every interval of the table, and their neighbours, at a few exponents."""
    hi = 0x3FE61000 + (np.arange(129, dtype=np.int64) << 13)
    first = np.concatenate([(hi << 32) + d for d in (-2, -1, 0, 1, 2)])
    return np.concatenate([first + (np.int64(e) << 52) for e in (-1000, -3, -1, 0, 1, 3, 900)]).view(np.float64)


@pytest.mark.parametrize("values", ["range", "one", "ends", "density"])
def test_log64_error(log64, values):
    rng = np.random.default_rng(5)
    x = {"range": lambda: 2.0 ** rng.uniform(-1021, 1023, 200000) * rng.uniform(1.0, 1.99, 200000),
         "one": lambda: np.concatenate([1.0 + s * 2.0 ** rng.uniform(-52, -5, 200000) for s in (-1, 1)]),
         "ends": _ends,
         "density": lambda: rng.uniform(0.3, 3.0, 400000)}[values]()
    x = x[x != 1.0]
    assert np.max(_ulps(log64(x), x)) < 1.2


def test_log64_outside_the_table(log64):
    assert log64(np.array([1.0]))[0] == 0.0
    tiny = np.array([5e-324, 1e-310, 2.2250738585072009e-308, 2.2250738585072014e-308, np.finfo(np.float64).max])
    assert np.max(_ulps(log64(tiny), tiny)) < 1.2
    with np.errstate(all="ignore"):
        y = log64(np.array([0.0, -0.0, -1.0, -1e-310, -np.inf, np.inf, np.nan]))
    assert y[0] == y[1] == -np.inf and y[5] == np.inf
    assert np.all(np.isnan(y[[2, 3, 4, 6]]))
