"""exp_df (csrc/sg_exp_df.h), the exponential of the sampled coefficients,
compiled for the host against the extended-precision exponential."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2310_14649_gb300", "csrc")
SOURCE = """
#include "sg_exp_df.h"
extern "C" void run(const double* a, float* out, long n) {
  for (long i = 0; i < n; ++i) {
    const float h = float(a[i]);
    out[i] = sg::exp_df(h, float(a[i] - double(h)));
  }
}
"""


@pytest.fixture(scope="module")
def exp_df(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("exp_df")
    (d / "e.cpp").write_text(SOURCE)
    so = str(d / "e.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC,
                    str(d / "e.cpp"), "-o", so], check=True)
    lib = ctypes.CDLL(so)

    def f(a):
        a = np.ascontiguousarray(a, dtype=np.float64)
        out = np.empty(a.shape, dtype=np.float32)
        lib.run(a.ctypes.data_as(ctypes.c_void_p), out.ctypes.data_as(ctypes.c_void_p), ctypes.c_long(a.size))
        return out
    return f


def test_normal_results_within_the_stated_bound(exp_df):
    r = np.random.default_rng(7)
    ln2 = np.log(2.0)
    a = np.concatenate([r.uniform(-60, 60, 1000000), r.uniform(-87, 88.7, 300000), r.uniform(-1, 1, 300000),
                        # both ends of every reduction interval
                        ((np.arange(-125, 127) + 0.5) * ln2)[:, None].repeat(400, 1).ravel()
                        + r.uniform(-1e-5, 1e-5, 252 * 400),
                        np.arange(-125, 128) * ln2, [0.0, 1e-30, -1e-30]])
    y = exp_df(a)
    exact = np.exp(a.astype(np.longdouble))
    ulp = np.spacing(exact.astype(np.float32)).astype(np.longdouble)
    below = exact < exact.astype(np.float32)          # a result just under a power of two has the smaller spacing
    ulp = np.where(below, np.spacing(np.nextafter(exact.astype(np.float32), np.float32(0))), ulp)
    assert np.max(np.abs(y.astype(np.longdouble) - exact) / ulp) <= 0.556


def test_ends_of_the_range(exp_df):
    y = exp_df(np.array([89.0, 99.9, 100.0, 1e30, np.inf, -110.5, -1e30, -np.inf, -104.0, np.nan]))
    assert np.all(np.isposinf(y[:5])) and np.all(y[5:9] == 0.0) and np.isnan(y[9])
    sub = np.linspace(-103.0, -88.0, 2001)            # subnormal results: one more rounding
    assert np.max(np.abs(exp_df(sub).astype(np.float64) - np.exp(sub))) <= 1.06 * 2.0 ** -149
