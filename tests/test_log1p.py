"""log(1 + x) of the packed softplus (csrc/pfc_log1p.h), compiled for the host in FP32: at most 1 ulp
on [0, 1], as CUDA's log1pf is documented, and a mean error below a twentieth of an ulp (an error
that leans one way adds up over the voxels)."""
import ctypes
import os
import subprocess

import numpy as np

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2103_04856_gb300", "csrc")
SOURCE = r"""
#include <cmath>
#include "pfc_log1p.h"
struct Scalar {
    using V = float;
    static float c(float x) { return x; }
    static float fma(float a, float b, float x) { return std::fmaf(a, b, x); }
};
extern "C" void run(const float* x, float* y, long n)
{
    for (long i = 0; i < n; ++i) y[i] = pfc::log1p01<Scalar>(x[i]);
}
"""


def test_log1p_is_accurate_to_an_ulp(tmp_path):
    src, lib = tmp_path / "log1p.cpp", tmp_path / "liblog1p.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, str(src), "-o",
                    str(lib)], check=True)
    # every 64th float of [2^-30, 1], and the ends
    bits = np.arange(np.float32(2.0 ** -30).view(np.uint32), np.float32(1.0).view(np.uint32) + 1, 64, dtype=np.uint32)
    x = np.concatenate([[np.float32(0.0), np.float32(1.0)], bits.view(np.float32)])
    y = np.empty_like(x)
    f = ctypes.CDLL(str(lib)).run
    f(x.ctypes.data_as(ctypes.c_void_p), y.ctypes.data_as(ctypes.c_void_p), ctypes.c_long(x.size))
    want = np.log1p(x.astype(np.float64))
    assert y[0] == 0.0
    err = (y.astype(np.float64) - want)[1:] / np.spacing(want[1:].astype(np.float32)).astype(np.float64)
    assert np.abs(err).max() <= 1.0
    near = x[1:] > 2.0 ** -8          # below, x itself is the value to within the rounding
    assert abs(err[near].mean()) <= 0.05
