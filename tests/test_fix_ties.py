"""Rounding of fixed-point populations to FP16 (csrc/kbc_fix.cuh by way of FP32, rounded to odd):
ties go to even, as the FP16 storage's rounding is stated."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1507_02518_gb300", "csrc")
WRAP = r'''
#define __host__
#define __device__
#define __forceinline__ inline
#include "kbc_fix.cuh"
extern "C" void to_odd(int n, const long long* v, float* o) {
  for (int k = 0; k < n; ++k) o[k] = kbc::fix::to_f32_odd<2>(v[k]);
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("ties")
    (d / "wrap.cpp").write_text(WRAP)
    so = str(d / "ties.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared",
                    "-I" + CSRC, str(d / "wrap.cpp"), "-o", so], check=True)
    return ctypes.CDLL(so)


def halves(lib, v):
    v = np.ascontiguousarray(v, dtype=np.int64)
    o = np.empty(len(v), np.float32)
    lib.to_odd(len(v), v.ctypes.data_as(ctypes.c_void_p), o.ctypes.data_as(ctypes.c_void_p))
    return o.astype(np.float16)


@pytest.mark.parametrize("k", range(38, 51))
def test_ties_go_to_even(lib, k):
    """12-bit numbers at every place of the format (normal halves): odd ones are ties."""
    m = np.arange(2 ** 11, 2 ** 12, dtype=np.int64)
    for v in (m << k, -(m << k)):
        want = (v.astype(np.float64) * 2.0 ** -62).astype(np.float16)  # exact in FP64
        assert np.array_equal(halves(lib, v), want)
        # a unit beside a tie is no tie
        for d in (-1, 1):
            got = halves(lib, v + d)
            near = np.where(m % 2 == 0, want,
                            ((v + d * 2.0 ** (k - 1)) * 2.0 ** -62).astype(np.float16))
            assert np.array_equal(got, near)
