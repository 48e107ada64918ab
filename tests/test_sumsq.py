"""Sum of squares in two FP32 words (csrc/sumsq.cuh), the norms of the GMRES vector kernels."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def sumsq(tmp_path_factory):
    d = tmp_path_factory.mktemp("sumsq")
    (d / "s.cpp").write_text('#include "sumsq.cuh"\nextern "C" double s(const float* x, int n) '
                             "{ SumSq q; for (int i = 0; i < n; ++i) q.add(x[i]); return q.value(); }\n")
    so = str(d / "s.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC",
                    "-I" + os.path.join(ROOT, "paper_1309_5994_gb300", "csrc"), str(d / "s.cpp"), "-o", so], check=True)
    lib = ctypes.CDLL(so)
    lib.s.restype = ctypes.c_double
    lib.s.argtypes = [ctypes.POINTER(ctypes.c_float), ctypes.c_int]
    return lambda x: lib.s(x.ctypes.data_as(ctypes.POINTER(ctypes.c_float)), len(x))


@pytest.mark.parametrize("n", [1, 2, 8, 16, 24, 400])
@pytest.mark.parametrize("span", [0.0, 3.0])
def test_sum_of_squares_keeps_more_than_fp32(sumsq, n, span):
    """n roundings of the low word at 2^-24 of 2^-24: n 2^-46 of the sum, far below FP32's 2^-24 an addition."""
    r = np.random.default_rng(n)
    x = (r.standard_normal(n) * 10.0 ** r.uniform(-span, 0.0, n)).astype(np.float32)
    want = float(sum(float(v) * float(v) for v in x))
    assert abs(sumsq(x) - want) <= n * 2.0 ** -46 * want
