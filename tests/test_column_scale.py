"""The fp16 projection's column scale (csrc/column_scale.cuh), compiled for the
host: finite, with a finite product with the weights' scale and a normal
reciprocal, for every column maximum from the smallest denormal to the largest
float and every weight scale a plan can have (2^8 to 2^41: at least one order
and node of weight 2 or less, at most 65536 nodes of 2048 angles)."""

import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2304_14492_gb300", "csrc")


@pytest.fixture(scope="module")
def column_scale(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("scale")
    (d / "s.cpp").write_text('#include "column_scale.cuh"\n'
                             'extern "C" float scale(float m, float a) { return zm::column_scale(m, a); }\n')
    lib = str(d / "s.so")
    subprocess.run([cxx, "-O2", "-shared", "-fPIC", "-I" + CSRC, str(d / "s.cpp"), "-o", lib], check=True)
    f = ctypes.CDLL(lib).scale
    f.restype, f.argtypes = ctypes.c_float, [ctypes.c_float, ctypes.c_float]
    return f


def test_every_exponent(column_scale):
    for ka in range(8, 42):
        for e in range(-149, 128):
            for frac in (1.0, 1.0 + 2.0 ** -23, 1.5, 2.0 - 2.0 ** -23):
                mx = float(np.float32(frac * 2.0 ** e))
                s = column_scale(mx, 2.0 ** ka)
                m, k = np.frexp(s)
                assert m == 0.5 and np.isfinite(s)                       # a power of two
                prod = np.float32(s) * np.float32(2.0 ** ka)
                assert np.isfinite(prod) and 2.0 ** -126 <= np.float32(1) / prod < np.inf
                assert mx * s < 2.0 ** 14
                assert mx * s >= 2.0 ** 13 or prod == 2.0 ** 126         # only the bound keeps it lower


@pytest.mark.parametrize("mx", [0.0, float("inf"), float("nan")])
def test_no_maximum_leaves_the_column(column_scale, mx):
    assert column_scale(mx, 2.0 ** 20) == 1.0
