"""The bracket of the fit's MAD (csrc/fit_bracket.h), compiled for the host: usable for every
distance that FP32 resolves around the median, whatever its size, and refused otherwise."""
import ctypes
import os
import struct
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "fit_bracket.h"
extern "C" int bracket(unsigned top, double med, double *out) {
  return vr::dist_bracket(top, med, out, out + 1, out + 2);
}
"""


@pytest.fixture(scope="module")
def bracket(tmp_path_factory):
    d = tmp_path_factory.mktemp("bracket")
    src, so = d / "b.cpp", d / "b.so"
    src.write_text(SRC)
    inc = os.path.join(ROOT, "paper_1902_01010_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", inc, str(src), "-o", str(so)], check=True)
    f = ctypes.CDLL(str(so)).bracket
    f.argtypes = [ctypes.c_uint, ctypes.c_double, ctypes.POINTER(ctypes.c_double)]

    def call(dist, med):
        out = (ctypes.c_double * 3)()
        ok = f(struct.unpack("<I", struct.pack("<f", dist))[0] >> 9, med, out)
        return bool(ok), list(out)

    return call


@pytest.mark.parametrize("dist", [1e-30, 0.03, 0.99, 1.0, 1.0001, 3.7, 1e4, 1e30, 3.3e36])
def test_usable_for_every_size_of_distance(bracket, dist):
    rng = np.random.default_rng(1)
    for med in dist * np.r_[0.0, rng.uniform(-50, 50, 20)]:
        ok, (lo, hi, err) = bracket(dist, med)
        assert ok, med
        # members whose FP32 distance has this key: the exact distance lies inside
        mf = np.float32(med)
        x = (mf + np.float32(dist) * (1 + rng.uniform(-2e-4, 2e-4, 500)).astype(np.float32)).astype(np.float32)
        df = np.abs(x - mf)
        same = (df.view(np.uint32) >> 9) == (np.float32(dist).view(np.uint32) >> 9)
        d = np.abs(x[same].astype(np.float64) - med)
        assert same.any() and (lo < d).all() and (d < hi).all()


def test_refused_at_infinity_and_where_fp32_does_not_resolve_the_distance(bracket):
    assert not bracket(float("inf"), 0.0)[0]
    assert not bracket(3.4028e38, 0.0)[0]  # the last slice below infinity has an infinite end
    for dist in (1e-3, 1.0, 50.0):
        assert not bracket(dist, 1000 * dist)[0]
    assert not bracket(0.0, 1.0)[0]
