"""The arithmetic of the spatially ordered mixed force that host code can run
(csrc/far_rule.h), compiled and checked on the CPU.

Coordinates about a block's centre are rounded once: at most half a unit of
their last place from the exact difference (plus what the two parts of x leave
out, 2^-48 of x), and their errors have no mean beyond what so many uniform
errors leave (five standard deviations of 0.29 units / sqrt(count)), with x's
upper part cut toward zero as the integrator cuts it, and rounded as the force
call does."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_1205_2288_gb300 import inputs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1205_2288_gb300", "csrc")

WRAP = r"""
#include "far_rule.h"
extern "C" void about_n(long long n, const float* h, const float* l, float c,
                        float* out) {
  for (long long i = 0; i < n; ++i) out[i] = tsbts::about(h[i], l[i], c);
}
"""

FP = C.POINTER(C.c_float)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("far_rule")
    src, so = d / "w.cpp", d / "libw.so"
    src.write_text(WRAP)
    subprocess.run([cxx, "-std=c++17", "-O2", "-shared", "-fPIC", "-I", CSRC,
                    str(src), "-o", str(so)], check=True)
    L = C.CDLL(str(so))
    L.about_n.argtypes = [C.c_longlong, FP, FP, C.c_float, FP]
    return L


def _split(x, cut):
    h = x.astype(np.float32)
    if cut:
        b = x.view(np.int64) & ~np.int64((1 << 29) - 1)
        h = b.view(np.float64).astype(np.float32)
    return h, (x - h).astype(np.float32)


def _about(lib, h, l, c):
    out = np.empty_like(h)
    lib.about_n(len(h), h.ctypes.data_as(FP), l.ctypes.data_as(FP), c,
                out.ctypes.data_as(FP))
    return out


@pytest.mark.parametrize("cut", [True, False])
@pytest.mark.parametrize("c,shift", [(0.3141, 0.0), (-1.7, 0.0), (0.0, 0.0),
                                     (1e-3, 0.0), (101.25, 100.0),
                                     (-3000.6, -3000.0)])
def test_one_rounding(lib, cut, c, shift):
    x = inputs.plummer(65536, 3)[1].ravel() + shift
    c = np.float32(c)
    h, l = _split(x, cut)
    got = _about(lib, h, l, c).astype(np.float64)
    want = x - np.float64(c)
    unit = np.spacing(np.abs(want).astype(np.float32)).astype(np.float64)
    err = got - want
    assert (np.abs(err) <= 0.5 * unit * (1 + 1e-6) +
            2.0 ** -48 * np.abs(x)).all()
    toward = (err / unit) * np.sign(x)
    assert abs(toward.mean()) < 5 * 0.29 / np.sqrt(len(x))
