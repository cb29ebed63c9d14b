"""The arithmetic of the spatially ordered mixed force that host code can run
(csrc/far_rule.h), compiled and checked on the CPU.

Coordinates about a block's centre are rounded once: at most half a unit of
their last place from the exact difference (plus what the two parts of x leave
out, 2^-48 of x), and their errors have no mean beyond what so many uniform
errors leave (five standard deviations of 0.29 units / sqrt(count)), with x's
upper part cut toward zero as the integrator cuts it, and rounded as the force
call does.

The split of a coordinate in ordered runs has its upper part rounded to nearest
and is exact to 2^-49. With it the distances of both forms of a pair, the
double-single difference and the one about a centre, have the same mean: none
beyond 5e-10 of the distance, where 300,000 pairs leave 1.2e-10 of their 3e-8
each (four standard deviations, both forms; cut upper parts leave 3e-9).

The curve's cells are the bodies' own: a Plummer sphere that was moved has as
many far pairs of a warp's bodies and a subtile as one about the coordinate
origin (within a tenth; the cells' edges lie elsewhere), also with a body far
outside."""
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
extern "C" void split_n(long long n, const double* x, float* h, float* l) {
  for (long long i = 0; i < n; ++i) tsbts::split_round(x[i], h[i], l[i]);
}
extern "C" void sample_n(int n, int* out) {
  for (int k = 0; k < tsbts::kCentreSample; ++k)
    out[k] = tsbts::centre_sample(k, n);
}
extern "C" void keys_n(long long n, const float* x, float scale,
                       unsigned* out) {
  for (long long i = 0; i < n; ++i)
    out[i] = tsbts::hilbert(tsbts::curve_cell(x[3 * i], scale),
                            tsbts::curve_cell(x[3 * i + 1], scale),
                            tsbts::curve_cell(x[3 * i + 2], scale));
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
    L.split_n.argtypes = [C.c_longlong, C.POINTER(C.c_double), FP, FP]
    L.sample_n.argtypes = [C.c_int, C.POINTER(C.c_int)]
    L.keys_n.argtypes = [C.c_longlong, FP, C.c_float, C.POINTER(C.c_uint32)]
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


def _split_round(lib, x):
    x = np.ascontiguousarray(x)
    h, l = np.empty(x.shape, np.float32), np.empty(x.shape, np.float32)
    lib.split_n(x.size, x.ctypes.data_as(C.POINTER(C.c_double)),
                h.ctypes.data_as(FP), l.ctypes.data_as(FP))
    return h, l


def test_split_rounds_to_nearest(lib):
    g = np.random.default_rng(4)
    x = g.choice([-1.0, 1.0], 200000) * 2.0 ** g.uniform(-70, 100, 200000)
    x[:4] = [1.0, -1.0, 1.0 + 2.0 ** -24, np.nextafter(2.0, 0.0)]
    h, l = _split_round(lib, x)
    unit = np.spacing(np.abs(x).astype(np.float32)).astype(np.float64)
    assert (np.abs(h - x) <= 0.5 * unit).all()
    assert (np.abs(h.astype(np.float64) + l - x) <=
            2.0 ** -49 * np.abs(x)).all()
    assert (h[4:] == x[4:].astype(np.float32)).all()


def test_both_forms_of_a_pair_have_the_same_mean(lib):
    r = inputs.plummer(36864, 1)[1]
    h, l = _split_round(lib, r)
    g = np.random.default_rng(0)
    err = {"near": [], "far": []}
    while len(err["far"]) < 75:
        d2 = ((r - r[g.integers(len(r))]) ** 2).sum(1)
        block = np.argsort(d2)[:256]
        lo, hi = h[block].min(0), h[block].max(0)
        cen = np.float32(0.5) * (lo + hi)
        rho2 = ((hi - lo).astype(np.float64) ** 2).sum() / 4
        j = np.flatnonzero(d2 > 6.25 * rho2)
        if len(j) < 1000:
            continue
        j, i = g.choice(j, 4000), g.choice(block, 4000)
        d = r[j] - r[i]
        far = np.stack([_about(lib, np.ascontiguousarray(h[:, k]),
                               np.ascontiguousarray(l[:, k]), cen[k])
                        for k in range(3)], 1)
        for name, x in (("near", (h[j] - h[i]) + (l[j] - l[i])),
                        ("far", far[j] - far[i])):
            err[name].append((((x - d) * d).sum(1) / (d * d).sum(1)).mean())
    for name, e in err.items():
        assert abs(np.mean(e)) < 5e-10, (name, np.mean(e))


def spatial_order(lib, r):
    """Bodies along the curve, as launch_spatial_order lists them."""
    n = len(r)
    pick = np.empty(1024, np.int32)
    lib.sample_n(n, pick.ctypes.data_as(C.POINTER(C.c_int)))
    assert (np.diff(pick) > 0).all() and pick[0] >= 0 and pick[-1] < n
    x = np.ascontiguousarray((r - np.sort(r[pick], 0)[512]), np.float32)
    scale = 0.5 * np.abs(x).sum() / n
    key = np.empty(n, np.uint32)
    lib.keys_n(n, x.ctypes.data_as(FP), scale,
               key.ctypes.data_as(C.POINTER(C.c_uint32)))
    return np.lexsort((np.arange(n), key))


def far_fraction(r, order):
    """Pairs of a warp's 64 bodies and a subtile of 32 that are further apart
    than the radius of the block's 256 bodies (all bodies active)."""
    x = r[order][:len(r) // 256 * 256]
    box = [(f(x.reshape(-1, k, 3), 1)) for k in (32, 64, 256)
           for f in (np.min, np.max)]
    jl, jh, wl, wh, bl, bh = box
    rho2 = np.repeat(((bh - bl) ** 2).sum(1) / 4, 4)
    far = 0
    for w in range(0, len(wl), 8):
        gap = np.maximum(0, np.maximum(jl - wh[w], wl[w] - jh))
        far += ((gap ** 2).sum(1) > rho2[w]).mean()
    return far / len(range(0, len(wl), 8))


@pytest.mark.parametrize("shift", [10.0, 100.0, 3000.0, 1e6])
def test_order_does_not_depend_on_the_origin(lib, shift):
    r = inputs.plummer(65536, 3)[1]
    r[77] = [1e5, -3e4, 2e4]
    want = far_fraction(r, spatial_order(lib, r))
    moved = r + shift * np.array([1.0, -0.6, 0.3])
    got = far_fraction(moved, spatial_order(lib, moved))
    assert want > 0.4 and got > 0.9 * want, (want, got)
