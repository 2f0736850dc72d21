"""The FP32-pair Box-Muller draw of csrc/noise.cuh (host build of the same source) against extended precision: random
53-bit uniforms, uniforms at both ends of the logarithm, and angles around every quarter turn."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2605_27231_gb300", "csrc")

WRAP = """
#define __host__
#define __device__
#define __forceinline__ inline
#include "noise.cuh"
extern "C" void draw(const uint64_t* a, const uint64_t* b, long n, float* g, float* r, float* c) {
  for (long i = 0; i < n; ++i) {
    g[i] = sigw::gauss_f32(a[i], b[i]);
    const sigw::ff x = sigw::ff_radius(a[i] + 1), y = sigw::ff_cos_turn(b[i]);
    r[2 * i] = x.h; r[2 * i + 1] = x.l;
    c[2 * i] = y.h; c[2 * i + 1] = y.l;
  }
}
"""


@pytest.fixture(scope="module")
def draw(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("noise")
    (d / "w.cpp").write_text(WRAP)
    so = str(d / "w.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, str(d / "w.cpp"), "-o", so],
                   check=True)
    lib = ctypes.CDLL(so)

    def f(a, b):
        n = len(a)
        a, b = (np.ascontiguousarray(x, dtype=np.uint64) for x in (a, b))
        g, r, c = np.zeros(n, np.float32), np.zeros((n, 2), np.float32), np.zeros((n, 2), np.float32)
        lib.draw(*(x.ctypes.data_as(ctypes.c_void_p) for x in (a, b)), ctypes.c_long(n),
                 *(x.ctypes.data_as(ctypes.c_void_p) for x in (g, r, c)))
        return g, r.astype(np.longdouble).sum(1), c.astype(np.longdouble).sum(1)

    return f


def _exact(a, b):
    one = np.longdouble(1)
    pi = np.longdouble("3.14159265358979323846264338327950288")
    # 1 - u1 is an integer over 2^53: log1p keeps the digits where u1 is near one
    c = (np.uint64(2 ** 53 - 1) - a).astype(np.longdouble) / 2 ** 53
    u1 = one - c
    ln = np.where(c < 0.5, np.log1p(-c), np.log(u1))
    quad = ((b + np.uint64(1 << 50)) >> np.uint64(51)).astype(np.int64)
    ang = (b.astype(np.int64) - (quad << 51)).astype(np.longdouble) * (2 * pi / 2 ** 53)
    cos = np.select([quad == 1, quad == 2, quad == 3], [-np.sin(ang), -np.cos(ang), np.sin(ang)], np.cos(ang))
    return np.sqrt(-2 * ln), cos


@pytest.mark.parametrize("which", ["random", "near one", "near zero", "quarter turns"])
def test_pair_draw_matches_extended_precision(draw, which):
    rng = np.random.default_rng(11)
    n = 200000
    a = rng.integers(0, 2 ** 53, n, dtype=np.uint64)
    b = rng.integers(0, 2 ** 53, n, dtype=np.uint64)
    small = rng.integers(0, 2 ** 53, n, dtype=np.uint64) >> rng.integers(0, 53, n, dtype=np.uint64)
    small[:3] = 0, 1, 2
    if which == "near one":
        a = np.uint64(2 ** 53 - 1) - small
    elif which == "near zero":
        a = small
    elif which == "quarter turns":
        off = (small >> np.uint64(3)).astype(np.int64) * rng.choice((-1, 1), n)
        b = ((rng.integers(0, 4, n) << 51) + off) % 2 ** 53
        b = b.astype(np.uint64)
    g, r, c = draw(a, b)
    R, C = _exact(a, b)
    assert np.all(np.abs(r - R) <= 2.0 ** -30 * np.abs(R))
    assert np.all(np.abs(c - C) <= 2.0 ** -30 * np.abs(C))
    # the rounded product: half an ulp, and the two pairs' errors
    ulp = np.spacing(np.abs((R * C).astype(np.float32))).astype(np.longdouble)
    assert np.all(np.abs(g - R * C) <= 0.52 * ulp + 2.0 ** -149)
