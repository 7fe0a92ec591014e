"""The fixed-point functions behind the FP64 mode's normals, compiled for the host, against
160-bit arithmetic: sine and cosine of the double 2 pi (m / 2^53) and sqrt(-2 ln((m + 1) /
2^53)) at octant borders, at both ends, at powers of two, close to u = 1 and at random. Each
result has at least 58 correct bits before one rounding to 53: relative error at most
2^-53 (1 + 2^-5), except for a sine or cosine below 2^-44, where the rounding of the angle is
added in double: at most that of 2^-44."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = """#include "fixed_normals.cuh"
extern "C" void eval(const uint64_t* m, long n, double* s, double* c, double* c1, double* r) {
  using namespace chem::fixedn;
  for (long i = 0; i < n; ++i) { sincos_2pi(m[i], s[i], c[i]); c1[i] = cos_2pi(m[i]); r[i] = radius(m[i]); }
}
"""


def _arguments(kind):
    top = 2 ** 53
    if kind == "borders":
        m = [k * 2 ** 49 + d for k in range(17) for d in (-2, -1, 0, 1, 2)]
    elif kind == "powers":
        m = [v for k in range(54) for v in (2 ** k - 1, 2 ** k, top - 2 ** k, top - 1 - 2 ** k)]
    elif kind == "near_one":
        m = [int(top * x) for x in np.linspace(0.98, 1.0, 1500, endpoint=False)]
    else:
        m = np.random.default_rng(3).integers(0, top, 4000).tolist()
    return np.array(sorted({int(v) for v in m if 0 <= v < top}), np.uint64)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed_normals")
    (d / "eval.cpp").write_text(SOURCE)
    so = str(d / "eval.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2509_03313_gb300", "csrc"), str(d / "eval.cpp"), "-o", so], check=True)
    return ctypes.CDLL(so)


@pytest.mark.parametrize("kind", ["borders", "powers", "near_one", "random"])
def test_against_160_bits(lib, kind):
    mp = pytest.importorskip("mpmath").mp
    m = _arguments(kind)
    s, c, c1, r = (np.zeros(m.size) for _ in range(4))
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    lib.eval(p(m), ctypes.c_long(m.size), p(s), p(c), p(c1), p(r))
    assert np.array_equal(c, c1)
    bound = 2.0 ** -53 * (1 + 2.0 ** -5)
    with mp.workprec(160):
        for i, v in enumerate(m.tolist()):
            t = mp.mpf(2.0 * math.pi * (v * 2.0 ** -53))
            want = [mp.sin(t), mp.cos(t),
                    mp.sqrt(-2 * mp.log(mp.mpf(v + 1) / 2 ** 53))]
            for name, got, ex in zip("scr", (s[i], c[i], r[i]), want):
                floor = 0.0 if name == "r" else 2.0 ** -44
                assert abs(mp.mpf(got) - ex) <= bound * max(abs(ex), floor), (name, v, got, ex)
