"""The radius of the FP64 mode's normals, compiled for the host: sqrt(-2 ln u) with the logarithm
and the root each rounded to double, as an FP64 evaluation rounds them. Before the roundings
both carry at least 58 bits, so against correctly rounded steps (160-bit arithmetic between
them) a result differs only where a value lies within 2^-5 units of a rounding border: by
one unit of the logarithm or of the root, and in at most 2 x 2 x 2^-5 of random cases."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

from test_fixed_normals import _arguments

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = """#include "fixed_normals.cuh"
extern "C" void eval(const uint64_t* m, long n, double* r) {
  for (long i = 0; i < n; ++i) r[i] = chem::fixedn::radius_fp64(m[i]);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("radius")
    (d / "eval.cpp").write_text(SOURCE)
    so = str(d / "eval.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2509_03313_gb300", "csrc"), str(d / "eval.cpp"), "-o", so], check=True)
    return ctypes.CDLL(so)


@pytest.mark.parametrize("kind", ["borders", "powers", "near_one", "random"])
def test_logarithm_and_root_are_rounded_to_double(lib, kind):
    mp = pytest.importorskip("mpmath").mp
    m = _arguments(kind)
    r = np.zeros(m.size)
    lib.eval(m.ctypes.data_as(ctypes.c_void_p), ctypes.c_long(m.size), r.ctypes.data_as(ctypes.c_void_p))
    equal = 0
    with mp.workprec(160):
        for i, v in enumerate(m.tolist()):
            want = math.sqrt(-2.0 * float(mp.log(mp.mpf(v + 1) / 2 ** 53)))
            equal += int(r[i] == want)
            assert abs(r[i] - want) <= 2.0 ** -52 * want + 2.0 ** -52 * want, (v, r[i], want)
    if kind == "random":
        assert equal >= (1.0 - 4 * 2.0 ** -5) * m.size, (equal, m.size)
