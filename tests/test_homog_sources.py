"""The rate equations divide by CUDA's own rounded operations, and their step-size factor
carries FP64 precision (its arithmetic compiled for the host against 80-bit arithmetic or more:
2^-52 relative within the limits that the factor is cut to)."""
import ctypes
import os
import re
import subprocess

import numpy as np
import pytest

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_03313_gb300", "csrc",
                      "homog.cu")


def _code():
    with open(SOURCE, encoding="utf-8") as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_reciprocals_are_rounded_ones():
    code = _code()
    assert "__frcp_rn" not in code and "hx_recip" not in code
    assert "__drcp_rn" in code


def test_step_size_factor_is_fp64(tmp_path):
    m = re.search(r"__device__ __forceinline__ (double hx_root\(.*?\n})", _code(), re.S)
    assert m, "no FP64 step-size factor"
    (tmp_path / "root.cpp").write_text(
        "#include <cmath>\nusing std::fma;\nconstexpr int HX_K = 6;\n%s\n"
        "extern \"C\" void roots(const double* a, const double* b, double* r, long n) {\n"
        "  for (long i = 0; i < n; ++i) r[i] = hx_root(a[i], b[i]);\n}\n" % m.group(1))
    so = str(tmp_path / "root.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", str(tmp_path / "root.cpp"),
                    "-o", so], check=True)
    rng = np.random.default_rng(4)
    sc = 10.0 ** rng.uniform(-8, 0, 100_000)
    x = np.concatenate([10.0 ** rng.uniform(-3.99, 3.99, 90_000), 10.0 ** rng.uniform(-60, -4.1, 5000),
                        10.0 ** rng.uniform(4.1, 25, 5000)])
    de, r = x * sc, np.zeros(x.size)
    at = lambda v: v.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    ctypes.CDLL(so).roots(at(de), at(sc), at(r), ctypes.c_long(x.size))
    mp = pytest.importorskip("mpmath").mp
    inside = np.abs(np.log10(x)) < 4.0
    with mp.workprec(100):
        for i in np.flatnonzero(inside)[::30]:
            want = (mp.mpf(de[i]) / mp.mpf(sc[i])) ** (mp.mpf(-1) / 6)
            assert abs(mp.mpf(r[i]) - want) <= mp.mpf(2) ** -52 * want
    assert np.all(r[~inside & (x < 1.0)] > 4.0 / 0.9) and np.all(r[~inside & (x > 1.0)] < 0.2 / 0.9)
    r0 = np.zeros(1)
    ctypes.CDLL(so).roots(at(np.zeros(1)), at(np.ones(1)), at(r0), ctypes.c_long(1))
    assert r0[0] > 4.0 / 0.9
