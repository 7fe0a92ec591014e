"""The fixed-point functions behind the FP64 mode's normals as the GPU evaluates them (its own
multiply-high, count of leading zeros, table reads and reciprocal square root seed), at the
bits they claim: sine and cosine of the double 2 pi (m / 2^53) and the radius with at least
58 bits before one rounding, the radius of the normals with the logarithm and the root each
rounded. Against long double (64 bits of significand or more); and the normals themselves
against the FP64 reference's."""
import math

import numpy as np
import pytest

import device_code
from harness import cuda_available
from oracle import sbs
from test_fixed_normals import _arguments

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not cuda_available(), reason="needs a CUDA GPU")]

SOURCE = """#include "phases.cuh"
using namespace chem;
__global__ void k_eval(long n, const unsigned long long* m, double* s, double* c, double* c1, double* r, double* rf) {
  for (long i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    fixedn::sincos_2pi(m[i], s[i], c[i]);
    c1[i] = fixedn::cos_2pi(m[i]);
    r[i] = fixedn::radius(m[i]);
    rf[i] = fixedn::radius_fp64(m[i]);
  }
}
__global__ void k_normals(long n, const uint32_t* id, uint32_t step, uint32_t k0, uint32_t k1, double* g) {
  for (long i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    gauss3_f64(id[i], step, k0, k1, g[3 * i], g[3 * i + 1], g[3 * i + 2]);
}
extern "C" int eval(long n, const unsigned long long* m, double* s, double* c, double* c1, double* r, double* rf) {
  Arrays a;
  const unsigned long long* dm = a.in(m, n);
  double *ds = a.out(s, n), *dc = a.out(c, n), *d1 = a.out(c1, n), *dr = a.out(r, n), *df = a.out(rf, n);
  if (a.err) return a.err;
  k_eval<<<256, 128>>>(n, dm, ds, dc, d1, dr, df);
  a.back(s, ds, n); a.back(c, dc, n); a.back(c1, d1, n); a.back(r, dr, n); a.back(rf, df, n);
  return a.err;
}
extern "C" int normals(long n, const uint32_t* id, long step, long k0, long k1, double* g) {
  Arrays a;
  const uint32_t* d = a.in(id, n);
  double* o = a.out(g, 3 * n);
  if (a.err) return a.err;
  k_normals<<<256, 128>>>(n, d, static_cast<uint32_t>(step), static_cast<uint32_t>(k0), static_cast<uint32_t>(k1), o);
  a.back(g, o, 3 * n);
  return a.err;
}
"""
BOUND = 2.0 ** -53 * (1 + 2.0 ** -5)  # 58 bits, then one rounding


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return device_code.load(tmp_path_factory.mktemp("normals"), SOURCE)


@pytest.mark.parametrize("kind", ["borders", "powers", "near_one", "random", "many"])
def test_device_functions_at_the_claimed_bits(lib, kind):
    m = np.random.default_rng(8).integers(0, 2 ** 53, 1_000_000).astype(np.uint64) if kind == "many" else _arguments(kind)
    s, c, c1, r, rf = (np.zeros(m.size) for _ in range(5))
    device_code.call(lib.eval, m.size, m, s, c, c1, r, rf)
    np.testing.assert_array_equal(c, c1)
    ld = np.longdouble
    t = (2.0 * math.pi * (m.astype(np.float64) * 2.0 ** -53)).astype(ld)
    with np.errstate(divide="ignore"):
        log = -np.log((m.astype(ld) + ld(1)) / ld(2) ** 53)
    for got, want, floor in ((s, np.sin(t), 2.0 ** -44), (c, np.cos(t), 2.0 ** -44), (r, np.sqrt(2 * log), 0.0)):
        over = np.abs(got.astype(ld) - want) - BOUND * np.maximum(np.abs(want), floor)
        assert over.max() <= 0, (m[int(over.argmax())], float(over.max()))
    want = np.sqrt(2.0 * log.astype(np.float64))
    assert np.all(np.abs(rf - want) <= 2.0 ** -51 * want)
    if kind in ("random", "many"):
        assert (rf == want).mean() >= 1.0 - 4 * 2.0 ** -5


def test_device_normals_equal_the_references(lib):
    ids = np.random.default_rng(9).integers(0, 2 ** 29 - 1, 200_000).astype(np.uint32)
    for step in (0, 7, 2 ** 31 + 5):
        key = sbs.philox_key(0xABCDEF0123456789 + step, 5)
        g = np.zeros((ids.size, 3))
        device_code.call(lib.normals, ids.size, ids, step, key[0], key[1], g)
        want = sbs.gaussians(ids, step, key)
        # each factor within 2 units of a double evaluation's, the product rounded
        assert np.all(np.abs(g - want) <= 2.0 ** -50 * np.maximum(np.abs(want), 2.0 ** -40))
        assert (g == want).mean() > 0.8
