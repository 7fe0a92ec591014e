"""The FP32 tier of the FP64 mode's pair search, which may only reject a pair that the FP64 test
rejects. Its two parts, compiled from the library's device header: the start distance formed
from truncated displacements lies within its margin of the exact one, also where two large
displacements nearly cancel; and a pair whose uniform lies just below its probability is not
rejected for any FP32 distances within the stated error of its own, from the smallest errors
to ones past a quarter of the reaction radius, for steps from 0.1 ps to 10 us."""
import numpy as np
import pytest

import device_code
from harness import cuda_available
from oracle import sbs
from paper_2509_03313_gb300 import workloads as W

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not cuda_available(), reason="needs a CUDA GPU")]

SOURCE = """#include "phases.cuh"
using namespace chem;
__global__ void k_start(long n, const float* f, const double* ei, const double* ej, float* d0, float* margin) {
  for (long i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    d0[i] = start_distance_f32(f[3 * i], f[3 * i + 1], f[3 * i + 2], ei[3 * i], ei[3 * i + 1], ei[3 * i + 2],
                               ej[3 * i], ej[3 * i + 1], ej[3 * i + 2], margin[i]);
}
__global__ void k_reject(long n, const float* d0, const float* d1, const float* eps, const double* Rd, const double* ddt,
                         const uint32_t* lo, const uint32_t* hi, uint32_t step, uint32_t k0, uint32_t k1, uint8_t* out) {
  __shared__ Tables tb[8];
  __shared__ Train tr[8];
  Tables& t = tb[threadIdx.x];
  Train& r = tr[threadIdx.x];
  for (long i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    t.Rf[0] = static_cast<float>(Rd[i]);
    r.inv_ddt_f[0] = 1.0f / static_cast<float>(ddt[i]);
    r.step = step; r.key0 = k0; r.key1 = k1;
    out[i] = surely_rejected(d0[i], d1[i], eps[i], 0, t, r, lo[i], hi[i]) ? 1 : 0;
  }
}
extern "C" int start(long n, const float* f, const double* ei, const double* ej, float* d0, float* margin) {
  Arrays a;
  const float* df = a.in(f, 3 * n); const double *di = a.in(ei, 3 * n), *dj = a.in(ej, 3 * n);
  float *r = a.out(d0, n), *m = a.out(margin, n);
  if (a.err) return a.err;
  k_start<<<256, 128>>>(n, df, di, dj, r, m);
  a.back(d0, r, n); a.back(margin, m, n);
  return a.err;
}
extern "C" int reject(long n, const float* d0, const float* d1, const float* eps, const double* R, const double* ddt,
                      const uint32_t* lo, const uint32_t* hi, long step, long k0, long k1, uint8_t* out) {
  Arrays a;
  const float *p0 = a.in(d0, n), *p1 = a.in(d1, n), *e = a.in(eps, n);
  const double *r = a.in(R, n), *t = a.in(ddt, n);
  const uint32_t *l = a.in(lo, n), *h = a.in(hi, n);
  uint8_t* o = a.out(out, n);
  if (a.err) return a.err;
  k_reject<<<1024, 8>>>(n, p0, p1, e, r, t, l, h, static_cast<uint32_t>(step), static_cast<uint32_t>(k0),
                        static_cast<uint32_t>(k1), o);
  a.back(out, o, n);
  return a.err;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return device_code.load(tmp_path_factory.mktemp("rejection"), SOURCE)


@pytest.mark.parametrize("cancel", [0.0, 1e-3, 1e-6, 1.0])
def test_start_distance_is_within_its_margin(lib, cancel):
    rng = np.random.default_rng(5)
    n = 200_000
    f = (rng.normal(size=(n, 3)) * 10.0 ** rng.uniform(-3, 2, (n, 1))).astype(np.float32)
    size = 10.0 ** rng.uniform(-4, 5, (n, 1))
    ei = rng.normal(size=(n, 3)) * size
    ej = ei + cancel * rng.normal(size=(n, 3)) * size
    d0, margin = np.zeros(n, np.float32), np.zeros(n, np.float32)
    device_code.call(lib.start, n, f, ei, ej, d0, margin)
    x = f.astype(np.longdouble) - (ej.astype(np.longdouble) - ei.astype(np.longdouble))
    err = np.abs(d0.astype(np.longdouble) - np.sqrt((x * x).sum(1)))
    worst = int(np.argmax(err / margin))
    assert err[worst] <= margin[worst], (f[worst], ei[worst], ej[worst], float(err[worst]), margin[worst])


def _probability_one_side(d0, u, R, ddt):
    """The largest d1 with touch_probability(d0, d1) > u, by bisection (it falls as d1 grows)."""
    lo, hi = R.copy(), R + 60.0 * np.sqrt(ddt) + 2.0 * d0
    for _ in range(120):
        mid = 0.5 * (lo + hi)
        up = sbs.touch_probability(d0, mid, R, ddt) > u
        lo, hi = np.where(up, mid, lo), np.where(up, hi, mid)
    return lo


def test_no_pair_is_rejected_that_the_exact_test_accepts(lib):
    rng = np.random.default_rng(6)
    n, step, key = 400_000, 41, sbs.philox_key(0x123456789ABC, 3)
    DAB = np.array([W.D_NM2_S[r.a] + W.D_NM2_S[r.b] for r in W.WATER_REACTIONS])
    radii = np.array([sbs.reaction_radius(r.k_tab, d) for r, d in zip(W.WATER_REACTIONS, DAB)])
    r = rng.integers(0, DAB.size, n)
    R, ddt = radii[r], DAB[r] * 10.0 ** rng.uniform(-13, -5, n)
    lo = rng.integers(0, 1 << 28, n).astype(np.uint32)
    hi = (lo + 1 + rng.integers(0, 1 << 20, n)).astype(np.uint32)
    u = sbs.acceptance_uniform(lo, hi, step, key)
    s = np.sqrt(ddt)
    d0 = R * (1.0 + rng.uniform(0.0, 0.01, n)) + s * 10.0 ** rng.uniform(-3, 0.7, n)
    d1 = R + (_probability_one_side(d0, u, R, ddt) - R) * (1.0 - 1e-9)
    true_p = sbs.touch_probability(d0, d1, R, ddt)
    # errors from FP32 rounding up to 0.9 of the radius; the FP32 distances anywhere within them
    eps = np.maximum(R * 10.0 ** rng.uniform(-7, -0.05, n), 2e-7 * np.maximum(d0, d1)).astype(np.float32)
    pick = rng.choice([-0.999, 0.0, 0.5, 0.999], (2, n))
    f0, f1 = ((d + p * eps).astype(np.float32) for d, p in zip((d0, d1), pick))
    ok = (u < true_p) & (np.abs(f0 - d0) <= eps) & (np.abs(f1 - d1) <= eps) & (f0 > 0) & (f1 > 0)
    assert ok.sum() > 0.8 * n
    out = np.zeros(n, np.uint8)
    device_code.call(lib.reject, n, f0, f1, eps, R, ddt, lo, hi, step, key[0], key[1], out)
    bad = np.flatnonzero(ok & (out != 0))
    assert bad.size == 0, (bad.size, d0[bad[0]], d1[bad[0]], f0[bad[0]], f1[bad[0]], eps[bad[0]], R[bad[0]], ddt[bad[0]],
                           u[bad[0]], true_p[bad[0]])
    # and it does decide: pairs well past their probability with the search's usual errors
    far = d1 + 3.0 * s
    small = np.maximum(1e-5 * R, 2e-7 * np.maximum(d0, far)).astype(np.float32)
    device_code.call(lib.reject, n, d0.astype(np.float32), far.astype(np.float32), small, R, ddt, lo, hi, step, key[0],
                     key[1], out)
    sure = u > 1.1 * sbs.touch_probability(d0, far, R, ddt)
    assert out[sure].mean() > 0.9
