"""chem_get_state of few species (one launch, from page-locked memory) on either side of its limits:
4,096 slots, and the species whose positions fit the first working buffer (two thirds of the
capacity); no species, reacted ones between the live, arrays that are not wanted, arrays
smaller than the species, and nothing written past them."""
import ctypes

import numpy as np
import pytest

from harness import cuda_available
from paper_2509_03313_gb300 import chem, workloads as W
from test_gpu_state import _check, _config, _pulse

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not cuda_available(), reason="needs a CUDA GPU")]


def _p(a):
    return None if a is None else a.ctypes.data_as(ctypes.c_void_p)


def _state(ctx, rows, want=(True, True, True)):
    arrays = [np.full(rows + 5, 77, np.int32), np.full(rows + 5, 77, np.uint32), np.full((rows + 5, 3), 77.0)]
    total = np.full(1, -1, np.int64)
    st = chem.lib().chem_get_state(ctx, rows, *[_p(a if w else None) for a, w in zip(arrays, want)], _p(total))
    return st, arrays, int(total[0])


@pytest.mark.parametrize("precision", [chem.CHEM_FP64, chem.CHEM_FP32_LOCAL])
@pytest.mark.parametrize("n,cap", [(1, 64), (2000, 3000), (2011, 3000), (4095, 9000), (4096, 9000), (4097, 9000)])
def test_state_at_the_limits(n, cap, precision):
    cfg, keep = _config(n, precision, cap)
    types, xyz = _pulse(n, n)
    ctx = chem.chem_init(cfg)
    try:
        st, a, total = _state(ctx, 10)
        assert st == chem.CHEM_OK and total == 0 and all(np.all(v == 77) for v in a)
        chem.chem_inject_pulse(ctx, types, xyz, np.zeros(n))
        chem.chem_run_until(ctx, 1e-18)
        st, (t, i, x), total = _state(ctx, n)
        assert st == chem.CHEM_OK and total == n
        assert np.all(t[n:] == 77) and np.all(i[n:] == 77) and np.all(x[n:] == 77.0)
        _check(i[:n], t[:n], x[:n], types, xyz)
        for want in ((False, True, False), (True, False, True), (False, False, False)):
            st, b, total = _state(ctx, n, want)
            assert st == chem.CHEM_OK and total == n
            for v, ref, w in zip(b, (t, i, x), want):
                assert np.array_equal(v, ref if w else np.full_like(v, 77))
        m = n // 2
        st, (t2, i2, x2), total = _state(ctx, m)
        assert st == chem.CHEM_EINVAL and total == n
        assert np.array_equal(t2[:m], t[:m]) and np.array_equal(i2[:m], i[:m]) and np.array_equal(x2[:m], x[:m])
        assert np.all(t2[m:] == 77) and np.all(i2[m:] == 77) and np.all(x2[m:] == 77.0)
    finally:
        chem.chem_destroy(ctx)


@pytest.mark.parametrize("precision", [chem.CHEM_FP64, chem.CHEM_FP32_LOCAL])
def test_reacted_species_are_left_out(precision):
    wl = W.uniform_2000(seed=9, L=150.0, n_steps=16)
    s = wl.schedule
    cfg, keep = chem.make_config(wl.L, wl.D, wl.reactions, seed=4, precision=precision, dt_min=s.dt_min, dt_max=s.dt_max,
                                 capacity_species=8192, launch_mode=chem.CHEM_LAUNCH_PHASES)
    ctx = chem.chem_init(cfg)
    try:
        p = wl.pulses[0]
        chem.chem_inject_pulse(ctx, p.types, p.xyz, p.t_arrival, p.energy_eV)
        chem.chem_run_until(ctx, wl.t_end)  # (a whole graph of steps: the last reacted are still among the slots)
        counts = chem.chem_tally(ctx, 7, 9)["counts"]
        st, (t, i, _), total = _state(ctx, 8192)
        assert st == chem.CHEM_OK and total == counts.sum() < p.n
        assert np.array_equal(np.bincount(t[:total], minlength=7), counts) and np.unique(i[:total]).size == total
    finally:
        chem.chem_destroy(ctx)
