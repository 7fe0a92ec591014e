"""chem_get_state's packing on the device: around its chunks of 1,024 slots, with the positions
spread over its buffers (a context filled to its capacity), with a caller's arrays smaller
than the species, and for single trains of a batch. One step of 1e-18 s moves no species by
more than 0.01 nm, so every position is known."""
import ctypes

import numpy as np
import pytest

from harness import cuda_available
from paper_2509_03313_gb300 import chem, workloads as W

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not cuda_available(), reason="needs a CUDA GPU")]
L = 500.0


def _config(n, precision, cap, train_id=0):
    return chem.make_config(L, W.D_NM2_S, [], seed=3, train_id=train_id, precision=precision, dt_min=1e-18,
                            dt_max=1e-18, capacity_species=cap, capacity_pending=n)


def _pulse(n, seed):
    rng = np.random.default_rng(seed)
    return rng.integers(0, 7, n).astype(np.int32), rng.uniform(-0.5 * L, 0.5 * L, (n, 3))


def _check(ids, types, xyz, want_types, want_xyz):
    o = np.argsort(ids)
    assert np.array_equal(ids[o], np.arange(want_types.size))
    assert np.array_equal(types[o], want_types)
    d = xyz[o] - want_xyz
    assert np.abs(d - L * np.round(d / L)).max() < 0.01


@pytest.mark.parametrize("precision", [chem.CHEM_FP64, chem.CHEM_FP32_LOCAL])
@pytest.mark.parametrize("n,cap", [(1, 1), (1023, 4096), (1024, 1024), (1025, 1100), (5000, 5000)])
def test_packed_state(n, cap, precision):
    cfg, keep = _config(n, precision, cap)
    types, xyz = _pulse(n, n)
    ctx = chem.chem_init(cfg)
    try:
        chem.chem_inject_pulse(ctx, types, xyz, np.zeros(n))
        chem.chem_run_until(ctx, 1e-18)
        i, t, x = chem.chem_get_state(ctx)
        _check(i, t, x, types, xyz)
        m = n // 2 + 1  # room for fewer: the first ones, and CHEM_EINVAL when there are more
        ids, ty, pos, total = np.zeros(m, np.uint32), np.zeros(m, np.int32), np.zeros((m, 3)), np.zeros(1, np.int64)
        p = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
        st = chem.lib().chem_get_state(ctx, m, p(ty), p(ids), p(pos), p(total))
        assert st == (chem.CHEM_OK if m >= n else chem.CHEM_EINVAL) and total[0] == n
        assert np.array_equal(ids, i[:m]) and np.array_equal(ty, t[:m]) and np.array_equal(pos, x[:m])
    finally:
        chem.chem_destroy(ctx)


def test_packed_state_of_the_trains_of_a_batch():
    sizes = [3, 1500, 0, 700]
    cfgs, keep = zip(*(_config(max(n, 1), chem.CHEM_FP32_LOCAL, n + 10, b) for b, n in enumerate(sizes)))
    ctx = chem.chem_batch_init(cfgs)
    try:
        pulses = [_pulse(n, 90 + b) for b, n in enumerate(sizes)]
        for b, (t, x) in enumerate(pulses):
            chem.chem_batch_inject(ctx, b, t, x, np.zeros(t.size))
        # trains 0 and 1 stop first and are parked while the others go on
        for ends in ([1e-18] * 4, [1e-18, 1e-18, 3e-18, 3e-18]):
            chem.chem_batch_run_until(ctx, ends)
            for b, (t, x) in enumerate(pulses):
                if t.size:
                    _check(*chem.chem_batch_get_state(ctx, b), t, x)
    finally:
        chem.chem_destroy(ctx)
