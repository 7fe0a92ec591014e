"""The pending queue over several injections: behind what is pending (appended where it lies),
before it, among it and at equal arrivals (merged), after a release, with the queue's room used
up so that it moves to the front, with a refused pulse in between, and past its capacity.
Species get their ids in release order: by arrival, then earlier calls first, then by index.
The whole run lasts 1e-16 s, in which no species moves by more than 0.01 nm."""
import numpy as np
import pytest

from harness import cuda_available
from paper_2509_03313_gb300 import chem, workloads as W

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not cuda_available(), reason="needs a CUDA GPU")]
L = 500.0
U = 1e-18  # unit of the arrival times


class Queue:
    """One train and the queue it should have."""

    def __init__(self, ctx, b, seed):
        self.ctx, self.b, self.rng, self.items = ctx, b, np.random.default_rng(seed), []

    def inject(self, t):
        t = np.asarray(t, np.float64) * U
        types = self.rng.integers(0, 7, t.size).astype(np.int32)
        xyz = self.rng.uniform(-0.5 * L, 0.5 * L, (t.size, 3))
        chem.chem_batch_inject(self.ctx, self.b, types, xyz, t)
        self.items += list(zip(t, types, xyz))

    def check(self, released):
        want = sorted(self.items, key=lambda s: s[0])  # (stable: call order, then index)
        ids, types, xyz = chem.chem_batch_get_state(self.ctx, self.b)
        o = np.argsort(ids)
        assert np.array_equal(ids[o], np.arange(released))
        assert np.array_equal(types[o], [s[1] for s in want[:released]])
        if released:
            d = xyz[o] - np.array([s[2] for s in want[:released]])
            assert np.abs(d - L * np.round(d / L)).max() < 0.01


@pytest.mark.parametrize("n", [5, 3000])
def test_queue_order_over_injections(n):
    cap = 4 * n  # of the queue
    cfgs, keep = zip(*(chem.make_config(L, W.D_NM2_S, [], seed=3, train_id=b, precision=chem.CHEM_FP64, dt_min=U,
                                        dt_max=U, capacity_species=8 * n, capacity_pending=cap) for b in range(2)))
    ctx = chem.chem_batch_init(cfgs)
    try:
        a, other = Queue(ctx, 0, 1), Queue(ctx, 1, 2)
        other.inject(np.full(n, 60))
        a.inject(np.zeros(n))
        a.inject(np.linspace(2, 20, n))          # behind it
        a.inject(np.linspace(20, 2, n))          # out of order, among it, one equal arrival
        chem.chem_batch_run_until(ctx, [U, U])   # n are released
        a.check(n)
        a.inject(np.linspace(30, 40, n))         # behind it, fills the queue's room
        with pytest.raises(chem.ChemError):      # refused: the last one lies outside the volume
            chem.chem_batch_inject(ctx, 0, np.zeros(n, np.int32), np.r_[np.zeros((n - 1, 3)), [[L, 0, 0]]],
                                   np.full(n, 50 * U))
        a.inject(np.linspace(40, 45, n))         # behind it, no room there: moves to the front
        a.check(n)
        chem.chem_batch_run_until(ctx, [100 * U, 100 * U])
        a.check(5 * n)
        other.check(n)
        other.inject(np.full(cap, 200))          # as many as the queue holds
        with pytest.raises(chem.ChemError):      # one more
            other.inject([200])
    finally:
        chem.chem_destroy(ctx)


@pytest.mark.parametrize("n", [5, 3000, 140000])  # (from 65,536 on several host threads share the work)
def test_every_species_is_released_once_and_in_order(n):
    cfg, keep = chem.make_config(L, W.D_NM2_S, [], seed=4, precision=chem.CHEM_FP32_LOCAL, dt_min=U, dt_max=U,
                                 capacity_species=8 * n, capacity_pending=4 * n)
    ctx = chem.chem_init(cfg)
    try:
        a = Queue(ctx, 0, 5)
        a.inject(np.repeat([0, 10], [n - n // 2, n // 2]))
        a.inject([])
        a.inject(np.full(n, 10))                 # behind it, at an equal arrival
        chem.chem_run_until(ctx, 5 * U)
        a.inject(np.full(n, 12))
        a.inject(np.full(n, 11))                 # among it
        chem.chem_run_until(ctx, 10.5 * U)
        a.inject(np.full(n, 20))                 # behind what is left
        chem.chem_run_until(ctx, 30 * U)
        a.check(5 * n)
    finally:
        chem.chem_destroy(ctx)
