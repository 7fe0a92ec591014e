"""The launch forms of a step (one kernel per phase; many steps per launch, as one cluster or
one CTA per SM) give the same results down to the order of the species, at the sizes where
the forms and their parts change: one cluster / the whole grid (2,560 species), the one-CTA
sort (4,096 keys) and its multi-tile form, runs that end inside, at and after a launch of
16 steps, and batches whose next step is planned ahead (up to 8 trains) or not. FP32-local
results are compared bit for bit, FP64 events with the reference."""
import numpy as np
import pytest

from harness import assert_fp64_parity, cuda_available, gpu_batch_run, gpu_run, oracle_run
from paper_2509_03313_gb300 import chem, workloads as W

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not cuda_available(), reason="needs a CUDA GPU")]
PH, PE = chem.CHEM_LAUNCH_PHASES, chem.CHEM_LAUNCH_PERSISTENT


def _mixture(n, seed, steps, dt=1e-9):
    counts = (W.MIX_COUNTS * n // W.MIX_COUNTS.sum()).astype(np.int64)
    counts[0] += n - counts.sum()
    L = max(160.0, 200.0 * (n / 2000.0) ** (1 / 3))
    return W.Workload("mix", L, [W.uniform_mixture(counts, L, seed)], W.Schedule(dt, dt), t_end=steps * dt)


def _raw(wl, seed, mode, precision=chem.CHEM_FP32_LOCAL, stops=()):
    import torch
    s, n = wl.schedule, wl.n_species
    cfg, keep = chem.make_config(wl.L, wl.D, wl.reactions, seed=seed, precision=precision, dt_min=s.dt_min,
                                 dt_max=s.dt_max, dt_growth=s.dt_growth, capacity_species=max(4096, 2 * n),
                                 capacity_pending=n, capacity_candidates=max(4096, n),
                                 capacity_event_log=4 * n + 64, launch_mode=mode,
                                 stream=torch.cuda.current_stream().cuda_stream)
    ctx = chem.chem_init(cfg)
    try:
        for p in wl.pulses:
            chem.chem_inject_pulse(ctx, p.types, p.xyz, p.t_arrival, p.energy_eV)
        for t in (*stops, wl.t_end):
            chem.chem_run_until(ctx, t)
        t = chem.chem_tally(ctx, 7, 9)
        return [*chem.chem_get_state(ctx), chem.chem_get_events(ctx), t["counts"], t["events"],
                np.array([t["t"], t["species_steps"]])]
    finally:
        chem.chem_destroy(ctx)


def _same(a, b):
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("n,steps", [(1, 3), (2, 16), (33, 17), (511, 15), (2000, 33), (2559, 20), (2561, 20),
                                     (4096, 18), (4097, 18), (7681, 17), (40000, 5)])
def test_forms_agree_bit_for_bit(n, steps):
    wl = _mixture(n, 300 + n, steps)
    ref = _raw(wl, 7, PH)
    _same(_raw(wl, 7, PE), ref)
    _same(_raw(wl, 7, chem.CHEM_LAUNCH_AUTO), ref)


@pytest.mark.parametrize("steps", [1, 15, 16, 17, 128, 129])
def test_order_after_runs_that_end_anywhere(steps):
    wl = _mixture(700, 41, steps)
    stops = [3e-9, 3e-9] if steps > 3 else []  # (the second has nothing to do)
    ref = _raw(wl, 9, PH, stops=stops)
    _same(_raw(wl, 9, PE, stops=stops), ref)


@pytest.mark.parametrize("n", [1500, 3500, 6000])
def test_fp64_forms_equal_reference(n):
    wl = _mixture(n, 77, 40)
    o = oracle_run(wl, 5, impl="cxx")
    for mode in (PH, PE):
        assert_fp64_parity(gpu_run(wl, 5, launch_mode=mode), o, wl.L)


@pytest.mark.parametrize("trains", [8, 9])
def test_batches_planned_ahead_or_not(trains):
    wls = [_mixture(150 + 60 * b, 500 + b, 10 + 3 * b) for b in range(trains)]
    seeds, tids = [20 + b for b in range(trains)], list(range(trains))
    outs = gpu_batch_run(wls, seeds, tids, launch_mode=PE)
    for b, (wl, g) in enumerate(zip(wls, outs)):
        assert_fp64_parity(g, oracle_run(wl, seeds[b], train_id=b), wl.L)
