"""The autotuner times the launch form that a run from the same state takes, also right after
injection into a fresh context (where no step has been taken and the species are still in
the pending queue): at 32,000 species one CTA per SM takes 20 % less time than a kernel per
phase, one cluster of 16 CTAs 40 to 80 % more, so the choice shows which form was timed."""
import numpy as np
import pytest

from harness import cuda_available
from paper_2509_03313_gb300 import chem, workloads as W

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not cuda_available(), reason="needs a CUDA GPU")]


def _context(wl, mode):
    import torch
    s, n = wl.schedule, wl.n_species
    cfg, keep = chem.make_config(wl.L, wl.D, wl.reactions, seed=1, precision=chem.CHEM_FP32_LOCAL, dt_min=s.dt_min,
                                 dt_max=s.dt_max, dt_growth=s.dt_growth, capacity_species=2 * n, capacity_pending=n,
                                 capacity_candidates=n, launch_mode=mode,
                                 stream=torch.cuda.current_stream().cuda_stream, allocator=chem.torch_allocator(0))
    return chem.chem_init(cfg), (cfg, keep)


@pytest.mark.parametrize("mode", [chem.CHEM_LAUNCH_AUTO, chem.CHEM_LAUNCH_PERSISTENT])
@pytest.mark.parametrize("late", [0.0, 1e-12])
def test_a_fresh_context_is_tuned_in_the_form_that_runs(mode, late):
    wl = W.tracks_same_density(3, 1600.0, t_end=1e-7)  # 32,000 species
    p = wl.pulses[0]
    assert 30_000 < p.n < 34_000
    ctx, keep = _context(wl, mode)
    try:
        chem.chem_inject_pulse(ctx, p.types, p.xyz, p.t_arrival + late, p.energy_eV)
        spl, n_lim, ih, form = chem.chem_autotune(ctx, 2000.0)
        assert form == chem.CHEM_LAUNCH_PERSISTENT and spl in (8, 32)
        assert chem.chem_tally(ctx, 7, 9)["t"] == 0.0
        chem.chem_run_until(ctx, wl.t_end)
        st = chem.chem_get_stats(ctx)
        assert st["graph_replays"] == 0 and st["phase_launches"]["persistent"] >= 1
    finally:
        chem.chem_destroy(ctx)


def test_the_automatic_mode_goes_on_choosing_after_tuning():
    # tuned on 300,000 species (a kernel per phase), then few: many steps per launch again
    n = 300_000
    counts = (W.MIX_COUNTS * n // W.MIX_COUNTS.sum()).astype(np.int64)
    wl = W.Workload("mix", 1200.0, [W.uniform_mixture(counts, 1200.0, 5)], W.Schedule(1e-9, 1e-9), t_end=5e-9)
    p = wl.pulses[0]
    ctx, keep = _context(wl, chem.CHEM_LAUNCH_AUTO)
    try:
        chem.chem_inject_pulse(ctx, p.types, p.xyz, p.t_arrival, p.energy_eV)
        form = chem.chem_autotune(ctx, 1000.0)[3]
        chem.chem_reset(ctx, 2)
        chem.chem_inject_pulse(ctx, p.types[:2000], p.xyz[:2000], p.t_arrival[:2000], 0.0)
        chem.chem_run_until(ctx, wl.t_end)
        st = chem.chem_get_stats(ctx)
        if form == chem.CHEM_LAUNCH_PHASES:
            assert st["graph_replays"] == 0 and st["phase_launches"]["persistent"] == 1
    finally:
        chem.chem_destroy(ctx)
