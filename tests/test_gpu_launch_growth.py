"""Species that arrive while a launch of many steps runs: the launch ends before the first step
whose species are more than its form is for (2,560 for one cluster, 65,536 for one CTA per
SM, 131,072 in batches), and the next steps take the form for them. The results, the order of the species
included, are those of the per-phase form; the counters show which launches ran."""
import dataclasses

import numpy as np
import pytest

from harness import assert_fp64_parity, cuda_available, gpu_batch_run, gpu_run, oracle_run
from paper_2509_03313_gb300 import chem, workloads as W

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not cuda_available(), reason="needs a CUDA GPU")]
PH, PE, AUTO = chem.CHEM_LAUNCH_PHASES, chem.CHEM_LAUNCH_PERSISTENT, chem.CHEM_LAUNCH_AUTO


def _growing(pulses, steps, seed):
    """(species, step of arrival) pulses of one box, steps of 1 ns."""
    L = max(160.0, 400.0 * (sum(n for n, _ in pulses) / 2000.0) ** (1 / 3))  # (few reactions: sizes stay)
    out = []
    for k, (n, at) in enumerate(pulses):
        counts = (W.MIX_COUNTS * n // W.MIX_COUNTS.sum()).astype(np.int64)
        counts[0] += n - counts.sum()
        p = W.uniform_mixture(counts, L, seed + k)
        # (half a step early: released by the step that begins at `at` ns)
        out.append(dataclasses.replace(p, t_arrival=np.full(n, max(0.0, at - 0.5) * 1e-9)))
    return W.Workload("grow", L, out, W.Schedule(1e-9, 1e-9), t_end=steps * 1e-9)


def _raw(wl, seed, mode, steps_per_launch=0):
    import torch
    n = wl.n_species
    cfg, keep = chem.make_config(wl.L, wl.D, wl.reactions, seed=seed, precision=chem.CHEM_FP32_LOCAL, dt_min=1e-9,
                                 dt_max=1e-9, capacity_species=max(4096, 2 * n), capacity_pending=n,
                                 capacity_candidates=max(4096, n), capacity_event_log=4 * n + 64, launch_mode=mode,
                                 steps_per_launch=steps_per_launch, stream=torch.cuda.current_stream().cuda_stream)
    ctx = chem.chem_init(cfg)
    try:
        for p in wl.pulses:
            chem.chem_inject_pulse(ctx, p.types, p.xyz, p.t_arrival, p.energy_eV)
        chem.chem_run_until(ctx, wl.t_end)
        t = chem.chem_tally(ctx, 7, 9)
        out = [*chem.chem_get_state(ctx), chem.chem_get_events(ctx), t["counts"], t["events"],
               np.array([t["t"], t["species_steps"]])]
        st = chem.chem_get_stats(ctx)
        return out, (st["phase_launches"]["persistent"], st["graph_replays"])
    finally:
        chem.chem_destroy(ctx)


def _same(a, b):
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x, y)


# pulses, steps, persistent launches and graph replays by default: a launch per form and 128 steps;
# after a persistent form the per-phase one fills up to 16 steps without a graph
@pytest.mark.parametrize("pulses,steps,launches", [
    ([(500, 0), (4000, 5)], 40, (2, 0)),           # one cluster, then one CTA per SM
    ([(4000, 1)], 33, (2, 0)),                     # a fresh context: nothing is there at first
    ([(4000, 16)], 17, (2, 0)), ([(700, 0), (1800, 15)], 48, (1, 0)),
    ([(280_000, 1)], 40, (1, 2)), ([(300, 0), (264_000, 16)], 32, (1, 1)), ([(5000, 0), (270_000, 37)], 50, (1, 1)),
    ([(300, 0), (9000, 3), (270_000, 7)], 16, (2, 0)),
    ([(60_000, 0), (9000, 17)], 50, (1, 2)),       # in the per-phase form: one CTA reacts, then all SMs
])
def test_a_launch_ends_where_its_species_outgrow_it(pulses, steps, launches):
    wl = _growing(pulses, steps, 900 + steps)
    ref, _ = _raw(wl, 11, PH)
    got, ran = _raw(wl, 11, AUTO)
    _same(got, ref)
    assert ran == launches
    got, ran = _raw(wl, 11, PE)
    _same(got, ref)
    assert ran[1] == 0


@pytest.mark.parametrize("spl", [1, 8])
def test_with_a_given_number_of_steps_per_launch(spl):
    wl = _growing([(800, 0), (6000, 3), (270_000, 13)], 21, 77)
    ref, _ = _raw(wl, 12, PH, spl)
    _same(_raw(wl, 12, AUTO, spl)[0], ref)


def test_fp64_and_batches_equal_the_reference():
    wl = _growing([(600, 0), (3000, 4)], 24, 41)
    assert_fp64_parity(gpu_run(wl, 3), oracle_run(wl, 3, impl="cxx"), wl.L)
    for trains in (3, 9):  # the next step planned ahead, or not
        wls = [_growing([(150 + 20 * b, 0), (200 + 300 * b, 3 + 2 * b)], 12 + 2 * b, 500 + b) for b in range(trains)]
        outs = gpu_batch_run(wls, [50 + b for b in range(trains)])
        for b, (w, g) in enumerate(zip(wls, outs)):
            assert_fp64_parity(g, oracle_run(w, 50 + b, train_id=b, impl="cxx"), w.L)


def test_a_batch_that_outgrows_its_form_equals_the_per_phase_form():
    # 103,000 species, then 139,000 (one CTA per SM up to 131,072 in batches), and few after 40 steps: steps 0 to 5,
    # then 10 without a graph and two of 16 with one, and the rest
    wls = [_growing([(3000, 0), (2000, 9)], 50, 61), _growing([(100_000, 0), (34_000, 6)], 40, 62)]
    stats = {}
    got = gpu_batch_run(wls, [5, 6], precision=chem.CHEM_FP32_LOCAL, stats=stats)
    ref = gpu_batch_run(wls, [5, 6], precision=chem.CHEM_FP32_LOCAL, launch_mode=PH)
    assert (stats["phase_launches"]["persistent"], stats["graph_replays"]) == (2, 2)
    for a, b in zip(got, ref):
        _same(a["state"], b["state"])
        _same([a["events"], a["tally"]["counts"], a["tally"]["events"]],
              [b["events"], b["tally"]["counts"], b["tally"]["events"]])
