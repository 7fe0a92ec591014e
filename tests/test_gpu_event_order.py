"""Event order of large contexts (more than 262,144 species of capacity, one kernel per phase):
ranks for up to 1,024 events of a step, event buckets beyond, and the general sorts when a
bucket overflows (the reacting species' ids a small part of all ids). Event lists, counts
and positions against the FP64 reference."""
import numpy as np
import pytest

from harness import assert_fp64_parity, cuda_available, gpu_batch_run, gpu_run, oracle_run
from paper_2509_03313_gb300 import chem, workloads as W

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not cuda_available(), reason="needs a CUDA GPU")]


def _workload(n, n_inert, L, seed, steps):
    counts = (W.MIX_COUNTS * n / W.MIX_COUNTS.sum()).astype(np.int64)
    pulses = [W.uniform_mixture(counts, L, seed)]
    if n_inert:  # H2 reacts with nothing; its ids come first
        pulses.insert(0, W.uniform_mixture([0] * W.H2 + [n_inert, 0], L, seed + 1))
    return W.Workload("order", L, pulses, W.Schedule(1e-9, 1e-9), t_end=steps * 1e-9)


# reacting species, inert species, box, capacity: ranks; buckets; an overflow with the events in
# shared memory, and in global memory
@pytest.mark.parametrize("n,n_inert,L,cap", [(3000, 0, 120.0, 300_000), (40_000, 0, 100.0, 2_000_000),
                                             (12_000, 100_000, 80.0, 300_000), (40_000, 100_000, 100.0, 300_000)])
def test_event_order_of_large_contexts(n, n_inert, L, cap):
    wl = _workload(n, n_inert, L, 31, 3)
    g = gpu_run(wl, 4, capacity=cap, launch_mode=chem.CHEM_LAUNCH_PHASES)
    o = oracle_run(wl, 4, impl="cxx")
    assert o.events_total.sum() > 100
    assert_fp64_parity(g, o, wl.L)


def test_event_order_of_a_large_batch():
    # three trains of very different sizes share the buckets; train 1's step has over 1,024 events
    wls = [_workload(400, 0, 150.0, 51, 4), _workload(30_000, 0, 100.0, 52, 2), _workload(2000, 150_000, 150.0, 53, 3)]
    outs = gpu_batch_run(wls, [6, 7, 8], [0, 1, 2], launch_mode=chem.CHEM_LAUNCH_PHASES)
    for b, (wl, g) in enumerate(zip(wls, outs)):
        assert_fp64_parity(g, oracle_run(wl, 6 + b, train_id=b, impl="cxx"), wl.L)
