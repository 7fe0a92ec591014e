"""Which branch orders the events of a step in the per-phase form of large contexts (more than
262,144 species of capacity), shown by the library's counters. The events' buckets serve any
number of events; only when one of a bucket's 8 places is missing do the sorts of the small
contexts run, in shared memory (8,192 events) or global memory. So:
* crowded steps of over 8,192 events that count no global order were ordered by buckets;
* with the reacting species' ids in a small part of all ids the buckets overflow: over 8,192
  events then count a global order, and with fewer of several trains a radix order (a train's
  keys share one bucket of the sort in shared memory, which buckets never come to).
The conflict rounds leave shared memory past 1,536 conflicting pairs in either case."""
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


@pytest.mark.parametrize("n_inert,cap,in_global", [(0, 2_000_000, False), (100_000, 300_000, True)])
def test_crowded_steps_by_buckets_or_in_global_memory(n_inert, cap, in_global):
    wl = _workload(40_000, n_inert, 100.0, 71, 2)
    g = gpu_run(wl, 14, capacity=cap, launch_mode=chem.CHEM_LAUNCH_PHASES)
    st = g["stats"]
    assert st["max_step_events"] > 8192 and st["graph_replays"] >= 1
    assert (st["react_order_global"] > 0) == in_global, st
    assert st["max_conflict_pairs"] > 1536 and st["react_rounds_global"] >= 1, st
    assert_fp64_parity(g, oracle_run(wl, 14, impl="cxx"), wl.L)


@pytest.mark.parametrize("n_inert,L,in_shared", [(0, 150.0, False), (120_000, 90.0, True)])
def test_a_batch_by_buckets_or_in_shared_memory(n_inert, L, in_shared):
    wls = [_workload(5000, n_inert, L, 81 + b, 3) for b in range(2)]
    if not n_inert:  # (capacities of twice the species: a third train makes the context a large one)
        wls.append(_workload(400, 130_000, 200.0, 91, 3))
    stats = {}
    outs = gpu_batch_run(wls, [24 + b for b in range(len(wls))], launch_mode=chem.CHEM_LAUNCH_PHASES, stats=stats)
    # more than 64 events of a train: a radix order, if it is sorted in shared memory
    assert max(int(g["steps"]["n_events"].max()) for g in outs) > 64
    assert stats["max_step_events"] <= 8192 and stats["react_order_global"] == 0
    assert (stats["react_order_radix"] > 0) == in_shared, stats
    for b, (wl, g) in enumerate(zip(wls, outs)):
        assert_fp64_parity(g, oracle_run(wl, 24 + b, train_id=b, impl="cxx"), wl.L)
