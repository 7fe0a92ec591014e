"""The per-phase form of batches plans the next step ahead for up to 86 trains (their records in
the shared memory of the reaction kernel) and begins it after the reactions beyond: 64, 65, 86
and 87 trains of different sizes and lengths, one of them with a second pulse, events, counts
and positions against the reference."""
import dataclasses

import numpy as np
import pytest

from harness import assert_fp64_parity, cuda_available, gpu_batch_run, oracle_run
from paper_2509_03313_gb300 import chem, workloads as W

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not cuda_available(), reason="needs a CUDA GPU")]


def _workload(b):
    counts = (W.MIX_COUNTS * (100 + 5 * b) // W.MIX_COUNTS.sum()).astype(np.int64)
    pulses = [W.uniform_mixture(counts, 90.0, 700 + b)]
    if b % 8 == 3:
        p = W.uniform_mixture(counts, 90.0, 800 + b)
        pulses.append(dataclasses.replace(p, t_arrival=np.full(p.n, 3.5e-9)))
    return W.Workload("plan", 90.0, pulses, W.Schedule(1e-9, 1e-9), t_end=(4 + b % 7) * 1e-9)


@pytest.mark.parametrize("trains", [64, 65, 86, 87])
def test_batches_planned_ahead_or_begun_after(trains):
    wls = [_workload(b) for b in range(trains)]
    outs = gpu_batch_run(wls, [40 + b for b in range(trains)], launch_mode=chem.CHEM_LAUNCH_PHASES)
    for b, (wl, g) in enumerate(zip(wls, outs)):
        assert_fp64_parity(g, oracle_run(wl, 40 + b, train_id=b, impl="cxx"), wl.L)
