"""The one-CTA event order of 1,024 threads falling back from its bucket sort to the block
radix sort. The two share one buffer: the radix sort clears the words from which the bucket
sort's threads read that a bucket is too large, so all of them must have read before any
goes on. Batches in the per-phase form whose event keys carry the train in their top bits put
the events of a train into one bucket of 2,048, or two: the steps that fall back are those
with more than 64 events in a bucket, counted here from the reference's event lists."""
import numpy as np
import pytest

from harness import assert_fp64_parity, cuda_available, gpu_batch_run, oracle_run
from paper_2509_03313_gb300 import chem, workloads as W

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not cuda_available(), reason="needs a CUDA GPU")]


def _dense(n, L, seed, n_steps):
    counts = (W.MIX_COUNTS * n / W.MIX_COUNTS.sum()).astype(np.int64)
    return W.Workload("dense", L, [W.uniform_mixture(counts, L, seed=seed)], W.Schedule(1e-9, 1e-9),
                      t_end=n_steps * 1e-9)


def _largest_bucket(keys):
    """Most keys in one of the bucket sort's 2,048 equal parts of the keys' range."""
    span = int(keys.max() - keys.min())
    return int(np.bincount((keys - keys.min()) >> max(0, span.bit_length() - 11)).max())


@pytest.mark.parametrize("sizes", [(3000, 2500), (1200, 5000, 2000), (4000, 300, 900, 3500)])
def test_every_fallback_of_a_batch(sizes):
    wls = [_dense(n, 100.0, 60 + 7 * b + n, 16) for b, n in enumerate(sizes)]
    stats = {}
    outs = gpu_batch_run(wls, [30 + b for b in range(len(wls))], launch_mode=chem.CHEM_LAUNCH_PHASES, stats=stats)
    refs = [oracle_run(wl, 30 + b, train_id=b, impl="cxx") for b, wl in enumerate(wls)]
    for wl, g, o in zip(wls, outs, refs):
        assert_fp64_parity(g, o, wl.L)
    shift = 32 - (len(wls) - 1).bit_length()  # the train's bits on top of the ids
    keys = {}
    for b, o in enumerate(refs):
        for e in o.events():
            keys.setdefault(int(e[0]), []).append((b << shift) | int(e[2]))
    want = sum(_largest_bucket(np.array(k)) > 64 for k in keys.values())
    assert 0 < want and stats["react_order_radix"] == want, (stats["react_order_radix"], want)
    assert stats["react_order_global"] == 0
