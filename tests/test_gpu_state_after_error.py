"""chem_get_state after a train could not park its species (more of them than its own capacity, in
room that other trains of the batch left): the species still lie in the stepped slots, and as
many as the train's capacity in the parking buffers too, together more than the packing's
working memory holds. The calls return the sticky error with what fits, write nothing past the
caller's rows, and a reset makes the context whole again."""
import ctypes

import numpy as np
import pytest

from harness import cuda_available
from paper_2509_03313_gb300 import chem
from test_gpu_state import _check, _config, _pulse

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not cuda_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("precision", [chem.CHEM_FP64, chem.CHEM_FP32_LOCAL])
@pytest.mark.parametrize("caps,sizes", [((4700, 400), (100, 5000)), ((400, 4700), (5000, 100)), ((60, 8000), (3000, 50))])
def test_state_after_a_failed_parking(caps, sizes, precision):
    big = int(np.argmax(sizes))
    cfgs, keep = zip(*(_config(n, precision, cap, b) for b, (n, cap) in enumerate(zip(sizes, caps))))
    pulses = [_pulse(n, 7 + b) for b, n in enumerate(sizes)]
    ctx = chem.chem_batch_init(cfgs)

    def start():
        for b, (t, x) in enumerate(pulses):
            chem.chem_batch_inject(ctx, b, t, x, np.zeros(t.size))
        chem.chem_batch_run_until(ctx, [1e-18] * 2)

    try:
        start()
        _check(*chem.chem_batch_get_state(ctx, big), *pulses[big])
        with pytest.raises(chem.ChemError) as e:
            chem.chem_batch_run_until(ctx, [1e-18 if b == big else 3e-18 for b in range(2)])
        assert e.value.status == chem.CHEM_ECAPACITY
        rows, guard = sum(caps) + 1000, 7
        p = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
        for b in range(2):
            ids, ty = np.full(rows + guard, 123, np.uint32), np.full(rows + guard, 123, np.int32)
            pos, total = np.full((rows + guard, 3), 123.0), np.zeros(1, np.int64)
            st = chem.lib().chem_batch_get_state(ctx, b, rows, p(ty), p(ids), p(pos), p(total))
            assert st == chem.CHEM_ECAPACITY and sizes[b] <= total[0] <= sum(caps), (st, total)
            n = int(total[0])
            assert np.all(ids[n:] == 123) and np.all(ty[n:] == 123) and np.all(pos[n:] == 123.0)
            assert set(ids[:n].tolist()) == set(range(sizes[b])) and np.all(np.abs(pos[:n]) <= 250.0)
        chem.chem_batch_reset(ctx, [3, 4])
        start()
        for b in range(2):
            _check(*chem.chem_batch_get_state(ctx, b), *pulses[b])
    finally:
        chem.chem_destroy(ctx)
