"""The rate-equation integrator on reaction tables of other sizes than the water table:
one row, an odd and an even number of rows, a full half warp (16 rows, 8 species), and
zero rows. Extents against the reference (same tolerances as the water-table tests: both
integrators' errors are far below 1e-8 relative + 1e-5 events)."""
import numpy as np
import pytest

from harness import cuda_available
from oracle import homogeneous as H
from oracle.sbs import philox_key
from paper_2509_03313_gb300 import chem

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not cuda_available(), reason="needs a CUDA GPU")]


def _table(n_types, n_rxn, seed):
    rng = np.random.default_rng(seed)
    pairs = [(a, b) for a in range(n_types) for b in range(a, n_types)]
    rng.shuffle(pairs)
    return [(int(a), int(b), float(10.0 ** rng.uniform(9.0, 11.0)),
             tuple(int(p) for p in rng.integers(0, n_types, rng.integers(0, 3))), 0)
            for a, b in pairs[:n_rxn]]


@pytest.mark.parametrize("n_types,n_rxn", [(2, 0), (1, 1), (2, 2), (4, 7), (5, 10), (8, 15), (8, 16)])
def test_extents_of_other_reaction_tables(n_types, n_rxn):
    rx = _table(n_types, n_rxn, 100 * n_types + n_rxn)
    L, T, seed = 400.0, 1e-3, 9
    rng = np.random.default_rng(n_rxn)
    types = np.repeat(np.arange(n_types, dtype=np.int32), rng.integers(50, 900, n_types))
    n0 = np.bincount(types, minlength=n_types)
    xyz = rng.uniform(-0.5 * L, 0.5 * L, (types.size, 3))
    cfg, keep = chem.make_config(L, np.full(n_types, 5e9), rx, seed=seed, capacity_species=16384)
    ctx = chem.chem_init(cfg)
    try:
        chem.chem_inject_pulse(ctx, types, xyz, np.zeros(types.size))
        chem.chem_run_homogeneous(ctx, T)
        e, E, _ = chem.chem_batch_homogeneous_report(ctx, 0)
        counts = chem.chem_tally(ctx, n_types, max(n_rxn, 1))["counts"]
    finally:
        chem.chem_destroy(ctx)
    if n_rxn == 0:
        np.testing.assert_array_equal(counts, n0)
        return
    e_ref, E_ref, n_ref = H.stage(n0, L, T, rx, 0, philox_key(seed, 0))
    np.testing.assert_allclose(e[:n_rxn], e_ref, rtol=1e-8, atol=1e-5)
    x = np.maximum(e_ref, 0.0)
    u = H.rounding_uniforms(n_rxn, 0, philox_key(seed, 0))
    if np.all(np.abs(x - np.floor(x) - u) > 2e-5 + 2e-8 * x):  # no rounding decision at the margin
        np.testing.assert_array_equal(E[:n_rxn], E_ref)
        np.testing.assert_array_equal(counts, n_ref)
