"""Layer counts about the number of records that the allocation-free entry
point uploads at once, against the context entry points."""
import numpy as np
import pytest

from paper_2203_09467_gb300 import workloads as W
from test_zz_no_alloc import TOL, _context_run, _static_call

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_layers", [1, 511, 512, 513, 1100, 4096])
def test_layer_counts_match_the_context_path(n_layers):
    from paper_2203_09467_gb300 import emt

    s = W.calo_setup()
    s.materials = np.array([W.LEAD, W.VACUUM, W.LIQUID_ARGON], np.float64)
    depth = float(s.layers[:, 1].sum())
    k = np.arange(n_layers)
    s.layers = np.stack([k % 3, np.full(n_layers, depth / n_layers), k % 100], axis=1).astype(np.float64)
    n = 12
    prim = W.calo_primaries(n, energy=500.0, seed=41)
    ids = np.arange(n, dtype=np.uint64) + 100
    want_hist, want_summ, _ = _context_run(emt, s, prim, ids, 1 << 18)
    rc, h, sm = _static_call(emt, s, prim, ids)
    assert rc == 0, rc
    e_in = want_summ[:, 3]
    assert np.array_equal(sm[:, 4:], want_summ[:, 4:])
    assert np.all(np.abs(sm[:, :3] - want_summ[:, :3]) <= TOL * e_in[:, None])
    assert np.all(np.abs(h - want_hist) <= TOL * e_in[:, None])
