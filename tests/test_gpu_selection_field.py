"""Track selection in a field: warp-sized chunks of the charged tracks in
cost order, some of them held.  Under a budget (both policies, with and
without the host spill) every result equals the unlimited run's."""
import numpy as np
import pytest

from paper_2203_09467_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _run(precision, block, **kw):
    from paper_2203_09467_gb300 import emt
    n = 45
    s = W.calo_field_setup(seed=31)
    prim = W.multi_primaries(n, 1, 3, 200.0, 30.0, seed=37)
    ctx = emt.context_for(s, precision=precision, slot_capacity=1 << 16, max_events=n, schedule="split",
                          block_size=block, **kw)
    ctx.submit(np.arange(n, dtype=np.uint64), prim)
    st = ctx.run()
    hist, summ, _ = ctx.read_all()
    ctx.close()
    return st, hist, summ


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("kw", [dict(max_active=33, select="order"), dict(max_active=700, select="low_energy"),
                                dict(max_active=700, select="low_energy", loop_mode="graph", graph_steps=6),
                                dict(max_active=500, select="low_energy", spill_above=800)])
def test_selection_in_a_field_changes_no_result(precision, kw):
    _, h0, s0 = _run(precision, 256)
    for block in (128, 256):
        st, h, s = _run(precision, block, **kw)
        assert st["held"] > 0 or st["spilled"] > 0
        assert np.array_equal(s[:, 4:], s0[:, 4:])
        assert np.allclose(s, s0, rtol=1e-12, atol=0) and np.allclose(h, h0, rtol=1e-12, atol=1e-12)
