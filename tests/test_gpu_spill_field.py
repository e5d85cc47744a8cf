"""Host spill in a field: the tracks that leave the device are taken from
warp-sized chunks in cost order.  More primaries than may stay are admitted,
so that the first step already moves some to host memory; every result equals
the run without a budget."""
import numpy as np
import pytest

from paper_2203_09467_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("block", [128, 256])
def test_spill_in_a_field_changes_no_result(precision, block):
    from paper_2203_09467_gb300 import emt
    n = 45
    s = W.calo_field_setup(seed=31)
    prim = W.multi_primaries(n, 2, 3, 200.0, 30.0, seed=37)
    out = []
    for kw in ({}, dict(max_active=40, select="low_energy", spill_above=64)):
        ctx = emt.context_for(s, precision=precision, slot_capacity=1 << 16, max_events=n, schedule="split",
                              block_size=block, **kw)
        ctx.submit(np.arange(n, dtype=np.uint64), prim)
        out.append((ctx.run(), *ctx.read_all()))
        ctx.close()
    (st0, h0, s0, _), (st, h, sm, _) = out
    assert len(prim["T"]) > 64 and st["held"] > 0 and st["spilled"] > 0
    assert st0["held"] == st0["spilled"] == 0
    assert np.array_equal(sm[:, 4:], s0[:, 4:])
    assert np.allclose(sm, s0, rtol=1e-12, atol=0) and np.allclose(h, h0, rtol=1e-12, atol=1e-12)
