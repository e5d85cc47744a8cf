"""The pipelined schedule's field kernel for the forms of a uniform field that
its own code paths take (an axis other than the calorimeter's, any direction,
turns large enough for the renormalisation in every substep): FP64 against the
oracle event by event, mixed precision against the split schedule, equal up to
the summation order of deposits."""
import numpy as np
import pytest

from paper_2203_09467_gb300 import workloads as W

pytestmark = pytest.mark.gpu

FIELDS = [((0.0, 1.5, 0.0), 1e-5), ((1.2, -0.7, 1.1), 1e-5), ((1.2, -0.7, 1.1), 1e-2)]


def _run(B, rk_delta, prim, n, **kw):
    from paper_2203_09467_gb300 import emt
    s = W.calo_field_setup(seed=17)
    s.world[9:12] = B
    s.world[12] = rk_delta
    ctx = emt.context_for(s, slot_capacity=1 << 18, max_events=n, **kw)
    ctx.submit(np.arange(n, dtype=np.uint64), prim)
    ctx.run()
    hist, summ, _ = ctx.read_all()
    ctx.close()
    return s, hist, summ


@pytest.mark.parametrize("B,rk_delta", FIELDS)
def test_fp64_pipelined_field_matches_oracle(B, rk_delta):
    import oracle
    n = 33
    prim = W.multi_primaries(n, 1, 3, 200.0, 20.0, seed=43)
    s, hist, summ = _run(B, rk_delta, prim, n, schedule="pipelined")
    orc = oracle.Oracle(s.materials, s.physics, s.layers, s.world, s.seed)
    oh, os_ = orc.run(prim, n, np.arange(n, dtype=np.uint64))
    orc.close()
    assert np.array_equal(summ[:, 4:], os_[:, 4:])
    assert np.all(np.abs(summ[:, :3] - os_[:, :3]) <= 1e-9 * os_[:, 3:4])
    assert np.all(np.abs(hist - oh) <= 1e-9 * os_[:, 3:4])


@pytest.mark.parametrize("B,rk_delta", FIELDS)
def test_mixed_pipelined_field_equals_split(B, rk_delta):
    n = 64
    prim = W.multi_primaries(n, 1, 4, 300.0, 30.0, seed=47)
    _, h1, s1 = _run(B, rk_delta, prim, n, precision="mixed", schedule="pipelined")
    _, h2, s2 = _run(B, rk_delta, prim, n, precision="mixed", schedule="split")
    assert np.array_equal(s1[:, 4:], s2[:, 4:])
    assert np.allclose(s1, s2, rtol=1e-12, atol=0) and np.allclose(h1, h2, rtol=1e-12, atol=1e-12)
