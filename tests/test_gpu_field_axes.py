"""Field propagation for every form of the uniform field: along each
coordinate axis (the step kernels leave out the products with the zero
components), in a general direction, and with a miss distance so large that a
substep's norm needs the full renormalisation.  FP64 against the oracle event
by event (1e-9 E_in, identical counts); mixed precision along an axis against
the same field with a second component of 1e-300 T, which takes the general
code and whose products vanish: equal up to the summation order of deposits."""
import numpy as np
import pytest

from paper_2203_09467_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _setup(B, rk_delta=1e-5):
    s = W.calo_field_setup(seed=17)
    s.world[9:12] = B
    s.world[12] = rk_delta
    return s


def _run(s, prim, n, **kw):
    from paper_2203_09467_gb300 import emt
    ctx = emt.context_for(s, slot_capacity=1 << 18, max_events=n, **kw)
    ctx.submit(np.arange(n, dtype=np.uint64), prim)
    ctx.run()
    hist, summ, _ = ctx.read_all()
    ctx.close()
    return hist, summ


@pytest.mark.parametrize("schedule", ["split", "fused"])
@pytest.mark.parametrize("B,rk_delta", [((-2.0, 0.0, 0.0), 1e-5), ((0.0, 1.5, 0.0), 1e-5), ((0.0, 0.0, -2.0), 1e-5),
                                        ((1.2, -0.7, 1.1), 1e-5), ((0.0, 2.0, 0.0), 1e-2), ((1.2, -0.7, 1.1), 1e-2)])
def test_fp64_field_direction_matches_oracle(B, rk_delta, schedule):
    import oracle
    n = 37
    s = _setup(B, rk_delta)
    prim = W.multi_primaries(n, 1, 3, 200.0, 20.0, seed=23)
    hist, summ = _run(s, prim, n, schedule=schedule)
    orc = oracle.Oracle(s.materials, s.physics, s.layers, s.world, s.seed)
    oh, os_ = orc.run(prim, n, np.arange(n, dtype=np.uint64))
    orc.close()
    assert np.array_equal(summ[:, 4:], os_[:, 4:])
    assert np.all(np.abs(summ[:, :3] - os_[:, :3]) <= 1e-9 * os_[:, 3:4])
    assert np.all(np.abs(hist - oh) <= 1e-9 * os_[:, 3:4])


@pytest.mark.parametrize("axis", [0, 1, 2])
def test_mixed_field_axis_equals_general_direction(axis):
    n = 64
    prim = W.multi_primaries(n, 1, 4, 300.0, 30.0, seed=29)
    B = np.zeros(3)
    B[axis] = 1.7
    C = B.copy()
    C[(axis + 1) % 3] = 1e-300
    h1, s1 = _run(_setup(B), prim, n, precision="mixed", schedule="split")
    h2, s2 = _run(_setup(C), prim, n, precision="mixed", schedule="split")
    assert np.array_equal(s1[:, 4:], s2[:, 4:])
    assert np.allclose(s1, s2, rtol=1e-12, atol=0) and np.allclose(h1, h2, rtol=1e-12, atol=1e-12)
