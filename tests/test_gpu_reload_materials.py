"""Materials loaded again after the geometry: the layers follow the new
densities (a layer may turn into vacuum or back), as in a context that loads
them first."""
import numpy as np
import pytest

from paper_2203_09467_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_materials_reloaded_after_geometry(precision):
    from paper_2203_09467_gb300 import emt
    n = 12
    s = W.calo_setup(seed=5)
    prim = W.calo_primaries(n, energy=2000.0)
    ids = np.arange(n, dtype=np.uint64)
    hollow = s.materials.copy()
    hollow[1] = W.VACUUM

    def run(ctx):
        ctx.submit(ids, prim)
        ctx.run()
        h, sm, _ = ctx.read_all()
        return h, sm

    def fresh(materials):
        ctx = emt.Context(precision=precision, slot_capacity=1 << 16, max_events=n, max_bins=100, seed=s.seed)
        ctx.load_materials(materials, s.physics)
        ctx.load_geometry(s.layers, s.world)
        out = run(ctx)
        ctx.close()
        return out

    ctx = emt.Context(precision=precision, slot_capacity=1 << 16, max_events=n, max_bins=100, seed=s.seed)
    ctx.load_materials(s.materials, s.physics)
    ctx.load_geometry(s.layers, s.world)
    for materials in (s.materials, hollow, s.materials):
        ctx.load_materials(materials, s.physics)
        (h, sm), (h0, sm0) = run(ctx), fresh(materials)
        assert np.array_equal(sm[:, 4:], sm0[:, 4:])
        assert np.allclose(sm, sm0, rtol=1e-12, atol=0) and np.allclose(h, h0, rtol=1e-12, atol=1e-12)
    ctx.close()
