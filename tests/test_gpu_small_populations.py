"""Chunk and round sizes that follow the population: from one track to a few
thousand, on every schedule and both block sizes, the chunks shrink to one
warp and the interactions of a chunk fill rounds of one model each.  FP64
against the oracle event by event (1e-9 E_in, identical counts)."""
import numpy as np
import pytest

from paper_2203_09467_gb300 import workloads as W

pytestmark = pytest.mark.gpu

LOOPS = [dict(schedule="fused", loop_mode="plain"), dict(schedule="fused", loop_mode="graph", graph_steps=6),
         dict(schedule="fused", loop_mode="persistent", graph_steps=32), dict(schedule="split", loop_mode="plain"),
         dict(schedule="split", loop_mode="graph", graph_steps=12),
         dict(schedule="pipelined", loop_mode="graph", graph_steps=6)]


@pytest.mark.parametrize("n", [1, 3, 33, 257, 1200])
def test_small_population_matches_oracle(n):
    import oracle
    from paper_2203_09467_gb300 import emt
    s = W.calo_setup(seed=41)
    prim = W.multi_primaries(n, 1, 2, 50.0, 30.0, seed=43)
    ids = np.arange(n, dtype=np.uint64)
    orc = oracle.Oracle(s.materials, s.physics, s.layers, s.world, s.seed)
    oh, os_ = orc.run(prim, n, ids)
    orc.close()
    for loop in LOOPS:
        for block in (128, 256):
            ctx = emt.context_for(s, slot_capacity=1 << 17, max_events=n, block_size=block, **loop)
            ctx.submit(ids, prim)
            ctx.run()
            hist, summ, _ = ctx.read_all()
            ctx.close()
            assert np.array_equal(summ[:, 4:], os_[:, 4:]), (loop, block)
            assert np.all(np.abs(summ[:, :3] - os_[:, :3]) <= 1e-9 * os_[:, 3:4]), (loop, block)
            assert np.all(np.abs(hist - oh) <= 1e-9 * os_[:, 3:4]), (loop, block)
