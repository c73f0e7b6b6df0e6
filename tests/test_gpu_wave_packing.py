"""Packing of phase blocks into the multi-step kernel's waves: a block's result does not
depend on the wave it runs in, so solves of different block subsets (other waves, other
orders) give the same bits."""
import numpy as np
import pytest

from paper_2603_25762_gb300 import qhap, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_blocks,R", [(30, 256), (48, 256), (48, 384), (64, 128)])
def test_blocks_equal_in_any_wave(n_blocks, R):
    ctx = qhap.Context(0)
    g = ctx.build_graph(synth.batched_blocks(7, n_blocks=n_blocks), mode=qhap.MODE_READ)
    kw = dict(replicas=R, steps=25, precision=qhap.PREC_BF16, seed=3,
              step_kernel="multistep-stream-tile")
    full = ctx.solve(g, **kw)
    cuts, waves = full.cuts(), full.timing()["n_step_launches"]
    for part in (np.arange(0, g.n_blocks, 3), np.arange(g.n_blocks)[::-1][: g.n_blocks // 2],
                 np.arange(1)):
        sub = ctx.solve(g, blocks=part, **kw)
        assert np.array_equal(sub.cuts()[part], cuts[part])
        assert sub.timing()["n_step_launches"] <= waves
        sub.free()
    full.free()
    g.free()
    ctx.close()
