"""The tuner stays with the multi-step family where a per-step kernel is close: the two round
differently, and the replicas' cuts must not depend on a close race of timings."""
import numpy as np
import pytest

from paper_2603_25762_gb300 import qhap, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("reads,R", [(300, 128), (633, 384), (1200, 128)])
def test_close_race_keeps_the_family(reads, R):
    fr = synth.region_reads(5, n_snps=round(reads * 10 / 3), region=reads * 1111, n_reads=reads,
                            len_mean=30_000, len_sd=20_000, len_max=150_000, flip_p=0.06,
                            miss_p=0.0, qual=(7, 30))
    kw = dict(replicas=R, steps=200, precision=qhap.PREC_BF16X2, seed=1, refine_max=1)
    cuts = []
    for kernel in (None, None, "multistep-stream-tile"):
        ctx = qhap.Context(0)
        g = ctx.build_graph(fr, mode=qhap.MODE_SNP)
        sol = ctx.solve(g, step_kernel=kernel, **kw)
        assert sol.timing()["kernel"].startswith("multistep")
        cuts.append(sol.cuts())
        sol.free()
        g.free()
        ctx.close()
    assert np.array_equal(cuts[0], cuts[1]) and np.array_equal(cuts[0], cuts[2])
