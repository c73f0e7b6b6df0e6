"""The tuner's kept choices: a solve must not depend on what the context solved before.
Solves of one graph in BF16 and BF16X2 (which walks the remainder entries too), and with a c0
that the multi-step kernels cannot hold, in both orders in one context against a context of
their own.  The kernels of one family give the same bits (tolerance 0)."""
import numpy as np
import pytest

from paper_2603_25762_gb300 import qhap, synth

pytestmark = pytest.mark.gpu

KW = dict(replicas=128, steps=60, seed=3, refine_max=1)


def _solve(ctx, g, **kw):
    sol = ctx.solve(g, **{**KW, **kw})
    out = sol.timing()["kernel"].split("-")[0] == "multistep", sol.cuts()
    sol.free()
    return out


def _check(fr, pair):
    alone = []
    for kw in pair:
        ctx = qhap.Context(0)
        g = ctx.build_graph(fr, mode=qhap.MODE_SNP)
        alone.append(_solve(ctx, g, **kw))
        g.free()
        ctx.close()
    for order in ((0, 1), (1, 0)):
        ctx = qhap.Context(0)
        g = ctx.build_graph(fr, mode=qhap.MODE_SNP)
        for k in order + order:
            multi, cuts = _solve(ctx, g, **pair[k])
            assert multi == alone[k][0]
            assert np.array_equal(cuts, alone[k][1])
        g.free()
        ctx.close()


def _region(reads):
    return synth.region_reads(5, n_snps=round(reads * 10 / 3), region=reads * 1111, n_reads=reads,
                              len_mean=30_000, len_sd=20_000, len_max=150_000, flip_p=0.06,
                              miss_p=0.0, qual=(7, 30))


# 60: J and its remainder both stay resident; 100, 150: J alone does (3 and 4 tiles a row);
# 300: neither
@pytest.mark.parametrize("reads", [60, 100, 150, 300])
def test_precisions_of_one_graph(reads):
    _check(_region(reads), [dict(precision=qhap.PREC_BF16), dict(precision=qhap.PREC_BF16X2)])


def test_c0_outside_the_multistep_range():
    _check(_region(60), [dict(precision=qhap.PREC_BF16), dict(precision=qhap.PREC_BF16, c0=1e-39)])
