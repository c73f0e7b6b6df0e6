"""The captured step loop of a solve with checks belongs to the graph it was captured for: a
graph rebuilt at the same addresses, with the same counts but other block sizes or weights,
gives the energy trace, steps and cuts of a context of its own (tolerance 0)."""
import numpy as np
import pytest

from paper_2603_25762_gb300 import qhap, synth

pytestmark = pytest.mark.gpu


def _chains(sizes, rng):
    """One chain of SNPs per block: vertices, entries and stored tiles depend on the sum of
    the sizes alone (sizes multiples of 128)."""
    rows, base = [], 0
    for n in sizes:
        rows += [(base + i, base + i + 1) for i in range(n - 1)]
        base += n
    snp = np.array(rows, np.int32).ravel()
    return synth.Fragments(base, 2 * np.arange(len(rows) + 1, dtype=np.int64), snp,
                           np.where(rng.random(snp.size) < 0.3, -1, 1).astype(np.int8),
                           rng.integers(7, 31, size=snp.size).astype(np.uint8),
                           np.ones(len(rows), np.uint8), np.arange(base), np.ones(base, np.int8))


def _solve(ctx, sizes, mode, alpha, precision, R):
    g = ctx.build_graph(_chains(sizes, np.random.default_rng(5)), mode=mode, porec_alpha=alpha)
    assert g.n_blocks == len(sizes)
    sol = ctx.solve(g, replicas=R, steps=120, precision=precision, seed=2, refine_max=1,
                    check_every=10, patience=3)
    steps, trace = sol.check_trace()
    out = (np.asarray(steps), np.asarray(trace), sol.cuts(),
           [sol.block(b)["steps_run"] for b in range(g.n_blocks)])
    sol.free()
    g.free()
    return out


# real weights (gathered cuts) and integer weights (cuts from the product, R % 64 = 0), with
# other chunks of 512 vertices; then weights 2^40 times as large
@pytest.mark.parametrize("mode,precision,R", [("snp", qhap.PREC_FP32, 12),
                                              ("read", qhap.PREC_FP32, 12),
                                              ("read", qhap.PREC_FP32, 64),
                                              ("read", qhap.PREC_FP8, 64)])
@pytest.mark.parametrize("sizes", [[(512, 512), (640, 384), (896, 128), (512, 512)],
                                   [(384, 384, 384), (128, 128, 896)]])
def test_block_sizes(mode, precision, R, sizes):
    m = qhap.MODE_SNP if mode == "snp" else qhap.MODE_READ
    if mode == "read":  # a read per pair of neighbouring SNPs: one vertex fewer per block
        sizes = [tuple(n + 1 for n in s) for s in sizes]
    ctx = qhap.Context(0)
    got = [_solve(ctx, s, m, 1.0, precision, R) for s in sizes]
    ctx.close()
    for s, out in zip(sizes, got):
        own = qhap.Context(0)
        want = _solve(own, s, m, 1.0, precision, R)
        own.close()
        for a, b in zip(out, want):
            assert np.array_equal(a, b, equal_nan=True)


def test_weights():
    ctx = qhap.Context(0)
    alphas = [1.0, 2.0**40, 2.0**-40, 1.0]
    got = [_solve(ctx, (640, 384), qhap.MODE_SNP, a, qhap.PREC_FP32, 12) for a in alphas]
    ctx.close()
    for alpha, out in zip(alphas, got):
        own = qhap.Context(0)
        want = _solve(own, (640, 384), qhap.MODE_SNP, alpha, qhap.PREC_FP32, 12)
        own.close()
        for a, b in zip(out, want):
            assert np.array_equal(a, b, equal_nan=True)
