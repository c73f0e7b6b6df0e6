"""SNP rows: the warp kernel's edges (32 covering fragments per round, the near window, the
far list and the rows it defers) against the oracle's FP64 graph.

Both sides add the same terms in the same order; a term differs by the rounding of the log
likelihood ratio (log10, a few ulp), so 1e-12 relative holds with room, and the edge lists
are equal."""
import numpy as np
import pytest

from paper_2603_25762_gb300 import qhap, synth

pytestmark = pytest.mark.gpu


def _fragments(rows, n_snps, porec, rng):
    ptr = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    snp = np.concatenate(rows).astype(np.int32)
    allele = np.where(rng.random(snp.size) < 0.5, 1, -1).astype(np.int8)
    qual = rng.integers(4, 94, size=snp.size).astype(np.uint8)
    return synth.Fragments(n_snps, ptr, snp, allele, qual, np.asarray(porec, np.uint8),
                           np.arange(n_snps), np.ones(n_snps, np.int8))


def _contacts(rng, n_snps, count):
    return [np.sort(rng.choice(n_snps, size=k, replace=False))
            for k in rng.integers(2, 7, size=count)]


@pytest.mark.parametrize("case", ["cover31", "cover32", "cover33", "cover65", "window", "far",
                                  "far-deferred", "many-terms", "pairs"])
@pytest.mark.parametrize("alpha,k", [(0.1, 10), (1.0, 4)])
def test_snp_rows_match_oracle(case, alpha, k):
    from oracle import oracle as o

    o.build()
    rng = np.random.default_rng(17)
    porec = None
    if case.startswith("cover"):  # every SNP in exactly that many fragments
        n, rows = 40, [np.arange(40)] * int(case[5:])
    elif case == "window":  # partners on both edges of the near window (u -+ 512)
        n = 1400
        rows = [np.array([u, u + d]) for u in range(0, 800, 7) for d in (511, 512, 513)]
        rows += [np.arange(a, a + 600) for a in (0, 300, 700)]
    elif case == "far":  # some hundred contacts, a few far terms per row
        n = 4000
        rows = _contacts(rng, n, 3000) + [np.arange(a, a + 30) for a in range(0, 3900, 10)]
        porec = [1] * 3000 + [0] * (len(rows) - 3000)
    elif case == "far-deferred":  # over 256 far terms in most rows: the CTA kernel
        n = 2500
        rows = _contacts(rng, n, 90000)
        porec = [1] * len(rows)
    elif case == "many-terms":  # over 8,192 terms in a narrow window: the CTA kernel
        n, rows = 300, [np.arange(300)] * 60
    else:  # two-SNP fragments and fragments of one SNP
        n = 200
        rows = [np.array([a, a + 1]) for a in range(199)] + [np.array([a]) for a in range(200)]
    fr = _fragments(rows, n, porec or [0] * len(rows), rng)
    ctx = qhap.Context(0)
    g = ctx.build_graph(fr, mode=qhap.MODE_SNP, porec_alpha=alpha, linkage_k=k)
    rp, col, w = g.edges()
    og = o.snp_graph(fr, alpha, k)
    assert np.array_equal(rp, og.row_ptr) and np.array_equal(col, og.col)
    np.testing.assert_allclose(w, og.w, rtol=1e-12, atol=1e-14)
    g.free()
    ctx.close()
