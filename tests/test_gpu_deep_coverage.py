"""Deep coverage: covering lists longer than the shared-memory sort (256 fragments) with
either payload, and SNP rows of more than 8,192 terms, which are summed where their window
allows it and refused where it does not.

Weights as in the SNP-row tests: the same terms in the same order, a term off by the
rounding of its log10, so 1e-12 relative; edges, votes and refusals are equal."""
import numpy as np
import pytest

from paper_2603_25762_gb300 import qhap, synth

pytestmark = pytest.mark.gpu


def _fragments(rows, rng):
    ptr = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    snp = np.concatenate(rows).astype(np.int32)
    n = int(snp.max()) + 1
    return synth.Fragments(n, ptr, snp, np.where(rng.random(snp.size) < 0.4, 1, -1).astype(np.int8),
                           rng.integers(4, 94, size=snp.size).astype(np.uint8),
                           np.zeros(len(rows), np.uint8), np.arange(n), np.ones(n, np.int8))


def _nested(cover, n, rng):  # SNP n / 2 under every fragment, the others under fewer
    lo = rng.integers(0, n // 2 + 1, size=cover)
    hi = rng.integers(n // 2 + 1, n + 1, size=cover)
    return [np.arange(a, b) for a, b in zip(lo, hi)]


@pytest.mark.parametrize("cover", [256, 257, 300, 511, 512, 513, 1100])
def test_snp_rows(cover):
    from oracle import oracle as o

    o.build()
    rng = np.random.default_rng(cover)
    fr = _fragments(_nested(cover, 60, rng), rng)
    ctx = qhap.Context(0)
    g = ctx.build_graph(fr, mode=qhap.MODE_SNP)
    rp, col, w = g.edges()
    og = o.snp_graph(fr)
    assert np.array_equal(rp, og.row_ptr) and np.array_equal(col, og.col)
    np.testing.assert_allclose(w, og.w, rtol=1e-12, atol=1e-14)
    g.free()
    ctx.close()


@pytest.mark.parametrize("cover", [256, 257, 513, 1100])
def test_read_votes(cover):
    from oracle import oracle as o

    o.build()
    rng = np.random.default_rng(cover)
    fr = _fragments(_nested(cover, 40, rng), rng)
    ctx = qhap.Context(0)
    g = ctx.build_graph(fr, mode=qhap.MODE_READ)
    sol = ctx.solve(g, replicas=8, steps=20, seed=1)
    bo, _ = g.blocks()
    hap1, _, block_id = ctx.phase(g, sol, fr.n_snps)
    want, block = o.vote(fr, sol.spins(g.n_nodes), bo, g.n_blocks)
    assert np.array_equal(hap1, want) and np.array_equal(block_id, block)
    sol.free()
    g.free()
    ctx.close()


# SNP 0: 40 x 299 terms of its neighbourhood and one partner at the window's far end; a
# window of 12,288 SNPs is the widest that takes any number of terms
@pytest.mark.parametrize("last,refused", [(12_287, False), (12_288, True)])
def test_many_terms_in_a_wide_window(last, refused):
    from oracle import oracle as o

    o.build()
    rng = np.random.default_rng(9)
    fr = _fragments([np.arange(300)] * 40 + [np.array([0, last])], rng)
    ctx = qhap.Context(0)
    if refused:
        with pytest.raises(qhap.QhError) as e:
            ctx.build_graph(fr, mode=qhap.MODE_SNP)
        assert e.value.status == qhap.QH_EUNSUPPORTED
    else:
        g = ctx.build_graph(fr, mode=qhap.MODE_SNP)
        rp, col, w = g.edges()
        og = o.snp_graph(fr)
        assert np.array_equal(rp, og.row_ptr) and np.array_equal(col, og.col)
        np.testing.assert_allclose(w, og.w, rtol=1e-12, atol=1e-14)
        g.free()
    ctx.close()
