"""SNP rows with many long-range contacts: the small CTA tier (window or terms up to 2,048),
the large one (window up to 12,288 SNPs, else 8,192 sorted terms) and what it refuses.
Weights as in the SNP-row tests: the same terms in the same order, a term off by the
rounding of its log10, so 1e-12 relative; edges and refusals are equal."""
import numpy as np
import pytest

from paper_2603_25762_gb300 import qhap, synth

pytestmark = pytest.mark.gpu


def _hub(window, terms, rng):
    """SNP 0 in `terms` two-SNP contacts, most of them over 512 SNPs away, the last one at
    the window's end; every other SNP in a read of its neighbourhood."""
    far = np.append(rng.integers(600, window, size=terms - 1), window - 1)
    rows = [np.array([0, v]) for v in far]
    rows += [np.arange(a, min(a + 4, window)) for a in range(1, window - 1, 3)]
    ptr = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    snp = np.concatenate(rows).astype(np.int32)
    return synth.Fragments(window, ptr, snp,
                           np.where(rng.random(snp.size) < 0.5, 1, -1).astype(np.int8),
                           rng.integers(4, 94, size=snp.size).astype(np.uint8),
                           np.array([1] * terms + [0] * (len(rows) - terms), np.uint8),
                           np.arange(window), np.ones(window, np.int8))


# small dense, small sorted (2,048 terms), large dense, large sorted (8,192 terms), refused
@pytest.mark.parametrize("window,terms,refused", [
    (2048, 3000, False), (2049, 2048, False), (2049, 2049, False), (12_288, 9000, False),
    (12_289, 2048, False), (12_289, 2049, False), (12_289, 8192, False), (12_289, 8193, True)])
def test_hub_row(window, terms, refused):
    from oracle import oracle as o

    o.build()
    fr = _hub(window, terms, np.random.default_rng(terms))
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
