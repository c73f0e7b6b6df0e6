"""Read-graph weights from 32-SNP words: word edges, reads without words (sparse, or over
2,048 SNPs), and pairs of both kinds, against the oracle (integers: equal)."""
import numpy as np
import pytest

from paper_2603_25762_gb300 import qhap, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("case", ["edges", "gaps", "sparse", "long", "unsorted"])
@pytest.mark.parametrize("weights", ["signed", "conflict"])
def test_read_weights_match_oracle(case, weights):
    from oracle import oracle as o

    o.build()
    rng = np.random.default_rng(23)
    if case == "edges":  # reads that start and end on both sides of a word's edge
        n = 200
        rows = [np.arange(a, a + s) for a in (0, 1, 30, 31, 32, 33, 63, 64, 65, 95, 96)
                for s in (1, 2, 31, 32, 33, 64, 65, 97)]
    elif case == "gaps":  # missing observations inside the reads
        n = 400
        rows = [np.flatnonzero(rng.random(n) < 0.5) for _ in range(20)]
        rows += [np.arange(a, a + 40)[rng.random(40) < 0.7] for a in range(0, 360, 4)]
        rows = [r for r in rows if r.size]
    elif case == "sparse":  # two to six SNPs far apart beside dense reads
        n = 3000
        rows = [np.sort(rng.choice(n, size=k, replace=False)) for k in rng.integers(2, 7, 300)]
        rows += [np.arange(a, a + 50) for a in range(0, 2950, 25)]
    elif case == "long":  # at most 64 words, and more
        n = 2300
        rows = [np.arange(a, b) for a, b in ((0, 2048), (0, 2049), (1, 2048), (31, 2080),
                                             (100, 2300), (5, 90), (2040, 2060), (2047, 2300))]
    else:  # fragments in no order, one empty
        n = 150
        rows = [np.arange(a, a + 30) for a in rng.permutation(120)] + [np.arange(0)]
    ptr = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    snp = np.concatenate(rows).astype(np.int32)
    al = np.where(rng.random(snp.size) < 0.5, 1, -1).astype(np.int8)
    fr = synth.Fragments(n, ptr, snp, al, np.full(snp.size, 30, np.uint8),
                         np.zeros(len(rows), np.uint8), np.arange(n), np.ones(n, np.int8))
    ctx = qhap.Context(0)
    g = ctx.build_graph(fr, mode=qhap.MODE_READ,
                        weight_mode=qhap.WEIGHT_SIGNED if weights == "signed"
                        else qhap.WEIGHT_CONFLICT)
    og = o.read_graph(fr, o.READ_SIGNED if weights == "signed" else o.READ_CONFLICT)
    rp, col, w = g.edges()

    def dense(rp, col, w):
        out = np.zeros((len(rows), len(rows)))
        out[np.repeat(np.arange(len(rows)), np.diff(rp)), col] = w
        return out

    assert np.array_equal(dense(rp, col, w), dense(og.row_ptr, og.col, og.w))
    g.free()
    ctx.close()


@pytest.mark.parametrize("m", [1, 2, 63, 64, 65, 2047, 2048, 2049, 4097, 9000])
def test_fragment_order_does_not_change_the_graph(m):
    """Shuffled fragments go through the whole key sort: the same graph, renumbered."""
    rng = np.random.default_rng(m)
    starts = np.sort(rng.integers(0, 4 * m + 8, size=m))
    rows = [np.arange(a, a + 6) for a in starts]
    n = int(starts.max()) + 6
    perm = rng.permutation(m)
    al = [np.where(rng.random(6) < 0.5, 1, -1).astype(np.int8) for _ in rows]
    ctx = qhap.Context(0)
    edges = []
    for order in (np.arange(m), perm):
        snp = np.concatenate([rows[i] for i in order]).astype(np.int32)
        ptr = np.arange(m + 1, dtype=np.int64) * 6
        fr = synth.Fragments(n, ptr, snp, np.concatenate([al[i] for i in order]),
                             np.full(snp.size, 30, np.uint8), np.zeros(m, np.uint8),
                             np.arange(n), np.ones(n, np.int8))
        g = ctx.build_graph(fr, mode=qhap.MODE_READ)
        rp, col, w = g.edges()
        a = order[np.repeat(np.arange(m), np.diff(rp))]
        b = order[col]
        k = np.lexsort((b, a))
        edges.append((a[k], b[k], w[k]))
        bo, lo = g.blocks()
        for blk in range(g.n_blocks):  # block members in ascending order
            assert np.array_equal(lo[bo == blk], np.arange((bo == blk).sum()))
        g.free()
    for x, y in zip(*edges):
        assert np.array_equal(x, y)
    ctx.close()
