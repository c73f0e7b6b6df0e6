"""The chunked cut reduction over blocks on both sides of its 512-vertex chunks in one graph:
every replica's cut against FP64 sums of the same states, real weights (bound as in
test_gpu_cut_scales) and integer weights (exact)."""
import numpy as np
import pytest

from paper_2603_25762_gb300 import qhap, synth
from test_gpu_cut_scales import _check

pytestmark = pytest.mark.gpu

SIZES = [2, 513, 130, 512, 3, 1025, 511, 1024, 128, 1600, 2]


# replica groups of 32: one, a part of a second, several
@pytest.mark.parametrize("mode", ["snp", "read"])
@pytest.mark.parametrize("R", [12, 40, 100])
def test_block_sizes(mode, R):
    rng = np.random.default_rng(8)
    rows, base = [], 0
    for n in SIZES:  # a chain: vertices i and i + 1 share a fragment (snp) or a SNP (read)
        m = n - 1 if mode == "snp" else n
        rows += [np.array([base + i, base + i + 1]) for i in range(m)]
        base += m + 1
    snp = np.concatenate(rows).astype(np.int32)
    fr = synth.Fragments(base, 2 * np.arange(len(rows) + 1, dtype=np.int64), snp,
                         np.where(rng.random(snp.size) < 0.3, -1, 1).astype(np.int8),
                         rng.integers(7, 31, size=snp.size).astype(np.uint8),
                         np.zeros(len(rows), np.uint8), np.arange(base), np.ones(base, np.int8))
    ctx = qhap.Context(0)
    g = ctx.build_graph(fr, mode=qhap.MODE_SNP if mode == "snp" else qhap.MODE_READ)
    _, bo, w = _check(ctx, g, R)
    assert np.bincount(bo[bo >= 0]).tolist() == SIZES
    assert (np.abs(w) == 1).all() == (mode == "read")
    g.free()
    ctx.close()
