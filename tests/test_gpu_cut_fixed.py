"""Every replica's cut of a SNP graph (real weights): the fixed-point node sums and the
chunked reduction against FP64 sums of the same states.

Bound, derived: a weight is rounded by at most 2^-47 of the largest |w|, so a cut by at
most nnz 2^-47 max|w| / 4 over its directed entries; the FP64 additions on either side add
at most (n + degree) 2^-53 sum|w|."""
import numpy as np
import pytest

from paper_2603_25762_gb300 import qhap, synth

pytestmark = pytest.mark.gpu


def _graph(ctx, reads):
    if reads == 0:  # rows of more than 256 entries (the fold) in one narrow window
        rng = np.random.default_rng(3)
        n, rows = 601, [np.arange(601)] * 4
        ptr = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
        snp = np.concatenate(rows).astype(np.int32)
        al = np.where(rng.random(snp.size) < 0.5, 1, -1).astype(np.int8)
        q = rng.integers(7, 31, size=snp.size).astype(np.uint8)
        fr = synth.Fragments(n, ptr, snp, al, q, np.zeros(4, np.uint8), np.arange(n),
                             np.ones(n, np.int8))
    else:
        fr = synth.region_reads(5, n_snps=round(reads * 10 / 3), region=reads * 1111,
                                n_reads=reads, len_mean=30_000, len_sd=20_000, len_max=150_000,
                                flip_p=0.06, miss_p=0.0, qual=(7, 30))
    return ctx.build_graph(fr, mode=qhap.MODE_SNP)


# replicas: FP64 (<= 4), bytes (R % 4), one word, two words a lane; vertices on both sides
# of one 512-row chunk
@pytest.mark.parametrize("reads", [60, 150, 160, 700, 0])
@pytest.mark.parametrize("R", [3, 5, 12, 100, 264])
def test_replica_cuts(reads, R):
    import torch

    ctx = qhap.Context(0)
    g = _graph(ctx, reads)
    steps = 30
    sol = ctx.solve(g, replicas=R, steps=steps, precision=qhap.PREC_FP32, seed=2, refine_max=1)
    n_pad, pidx, _ = g.layout()
    x = torch.empty(R, n_pad, device="cuda")
    y = torch.empty(R, n_pad, device="cuda")
    ctx.debug_init_state(g, R, x, y, seed=2)
    ctx.debug_steps(g, qhap.PREC_FP32, R, x, y, 0, steps, steps)
    live = np.flatnonzero(pidx >= 0)
    spins = np.zeros((R, g.n_nodes))
    spins[:, live] = np.where(x.cpu().numpy()[:, pidx[live]] >= 0, 1.0, -1.0)
    rp, col, w = g.edges()
    row = np.repeat(np.arange(g.n_nodes), np.diff(rp))
    bo, _ = g.blocks()
    cuts = sol.cuts()
    for b in range(g.n_blocks):
        e = bo[row] == b
        n, deg = (bo == b).sum(), np.diff(rp)[bo == b].max()
        tol = e.sum() * 2.0**-47 * np.abs(w[e]).max() / 4 \
            + (n + deg) * 2.0**-53 * np.abs(w[e]).sum()
        want = ((spins[:, row[e]] != spins[:, col[e]]) * w[e]).sum(1) / 2
        assert np.abs(cuts[b] - want).max() <= tol
    sol.free()
    g.free()
    ctx.close()
