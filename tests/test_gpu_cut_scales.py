"""Replica cuts of a SNP graph whose blocks, or whose size, do not suit one fixed-point scale.

Bound, derived: a row of d entries is scaled by its own largest |w| to b = min(53, 62 -
ceil(log2 d)) bits, so each of its weights is rounded by at most 2^-b of that maximum, and a
cut by a quarter of the sum of d 2^-b max|w| over the block's rows; the FP64 additions on
either side add at most (n + degree) 2^-53 sum|w|."""
import numpy as np
import pytest

from paper_2603_25762_gb300 import qhap, synth

pytestmark = pytest.mark.gpu

LONG = 66_000  # SNPs of one block, past 2^16


def _fragments(kind, rng):
    if kind == "blocks":  # 300 SNPs under ordinary reads, then 300 under contacts alone
        groups = [(lo + base, 6, base > 0) for base in (0, 300) for lo in range(0, 295, 2)]
    elif kind == "long":
        groups = [(lo, 3, False) for lo in range(0, LONG - 2, 2)]
    else:  # rows of more than 512 entries beside short ones, all of one block
        groups = [(0, 700, False), (0, 700, True)] + [(lo, 4, True) for lo in range(698, 790, 3)]
    snp = np.concatenate([np.arange(lo, lo + k) for lo, k, _ in groups]).astype(np.int32)
    ptr = np.concatenate([[0], np.cumsum([k for _, k, _ in groups])]).astype(np.int64)
    n = int(snp.max()) + 1
    return synth.Fragments(n, ptr, snp, np.where(rng.random(snp.size) < 0.3, -1, 1).astype(np.int8),
                           rng.integers(7, 31, size=snp.size).astype(np.uint8),
                           np.array([p for *_, p in groups], np.uint8), np.arange(n),
                           np.ones(n, np.int8))


def _check(ctx, g, R):
    import torch

    steps = 12
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
    deg = np.diff(rp)
    row = np.repeat(np.arange(g.n_nodes), deg)
    bo, _ = g.blocks()
    top = np.zeros(g.n_nodes)
    np.maximum.at(top, row, np.abs(w))
    bits = np.minimum(53, 62 - np.ceil(np.log2(np.maximum(deg, 1))))
    cuts = sol.cuts()
    for b in range(g.n_blocks):
        e, v = bo[row] == b, bo == b
        tol = (deg * 2.0**-bits * top)[v].sum() / 4 \
            + (v.sum() + deg[v].max()) * 2.0**-53 * np.abs(w[e]).sum()
        want = ((spins[:, row[e]] != spins[:, col[e]]) * w[e]).sum(1) / 2
        assert np.abs(cuts[b] - want).max() <= tol
    sol.free()
    return row, bo, w


@pytest.mark.parametrize("kind,alpha,R", [("blocks", 2.0**-50, 12), ("blocks", 2.0**-50, 264),
                                          ("blocks", 2.0**60, 9), ("rows", 2.0**-30, 12),
                                          ("rows", 2.0**40, 256), ("long", 1.0, 12)])
def test_cuts_of_unlike_weights(kind, alpha, R):
    ctx = qhap.Context(0)
    fr = _fragments(kind, np.random.default_rng(4))
    g = ctx.build_graph(fr, mode=qhap.MODE_SNP, porec_alpha=alpha)
    row, bo, w = _check(ctx, g, R)
    assert g.n_blocks == (2 if kind == "blocks" else 1)
    if kind == "long":
        assert (bo == 0).sum() > 65_536
    g.free()
    ctx.close()


def test_largest_significand():
    """Weights of +-(2 - 2^-30): rounded to 53 bits their last digit is 2^17."""
    ctx = qhap.Context(0)
    n = 200
    snp = (np.arange(n - 1)[:, None] + np.arange(2)).astype(np.int32).ravel()
    fr = synth.Fragments(n, 2 * np.arange(n, dtype=np.int64), snp,
                         np.where(np.random.default_rng(6).random(snp.size) < 0.3, -1, 1)
                         .astype(np.int8), np.full(snp.size, 20, np.uint8),
                         np.ones(n - 1, np.uint8), np.arange(n), np.ones(n, np.int8))
    g = ctx.build_graph(fr, mode=qhap.MODE_SNP, porec_alpha=1.0)
    unit = np.abs(g.edges()[2]).max()
    g.free()
    g = ctx.build_graph(fr, mode=qhap.MODE_SNP, porec_alpha=(2 - 2.0**-30) / unit)
    _, _, w = _check(ctx, g, 12)
    assert (np.abs(w) >= 2 - 2.0**-17).all() and (np.abs(w) < 2).all()
    g.free()
    ctx.close()
