"""A state with an infinity or a NaN: 0 * x is then NaN, so the product covers every stored
tile, also its parts without a nonzero of J."""
import numpy as np
import pytest

from paper_2603_25762_gb300 import qhap, synth

pytestmark = pytest.mark.gpu


def _graph(ctx):
    g = ctx.build_graph(synth.region_reads(11, n_snps=1000, region=333_000, n_reads=600),
                        mode=qhap.MODE_READ)
    n_pad, pidx, _ = g.layout()
    rp, col, _ = g.edges()
    live = pidx >= 0
    row = np.repeat(np.arange(g.n_nodes), np.diff(rp))
    tiles = np.zeros((n_pad // 128, n_pad // 128), bool)  # stored: tiles with an edge
    on = live[row] & live[col]
    tiles[pidx[row[on]] // 128, pidx[col[on]] // 128] = True
    return g, n_pad, pidx[live], tiles


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("precision,kernel", [
    (qhap.PREC_FP32, None), (qhap.PREC_BF16, "cta-bn128-s3"), (qhap.PREC_BF16, "cta-bn64-s2-x4"),
    (qhap.PREC_BF16, "persistent-bn128"), (qhap.PREC_BF16, "persistent-bn64-tma-state"),
    (qhap.PREC_BF16, "multistep-stream-tile"), (qhap.PREC_BF16, "multistep-stream-group")])
def test_step_from_a_nonfinite_state(precision, kernel, value):
    import torch

    R, r = 128, 37
    ctx = qhap.Context(0)
    g, n_pad, rows, tiles = _graph(ctx)
    c = int(rows[len(rows) // 2])
    hit = tiles[rows // 128, c // 128]  # rows whose row tile stores c's column tile
    assert hit.any() and not hit.all()
    x = torch.zeros(R, n_pad, device="cuda")
    y = torch.zeros(R, n_pad, device="cuda")
    x[r, c] = float(value)
    ctx.debug_steps(g, precision, R, x, y, 0, 1, 40, step_kernel=kernel)
    got = torch.isfinite(y).cpu().numpy()[:, rows]
    assert got[np.arange(R) != r].all()
    # 0 * value is NaN in every row of the tile; the rows with an edge to c hold an infinity
    # or, where it hit the wall, y = 0: all others of the tile are NaN
    xs = x.cpu().numpy()[:, rows]
    assert np.isfinite(xs[r][~hit & (rows != c)]).all() and got[r][~hit & (rows != c)].all()
    rp, col, _ = g.edges()
    _, pidx, _ = g.layout()
    node = {int(p): i for i, p in enumerate(pidx) if p >= 0}
    edge = np.isin(rows, pidx[col[rp[node[c]]:rp[node[c] + 1]]])
    nan = np.isnan(xs[r])
    assert nan[hit & ~edge & (rows != c)].all()
    z = torch.zeros(R, n_pad, device="cuda")
    x.zero_()
    x[r, c] = float(value)
    ctx.debug_matvec(g, precision, R, x, z)
    zf = np.isfinite(z.cpu().numpy()[:, rows])
    assert np.array_equal(~zf[r], hit) and zf[np.arange(R) != r].all()
    g.free()
    ctx.close()
