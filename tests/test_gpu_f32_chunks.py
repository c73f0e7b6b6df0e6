"""FP32 step on tile storage: the chunk lists and the tile edges of k_step_f32.

The states are multiples of 1/64 in [-1, 1] and the weights small integers, so every
product and partial sum is a multiple of 1/64 below 2^18 in magnitude: FP32 holds each
exactly and J x X must equal the FP64 product bit for bit (tolerance 0)."""
import numpy as np
import pytest

from paper_2603_25762_gb300 import qhap, synth

pytestmark = pytest.mark.gpu


def _graph(ctx, reads):
    if reads <= 80:
        fr = synth.tiny_reads(7, n_snps=40, n_reads=reads)
    else:
        fr = synth.region_reads(7, n_snps=round(reads * 5 / 3), region=reads * 555,
                                n_reads=reads)
    return ctx.build_graph(fr, mode=qhap.MODE_READ)


def _dense(g, n_pad, pidx):
    rp, col, w = g.edges()
    row = np.repeat(np.arange(g.n_nodes), np.diff(rp))
    J = np.zeros((n_pad, n_pad))
    J[pidx[row], pidx[col]] = -w
    return J


# row counts around the 32-row groups and the 128-row tiles; replicas around the 8, 32 and
# 64 a CTA takes (400 reads x 1,600 replicas reach the last)
@pytest.mark.parametrize("reads,R", [(2, 1), (33, 8), (96, 9), (31, 15), (32, 16), (33, 17), (64, 33), (127, 64),
                                     (129, 65), (257, 300), (400, 1600), (400, 1633), (700, 100)])
def test_product_exact_at_edges(reads, R):
    import torch

    ctx = qhap.Context(0)
    g = _graph(ctx, reads)
    n_pad, pidx, _ = g.layout()
    J = _dense(g, n_pad, pidx)
    rng = np.random.default_rng(reads * 1000 + R)
    x = np.zeros((R, n_pad), np.float32)
    live = pidx[pidx >= 0]
    x[:, live] = rng.integers(-64, 65, size=(R, live.size)) / 64.0
    want = x.astype(np.float64) @ J.T
    xt = torch.from_numpy(x).cuda()
    buf = torch.full((R * n_pad + 1,), 9.0, device="cuda")
    for off in (0, 1):  # 16-byte aligned output, and one that is not
        z = buf[off:off + R * n_pad]
        ctx.debug_matvec(g, qhap.PREC_FP32, R, xt, z)
        got = z.cpu().numpy().reshape(R, n_pad)
        assert np.array_equal(got[:, live].astype(np.float64), want[:, live])
    g.free()
    ctx.close()


@pytest.mark.parametrize("variant,reads,R", [("ballistic", 129, 17), ("discrete", 161, 40),
                                             ("adiabatic", 97, 9), ("ballistic", 400, 1633)])
def test_unaligned_momentum_equals_aligned(variant, reads, R):
    """y from a buffer that is only 4-byte aligned takes scalar accesses: the same bits."""
    import torch

    ctx = qhap.Context(0)
    g = _graph(ctx, reads)
    n_pad, _, _ = g.layout()
    x0 = torch.empty(R, n_pad, device="cuda")
    y0 = torch.empty(R, n_pad, device="cuda")
    ctx.debug_init_state(g, R, x0, y0)
    out = []
    for off in (0, 1):
        x = x0.clone()
        buf = torch.zeros(R * n_pad + 1, device="cuda")
        y = buf[off:off + R * n_pad].view(R, n_pad)
        y.copy_(y0)
        torch.cuda.synchronize()
        ctx.debug_steps(g, qhap.PREC_FP32, R, x, y, 0, 5, 50, dt=0.5, variant=variant)
        out.append((x.cpu().numpy(), y.cpu().numpy()))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    assert not np.array_equal(out[0][0], x0.cpu().numpy())
    g.free()
    ctx.close()
