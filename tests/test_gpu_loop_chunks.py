"""The solve's step loop, replayed in chunks from a device-held step base plus a remainder
of direct launches, against the same steps launched one by one from the same start."""
import numpy as np
import pytest

from paper_2603_25762_gb300 import qhap, synth

pytestmark = pytest.mark.gpu


# around the 64 steps below which nothing is captured, one chunk (64 + 1, 66 = 66 % 34 ..),
# several chunks with and without a remainder
@pytest.mark.parametrize("steps", [1, 63, 64, 65, 66, 127, 130, 211])
@pytest.mark.parametrize("precision,kernel", [(qhap.PREC_FP32, None),
                                              (qhap.PREC_BF16, "cta-bn64-s2-x4"),
                                              (qhap.PREC_BF16, "persistent-bn64-tma-state"),
                                              (qhap.PREC_FP8, None)])
def test_chunked_loop_equals_single_steps(steps, precision, kernel):
    import torch

    R = 64
    ctx = qhap.Context(0)
    g = ctx.build_graph(synth.hifi_region(3, scale=0.03), mode=qhap.MODE_READ)
    sol = ctx.solve(g, replicas=R, steps=steps, precision=precision, seed=5, step_kernel=kernel)
    n_pad, pidx, _ = g.layout()
    x = torch.empty(R, n_pad, device="cuda")
    y = torch.empty(R, n_pad, device="cuda")
    ctx.debug_init_state(g, R, x, y, seed=5)
    ctx.debug_steps(g, precision, R, x, y, 0, steps, steps, step_kernel=kernel)
    spins = np.where(x.cpu().numpy()[:, pidx[pidx >= 0]] >= 0, 1.0, -1.0)
    live = np.flatnonzero(pidx >= 0)
    bo, _ = g.blocks()
    rp, col, w = g.edges()
    row = np.repeat(np.arange(g.n_nodes), np.diff(rp))
    full = np.zeros((R, g.n_nodes))
    full[:, live] = spins
    cuts = sol.cuts()
    for b in range(g.n_blocks):  # integer weights: the cuts are exact
        e = bo[row] == b
        cross = full[:, row[e]] != full[:, col[e]]
        assert np.array_equal(cuts[b], (cross * w[e]).sum(1) / 2)
    sol.free()
    g.free()
    ctx.close()
