"""The schedule's step coefficients: the table's two lengths (AUTO schedule) and the schedules
too long for it."""
import numpy as np
import pytest

from paper_2603_25762_gb300 import qhap, synth

pytestmark = pytest.mark.gpu


def _two_blocks():
    parts, snps, ptr = [], 0, [np.zeros(1, np.int64)]
    for i, n in enumerate((5100, 200)):  # on both sides of AUTO's 5,000 vertices
        fr = synth.region_reads(20 + i, n_snps=round(n * 5 / 3), region=n * 555, n_reads=n)
        ptr.append(fr.frag_ptr[1:] + ptr[-1][-1])
        parts.append((fr.snp + np.int32(snps), fr.allele, fr.qual, fr.is_porec))
        snps += fr.n_snps
    snp, al, q, pc = (np.concatenate(c) for c in zip(*parts))
    return synth.Fragments(snps, np.concatenate(ptr), snp, al, q, pc, np.arange(snps),
                           np.ones(snps, np.int8))


@pytest.mark.parametrize("precision,R", [(qhap.PREC_FP32, 16), (qhap.PREC_BF16, 64),
                                         (qhap.PREC_BF16, 128), (qhap.PREC_FP8, 64)])
def test_auto_schedule_equals_each_length(precision, R):
    """A block's result does not depend on the other blocks' schedule length (same bits)."""
    ctx = qhap.Context(0)
    g = ctx.build_graph(_two_blocks(), mode=qhap.MODE_READ)
    sizes = g.block_sizes()
    kernel = "cta-bn64-s2-x4" if (precision, R) == (qhap.PREC_BF16, 64) else \
        "multistep-stream-tile" if precision == qhap.PREC_BF16 else None
    kw = dict(replicas=R, precision=precision, seed=4, step_kernel=kernel)
    auto = ctx.solve(g, schedule=qhap.SCHED_AUTO, **kw).cuts()
    want = {n: ctx.solve(g, steps=n, **kw).cuts() for n in (500, 1000)}
    assert (sizes >= 5000).any() and (sizes < 5000).any()
    for b in range(g.n_blocks):
        assert np.array_equal(auto[b], want[1000 if sizes[b] >= 5000 else 500][b])
    g.free()
    ctx.close()


@pytest.mark.parametrize("precision,kernel", [(qhap.PREC_FP32, None),
                                              (qhap.PREC_BF16, "cta-bn64-s2-x4"),
                                              (qhap.PREC_BF16, "multistep-stream-tile")])
@pytest.mark.parametrize("steps", [3, 1000, 1 << 20, (1 << 20) + 1])
def test_coefficients_of_one_step(precision, kernel, steps):
    """One step from a known state against the update in FP64 from the library's own product.
    FP32 rounds y' and x' at most five times each, at magnitudes below 0.5: 5 2^-25 < 2e-7
    absolute (the multi-step kernel rounds y once more through y / (dt c0): 3e-7)."""
    import torch

    R, dt = 128, 0.1
    ctx = qhap.Context(0)
    g = ctx.build_graph(synth.hifi_region(6, scale=0.02), mode=qhap.MODE_READ)
    n_pad, pidx, c0 = g.layout()
    live = pidx[pidx >= 0]
    bo, _ = g.blocks()
    cb = c0[bo[pidx >= 0]]
    for t in sorted({0, steps // 2, steps - 1}):
        x = torch.empty(R, n_pad, device="cuda")
        y = torch.empty(R, n_pad, device="cuda")
        ctx.debug_init_state(g, R, x, y, seed=9)
        z = torch.zeros(R, n_pad, device="cuda")
        ctx.debug_matvec(g, precision, R, x, z)
        x0, y0, z0 = (a.cpu().numpy().astype(np.float64)[:, live] for a in (x, y, z))
        ctx.debug_steps(g, precision, R, x, y, t, 1, steps, dt=dt, step_kernel=kernel)
        y1 = y0 + np.float64(np.float32(dt)) * (-(1.0 - t / steps) * x0 +
                                                cb.astype(np.float32).astype(np.float64) * z0)
        x1 = x0 + np.float64(np.float32(dt)) * y1
        assert np.abs(x1).max() < 0.5 and np.abs(y1).max() < 0.5
        assert np.abs(y.cpu().numpy()[:, live] - y1).max() < 3e-7
        assert np.abs(x.cpu().numpy()[:, live] - x1).max() < 3e-7
    g.free()
    ctx.close()
