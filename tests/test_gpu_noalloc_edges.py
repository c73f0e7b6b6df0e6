"""qh_matvec_bf16_noalloc: inputs that are only 4-byte aligned, outputs that held other
values (padding vertices get zeros), several blocks; equal to the debug product."""
import numpy as np
import pytest

from paper_2603_25762_gb300 import qhap, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("reads,R", [(2, 64), (127, 128), (129, 64), (700, 192), (0, 64)])
@pytest.mark.parametrize("off", [0, 1])
def test_product_alignment_and_padding(reads, R, off):
    import torch

    ctx = qhap.Context(0)
    fr = synth.batched_blocks(5, n_blocks=3, n_max=300) if reads == 0 else \
        synth.region_reads(5, n_snps=max(8, reads * 2), region=max(15_000, reads * 555),
                           n_reads=reads)
    g = ctx.build_graph(fr, mode=qhap.MODE_READ)
    n_pad, pidx, _ = g.layout()
    n = R * n_pad
    gen = torch.Generator().manual_seed(reads + R)
    x = torch.zeros(n + 1, device="cuda")
    xv = x[off:off + n].view(R, n_pad)
    live = torch.from_numpy(pidx[pidx >= 0].astype(np.int64))
    xv[:, live.cuda()] = (2 * torch.rand(R, live.numel(), generator=gen) - 1).cuda()
    z = torch.full((n + 1,), 7.0, device="cuda")
    zv = z[off:off + n].view(R, n_pad)
    torch.cuda.synchronize()
    ctx.matvec_bf16_noalloc(g, R, xv, zv)
    want = torch.zeros(R, n_pad, device="cuda")
    ctx.debug_matvec(g, qhap.PREC_BF16, R, xv.contiguous().clone(), want)
    assert torch.equal(zv, want)
    pad = np.setdiff1d(np.arange(n_pad), pidx)
    assert not zv[:, torch.from_numpy(pad).cuda()].any()
    assert z[n if off == 0 else 0].item() == 7.0  # nothing outside the output
    g.free()
    ctx.close()
