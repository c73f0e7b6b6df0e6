"""The tensor-core steps walk only the 64-column K-slices of J that hold a nonzero.  A
slice of zeros adds exact zeros, so a graph stored with every tile and slice (dense) must
give the same bits (tolerance 0)."""
import numpy as np
import pytest

from paper_2603_25762_gb300 import qhap, synth

pytestmark = pytest.mark.gpu


# sizes around one tile and its halves (a last tile of 1, 63, 64, 65 rows), and several tiles
@pytest.mark.parametrize("reads,mode,precision", [
    (65, "read", qhap.PREC_BF16), (129, "read", qhap.PREC_BF16), (191, "read", qhap.PREC_BF16),
    (192, "read", qhap.PREC_BF16), (321, "read", qhap.PREC_BF16), (700, "read", qhap.PREC_BF16),
    (120, "snp", qhap.PREC_BF16), (250, "snp", qhap.PREC_BF16X2)])
def test_slices_equal_dense(reads, mode, precision):
    import torch

    R = 256
    if mode == "read":
        fr = synth.region_reads(11, n_snps=round(reads * 5 / 3), region=reads * 555, n_reads=reads)
    else:
        fr = synth.region_reads(11, n_snps=round(reads * 10 / 3), region=reads * 1111,
                                n_reads=reads, len_mean=30_000, len_sd=20_000, len_max=150_000,
                                flip_p=0.06, miss_p=0.0, qual=(7, 30))
    ctx = qhap.Context(0)
    m = qhap.MODE_READ if mode == "read" else qhap.MODE_SNP
    graphs = [ctx.build_graph(fr, mode=m, dense=d) for d in (False, True)]
    n_pad, _, _ = graphs[0].layout()
    ran = 0
    for kernel in qhap.STEP_KERNELS[:10]:
        out = []
        for g in graphs:
            x = torch.empty(R, n_pad, device="cuda")
            y = torch.empty(R, n_pad, device="cuda")
            ctx.debug_init_state(g, R, x, y)
            try:
                ctx.debug_steps(g, precision, R, x, y, 0, 7, 40, step_kernel=kernel)
            except qhap.QhError as e:  # this variant does not fit (resident tiles)
                assert e.status == qhap.QH_EINVAL and "jres" in kernel
                break
            out.append((x.cpu().numpy(), y.cpu().numpy()))
        if len(out) < 2:
            continue
        ran += 1
        assert np.array_equal(out[0][0], out[1][0]), kernel
        assert np.array_equal(out[0][1], out[1][1]), kernel
    assert ran >= 8
    for g in graphs:
        g.free()
    ctx.close()
