"""The FP32 step's chunk records beyond 2^20 stored tiles (64 GiB of FP32 tiles), where 32-bit
chunk offsets end: the packing on the host at tile counts that need no memory, and the
product of one dense block of 1,025 x 1,025 tiles on the GPU."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2603_25762_gb300", "csrc")

HARNESS = r"""
#include <stdio.h>
#include "chunk.cuh"
int main(void) {
  const int64_t begins[] = {0, 1, 47, (1 << 20) - 1025, (1 << 20) - 1, 1 << 20, (1 << 21) + 3, 3100000};
  const int32_t tiles[] = {0, 1, 1023, 1024, 4095};
  long bad = 0;
  for (int64_t b : begins)
    for (int32_t e : tiles)
      for (int32_t c = 0; c < 16; ++c) {
        const int32_t rec = qh::f32_chunk(e, c);
        const int64_t want = (b + e) * 16384 + 8 * c;  /* tiles of 128 x 128, chunks of 8 columns */
        const float* at = qh::f32_chunk_at((const float*)64, qh::f32_row_chunk((int32_t)b), rec);
        if (rec < 0 || (int64_t)(uintptr_t)at != 64 + 4 * want) ++bad;
      }
  printf("bad %ld\n", bad);
  return bad != 0;
}
"""


def test_chunk_offsets(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src = tmp_path / "chunk_check.cpp"
    src.write_text(HARNESS)
    exe = tmp_path / "chunk_check"
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "bad 0", out.stdout


@pytest.mark.gpu
def test_product_past_two_to_the_twenty_tiles():
    """A chain of reads (read i covers SNPs i and i + 1), stored dense: 103 GB of tiles.  x in
    multiples of 1/64 and weights +-1: every product and sum is exact (tolerance 0)."""
    import torch

    from paper_2603_25762_gb300 import qhap, synth

    if torch.cuda.mem_get_info()[0] < 140 << 30:
        pytest.skip("needs 140 GiB of free device memory")
    n, R = 131_100, 2
    rng = np.random.default_rng(1)
    snp = (np.arange(n)[:, None] + np.arange(2)).astype(np.int32).ravel()
    al = rng.choice(np.array([-1, 1], np.int8), size=2 * n)
    fr = synth.Fragments(n + 1, 2 * np.arange(n + 1, dtype=np.int64), snp, al,
                         np.full(2 * n, 30, np.uint8), np.zeros(n, np.uint8), np.arange(n + 1),
                         np.ones(n + 1, np.int8))
    ctx = qhap.Context(0)
    g = ctx.build_graph(fr, mode=qhap.MODE_READ, dense=True)
    n_pad, pidx, _ = g.layout()
    assert (n_pad // 128) ** 2 > 1 << 20
    live = np.flatnonzero(pidx >= 0)
    x = np.zeros((R, n_pad), np.float32)
    x[:, pidx[live]] = rng.integers(-64, 65, size=(R, live.size)) / 64.0
    rp, col, w = g.edges()
    row = np.repeat(np.arange(g.n_nodes), np.diff(rp))
    want = np.zeros((R, n_pad))
    for r in range(R):
        np.add.at(want[r], pidx[row], -w * x[r, pidx[col]])
    xt = torch.from_numpy(x).cuda()
    z = torch.zeros(R, n_pad, device="cuda")
    ctx.debug_matvec(g, qhap.PREC_FP32, R, xt, z)
    assert np.array_equal(z.cpu().numpy()[:, pidx[live]].astype(np.float64), want[:, pidx[live]])
    g.free()
    ctx.close()
