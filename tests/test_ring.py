"""The multi-step kernel's producer, once its waits give up: the ring uses it must see land
before the CTA exits (csrc/ring.cuh), against a simulation of batches of copies over ring
slots.  The header is plain C++; a GPU run in which a wait runs out mid-batch is not made."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2603_25762_gb300", "csrc")

HARNESS = r"""
#include <stdio.h>
#include "ring.cuh"
static uint64_t state = 1;
static uint32_t rnd(uint32_t n) {
  state = state * 6364136223846793005ULL + 1442695040888963407ULL;
  return (uint32_t)(state >> 33) % n;
}
int main(void) {
  long bad = 0;
  for (int trial = 0; trial < 200000; ++trial) {
    const uint32_t st = rnd(2) ? 4 : 6;
    int64_t last[6] = {-1, -1, -1, -1, -1, -1};  /* latest use of each slot */
    uint32_t q = 0, part = 0;
    const uint32_t batches = rnd(7);
    for (uint32_t b = 0; b < batches; ++b) {     /* whole batches of 1 .. st copies */
      const uint32_t n = 1 + rnd(st);
      for (uint32_t l = 0; l < n; ++l) last[(q + l) % st] = q + l;
      q += n;
    }
    if (rnd(2)) {                                /* then one given up: any of its copies */
      part = rnd(1u << st);
      for (uint32_t l = 0; l < st; ++l)
        if ((part >> l) & 1u) last[(q + l) % st] = q + l;
    }
    int64_t seen[6] = {-1, -1, -1, -1, -1, -1};
    for (uint32_t l = 0; l < st; ++l) {
      uint32_t use;
      if (qh::ring_last_use(q, part, l, st, &use)) {
        if (seen[use % st] >= 0) ++bad;          /* a slot is waited for once */
        seen[use % st] = use;
      }
    }
    for (uint32_t s = 0; s < st; ++s) bad += seen[s] != last[s];
  }
  printf("bad %ld\n", bad);
  return bad != 0;
}
"""


def test_every_slot_in_flight_is_waited_for(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src = tmp_path / "ring_check.cpp"
    src.write_text(HARNESS)
    exe = tmp_path / "ring_check"
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "bad 0", out.stdout
