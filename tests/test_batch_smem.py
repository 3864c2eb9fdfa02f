"""Shared memory of the batched FP32 sampler, on the host: what a plan reserves covers the layout
of every lattice in it.

The size is not monotonic in the bond pad (the ring of site tensors holds three up to a pad of
32 and two above), so a plan whose largest pad is 36 may hold a lattice of pad 32 that needs
more.  The host functions of the kernel's header are compiled into a small program and evaluated
over pads, widths, samples per lane and warps.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2104_13264_gb300", "csrc")

PROGRAM = r"""
#include <stdio.h>
#include "sample_f32_kernel.cuh"
int main() {
  using namespace tnmc;
  const int pads[] = {4, 8, 16, 20, 28, 32, 36, 40, 48, 64}, widths[] = {1, 8, 31, 32, 33, 64, 250, 1024};
  const int np = 10, nl = 8;
  long bad = 0, shrinks = 0, cases = 0;
  for (int edge = 0; edge < 2; ++edge)
  for (int SB = 1; SB <= 8; SB *= 2)
    for (int NW = 1; NW <= 4; NW *= 2)
      for (int i = 0; i < np * nl; ++i)
        for (int j = 0; j < np * nl; ++j, ++cases) {
          const int P[2] = {pads[i / nl], pads[j / nl]}, L[2] = {widths[i % nl], widths[j % nl]};
          const size_t r = f32_smem_largest(2, [&](int k) { return P[k]; }, [&](int k) { return L[k]; }, SB, NW, edge);
          for (int k = 0; k < 2; ++k) bad += f32_smem(P[k], L[k], SB, NW, edge).total > r;
          const size_t corner = f32_smem(P[0] > P[1] ? P[0] : P[1], L[0] > L[1] ? L[0] : L[1], SB, NW, edge).total;
          shrinks += r > corner;
        }
  printf("%ld %ld %ld\n", cases, bad, shrinks);
  return 0;
}
"""


def test_reservation_covers_every_lattice(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "smem.cu", tmp_path / "smem"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a",
                    "--expt-relaxed-constexpr", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    cases, bad, shrinks = map(int, out.split())
    assert cases == 2 * 4 * 3 * 80 * 80
    assert bad == 0
    # the pairs for which the layout of the largest pad and width would have been too small exist
    assert shrinks > 0
