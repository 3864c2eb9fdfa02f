"""Shared memory of the batched FP32 sampler, on the host: what a plan reserves covers the layout
of every lattice in it.

The size is not monotonic in the bond pad (the ring of site tensors holds three up to a pad of
32 and two above), so a plan whose largest pad is 36 may hold a lattice of pad 32 that needs
more.  The host functions of the kernel's header are compiled into a small program and evaluated
over pads, widths, samples per lane and warps.  A second program checks that every lattice the API
accepts (up to 4096 columns, pads up to 64) gets a launch that fits, whatever the number of samples.
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

PLANS = r"""
#include <stdio.h>
#include "sample_f32_kernel.cuh"
#include "sample_f64_kernel.cuh"
int main() {
  using namespace tnmc;
  const size_t block = 232448, sm = 233472;      // shared memory of a CTA and of an SM
  const int64_t totals[] = {1, 33, 700, 5000, 9001, 20000, 65536, 1 << 20};
  long cases = 0, bad = 0, edge = 0;
  for (int P = 4; P <= 64; P += 4)
    for (int Lx = 1; Lx <= 4096; Lx += Lx < 64 ? 21 : 167 + (Lx > 3800))
      for (int64_t total : totals) {
        const F64Plan d = f64_plan(total, P, 152, sm, [&](int S, bool e) { return f64_tile_smem(P, Lx, S, e); });
        ++cases;
        bad += d.smem > block || d.smem != f64_tile_smem(P, Lx, d.S, d.edge) || d.S / 8 * P > 64;
        edge += d.edge;
        for (int strong = 0; strong < 2; ++strong, ++cases) {
          const F32Plan f = f32_plan(total, P, strong, 152, block, sm,
                                     [&](int SB, int NW, bool e) { return f32_smem(P, Lx, SB, NW, e).total; },
                                     [&](int) { return 4; });
          bad += f.NW < 1 || f.smem > block || f.smem != f32_smem(P, Lx, f.SB, f.NW, f.edge).total ||
                 (strong && !f.edge) || (f.edge && f.SB == 8) || f.SB > f32_block(total, P, 152);
          edge += f.edge;
        }
      }
  printf("%ld %ld %ld\n", cases, bad, edge);
  return 0;
}
"""


def _run(tmp_path, program):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "smem.cu", tmp_path / "smem"
    src.write_text(program)
    subprocess.run([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a",
                    "--expt-relaxed-constexpr", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return map(int, subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())


def test_every_accepted_lattice_gets_a_launch(tmp_path):
    cases, bad, edge = _run(tmp_path, PLANS)
    assert cases > 10000 and bad == 0 and 0 < edge < cases


def test_reservation_covers_every_lattice(tmp_path):
    cases, bad, shrinks = _run(tmp_path, PROGRAM)
    assert cases == 2 * 4 * 3 * 80 * 80
    assert bad == 0
    # the pairs for which the layout of the largest pad and width would have been too small exist
    assert shrinks > 0
