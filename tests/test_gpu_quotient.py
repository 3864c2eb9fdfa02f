"""The FP64 sampler's division (needs a GB300): quotient_f64 against the compiler's division.

A small program over the kernel's header divides 2^24 pairs w <= t, t over the range the
sampler uses it in.  With a reciprocal within half a unit and a little, the residual step rounds to
nearest except next to a tie: at most one result in 2^20 may differ, by one unit in the last place.
"""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2104_13264_gb300", "csrc")

PROGRAM = r"""
#include <stdio.h>
#include "sample_f64_kernel.cuh"
using namespace tnmc;
__device__ unsigned long long mix(unsigned long long z) {
  z += 0x9e3779b97f4a7c15ull;
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}
// out: [0] quotients that differ, [1] by more than one unit, [2] products that differ
__global__ void compare(unsigned long long* out) {
  const unsigned long long i = blockIdx.x * 256ull + threadIdx.x;
  const unsigned long long a = mix(2 * i), b = mix(2 * i + 1);
  const int e = (int)(a >> 52) % 1800 - 900, d = (int)(b >> 52) % 40;
  const double t = __longlong_as_double((a & 0xfffffffffffffull) | (1023ull + e) << 52);
  double w = __longlong_as_double((b & 0xfffffffffffffull) | (1023ull + e - d) << 52);
  if (w > t) w *= 0.5;
  const double r = reciprocal_f64(t), q = quotient_f64(w, t, r), ref = w / t;
  const long long diff = llabs(__double_as_longlong(q) - __double_as_longlong(ref));
  if (diff) atomicAdd(out, 1ull);
  if (diff > 1) atomicAdd(out + 1, 1ull);
  if (w * r != ref) atomicAdd(out + 2, 1ull);
}
int main() {
  unsigned long long h[3], *d;
  if (cudaMalloc(&d, sizeof(h)) || cudaMemset(d, 0, sizeof(h))) return 1;
  compare<<<1 << 16, 256>>>(d);
  if (cudaMemcpy(h, d, sizeof(h), cudaMemcpyDeviceToHost)) return 1;
  printf("%llu %llu %llu\n", h[0], h[1], h[2]);
  return 0;
}
"""


def test_quotient_rounds_to_nearest(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    src, exe = tmp_path / "quotient.cu", tmp_path / "quotient"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-O3", "-gencode", "arch=compute_103a,code=sm_103a",
                    "--expt-relaxed-constexpr", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    differ, far, products = map(int, out.split())
    print(differ, far, products)
    assert far == 0 and differ <= 16
    assert products > 1000000        # what the residual step is for
