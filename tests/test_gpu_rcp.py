"""rcp_fp64 (the FP64 steps' reciprocal) against the correctly rounded 1.0 / x: at most one
unit in the last place over [2^-32, 2^32], the residual of the hardware's approximation that
this rests on below 2^-19.9, and what it gives outside (no NaN from a finite normal x)."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# 2^20 pseudo-random mantissas and the 64 next to each power of two, for every exponent.
PROGRAM = r"""
#include <cstdio>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include "lbm.h"
#include "lbm_device.cuh"

__global__ void k_check(int e0, unsigned long long* ulps, unsigned* resid, int* nans) {
  const unsigned n = blockIdx.x * blockDim.x + threadIdx.x;
  const long long m = n < 64 ? n : n < 128 ? (1ll << 52) - 1 - (n - 64)
                               : ((long long)lbm::mix32(n) << 20 ^ lbm::mix32(n * 2654435761u + blockIdx.y)) & ((1ll << 52) - 1);
  const double x = __longlong_as_double((long long)(e0 + int(blockIdx.y) + 1023) << 52 | m);
  const double r = lbm::rcp_fp64(x), want = 1.0 / x;
  const long long d = __double_as_longlong(r) - __double_as_longlong(want);
  double a;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(a) : "d"(x));
  if (r != r) atomicAdd(nans, 1);
  const unsigned long long u = d < 0 ? -d : d;
  const unsigned e = __float_as_uint(float(fabs(__fma_rn(-x, a, 1.0))));
  if (u > *(volatile unsigned long long*)ulps) atomicMax(ulps, u);
  if (e > *(volatile unsigned*)resid) atomicMax(resid, e);
}

int main() {
  unsigned long long* ulps;
  unsigned* resid;
  int* nans;
  cudaMallocManaged(&ulps, 8), cudaMallocManaged(&resid, 4), cudaMallocManaged(&nans, 4);
  const int ranges[3][2] = {{-32, 65}, {-1000, 968}, {33, 967}};
  for (auto& r : ranges) {
    *ulps = 0, *resid = 0, *nans = 0;
    k_check<<<dim3(r[1] > 100 ? 16 : 4096, r[1]), 256>>>(r[0], ulps, resid, nans);
    if (cudaDeviceSynchronize() != cudaSuccess) return 1;
    float f;
    __builtin_memcpy(&f, resid, 4);
    std::printf("%llu %.9g %d\n", *ulps, double(f), *nans);
  }
  return 0;
}
"""


def test_reciprocal(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1809_02390_gb300 import build

    src, exe = tmp_path / "rcp.cu", tmp_path / "rcp"
    src.write_text(PROGRAM)
    subprocess.run([build.NVCC, *build.ARCH, "-O3", "-std=c++17", "-I" + os.path.join(ROOT, "include"),
                    "-I" + build.CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split("\n")
    (ulps, resid, nans), *others = [[float(v) for v in line.split()] for line in out[:3]]
    assert ulps <= 1 and resid < 2.0 ** -19.9 and nans == 0
    for u, _, n in others:
        assert u <= 1 and n == 0
