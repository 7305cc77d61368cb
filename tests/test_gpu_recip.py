"""The layout kernels' own reciprocals and reciprocal square roots (csrc/recip.cuh)
against CUDA's, over the exponents they are used at and beyond, in a small
program compiled from that header: FP32 and FP64 reciprocals and the FP64
reciprocal square root are at most one unit in the last place off, and the
special values are those of the plain formula."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <math.h>
#include <stdio.h>
#include <string.h>
#include "recip.cuh"
using namespace pprviz;

__device__ long long ulps(float a, float b) { return llabs((long long)__float_as_int(a) - __float_as_int(b)); }
__device__ long long ulps(double a, double b) { return llabs(__double_as_longlong(a) - __double_as_longlong(b)); }

// every FP32 mantissa at the exponent e
__global__ void k_rcp32(int e, unsigned long long *worst) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  const float a = __int_as_float(((127 + e) << 23) | m);
  atomicMax(worst, (unsigned long long)ulps(rcp_pos(a), __frcp_rn(a)));
}
// FP64: a mantissa from a counter (splitmix64), the exponent e
__device__ double number(long long i, int e) {
  unsigned long long z = (unsigned long long)i * 0x9e3779b97f4a7c15ull + 0x1234567ull;
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  z ^= z >> 31;
  return __longlong_as_double(((long long)(1023 + e) << 52) | (long long)(z & 0xfffffffffffffull));
}
__global__ void k_64(int e, unsigned long long *rcp, unsigned long long *rsq) {
  const double a = number((long long)blockIdx.x * blockDim.x + threadIdx.x + ((long long)(e + 1100) << 32), e);
  if (rcp) atomicMax(rcp, (unsigned long long)ulps(rcp_pos(a), __drcp_rn(a)));
  atomicMax(rsq, (unsigned long long)ulps(rsqrt_pos(a), rsqrt(a)));
}
__global__ void k_special(const double *in, double *out, int n) {
  if ((int)threadIdx.x < n) out[threadIdx.x] = rsqrt_pos(in[threadIdx.x]);
}

int main() {
  unsigned long long *d, h[3] = {0, 0, 0};
  if (cudaMalloc(&d, sizeof(h)) != cudaSuccess) return 2;
  cudaMemset(d, 0, sizeof(h));
  for (int e = -60; e <= 60; e += 4) k_rcp32<<<(1 << 23) / 256, 256>>>(e, d);
  for (int e = -1000; e <= 1000; e += 25) k_64<<<4096, 256>>>(e, d + 1, d + 2);
  for (int e = -1022; e <= 1023; ++e) k_64<<<16, 256>>>(e, nullptr, d + 2);
  if (cudaMemcpy(h, d, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
  const double in[8] = {0.0, -0.0, INFINITY, NAN, -1.0, 4.9e-324, 1e-310, 1.7976931348623157e308};
  double *di, *dout, out[8];
  cudaMalloc(&di, sizeof(in));
  cudaMalloc(&dout, sizeof(in));
  cudaMemcpy(di, in, sizeof(in), cudaMemcpyHostToDevice);
  k_special<<<1, 32>>>(di, dout, 8);
  if (cudaMemcpy(out, dout, sizeof(out), cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
  bool ok = true;
  for (int i = 0; i < 8; ++i) {
    const double want = in[i] > 0.0 ? 1.0 / sqrt(in[i]) : 0.0;
    ok = ok && fabs(out[i] - want) <= 4e-16 * want;
  }
  printf("%llu %llu %llu %d\n", h[0], h[1], h[2], (int)ok);
  return 0;
}
"""


def test_reciprocals_against_cudas(tmp_path):
    from paper_2112_14944_gb300 import build as b
    src, exe = tmp_path / "recip.cu", tmp_path / "recip"
    src.write_text(SOURCE)
    subprocess.run([b.nvcc(), *b.ARCH, "-std=c++17", "-O3", "-I", b.CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, env=dict(os.environ)).stdout.split()
    rcp32, rcp64, rsq64, special = map(int, out)
    assert rcp32 <= 1 and rcp64 <= 1 and rsq64 <= 1 and special == 1
