"""The training kernels' SiLU and its derivative divide by a reciprocal with one
Newton step and one correction (Markstein 1990) instead of the compiler's
division. Here both are compared for every FP32 argument: the same bits, but for
SiLU(-0), which is +0."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

PROBE = r"""
#include <cstdio>
#include "ezo_mlp_gemm_tc.cu"

namespace ezo {
namespace {

__device__ bool same(float a, float b) { return __float_as_uint(a) == __float_as_uint(b) || (a != a && b != b); }

// thread i: the arguments with the bits 16 i .. 16 i + 15, one by one and as
// the sixteen values of a thread
__global__ void k_compare(unsigned long long* bad) {
  const unsigned first = (blockIdx.x * blockDim.x + threadIdx.x) * 16u;
  float z[16], silu[16], dsilu[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) z[j] = __uint_as_float(first + j);
  silu_n(z, silu);
  dsilu_n(z, dsilu);
  unsigned n[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const float s = 1.f / (1.f + __expf(-z[j])), d = s * (1.f + z[j] * (1.f - s));
    const float y = first + j == 0x80000000u ? 0.f : z[j] / (1.f + __expf(-z[j]));
    const float one[1] = {z[j]};
    float silu1[1], dsilu1[1];
    silu_n(one, silu1);
    dsilu_n(one, dsilu1);
    n[0] += !same(silu[j], y);
    n[1] += !same(silu1[0], y);
    n[2] += !same(dsilu[j], d);
    n[3] += !same(dsilu1[0], d);
  }
  for (int k = 0; k < 4; ++k)
    if (n[k]) atomicAdd(bad + k, (unsigned long long)n[k]);
}

}  // namespace
}  // namespace ezo

int main() {
  unsigned long long *bad = nullptr, host[4];
  if (cudaMalloc(&bad, sizeof(host)) != cudaSuccess || cudaMemset(bad, 0, sizeof(host)) != cudaSuccess) return 2;
  ezo::k_compare<<<1u << 20, 256>>>(bad);
  if (cudaMemcpy(host, bad, sizeof(host), cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
  std::printf("%llu %llu %llu %llu\n", host[0], host[1], host[2], host[3]);
  return 0;
}
"""


def test_every_argument_divides_as_the_plain_division(tmp_path):
    from paper_2504_10783_gb300 import build
    src, exe = tmp_path / "probe.cu", tmp_path / "probe"
    src.write_text(PROBE)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.split() == ["0"] * 4
