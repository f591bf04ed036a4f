"""The PLIC geometry's quotients (rcp_of, div_by, inv_of, third_of of
csrc/vof_device.cuh: a reciprocal on the FP32 and integer units, then two fused
multiply-adds) against CUDA's division, bit for bit.

A small program is compiled with the library's own flags and run.  Operands:
random significands; significands at and next to 1, 1.5 and 2 (quotients next to
the middle of two numbers among them); both signs; exponents inside, at and just
outside the window of the fast path; zeros, subnormals, infinities and NaN; and
warps in which fast and fallback lanes mix."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include <cuda_runtime.h>
#include "vof_device.cuh"
using namespace vofgb;
__device__ unsigned long long mix(unsigned long long z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
__device__ double from(unsigned long long sign, int field, unsigned long long frac) {
  return __longlong_as_double((long long)((sign & 1ull) << 63 | (unsigned long long)field << 52 | (frac & 0xFFFFFFFFFFFFFull)));
}
// significands at and next to 1, 2, 1.5, and where the top 24 bits change
__device__ unsigned long long edge_frac(int k) {
  const unsigned long long b[8] = {0ull, 1ull, 2ull, 0xFFFFFFFFFFFFFull, 0xFFFFFFFFFFFFEull, 0x8000000000000ull, 0x1FFFFFFFull, 0x20000000ull};
  return b[k & 7];
}
// family 0: random; 1: edge significands; 2: edges of the exponent window;
// 3: special values mixed into warps of ordinary ones
__device__ double operand(int family, unsigned long long r, int i, bool numerator) {
  const unsigned long long f = mix(r);
  if (family == 0) return from(r, 1023 - 200 + (int)((r >> 8) % 400), f);
  if (family == 1) return from(r, 1023 - 3 + (int)((r >> 8) % 6), (r >> 20 & 1) ? edge_frac((int)(r >> 24)) : f);
  if (family == 2) {
    const int e[6] = {572, 573, 574, 1471, 1472, 1473};
    return from(r, e[(r >> 8) % 6], (r >> 20 & 3) ? f : edge_frac((int)(r >> 24)));
  }
  if ((r >> 12) % 5) return from(r, 1023 - 40 + (int)((r >> 8) % 80), f);
  switch ((r >> 30) % 6) {
    case 0: return numerator ? __longlong_as_double((long long)(r & 1ull) << 63) : 1.0;  // (zeros only above the line)
    case 1: return from(r, 0, f);       // subnormal
    case 2: return from(r, 2046, f);
    case 3: return from(r, 1, f);
    case 4: return from(r, 2047, 0);    // infinity
    default: return from(r, 2047, 1ull << 51);
  }
}
__device__ bool same(double a, double b) {  // (any NaN equals any NaN)
  const long long x = __double_as_longlong(a), y = __double_as_longlong(b), top = 0x7FF0000000000000ll;
  return x == y || ((x & 0x7FFFFFFFFFFFFFFFll) > top && (y & 0x7FFFFFFFFFFFFFFFll) > top);
}
__global__ void quotients(int family, unsigned long long seed, unsigned n, unsigned long long* bad) {
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    double b = operand(family, mix(seed + 2ull * i), (int)i, false);
    const double a = operand(family, mix(seed + 2ull * i + 1ull), (int)i, true);
    if (!dnz(a)) b = fabs(b);  // b > 0 wherever a may be 0 (the callers' promise)
    const Rcp R = rcp_of(b);
    if (!same(div_by(a, R), a / b)) atomicAdd(bad, 1ull);
    if (!same(inv_of(R), 1.0 / b)) atomicAdd(bad + 1, 1ull);
    // third_of has no fallback: its callers' values are ordinary
    if (family < 2 && !same(third_of(a), a / 3.0)) atomicAdd(bad + 2, 1ull);
  }
}
int main(int argc, char** argv) {
  unsigned long long* d;
  unsigned long long h[3];
  if (cudaMalloc(&d, sizeof(h)) != cudaSuccess) return 2;
  for (int f = 0; f < 4; ++f) {
    cudaMemset(d, 0, sizeof(h));
    quotients<<<152 * 4, 256>>>(f, 77ull + 1000003ull * f, 1u << 22, d);
    if (cudaMemcpy(h, d, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
    printf("%llu %llu %llu\n", h[0], h[1], h[2]);
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def mismatches(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2001_03477_gb300 import build as B
    d = tmp_path_factory.mktemp("division")
    (d / "q.cu").write_text(PROGRAM)
    exe = str(d / "q")
    flags = [f for f in B.FLAGS if f not in ("-Xcompiler", "-fPIC", "-fvisibility=hidden")]
    subprocess.run([B.nvcc(), *B.ARCH, *flags, "-I", B.CSRC, "-I", os.path.join(B.ROOT, "include"), "-o", exe, str(d / "q.cu")],
                   check=True, timeout=300)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout
    return [[int(x) for x in line.split()] for line in out.splitlines()]


@pytest.mark.parametrize("family", range(4), ids=["random", "edge significands", "edges of the window", "special values"])
def test_quotients_are_cudas(mismatches, family):
    assert mismatches[family] == [0, 0, 0]
