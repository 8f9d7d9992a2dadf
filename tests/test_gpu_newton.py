"""The selection's reciprocal root and quotient (csrc/newton.cuh) against float64 and against CUDA's own
1.0f / sqrtf(x) and a / r, by a small program built from the header with nvcc."""
import os
import shutil
import subprocess

import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_06411_gb300", "csrc")

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include "newton.cuh"
struct Result { unsigned long long root, cuda_root, quot, differ; };   // worst errors in ulp (bits of a double)
__device__ void worst(unsigned long long* p, double got, double exact) {
  const double u = fabs(got - exact) / ldexp(1.0, ilogb(exact) - 23);
  atomicMax(p, static_cast<unsigned long long>(__double_as_longlong(u)));
}
__device__ unsigned rnd(unsigned& s) { s ^= s << 13; s ^= s >> 17; s ^= s << 5; return s; }
__global__ void roots(Result* r) {   // every mantissa of [1, 4), at several powers of 4
  const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
  for (int e = -60; e <= 60; e += 20) {
    const float x = ldexpf(__uint_as_float(0x3f800000u + i), 2 * e);
    const double exact = 1.0 / sqrt(static_cast<double>(x));
    worst(&r->root, mapk::inv_sqrt(x), exact);
    worst(&r->cuda_root, 1.0f / sqrtf(x), exact);
  }
}
__global__ void quotients(Result* r) {
  unsigned s = 2654435761u * (blockIdx.x * blockDim.x + threadIdx.x + 1u);
  for (int k = 0; k < 64; ++k) {
    const float d = ldexpf(__uint_as_float(0x3f800000u | (rnd(s) >> 9)), static_cast<int>(rnd(s) % 61u) - 30);
    const float a = ldexpf(__uint_as_float(0x3f800000u | (rnd(s) >> 9)), static_cast<int>(rnd(s) % 61u) - 30) *
                    ((rnd(s) & 1u) ? -1.f : 1.f);
    const float q = mapk::quotient(a, d, 1.0f / d);
    worst(&r->quot, q, static_cast<double>(a) / static_cast<double>(d));
    if (q != a / d) atomicAdd(&r->differ, 1ull);
  }
}
__global__ void edges(Result* r, float* out) { out[0] = mapk::inv_sqrt(INFINITY); out[1] = mapk::inv_sqrt(1.0f); }
int main() {
  Result* r; float* out;
  if (cudaMalloc(&r, sizeof(Result)) || cudaMemset(r, 0, sizeof(Result)) || cudaMalloc(&out, 8)) return 1;
  roots<<<(1 << 24) / 256, 256>>>(r);
  quotients<<<(1 << 20) / 256, 256>>>(r);
  edges<<<1, 1>>>(r, out);
  Result h; float o[2];
  if (cudaMemcpy(&h, r, sizeof(h), cudaMemcpyDeviceToHost) || cudaMemcpy(o, out, 8, cudaMemcpyDeviceToHost)) return 1;
  auto d = [](unsigned long long b) { double x; __builtin_memcpy(&x, &b, 8); return x; };
  std::printf("%.9f %.9f %.9f %llu %g %g\n", d(h.root), d(h.cuda_root), d(h.quot), h.differ, o[0], o[1]);
  return 0;
}
"""


def test_reciprocal_root_and_quotient_errors(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    src = tmp_path / "newton.cu"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-I", CSRC, str(src),
                    "-o", str(tmp_path / "newton")], check=True, capture_output=True)
    out = subprocess.run([str(tmp_path / "newton")], check=True, capture_output=True, text=True).stdout.split()
    root, cuda_root, quot, differ, at_inf, at_one = (float(v) for v in out)
    # rsqrtf is 2 ulp off at most; the step squares that (2^-43) and rounds its correction and the sum
    assert root < 1.0 and root < cuda_root
    # the correction's own error is 2^-23 of it: half an ulp from the last rounding, and no more than 2^-20 beside
    assert quot <= 0.5 + 2.0 ** -20
    assert differ <= 64 * 2 ** 20 * 2.0 ** -20          # a last bit may differ next to a tie only
    assert at_inf == 0.0 and at_one == 1.0
