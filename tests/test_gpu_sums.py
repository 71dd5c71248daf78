"""The FP32 accumulators of the CG scalars (GPU), run in a program of their own against sums in 64 bits: each
product enters a compensated sum by itself, with one rounding."""
import subprocess

import numpy as np
import pytest

from paper_1411_0330_gb300 import build

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "common.cuh"
using namespace lsh;
__global__ void sums(int n, const float2* a, const float2* b, double* out) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  Acc2 two;
  Acc<float> one;
  for (int i = 0; i < n; ++i) {
    const float2 u = a[(long long)t * n + i], v = b[(long long)t * n + i];
    two.mac(u, v);
    one.mac(u.x, v.x);
    one.mac(u.y, v.y);
  }
  out[2 * t] = two.fold(2.f).get();
  out[2 * t + 1] = one.get();
}
int main(int, char** argv) {
  const int threads = 4096, n = 128;
  std::vector<float2> a(threads * n), b(threads * n);
  FILE* f = std::fopen(argv[1], "rb");
  if (!f || std::fread(a.data(), sizeof(float2), a.size(), f) != a.size() ||
      std::fread(b.data(), sizeof(float2), b.size(), f) != b.size())
    return 1;
  float2 *da, *db;
  double* d;
  const size_t bytes = sizeof(float2) * a.size();
  if (cudaMalloc(&da, bytes) || cudaMalloc(&db, bytes) || cudaMalloc(&d, 16 * threads)) return 2;
  cudaMemcpy(da, a.data(), bytes, cudaMemcpyHostToDevice);
  cudaMemcpy(db, b.data(), bytes, cudaMemcpyHostToDevice);
  sums<<<threads / 256, 256>>>(n, da, db, d);
  std::vector<double> h(2 * threads);
  if (cudaMemcpy(h.data(), d, 16 * threads, cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
  for (int t = 0; t < threads; ++t) std::printf("%.17g %.17g\n", h[2 * t], h[2 * t + 1]);
  return 0;
}
"""


@pytest.mark.parametrize("signs", [False, True])
def test_error_of_a_sum_of_products(tmp_path, signs):
    """One rounding of each product v: its error has a standard deviation of at most 2 u v / sqrt(12) = 0.578 u v
    (u = 2^-24), what an addition loses is kept (to u^2), so that a sum's error is at most 0.578 u sqrt(sum v^2)
    in the root mean square over many sums; 4096 of them know it to 1.1 %, four times that makes 0.604.
    Products summed four at a time in FP32 first would stand at about 1.9 without signs."""
    (tmp_path / "sums.cu").write_text(PROGRAM)
    exe = str(tmp_path / "sums")
    subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "-O3", "-I" + build.CSRC, "-o", exe,
                    str(tmp_path / "sums.cu")], check=True, capture_output=True)
    rng = np.random.default_rng(7)
    a, b = (rng.uniform(0.5, 2.0, (4096, 256)).astype(np.float32) for _ in range(2))
    if signs:
        b *= rng.choice([-1.0, 1.0], b.shape).astype(np.float32)
    with open(tmp_path / "data", "wb") as f:
        f.write(a.tobytes() + b.tobytes())
    out = subprocess.run([exe, str(tmp_path / "data")], check=True, capture_output=True, text=True).stdout
    two, one = np.array([[float(v) for v in line.split()] for line in out.splitlines()]).T
    p = a.astype(np.float64) * b
    exact, size = p.sum(1), np.sqrt((p * p).sum(1))
    for got in (two / 2, one):
        assert np.sqrt(np.mean(((got - exact) / size) ** 2)) < 0.604 * 2.0 ** -24
