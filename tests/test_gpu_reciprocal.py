"""The FP64 reciprocal that the bond, force and gradient passes take (a hardware
approximation and two Newton-Raphson steps where those hold, a division
elsewhere) against CUDA's division: over all exponents, both signs, denormals,
zeros, infinities and NaN, and densely about the ends of the approximation's
range and over the lengths and denominators of the potential."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

SOURCE = r'''
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>
#include "internal.cuh"
__global__ void k(int n, const double* x, double* a, double* b) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  a[i] = ct::inv(x[i]);
  b[i] = 1.0 / x[i];
}
int main() {
  std::vector<double> x;
  unsigned long long s = 88172645463325252ull;
  auto rnd = [&]() { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return s; };
  auto bits = [](unsigned long long u) { double d; memcpy(&d, &u, 8); return d; };
  const unsigned long long frac = (1ull << 52) - 1;
  for (unsigned long long e = 0; e < 2048; ++e)            // every exponent: ends, middle, random
    for (int k = 0; k < 64; ++k) {
      unsigned long long m = k == 0 ? 0 : k == 1 ? frac : k == 2 ? 1ull << 51 : k == 3 ? 1 : rnd() & frac;
      x.push_back(bits(e << 52 | m));
      x.push_back(bits(1ull << 63 | e << 52 | m));
    }
  for (unsigned long long e : {122ull, 123ull, 1922ull, 1923ull})   // about the ends of the window
    for (int k = 0; k < 4096; ++k) x.push_back(bits(e << 52 | (rnd() & frac)));
  for (int k = 0; k < 1 << 20; ++k) x.push_back(std::pow(10.0, -3.0 + 6.0 * k / (1 << 20)) * (1.0 + 1e-9 * (rnd() % 1000)));
  const int n = (int)x.size();
  double *dx, *da, *db;
  cudaMalloc(&dx, n * 8); cudaMalloc(&da, n * 8); cudaMalloc(&db, n * 8);
  cudaMemcpy(dx, x.data(), n * 8, cudaMemcpyHostToDevice);
  k<<<(n + 255) / 256, 256>>>(n, dx, da, db);
  if (cudaDeviceSynchronize() != cudaSuccess) return 1;
  std::vector<double> a(n), b(n);
  cudaMemcpy(a.data(), da, n * 8, cudaMemcpyDeviceToHost);
  cudaMemcpy(b.data(), db, n * 8, cudaMemcpyDeviceToHost);
  long long worst = 0, kind = 0, off = 0;
  for (int i = 0; i < n; ++i) {
    long long p, q;
    memcpy(&p, &a[i], 8); memcpy(&q, &b[i], 8);
    if (std::isnan(b[i])) { kind += !std::isnan(a[i]); continue; }
    if (std::isnan(a[i]) || std::signbit(a[i]) != std::signbit(b[i])) { ++kind; continue; }
    long long d = llabs(p - q);
    if (d > worst) worst = d;
    off += d != 0;
  }
  printf("%lld %lld %lld %d\n", worst, kind, off, n);
}
'''


def test_inv_is_within_one_unit_of_the_division(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    src = tmp_path / "inv.cu"
    src.write_text(SOURCE)
    exe = str(tmp_path / "inv")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-I",
                    os.path.join(ROOT, "paper_1802_07871_gb300", "csrc"), "-I", os.path.join(ROOT, "include"), str(src),
                    "-o", exe], check=True)
    worst, kind, off, n = map(int, subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split())
    # y (1 + e) in one rounding, e = 1 - x y exact to 2^-106: half a unit and a
    # little, so at most the neighbour of the correctly rounded quotient
    assert worst <= 1 and kind == 0, (worst, kind, off, n)
