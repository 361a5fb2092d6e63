"""div_rn and sqrt_rn (csrc/rounded.cuh) return the bits of the IEEE division and square root:
on the host against the compiler's, on the GPU against CUDA's.  Significands cover few bits,
many bits, all ones and powers of two, where a candidate lies closest to a rounding boundary;
exponents cover the range where the functions hand over to the built-in ones."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "%s/paper_1703_10973_gb300/csrc/rounded.cuh"
#include <cstdio>
#include <cstdlib>
using namespace sdpgb;
__host__ __device__ uint64_t mix(uint64_t z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
__host__ __device__ double make(uint64_t i) {
  const uint64_t a = mix(i), b = mix(a);
  uint64_t m = a & 0xFFFFFFFFFFFFFull;
  const int mode = (int)(b %% 6);
  if (mode == 1) m >>= (b >> 8) %% 53;
  if (mode == 2) m = 0xFFFFFFFFFFFFFull - (b >> 8) %% 16;
  if (mode == 3) m = (b >> 8) %% 16;
  if (mode == 4) m &= ~((1ull << ((b >> 8) %% 52)) - 1);
  const uint64_t e = (mode == 5) ? (b >> 20) %% 2048 : 1023 - 60 + (b >> 20) %% 120;
  return rd_double(((b & 8) << 60) | (e << 52) | m);
}
__host__ __device__ bool same(double x, double y) { return rd_bits(x) == rd_bits(y) || (x != x && y != y); }
__host__ __device__ int wrong(uint64_t i) {
  const double a = make(2 * i), b = make(2 * i + 1), s = fabs(a), q = fabs(b) * fabs(b);
  return !same(div_rn(a, b), a / b) + !same(div_rn(1.0, a), 1.0 / a) + !same(sqrt_rn(s), sqrt(s)) +
         !same(sqrt_rn(q), sqrt(q)) + !same(sqrt_rn(a), sqrt(a));
}
__global__ void k(uint64_t n, unsigned long long* bad) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    const int w = wrong(i);
    if (w) atomicAdd(bad, (unsigned long long)w);
  }
}
int main(int argc, char** argv) {
  const uint64_t n = strtoull(argv[2], nullptr, 10);
  unsigned long long bad = 0;
  if (argv[1][0] == 'h') {
    for (uint64_t i = 0; i < n; ++i) bad += wrong(i);
  } else {
    unsigned long long* d;
    if (cudaMalloc(&d, 8) != cudaSuccess) return 2;
    cudaMemset(d, 0, 8);
    k<<<608, 256>>>(n, d);
    if (cudaMemcpy(&bad, d, 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
  }
  printf("%%llu\n", bad);
  return 0;
}
"""


def _run(tmp_path, where, count):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src, exe = str(tmp_path / "t.cu"), str(tmp_path / "t")
    with open(src, "w") as f:
        f.write(SRC % ROOT)
    subprocess.run([nvcc, "-O2", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", src, "-o", exe], check=True)
    r = subprocess.run([exe, where, str(count)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr
    assert int(r.stdout) == 0


def test_rounded_on_the_host(tmp_path):
    _run(tmp_path, "host", 2_000_000)


@pytest.mark.gpu
def test_rounded_on_the_gpu(tmp_path):
    _run(tmp_path, "device", 400_000_000)
