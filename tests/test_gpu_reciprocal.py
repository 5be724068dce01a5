"""The reciprocal of the J2 and finite-strain updates (element.cuh, rcp64) against the IEEE division, in units in the
last place.  After its Householder step the relative error is e^3, with |e| < 2^-19 that of the hardware's approximation
(PTX: 20 significant bits), so below 2^-57, beside the last rounding: at most one unit from the correctly rounded
quotient."""
import subprocess

import pytest

from tests.helpers import engine

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <cstdio>
#include "element.cuh"

// argument k: random fraction and sign, or (one in eight) a power of two or a neighbour of one; exponent in [-1000, 1000]
__device__ double argument(uint64_t k) {
  uint64_t z = (k + 1) * 0x9e3779b97f4a7c15ull;  // SplitMix64 (Steele, Lea, Flood 2014)
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  z ^= z >> 31;
  uint64_t fraction = z & 0xfffffffffffffull;
  if ((k & 7) == 0) fraction = (k & 24) == 0 ? 0 : (k & 24) == 8 ? 1 : (k & 24) == 16 ? 0xfffffffffffffull : fraction & 0xff;
  const uint64_t exponent = 23 + (z >> 52) % 2001;
  return __longlong_as_double((long long)(fraction | exponent << 52 | (z << 10 & 0x8000000000000000ull)));
}

__global__ void compare(uint64_t n, unsigned long long* worst) {
  unsigned long long w = 0;
  for (uint64_t k = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; k < n; k += (uint64_t)gridDim.x * blockDim.x) {
    const double d = argument(k);
    const long long a = __double_as_longlong(fea::rcp64(d)), b = __double_as_longlong(1.0 / d);
    const unsigned long long diff = a > b ? a - b : b - a;
    w = diff > w ? diff : w;
  }
  atomicMax(worst, w);
}

int main() {
  unsigned long long *worst, h = 0;
  if (cudaMalloc(&worst, 8) != cudaSuccess || cudaMemset(worst, 0, 8) != cudaSuccess) return 1;
  compare<<<608, 256>>>(1ull << 28, worst);
  if (cudaMemcpy(&h, worst, 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
  std::printf("%llu\n", h);
  return 0;
}
"""


def test_reciprocal_within_one_unit(tmp_path):
    engine()
    from paper_1805_03949_gb300 import build
    src = tmp_path / "reciprocal.cu"
    src.write_text(SOURCE)
    exe = str(tmp_path / "reciprocal")
    subprocess.check_call([build.nvcc()] + build.ARCH + build.NVCC_FLAGS +
                          ["-I", build.INCLUDE, "-I", build.CSRC, str(src), "-o", exe])
    assert int(subprocess.check_output([exe], timeout=120)) <= 1
