"""GPU: the float-float sum of two path counts (sigma of a 2-degree vertex's run where both neighbours'
paths are equally long) is the exact sum cut once to 48 bits, also where the sum passes 2^64."""
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_1602_00963_gb300 import build

pytestmark = pytest.mark.gpu

MAIN = r"""
#include <cstdio>
#include <vector>
#include "bc_ff.cuh"
using u64 = unsigned long long;
__global__ void k(int n, const u64 *a, const u64 *b, float2 *out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = bcl::ff_sum_u64(a[i], b[i]);
}
int main(int argc, char **argv) {
  FILE *f = fopen(argv[1], "rb");
  int n = 0;
  if (!f || fread(&n, 4, 1, f) != 1 || n < 1 || n > 1 << 20) return 1;
  std::vector<u64> h(2 * (size_t)n);
  if (fread(h.data(), 8, h.size(), f) != h.size()) return 2;
  fclose(f);
  u64 *d;
  float2 *o;
  if (cudaMalloc(&d, h.size() * 8) != cudaSuccess || cudaMalloc(&o, (size_t)n * 8) != cudaSuccess) return 3;
  cudaMemcpy(d, h.data(), h.size() * 8, cudaMemcpyHostToDevice);
  k<<<(n + 255) / 256, 256>>>(n, d, d + n, o);
  std::vector<float2> r(n);
  if (cudaMemcpy(r.data(), o, (size_t)n * 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 4;
  f = fopen(argv[2], "wb");
  if (!f || fwrite(r.data(), 8, n, f) != (size_t)n) return 5;
  return fclose(f);
}
"""


def test_sum_is_cut_once(tmp_path):
    rng = np.random.Generator(np.random.PCG64(48))
    top = (1 << 64) - 1
    a = [1, 0, top, 1, top, 1 << 63, (1 << 60) + 4095, (1 << 48) + 1, (1 << 49) - 1]
    b = [0, 1, top, top, 1, 1 << 63, (1 << 60) - 4095, (1 << 48) - 1, (1 << 49) - 1]
    for bits in range(1, 65):
        a += [int(x) | 1 << bits - 1 for x in rng.integers(0, 1 << bits - 1, 50, dtype=np.uint64, endpoint=True)]
        b += [int(x) >> int(rng.integers(0, 64)) for x in rng.integers(0, top, 50, dtype=np.uint64, endpoint=True)]
    (tmp_path / "main.cu").write_text(MAIN)
    exe, inp, out = (str(tmp_path / x) for x in ("main", "in", "out"))
    subprocess.check_call([build.nvcc()] + build.ARCH + ["-O3", "-std=c++17", "-I", build.CSRC, "-o", exe,
                                                        os.path.join(str(tmp_path), "main.cu")])
    with open(inp, "wb") as f:
        f.write(np.int32(len(a)).tobytes() + np.array(a, np.uint64).tobytes() + np.array(b, np.uint64).tobytes())
    subprocess.check_call([exe, inp, out])
    r = np.fromfile(out, np.float32).reshape(-1, 2)
    for x, y, (hi, lo) in zip(a, b, r):
        cut = max((x + y).bit_length() - 48, 0)
        assert Fraction(float(hi)) + Fraction(float(lo)) == (x + y) >> cut << cut, (x, y, hi, lo)
