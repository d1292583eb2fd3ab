"""The FP32 reciprocal of the step's kernels (recip in lb_split.cuh) over every bit pattern, against the
division in double precision. One Newton step from an approximation of relative error 2^-23 leaves
2^-46, the rounding of its residual 2^-47 and of the result 2^-24: 2^-24 (1 + 2^-20) for a normal result;
for a subnormal one (|x| > 2^126) another rounding, to the subnormal spacing. Results beyond the largest
float, the zeros, infinities and NaN as IEEE has them."""
import subprocess
from pathlib import Path

import pytest

from paper_1111_0905_gb300 import build

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include <cstdio>
#include "lb_split.cuh"
// counts[0]: out of bounds; counts[1]: a pattern out of bounds; counts[2]: patterns checked
__global__ void check(unsigned long long* counts) {
  const unsigned long long total = 1ull << 32, step = (unsigned long long)gridDim.x * blockDim.x;
  unsigned long long seen = 0;
  for (unsigned long long k = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; k < total; k += step) {
    const float x = __uint_as_float((unsigned)k);
    const float r = tlbm::recip(x);
    ++seen;
    bool ok;
    if (isnan(x)) ok = isnan(r);
    else if (isinf(x) || x == 0.0f) ok = r == 1.0f / x && signbit(r) == signbit(x);
    else {
      const double q = 1.0 / (double)x, err = fabs((double)r - q);
      if (fabs(q) >= 0x1.ffffffp127) ok = isinf(r) && signbit(r) == signbit(x);
      else if (fabs(q) >= 0x1p-126) ok = err <= fabs(q) * 0x1p-24 * (1.0 + 0x1p-20);
      else ok = err <= fabs(q) * 0x1p-24 * (1.0 + 0x1p-20) + 0x1p-150;
    }
    if (!ok) { atomicAdd(&counts[0], 1ull); counts[1] = k; }
  }
  atomicAdd(&counts[2], seen);
}
int main() {
  unsigned long long *d, h[3] = {1, 0, 0};
  if (cudaMalloc(&d, sizeof(h)) != cudaSuccess || cudaMemset(d, 0, sizeof(h)) != cudaSuccess) return 2;
  check<<<1216, 256>>>(d);
  if (cudaGetLastError() != cudaSuccess || cudaMemcpy(h, d, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
  std::printf("%llu %llu %llu\n", h[0], h[1], h[2]);
  return 0;
}
"""


def test_fp32_reciprocal_over_every_bit_pattern(cuda, tmp_path):
    src, exe = tmp_path / "recip.cu", tmp_path / "recip"
    src.write_text(PROGRAM)
    flags = [f for f in build.FLAGS if f not in ("-Xcompiler", "-fPIC")]
    subprocess.run([build.nvcc(), *build.ARCH, *flags, "-I", str(Path(build.CSRC)), str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()
    assert int(out[2]) == 1 << 32
    assert int(out[0]) == 0, f"{out[0]} patterns, one of them {int(out[1]):#010x}"
