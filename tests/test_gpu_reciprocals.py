"""The kernels' FP32 reciprocal, all 2^32 arguments: correctly rounded wherever
the argument and the result are normal, exact for zeros and infinities, a signed
infinity for subnormal arguments, a signed zero where the result is subnormal."""
import subprocess

import pytest

torch = pytest.importorskip("torch")

from paper_2311_08927_gb300 import build as B  # noqa: E402

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include <cstdio>
#include "adm1_device.cuh"
using namespace chad;
__device__ unsigned long long wrong[5];
__global__ void check() {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < (1ull << 32); i += stride) {
    const float d = __uint_as_float((unsigned)i), ref = __frcp_rn(d), got = rcp<float>(d);
    const float tiny = 1.17549435e-38f;  // 2^-126
    int kind = 0;
    bool same;
    if (isnan(d)) {
      kind = 1;
      same = isnan(got);
    } else if (d == 0.0f || isinf(d)) {
      kind = 2;
      same = __float_as_uint(got) == __float_as_uint(ref);
    } else if (fabsf(d) < tiny) {
      kind = 3;
      same = __float_as_uint(got) == __float_as_uint(copysignf(INFINITY, d));
    } else if (fabsf(ref) < tiny) {
      kind = 4;
      same = __float_as_uint(got) == __float_as_uint(copysignf(0.0f, d));
    } else {
      same = __float_as_uint(got) == __float_as_uint(ref);
    }
    if (!same) atomicAdd(&wrong[kind], 1ull);
  }
}
int main() {
  check<<<1216, 256>>>();
  unsigned long long h[5];
  if (cudaMemcpyFromSymbol(h, wrong, sizeof(h)) != cudaSuccess) return 2;
  std::printf("normal %llu nan %llu zero or infinite %llu subnormal argument %llu result %llu\n", h[0],
              h[1], h[2], h[3], h[4]);
  return h[0] || h[1] || h[2] || h[3] || h[4];
}
"""


def test_fp32_reciprocal_is_correctly_rounded(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    src, exe = tmp_path / "rcp.cu", tmp_path / "rcp"
    src.write_text(PROGRAM)
    subprocess.run([B.nvcc(), *B.ARCH, *B.NVCC_FLAGS, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
