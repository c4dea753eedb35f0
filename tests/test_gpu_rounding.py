"""The push's reciprocal roots against the functions whose results they have to
give, for every float from 1 to infinity and for NaN."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "pic_dev.cuh"

using namespace pic;

__device__ bool same(float a, float b) {
  return __float_as_uint(a) == __float_as_uint(b) || (isnan(a) && isnan(b));
}

// bits lo .. hi inclusive; differences of the four, each from the function's result
__global__ void k_compare(unsigned lo, unsigned hi, unsigned long long* differ) {
  unsigned long long d[4] = {0, 0, 0, 0};
  for (unsigned long long b = lo + blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; b <= hi;
       b += gridDim.x * (unsigned long long)blockDim.x) {
    const float x = __uint_as_float((unsigned)b);
    d[0] += !same(inverse_sqrt_rn(x), __frcp_rn(__fsqrt_rn(x)));
    d[1] += !same(rsqrt_from_1(x), rsqrtf(x));
    d[2] += !same(2.0f * rcp_from_1(x), __fdividef(2.0f, x));
    d[3] += !same(rcp_from_1(x), __fdividef(1.0f, x));
  }
  for (int i = 0; i < 4; ++i)
    if (d[i]) atomicAdd(&differ[i], d[i]);
}

extern "C" int compare(unsigned lo, unsigned hi, unsigned long long* out) {
  unsigned long long* d;
  if (cudaMalloc(&d, 32) != cudaSuccess) return 1;
  cudaMemset(d, 0, 32);
  k_compare<<<1216, 256>>>(lo, hi, d);
  const cudaError_t e = cudaMemcpy(out, d, 32, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return e == cudaSuccess ? 0 : 2;
}
"""


@pytest.fixture(scope="module")
def compare(tmp_path_factory):
    from paper_1906_06306_gb300 import build as b

    d = tmp_path_factory.mktemp("rounding")
    src, lib = d / "rounding.cu", d / "librounding.so"
    src.write_text(SOURCE)
    flags = [f for f in b.NVCC_FLAGS if f != "-lineinfo"]
    subprocess.run([b._nvcc(), *b.ARCH, *flags, "-shared", "-cudart", "shared", "-Xlinker", "-rpath",
                    "-Xlinker", "/usr/local/cuda/lib64", "-o", str(lib), str(src)], check=True)
    fn = ctypes.CDLL(str(lib)).compare
    fn.argtypes = [ctypes.c_uint, ctypes.c_uint, ctypes.c_void_p]

    def run(lo, hi):
        out = np.zeros(4, dtype=np.uint64)
        assert fn(lo, hi, out.ctypes.data) == 0
        return out.tolist()

    return run


@pytest.mark.parametrize("lo,hi", [(0x3F800000, 0x7F800000),   # 1 .. infinity
                                   (0x7F800001, 0x7FFFFFFF)])  # NaN
def test_reciprocal_roots_give_the_functions_results(compare, lo, hi):
    assert compare(lo, hi) == [0, 0, 0, 0]
