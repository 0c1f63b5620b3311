"""The two forms of SiLU in csrc/cc_common.cuh, silu and silu_div, give the
same bits for every float: which of them finishes a scored row depends on the
tiles beside it, and a row's score must not."""
import ctypes
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "cc_common.cuh"
// out[0]: floats whose results differ; out[1], out[2]: the least and largest of
// their bit patterns.  Two NaNs are the same result.
__global__ void compare(unsigned long long *out) {
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
       i < (1ull << 32); i += (unsigned long long)gridDim.x * blockDim.x) {
    const float x = __uint_as_float((unsigned)i), a = cc::silu(x), b = cc::silu_div(x);
    if (__float_as_uint(a) == __float_as_uint(b) || (a != a && b != b)) continue;
    atomicAdd(&out[0], 1ull);
    atomicMin(&out[1], i);
    atomicMax(&out[2], i);
  }
}
extern "C" int run(unsigned long long *out) {
  compare<<<1024, 256>>>(out);
  return (int)cudaDeviceSynchronize();
}
"""


def test_both_forms_agree_on_every_float(tmp_path):
    from paper_2607_27600_gb300 import build
    src, lib = tmp_path / "silu.cu", tmp_path / "libsilu.so"
    src.write_text(SOURCE)
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-shared", str(src),
                    "-o", str(lib)], check=True, timeout=120)
    out = torch.tensor([0, 1 << 33, 0], dtype=torch.int64, device="cuda")
    assert ctypes.CDLL(str(lib)).run(ctypes.c_void_p(out.data_ptr())) == 0
    n, lo, hi = out.tolist()
    bounds = np.array([lo & 0xFFFFFFFF, hi], np.uint32).view(np.float32)
    assert n == 0, f"{n} floats differ, bit patterns {lo:#x} ({bounds[0]}) to {hi:#x} ({bounds[1]})"
