"""The GELU of the bf16 epilogues against 64 bits, compiled from the kernels' own header."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = """
#include "common.cuh"
__global__ void gelu_kernel(const float *v, unsigned short *one, unsigned short *two, int pairs) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= pairs) return;
  for (int k = 0; k < 2; ++k)
    one[2 * i + k] = __bfloat16_as_ushort(__float2bfloat16_rn(tsfm::gelu_erf_fast(v[2 * i + k])));
  const uint32_t p = tsfm::gelu_erf_fast2(v[2 * i], v[2 * i + 1]);
  two[2 * i] = (unsigned short)p;
  two[2 * i + 1] = (unsigned short)(p >> 16);
}
extern "C" int gelu(const float *v, unsigned short *one, unsigned short *two, int pairs) {
  gelu_kernel<<<(pairs + 127) / 128, 128>>>(v, one, two, pairs);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def gelu(tmp_path_factory):
    d = tmp_path_factory.mktemp("gelu")
    src, lib = d / "gelu.cu", d / "gelu.so"
    src.write_text(SOURCE)
    subprocess.run([os.environ.get("NVCC", "nvcc"), "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-shared",
                    "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "paper_2511_18191_b200", "csrc"), "-o", str(lib), str(src)],
                   check=True)
    f = ctypes.CDLL(str(lib)).gelu

    def run(v):
        n = len(v)
        v = torch.tensor(v, dtype=torch.float32, device="cuda")
        out = [torch.empty(n, dtype=torch.int16, device="cuda") for _ in range(2)]
        assert f(ctypes.c_void_p(v.data_ptr()), ctypes.c_void_p(out[0].data_ptr()), ctypes.c_void_p(out[1].data_ptr()),
                 ctypes.c_int(n // 2)) == 0
        return [o.view(torch.bfloat16).double().cpu().numpy() for o in out]

    return run


def test_gelu_of_finite_values(gelu):
    v = np.concatenate([np.linspace(-14.0, 14.0, 20001), np.logspace(-30, 37, 999), -np.logspace(-30, 37, 1000)]).astype(np.float32)
    want = np.array([x * 0.5 * math.erfc(-x / math.sqrt(2.0)) for x in v.astype(np.float64)])
    # rounding to bf16 (8 significant bits: half an ulp is at most 2^-8 of the value); the polynomial's 0.75e-7 |v| and
    # four roundings of an erfc of at most 1, 2.4e-7 |v| (beyond 14 the exact value on the negative side is below any of
    # this, on the positive side the result is v)
    tol = np.abs(want) * 2.0 ** -8 + np.minimum(np.abs(v), 14.0) * 3.2e-7 + 1e-38
    for got in gelu(v):
        assert (np.abs(got - want) <= tol).all()


def test_gelu_of_infinities_and_nan(gelu):
    for got in gelu([math.inf, 1.0, 2.0, math.inf, math.nan, 1.0, 3e38, math.inf, -3e38, math.nan]):
        assert got[0] == got[3] == got[7] == math.inf
        assert math.isnan(got[4]) and math.isnan(got[9])
        assert got[8] == 0.0 and np.isfinite(got[[1, 2, 5]]).all()
