"""The hidden layers' bf16 tanh (csrc/tc.cuh, tanh_bf16) against CUDA's tanhf
rounded to bf16: the same bits for every one of the 2^32 fp32 arguments, with
and without a bias.  The kernel is compiled here with nvcc from the library's
own header."""
import ctypes as C
import os
import subprocess

import pytest
import torch

from paper_2608_11226_gb300 import build as libbuild

pytestmark = pytest.mark.gpu

SRC = r"""
#include "common.cuh"
#include "tc.cuh"

// thread i: arguments with the bit patterns 16 i .. 16 i + 15; counts the
// results that differ from tanhf's (two NaNs are alike) without having been
// reported, and all that differ
__global__ void sweep_kernel(float bias_step, unsigned long long* differ) {
  __shared__ __align__(16) float bias[16];
  if (threadIdx.x < 16) bias[threadIdx.x] = bias_step * (float)threadIdx.x;
  __syncthreads();
  const uint32_t u = (blockIdx.x * blockDim.x + threadIdx.x) * 16u;
  float v[16];
  uint32_t pk[8];
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(u + (uint32_t)i);
  uint32_t least;
  pe::tc::tanh_bf16(v, bias, pk, least);
  int n = 0;
  for (int i = 0; i < 16; ++i) {
    const uint32_t got = (pk[i / 2] >> (16 * (i & 1))) & 0xFFFFu;
    const uint32_t want = __bfloat16_as_ushort(__float2bfloat16_rn(tanhf(v[i] + bias[i])));
    n += got != want && !((got & 0x7FFFu) > 0x7F80u && (want & 0x7FFFu) > 0x7F80u);
  }
  if (n && !pe::tc::near_midpoint(least)) atomicAdd(differ, (unsigned long long)n);
  if (n) atomicAdd(differ + 1, (unsigned long long)n);
}

extern "C" int sweep(float bias_step, unsigned long long* differ) {
  sweep_kernel<<<1 << 20, 256>>>(bias_step, differ);
  return (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def so(tmp_path_factory):
    d = tmp_path_factory.mktemp("tanh")
    src, lib = os.path.join(d, "tanh_sweep.cu"), os.path.join(d, "libtanh_sweep.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.check_call([libbuild.nvcc(), *libbuild.ARCH, *libbuild.FLAGS, "-shared", "-o", lib, src])
    s = C.CDLL(lib)
    s.sweep.argtypes = [C.c_float, C.c_void_p]
    return s


@pytest.mark.parametrize("bias_step", [0.0, 0.0371])
def test_bf16_tanh_is_tanhf_for_every_argument(so, bias_step):
    differ = torch.zeros(2, dtype=torch.int64, device="cuda")
    assert so.sweep(bias_step, differ.data_ptr()) == 0
    torch.cuda.synchronize()
    assert int(differ[0]) == 0 and int(differ[1]) < 1 << 12, differ
