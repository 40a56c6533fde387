"""The hidden layers' bf16 tanh (csrc/tc.cuh) against CUDA's tanhf rounded to
bf16.  tanh_bf16, compiled here with nvcc from the library's own header: for
every one of the 2^32 fp32 arguments the same bits, or reported.  The networks,
through pe_value: arguments around the rounding midpoints, in every row and
column of both layers."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2608_11226_gb300 import build as libbuild
from paper_2608_11226_gb300 import pe
from paper_2608_11226_gb300 import workloads as W

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


@pytest.mark.parametrize("D,H", [(32, 256), (64, 512)])
@pytest.mark.parametrize("layer", [1, 2])
def test_bf16_network_tanh_near_midpoints(D, H, layer):
    """Zero observations, so that a layer's pre-activations are its biases: the
    floats within four steps of where tanh crosses a midpoint between two bf16
    values, both signs.  Every row of a tile then has values for tanhf in every
    chunk.  The head picks one unit per call; behind layer 1 the second layer is
    the identity."""
    rng = np.random.default_rng(layer)
    t = rng.uniform(0.02, 0.995, H).astype(np.float32)
    mid = ((t.view(np.uint32) & 0xFFFF0000) | 0x8000).view(np.float32)
    z = np.arctanh(mid.astype(np.float64)).astype(np.float32)
    z = (z.view(np.int32) + rng.integers(-4, 5, H)).astype(np.int32).view(np.float32) * rng.choice([-1, 1], H)
    z = torch.from_numpy(z.astype(np.float32)).cuda()
    want = torch.tanh(z).bfloat16().float()
    p = torch.zeros(W.param_count(D, H, 16), device="cuda")
    v1 = H * D + H + H * H + H + 16 * H + 16  # the value network follows the policy
    c1, v2 = v1 + H * D, v1 + H * D + H
    c2, v3 = v2 + H * H, v2 + H * H + H
    if layer == 1:
        p[c1:c1 + H] = z
        p[v2:v2 + H * H] = torch.eye(H, device="cuda").flatten()
        want = torch.tanh(want).bfloat16().float()
    else:
        p[c2:c2 + H] = z
    obs = torch.zeros(300, D, dtype=torch.bfloat16, device="cuda")
    out = torch.empty(300, device="cuda")
    for i in range(0, H, 5):
        p[v3:v3 + H] = 0
        p[v3 + i] = 1
        pe.value(W.NetSpec(D, H, 16, pe.PE_BF16), p, obs, out)
        assert torch.equal(out, want[i].expand(300)), (i, float(z[i]), float(want[i]), out)
    pe.device_check()
