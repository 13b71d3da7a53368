"""silu in the general expert launch is the correctly rounded quotient z / (1 + exp(-z)) for every fp32
z, also where its divisor is near the end of fp32's range (a fast division gives 0 once the divisor is
above 2^126, and is up to 2 ulp off elsewhere)."""
import ctypes
import math
import os
import subprocess

import pytest
import torch

from dmoe_synth import ROUTE_TOKEN, TINY
from tests import parity as P
from tests.conftest import ROOT

pytestmark = pytest.mark.gpu

KERNEL = r"""
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include "silu.cuh"
using namespace dmoe;
// out[0]: values of the range whose corrected quotient is not the operator's; out[1]: values of z,
// one of two in a slice with 1, that silu_all gives another result for
__global__ void count(unsigned long long* out) {
  unsigned long long a = 0, b = 0;
  const uint64_t step = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (1ull << 32); i += step) {
    const float z = __uint_as_float((uint32_t)i), w = silu_divide(z);
    if (fabsf(z) <= kSiluMax)
      a += __float_as_uint(silu_corrected(z)) != __float_as_uint(w);
    float s[2] = {1.f, z};
    silu_all(s);
    b += isnan(w) ? !isnan(s[1]) : __float_as_uint(s[1]) != __float_as_uint(w);
    b += __float_as_uint(s[0]) != __float_as_uint(silu_divide(1.f));
  }
  atomicAdd(out, a);
  atomicAdd(out + 1, b);
}
extern "C" int run(unsigned long long* out) {
  count<<<1520, 256>>>(out);
  return (int)cudaDeviceSynchronize();
}
"""


def test_silu_of_every_number(tmp_path):
    from paper_2605_30876_gb300 import _build
    src, lib = tmp_path / "silu.cu", tmp_path / "silu.so"
    src.write_text(KERNEL)
    subprocess.run([_build._nvcc(), *_build.ARCH, *_build.FLAGS, "-I",
                    os.path.join(ROOT, "paper_2605_30876_gb300", "csrc"), "-shared", "-o", str(lib),
                    str(src)], check=True)
    out = torch.zeros(2, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    run = ctypes.CDLL(str(lib)).run
    run.argtypes = [ctypes.c_void_p]
    assert run(out.data_ptr()) == 0
    assert out.tolist() == [0, 0]


GATES = [-1.0, -60.0, -87.0, -87.5, -88.0, -88.5]   # exact in bf16; exp(87.5) is above 2^126


@pytest.mark.parametrize("Is", [0, 128])
def test_layer_with_large_negative_gates(Is):
    # token t is (1, 1, 0, ..): row i of W_gate gives the gate GATES[i % 6], row i of W_up 2^122,
    # and column i of the identity W_down hands H's element i to y
    T, I, d, E = 128, 128, 256, 8
    shape = TINY.with_(block_size=T, n_blocks=1, mode=ROUTE_TOKEN, n_experts=E, top_k=1, d_model=d,
                       d_ff=I, d_ff_shared=Is)
    dev, _ = P.make(shape, seed=1)
    z = torch.tensor([GATES[i % len(GATES)] for i in range(I)])
    up = 2.0 ** 122
    dev["x"].zero_()
    dev["x"][:, :2] = 1.0
    dev["w_r"].zero_()
    for p in ("w", "ws")[: 2 if Is else 1]:
        for key in ("gate", "up", "down"):
            dev[f"{p}_{key}"].zero_()
        dev[f"{p}_gate"][..., :, 0] = z.bfloat16().cuda()
        dev[f"{p}_up"][..., :, 1] = up
        dev[f"{p}_down"][..., :I, :] = torch.eye(I).bfloat16().cuda()
    from paper_2605_30876_gb300.layer import MoELayer
    layer = MoELayer.from_shape(shape, dev)
    y = layer.forward(dev["x"]).float().cpu()
    assert P.dm().dmoe_get_device_error(layer.ws)[0] == 0
    want = torch.tensor([v / (1 + math.exp(-v)) * up for v in z.tolist()]) * (2 if Is else 1)
    # H, the slot row and y are rounded to bf16 (2^-9 each); the exponential of 88 is 1.3e-5 off
    torch.testing.assert_close(y[:, :I], want.expand(T, I), rtol=3 * 2.0 ** -9 + 1e-4, atol=0.0)
    assert torch.all(y[:, I:] == 0)
