"""The double-word square root and reciprocal of the double-float panel
(panel.cuh: dw_sqrt_fast, dw_rcp_fast), compiled from the header and run on the
GPU.  Criterion: over the same arguments neither the largest nor the root mean
square relative error exceeds that of one correction step on IEEE quotient and
root (Dekker; float32 on the host), the form whose place they take, and the
result is a normalised pair.  References in numpy's long double (at least 64
significant bits).  Arguments: two binades (both parities of the exponent), and
1e-30 .. 1e30, where the low words are normal FP32 numbers.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_1708_06290_gb300 import build

pytestmark = pytest.mark.gpu

SRC = r'''
#include "panel.cuh"
__global__ void k(int n, const float2* x, float2* root, float2* rcp) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const ssv::dw v{x[i].x, x[i].y};
  const ssv::dw r = ssv::pan::dw_sqrt_fast(v), q = ssv::pan::dw_rcp_fast(v);
  root[i] = make_float2(r.hi, r.lo);
  rcp[i] = make_float2(q.hi, q.lo);
}
extern "C" int run(int n, const void* x, void* root, void* rcp) {
  k<<<(n + 255) / 256, 256>>>(n, (const float2*)x, (float2*)root, (float2*)rcp);
  return (int)cudaDeviceSynchronize();
}
'''
f32, LD = np.float32, np.longdouble


def fma(a, b, c):
    return f32(LD(a) * LD(b) + LD(c))


def fast(a, b):
    s = f32(a + b)
    return s, f32(b - f32(s - a))


def ieee_root(hi, lo):
    s = np.sqrt(hi)
    return fast(s, f32(f32(fma(-s, s, hi) + lo) / f32(f32(2) * s)))


def ieee_rcp(hi, lo):
    q = f32(f32(1) / hi)
    return fast(q, f32(f32(fma(-q, hi, f32(1)) + fma(-q, lo, f32(0))) / hi))


@pytest.fixture(scope="module")
def scalars(tmp_path_factory):
    d = tmp_path_factory.mktemp("dw")
    src, lib = d / "dw.cu", str(d / "dw.so")
    src.write_text(SRC)
    subprocess.run([build._nvcc()] + build.ARCH + build.NVCC_FLAGS + ["-shared", "-o", lib, str(src)], check=True)
    assert os.path.exists(lib)
    return ctypes.CDLL(lib)


@pytest.mark.parametrize("span", ["binades", "range"])
def test_root_and_reciprocal(scalars, span):
    rng = np.random.default_rng(41)
    n = 1 << 20
    hi = f32(rng.uniform(1.0, 4.0, n) if span == "binades" else 10.0 ** rng.uniform(-30, 30, n))
    hi, lo = fast(hi, f32(hi.astype(np.float64) * rng.uniform(-2.0 ** -25, 2.0 ** -25, n)))
    x = torch.from_numpy(np.stack([hi, lo], axis=1)).cuda()
    root, rcp = torch.empty_like(x), torch.empty_like(x)
    rc = scalars.run(n, *(ctypes.c_void_p(t.data_ptr()) for t in (x, root, rcp)))
    assert rc == 0
    X = LD(hi) + LD(lo)
    for got, old, exact in ((root, ieee_root, np.sqrt(X)), (rcp, ieee_rcp, 1 / X)):
        g = got.cpu().numpy()
        err = lambda a, b: np.abs((LD(a) + LD(b) - exact) / exact).astype(np.float64)  # noqa: E731
        e, o = err(g[:, 0], g[:, 1]), err(*old(hi, lo))
        assert e.max() <= o.max(), (np.log2(e.max()), np.log2(o.max()))
        assert np.sqrt((e ** 2).mean()) <= np.sqrt((o ** 2).mean())
        assert (np.abs(g[:, 1]) <= np.abs(g[:, 0]) * f32(2.0 ** -23)).all()
