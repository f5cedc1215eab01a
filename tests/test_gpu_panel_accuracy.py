"""Rounding errors of a double-float window panel of 128 rows (panel.cuh),
compiled from the header and run on the GPU: the panel goes through sub-blocks of
rows whose transforms are applied to all other rows at once.  Criterion: the error
of its coefficients (root mean square over a window, geometric mean over the
windows) is no larger than that of the plain form, one reflector at a time on all
rows in the same double-float arithmetic, its scalars by one correction step on
IEEE quotient and root.  1.1: two roundings of the same window differ by some 40 %
in that figure, the means over 64 windows by 5 %.  Reference: the plain form in
numpy's long double.
"""
import ctypes
import subprocess

import numpy as np
import pytest
import torch

from paper_1708_06290_gb300 import build

pytestmark = pytest.mark.gpu

NB, WINDOWS = 128, 64
SRC = r'''
#include "panel.cuh"
using namespace ssv;
constexpr int NB = 128, NT = 256;
// window rows Z (NB x m), H (n x n, n = NB + m) as pairs, coefficients ((NB + m) x m)
template <int M>
__global__ void __launch_bounds__(NT) panel(int m, const float* hi, const float* lo, const cd* sigma, const float4* Z,
                                            float4* out) {
  extern __shared__ __align__(16) unsigned char raw[];
  auto& sm = *reinterpret_cast<pan::Smem<pan::DF32, M, NB>*>(raw);
  constexpr int S = pan::Smem<pan::DF32, M, NB>::S;
  __shared__ int sing;
  const int w = blockIdx.x, n = NB + m;
  for (int e = threadIdx.x; e < NB * m; e += NT) sm.W[(e / m) * S + e % m] = Z[(size_t)w * NB * m + e];
  pan::run<pan::DF32, M, NB, NT, false>(pan::DF32::H{hi + (size_t)w * n * n, lo + (size_t)w * n * n, n}, m, 0, sigma[w],
                                        NB, m, sm, (pan::SmemR<pan::DF32, M, NB>*)nullptr, 0.0, &sing);
  for (int e = threadIdx.x; e < n * m; e += NT) out[(size_t)w * n * m + e] = sm.W[(e / m) * S + e % m];
}
// one correction step on IEEE quotient and root
__device__ dw quotient(dw x, dw y) {
  const float q = x.hi / y.hi;
  return dw_fast(q, (fmaf(-q, y.hi, x.hi) + fmaf(-q, y.lo, x.lo)) / y.hi);
}
__device__ dw root(dw x) {
  const float s = sqrtf(x.hi);
  return dw_fast(s, (fmaf(-s, s, x.hi) + x.lo) / (2.f * s));
}
// one reflector at a time; rows 0 .. NB - 1 of Y: window row, then coefficient row; NB ..: unit rows
__global__ void __launch_bounds__(NT) plain(int m, const float* hi, const float* lo, const cd* sigma, const float4* Z,
                                            float4* out) {
  using A = pan::DF32;
  const int w = blockIdx.x, n = NB + m, row = threadIdx.x;
  hi += (size_t)w * n * n;
  lo += (size_t)w * n * n;
  float4* Y = out + (size_t)w * n * m;
  for (int e = threadIdx.x; e < n * m; e += NT) {
    const int r = e / m, q = e % m;
    Y[e] = r < NB ? Z[(size_t)w * NB * m + e] : r - NB == q ? A::one() : A::zero();
  }
  __shared__ float4 v[17];
  __shared__ dw tau;
  for (int c = NB - 1; c >= 0; --c) {
    __syncthreads();
    if (row == 0) {
      dw rest2{0.f, 0.f};
      for (int q = 0; q < m; ++q) {
        const float4 x = Y[c * m + q];
        rest2 = dw_add(rest2, dw_add(dw_mul(dw{x.x, x.y}, dw{x.x, x.y}), dw_mul(dw{x.z, x.w}, dw{x.z, x.w})));
        v[q] = A::conj(x);
      }
      const dw xf{hi[(m + c) + (size_t)c * n], lo[(m + c) + (size_t)c * n]};
      const dw af{fabsf(xf.hi), xf.hi < 0.f ? -xf.lo : xf.lo}, nrm2 = dw_add(rest2, dw_mul(xf, xf));
      const dw nrm = root(nrm2), vf = dw_mul(xf, dw_add(dw{1.f, 0.f}, quotient(nrm, af)));
      tau = quotient(dw{1.f, 0.f}, dw_add(nrm2, dw_mul(af, nrm)));
      v[m] = make_float4(vf.hi, vf.lo, 0.f, 0.f);
    }
    __syncthreads();
    if (row < n) {
      float4* y = Y + row * m;
      if (row == c) for (int q = 0; q < m; ++q) y[q] = A::zero();
      float4 f = A::zero();
      if (row < c) f = row == c - m ? A::shifted(make_float2(hi[c + (size_t)c * n], lo[c + (size_t)c * n]), sigma[w])
                                    : make_float4(hi[(m + row) + (size_t)c * n], lo[(m + row) + (size_t)c * n], 0.f, 0.f);
      else if (row == c) f = A::one();
      A::Acc a{0.f, 0.f, 0.f, 0.f};
      for (int q = 0; q < m; ++q) A::mac(a, y[q], v[q]);
      A::mac(a, f, v[m]);
      const float4 t = A::scale(tau, a);
      for (int q = 0; q < m; ++q) y[q] = A::sub(y[q], t, v[q]);
    }
  }
}
template <int M>
int go(int nw, int m, const void* hi, const void* lo, const void* sg, const void* Z, void* o1, void* o2) {
  const int bytes = (int)sizeof(pan::Smem<pan::DF32, M, NB>);
  cudaError_t e = cudaFuncSetAttribute(panel<M>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess) return (int)e;
  panel<M><<<nw, NT, bytes>>>(m, (const float*)hi, (const float*)lo, (const cd*)sg, (const float4*)Z, (float4*)o1);
  plain<<<nw, NT>>>(m, (const float*)hi, (const float*)lo, (const cd*)sg, (const float4*)Z, (float4*)o2);
  return (int)cudaDeviceSynchronize();
}
extern "C" int run(int nw, int m, const void* hi, const void* lo, const void* sg, const void* Z, void* o1, void* o2) {
  return m <= 2 ? go<2>(nw, m, hi, lo, sg, Z, o1, o2) : m <= 4 ? go<4>(nw, m, hi, lo, sg, Z, o1, o2)
       : m <= 8 ? go<8>(nw, m, hi, lo, sg, Z, o1, o2) : go<16>(nw, m, hi, lo, sg, Z, o1, o2);
}
'''
LD, LC = np.longdouble, np.clongdouble


def exact(H, sigma, Z):
    """Coefficients of all windows: H (w, n, n), Z (w, NB, m)."""
    nw, n = H.shape[:2]
    m = n - NB
    Y = np.zeros((nw, n, m), LC)
    Y[:, :NB] = Z
    Y[:, NB:] = np.eye(m)
    for c in range(NB - 1, -1, -1):
        x, xf = Y[:, c].copy(), H[:, m + c, c]
        nrm2 = (x.real ** 2 + x.imag ** 2).sum(1) + xf ** 2
        nrm = np.sqrt(nrm2)
        vf = xf + np.where(xf < 0, -nrm, nrm)
        tau = 1 / (nrm2 + np.abs(xf) * nrm)
        v = x.conj()
        Y[:, c] = 0
        f = np.zeros((nw, n), LC)
        f[:, :c] = H[:, m:m + c, c]
        f[:, c] = 1
        if c >= m:
            f[:, c - m] -= sigma
        t = tau[:, None] * (np.einsum("wrq,wq->wr", Y, v) + f * vf[:, None])
        Y -= t[:, :, None] * v.conj()[:, None, :]
    return Y


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("panel")
    src, so = d / "panel.cu", str(d / "panel.so")
    src.write_text(SRC)
    subprocess.run([build._nvcc()] + build.ARCH + build.NVCC_FLAGS + ["-shared", "-o", so, str(src)], check=True)
    return ctypes.CDLL(so)


@pytest.mark.parametrize("m", [2, 3, 4, 8, 16])
def test_panel_errors(lib, m):
    rng = np.random.default_rng(900 + m)
    n = NB + m
    H = rng.standard_normal((WINDOWS, n, n)) / np.sqrt(n)
    H[:, np.arange(n), np.arange(n)] -= 2.0
    H[:, np.arange(m, n), np.arange(NB)] = 1.0 + 0.2 * rng.standard_normal((WINDOWS, NB))
    sigma = 1j * 10.0 ** rng.uniform(-2, 1, WINDOWS)
    Z = (rng.standard_normal((WINDOWS, NB, m)) + 1j * rng.standard_normal((WINDOWS, NB, m))) / np.sqrt(2)
    hi = H.astype(np.float32)
    lo = (H - hi).astype(np.float32)
    pair = lambda a: (a.astype(np.float32), (a - a.astype(np.float32)).astype(np.float32))  # noqa: E731
    zr, zi = pair(Z.real), pair(Z.imag)
    z4 = np.stack([zr[0], zr[1], zi[0], zi[1]], axis=-1)
    col = lambda a: torch.from_numpy(np.ascontiguousarray(a.transpose(0, 2, 1))).cuda()  # noqa: E731
    d = [col(hi), col(lo), torch.from_numpy(sigma).cuda(), torch.from_numpy(np.ascontiguousarray(z4)).cuda()]
    o = [torch.empty((WINDOWS, n, m, 4), dtype=torch.float32, device="cuda") for _ in range(2)]
    assert lib.run(WINDOWS, m, *(ctypes.c_void_p(t.data_ptr()) for t in d + o)) == 0
    ref = exact(hi.astype(LD) + lo, sigma.astype(LC),
                (z4[..., 0].astype(LD) + z4[..., 1]) + 1j * (z4[..., 2].astype(LD) + z4[..., 3]))
    err = []
    for t in o:
        a = t.cpu().numpy().astype(LD)
        e = np.abs((a[..., 0] + a[..., 1]) + 1j * (a[..., 2] + a[..., 3]) - ref).astype(float)
        err.append(np.exp(0.5 * np.log((e ** 2).mean((1, 2))).mean()))
    assert err[0] <= 1.1 * err[1], "sub-blocks %.2e, reflector by reflector %.2e" % tuple(err)
