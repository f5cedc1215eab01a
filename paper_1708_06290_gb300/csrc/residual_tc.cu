// FP64-accurate residual E = R - (H - sigma I) Xhat on the tensor cores.
//
// The certification step of the mixed path (the refinement residual of
// iterative refinement; the residual of Sec. 3.3's unreduced right-hand-side
// technique) needs H Xhat to about 2^-50 of ||H|| ||Xhat||.  It is formed by
// error-free splitting (Ozaki, Ogita, Oishi, Rump 2012):
//
//   * each row i of H (its structural part, columns j >= i - m) is written as
//     H(i, j) = (-1)^s 2^{E_i} sum_{k=1..8} d_k 2^{-7k}, d_k in [0, 127],
//     with 2^{E_i} > max_j |H(i, j)|, and likewise each real column c of Xhat
//     (Re and Im of every column q) with its own exponent E_c;
//   * the digits are exact in BF16, so every slice product H_k X_l is exact in
//     FP32 as long as each partial sum stays below 2^24: with windows of 128
//     terms and the (t - 1) products of one level t = k + l summed together,
//     |sum| <= 8 * 128 * 127^2 < 2^24;
//   * H X = 2^{E_i + E_c} sum_{t=2..9} 2^{-7t} L_t, L_t = sum_{k+l=t} H_k X_l
//     (the 36 products with k + l <= 9; the dropped ones are below
//     2^{-56} relative to the row and column scales).
//
// Persistent CTAs (one per SM) take work items of 128 rows of H and one group
// of shifts (N = 32 real columns: 32 / cs shifts of cs columns, 2m rounded up
// to a power of two), in three roles that only meet at mbarriers:
//   * a producer thread copies the sixteen digit tiles of a 32-deep K stage
//     (no-swizzle K-major core-matrix layout, stored tile by tile in global
//     memory) into one of two stage buffers with 1-D TMA bulk copies;
//   * an issuing thread multiplies a stage into one of two TMEM windows: the
//     eight digit tiles of Xhat lie side by side, so one tcgen05.mma (kind::f16,
//     BF16 x BF16 -> FP32, M = 128, K = 16) of H digit a against Xhat digits
//     0 .. 7 - a (N = 32 (8 - a) columns) lands digit b in level a + b; every
//     fourth stage completes a window;
//   * eight warps read a finished window's levels back (tcgen05.ld) and add
//     them, scaled by 2^{-7t}, into double-float sums while the other window
//     multiplies; after an item's last window they form E in FP64.
// What bounds it: shared memory, which takes a stage's 80 KB and gives 138 KB to
// the products (1.7 k clocks of its bandwidth; the products themselves 1.2 k, 2.6 k
// measured); the readout of a window hides under the next one's products.
#include <algorithm>

#include "cluster.cuh"
#include "ssv_internal.cuh"
#include "tc_common.cuh"

namespace ssv {

namespace {

constexpr int kM = 128;       // rows of H per tile = TMEM lanes
constexpr int kN = 32;        // real columns per group of shifts
constexpr int kKS = 32;       // K per shared-memory stage
constexpr int kSl = 8;        // digit slices of H and of Xhat
constexpr int kLev = 8;       // levels t = 2 .. 9
constexpr int kWin = 128 / kKS;  // stages per exact accumulation window (K = 128)
constexpr int kKG = kKS / 8;     // core matrices along K in a tile
constexpr int kAT = kM * kKS;    // BF16 elements of one H slice tile
constexpr int kBT = kN * kKS;    // BF16 elements of one Xhat slice tile
constexpr uint32_t kStageBytes = (uint32_t)kSl * (kAT + kBT) * 2;
constexpr int kWinCols = kLev * kN;  // TMEM columns of a window; two windows
constexpr int kDrain = 256;          // readout threads (row x half of the columns), warps 0 .. 7
constexpr int kH = kN * kM / kDrain;  // columns of a readout thread
constexpr int kT = kDrain + 64;      // + the producer's and the issuer's warp
constexpr size_t kSmem = 2 * (size_t)kStageBytes + 128;
static_assert(kSmem <= 227 * 1024, "shared memory");
static_assert(2 * kWinCols == 512, "TMEM columns of the two windows");
using namespace tcg;
static_assert(kSl == kDigits, "eight digit slices");

// column stride of one shift in a group: 2m real columns rounded up to a power of two
__host__ __device__ inline int group_cols(int m) {
  int c = 2;
  while (c < 2 * m) c <<= 1;
  return c;
}

// element offset inside a K-major core-matrix tile with kKG core matrices
// along K: core (row group g, K group kk) at (g * kKG + kk) * 64 elements,
// 8 rows of 8 contiguous elements each (byte strides: 128 along K, kKG * 128
// along rows)
__host__ __device__ __forceinline__ int tile_off(int row, int k) {
  return (((row >> 3) * kKG + (k >> 3)) * 8 + (row & 7)) * 8 + (k & 7);
}

// Row exponents of H's structural part: blocks of 128 rows x kHChunk columns
// (hexp preset to INT_MIN-like bytes, combined by atomicMax).  One thread per
// row over all n columns took 0.87 ms at n = 4000, a chain of n loads on 32 SMs.
constexpr int kHChunk = 64;
__global__ void __launch_bounds__(256) tc_hrow_kernel(int n, int m, const double* __restrict__ H,
                                                      int* __restrict__ hexp) {
  __shared__ int part[128];
  const int row = threadIdx.x & 127, half = threadIdx.x >> 7;
  const int i = blockIdx.x * 128 + row;
  const int j0 = blockIdx.y * kHChunk, j1 = min(n, j0 + kHChunk);
  // the chunk lies left of the structural part of every row of the block
  if (j1 <= (int)blockIdx.x * 128 - m) return;
  int mx = 0;  // as integers: a maximum of doubles holds the FP64 pipe
  if (i < n) {
#pragma unroll 8
    for (int j = max(j0, i - m) + half; j < j1; j += 2) mx = max(mx, abs_hi(H[i + (size_t)j * n]));
  }
  int E = i < n ? scale_exp_hi(mx) : 0;  // padding rows: 0
  if (half == 1) part[row] = E;
  __syncthreads();
  if (half == 0) atomicMax(hexp + i, max(E, part[row]));
}

// items (i, j8): rows i fastest (coalesced reads of column-major H)
__global__ void tc_hsplit_kernel(int n, int m, int npad, const double* __restrict__ H,
                                 const int* __restrict__ hexp, uint4* __restrict__ Hs) {
  const int KT = npad / kKS, RB = npad / kM;
  const long long items = (long long)npad * (npad / 8);
  for (long long it = blockIdx.x * (long long)blockDim.x + threadIdx.x; it < items;
       it += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(it % npad), j8 = (int)(it / npad);
    const int E = hexp[i];
    unsigned short dg[8][kSl];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int j = j8 * 8 + e;
      const double v = (i < n && j < n && j >= i - m) ? H[i + (size_t)j * n] : 0.0;
      digits8(v, E, dg[e]);
    }
    const int I = i / kM, J = (j8 * 8) / kKS;
    const int off = tile_off(i % kM, (j8 * 8) % kKS);
#pragma unroll
    for (int l = 0; l < kSl; ++l) {
      uint4 w;
      w.x = dg[0][l] | ((unsigned)dg[1][l] << 16);
      w.y = dg[2][l] | ((unsigned)dg[3][l] << 16);
      w.z = dg[4][l] | ((unsigned)dg[5][l] << 16);
      w.w = dg[6][l] | ((unsigned)dg[7][l] << 16);
      const size_t base = ((size_t)(l * RB + I) * KT + J) * kAT + off;
      Hs[base / 8] = w;
    }
  }
}

// Digits of Xhat: a cluster of R CTAs per active shift finds the column
// exponents (each CTA over its share of the K tiles, combined through
// distributed shared memory), then writes its share of the digit tiles.
// Bound by memory: reads X twice (16 m bytes a row) and writes 16 digits of
// 2 m columns.  A warp takes 8 real columns x 32 rows of X, so that a digit
// plane's store is 512 contiguous bytes (one block per shift, 16-byte pieces
// 128 bytes apart: 6.4 ms for 2000 shifts at n = 5000, m = 16, and 0.33 ms for
// 40 at n = 4000).
// Entry w of the list takes columns (w mod S) cs .. of group w / S (S = 32 / cs).
__global__ void __launch_bounds__(256) tc_xsplit_kernel(int n, int m, int npad, int cs, int R,
                                                        const int* __restrict__ list,
                                                        const int* __restrict__ count,
                                                        const cd* __restrict__ X, long long ldx,
                                                        uint4* __restrict__ Xs,
                                                        int* __restrict__ xexp) {
  const int w = blockIdx.x / R;
  if (w >= *count) return;  // the whole cluster
  const int sh = list[w];
  const int rank = cluster_rank();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int KT = npad / kKS;
  const cd* Xh = X + (size_t)sh * m * ldx;
  const int S = kN / cs, grp = w / S, r0 = (w % S) * cs;  // this shift's rows of the group's tiles
  __shared__ int sE[kN], tE[kN];
  if (tid < kN) sE[tid] = tid < 2 * m ? -0x7fffffff : 0;
  __syncthreads();
  const int per = (KT + R - 1) / R;
  const int J0 = min(KT, rank * per), J1 = min(KT, J0 + per);
  {
    // complex column q by `parts` warps, lanes along the rows
    const int parts = max(1, 8 / m);
    const int ja = J0 * kKS, jb = min(n, J1 * kKS);
    for (int u = warp; u < m * parts; u += 8) {
      const int q = u % m, part = u / m;
      int mr = 0, mi = 0;
#pragma unroll 4
      for (int j = ja + part * 32 + lane; j < jb; j += parts * 32) {
        const cd x = Xh[j + (size_t)q * ldx];
        mr = max(mr, abs_hi(x.x));
        mi = max(mi, abs_hi(x.y));
      }
      const int er = scale_exp_hi(__reduce_max_sync(0xffffffffu, mr));
      const int ei = scale_exp_hi(__reduce_max_sync(0xffffffffu, mi));
      if (lane == 0) {
        atomicMax(&sE[2 * q], er);
        atomicMax(&sE[2 * q + 1], ei);
      }
    }
  }
  __syncthreads();
  if (R > 1) {
    cluster_sync_all();
    if (tid < kN) {
      int E = sE[tid];
      for (int r = 0; r < R; ++r) E = max(E, cluster_ld(sE + tid, r));
      tE[tid] = E;
    }
  } else if (tid < kN) {
    tE[tid] = sE[tid];
  }
  __syncthreads();
  if (tid < cs && rank == 0) xexp[(size_t)grp * kN + r0 + tid] = tE[tid];
  // lane = (real column c0 + lane mod 8, K group lane / 8 of the 32-deep tile)
  const int cl = lane & 7, kg = lane >> 3;
  const int nc8 = (cs + 7) / 8;
  for (int u = warp; u < (J1 - J0) * nc8; u += 8) {
    const int J = J0 + u / nc8, c = (u % nc8) * 8 + cl;
    if (c >= cs) continue;
    const int E = tE[c];
    const bool act = c < 2 * m;
    const double* xp = reinterpret_cast<const double*>(Xh + (size_t)(c >> 1) * ldx) + (c & 1);
    unsigned short dg[8][kSl];
    const int j = J * kKS + kg * 8;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      double v = 0.0;
      if (act && j + e < n) v = xp[2 * (size_t)(j + e)];
      digits8(v, E, dg[e]);
    }
    const int off = tile_off(r0 + c, kg * 8);
#pragma unroll
    for (int l = 0; l < kSl; ++l) {
      uint4 o;
      o.x = dg[0][l] | ((unsigned)dg[1][l] << 16);
      o.y = dg[2][l] | ((unsigned)dg[3][l] << 16);
      o.z = dg[4][l] | ((unsigned)dg[5][l] << 16);
      o.w = dg[6][l] | ((unsigned)dg[7][l] << 16);
      const size_t base = ((size_t)(grp * kSl + l) * KT + J) * kBT + off;
      Xs[base / 8] = o;
    }
  }
  if (R > 1) cluster_sync_all();  // no CTA leaves while its maxima may still be read
}

// Work item = (row block I, group g of shifts), 16 groups at a time so that
// the CTAs resident together share H and Xhat tiles in L2.
constexpr int kGroup = 16;
__device__ __forceinline__ void task_coords(long long t, int RB, int cnt, int* I, int* w) {
  const long long full = (long long)(cnt / kGroup) * kGroup * RB;
  if (t < full) {
    const long long g = t / ((long long)kGroup * RB), r = t % ((long long)kGroup * RB);
    *I = (int)(r / kGroup);
    *w = (int)(g * kGroup + r % kGroup);
  } else {
    const int gl = cnt - (cnt / kGroup) * kGroup;
    const long long r = t - full;
    *I = (int)(r / gl);
    *w = (cnt / kGroup) * kGroup + (int)(r % gl);
  }
}

// a bounded wait of one role: gives up at the poll limit or when another role
// has (the block then leaves together)
__device__ __forceinline__ bool role_wait(uint32_t mbar, uint32_t parity, volatile int* fail) {
  for (long long it = 0; it < kWaitLimit / 64; ++it) {
    if (mbar_wait(mbar, parity, 64)) return true;
    if (*fail) return false;
  }
  *fail = 1;
  return false;
}

template <int CS>
__global__ void __launch_bounds__(kT, 1) tc_residual_kernel(
    int n, int m, int npad, const uint4* __restrict__ Hs, const int* __restrict__ hexp,
    const uint4* __restrict__ Xs, const int* __restrict__ xexp, const double* __restrict__ R,
    const cd* __restrict__ shifts, const int* __restrict__ list, const int* __restrict__ count,
    const cd* __restrict__ X, long long ldx, float2* __restrict__ E, double* __restrict__ acc,
    int* __restrict__ err) {
  constexpr int S = kN / CS;  // shifts of a group
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) unsigned long long mbar[8];
  __shared__ uint32_t tslot;
  __shared__ volatile int fail;
  __shared__ int issued[2];  // stages copied, stages multiplied (read when a wait gave up)
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int KT = npad / kKS, RB = npad / kM;
  const int cnt = *count;
  const int ngrp = (cnt + S - 1) / S;
  const long long items = (long long)ngrp * RB;
  // full[b] / empty[b]: stage buffer b copied / multiplied; tfull[t] / tempty[t]:
  // TMEM window t complete / read back
  const uint32_t full = smem_addr(mbar), empty = full + 16, tfull = full + 32, tempty = full + 48;
  const uint32_t sBase = smem_addr(smem);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tslot)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int q = 0; q < 8; ++q)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(full + 8u * q), "r"(q >= 6 ? kDrain / 32 : 1));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fail = 0;
    issued[0] = 0;
    issued[1] = 0;
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tslot;
  if (warp == kDrain / 32) {
    if (lane == 0) {
      // ---- producer: stage i (counted over all items) into buffer i & 1
      unsigned i = 0;
      bool ok = true;
      for (long long t = blockIdx.x; t < items && ok; t += gridDim.x) {
        int I, g;
        task_coords(t, RB, ngrp, &I, &g);
        for (int J = max(0, I * kM - m) / kKS; J < KT; ++J, ++i) {
          const uint32_t b = i & 1u;
          if (!role_wait(empty + 8u * b, ((i >> 1) & 1u) ^ 1u, &fail)) {
            ok = false;
            break;
          }
          const uint32_t dst = sBase + b * kStageBytes, lb = full + 8u * b;
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(lb), "r"(kStageBytes)
                       : "memory");
          for (int k = 0; k < kSl; ++k)
            bulk_copy(dst + (uint32_t)(k * kAT * 2), Hs + ((size_t)(k * RB + I) * KT + J) * (kAT / 8),
                      (uint32_t)(kAT * 2), lb);
          for (int l = 0; l < kSl; ++l)
            bulk_copy(dst + (uint32_t)(kSl * kAT * 2 + l * kBT * 2),
                      Xs + ((size_t)(g * kSl + l) * KT + J) * (kBT / 8), (uint32_t)(kBT * 2), lb);
          issued[0] = (int)(i + 1);
        }
      }
    }
  } else if (warp == kDrain / 32 + 1) {
    if (lane == 0) {
      // ---- issuer: window v (counted over all items) into TMEM half v & 1
      unsigned i = 0, v = 0;
      bool ok = true;
      for (long long t = blockIdx.x; t < items && ok; t += gridDim.x) {
        int I, g;
        task_coords(t, RB, ngrp, &I, &g);
        const int nst = KT - max(0, I * kM - m) / kKS;
        for (int st = 0; st < nst; ++st, ++i) {
          const uint32_t b = i & 1u, h = v & 1u;
          const bool fresh = (st % kWin) == 0;
          if (fresh && !role_wait(tempty + 8u * h, ((v >> 1) & 1u) ^ 1u, &fail)) ok = false;
          if (ok && !role_wait(full + 8u * b, (i >> 1) & 1u, &fail)) ok = false;
          if (!ok) break;
          fence_after();
          const uint32_t aBase = sBase + b * kStageBytes;
          const uint32_t bBase = aBase + (uint32_t)(kSl * kAT * 2);
          const uint32_t d = tmem + h * (uint32_t)kWinCols;
          constexpr uint32_t kSbo = (uint32_t)kKG * 128u;
#pragma unroll
          for (int ks = 0; ks < kKS / 16; ++ks) {
#pragma unroll
            for (int da = 0; da < kSl; ++da) {
              const uint64_t ad = mat_desc(aBase + (uint32_t)(da * kAT * 2 + ks * 256), 128u, kSbo);
              const uint64_t bd = mat_desc(bBase + (uint32_t)(ks * 256), 128u, kSbo);
              // a = 0 reaches every level: its first product opens the window
              mma_bf16(d + (uint32_t)(da * kN), ad, bd, idesc_bf16(kM, kN * (kSl - da)),
                       (fresh && ks == 0 && da == 0) ? 0u : 1u);
            }
          }
          mma_commit(empty + 8u * b);
          issued[1] = (int)(i + 1);
          if ((st % kWin) == kWin - 1 || st == nst - 1) {
            mma_commit(tfull + 8u * h);
            ++v;
          }
        }
      }
    }
  } else {
    // ---- readout and epilogue: thread = (row, half of the columns).  Two warps to
    // a scheduler: with one, 2000 shifts at n = 5000, m = 16 took 60.3 ms (55.1)
    const int hf = warp >> 2, cb = kH * hf;
    // shifts of this half: lb .. lb + SH - 1 of the group, CL columns each from cz on
    constexpr int SH = CS >= kH ? 1 : kH / CS, CL = CS < kH ? CS : kH;
    const int lb = cb / CS, cz = cb % CS;
    unsigned v = 0;
    bool ok = true;
    for (long long t = blockIdx.x; t < items && ok; t += gridDim.x) {
      int I, g;
      task_coords(t, RB, ngrp, &I, &g);
      const int i0 = I * kM;
      const int nst = KT - max(0, i0 - m) / kKS;
      float ah[kH], al[kH];
#pragma unroll
      for (int c = 0; c < kH; ++c) { ah[c] = 0.f; al[c] = 0.f; }
      for (int st = 0; st < nst; st += kWin, ++v) {
        const uint32_t h = v & 1u;
        // every lane polls; the warp agrees (it reads TMEM together)
        ok = __all_sync(0xffffffffu, role_wait(tfull + 8u * h, (v >> 1) & 1u, &fail));
        if (!ok) break;
        fence_after();
        float sc = 0.0078125f * 0.0078125f;  // 2^{-7t}, t = 2
#pragma unroll 1
        for (int lv = 0; lv < kLev; ++lv) {
          uint32_t r[kH];
          tmem_ld16(tmem + ((uint32_t)((warp & 3) * 32) << 16) + h * (uint32_t)kWinCols + (uint32_t)(lv * kN + cb), r);
#pragma unroll
          for (int c = 0; c < kH; ++c) {
            const float pv = __uint_as_float(r[c]) * sc;
            const float s = ah[c] + pv;
            const float bp = s - ah[c];
            al[c] += (ah[c] - (s - bp)) + (pv - bp);
            ah[c] = s;
          }
          sc *= 0.0078125f;
        }
        fence_before();
        __syncwarp();
        if (lane == 0)
          asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tempty + 8u * h) : "memory");
      }
      if (!ok) break;
      // E(i, q) = R(i, q) - (H Xhat)(i, q) + sigma Xhat(i, q) of the group's shifts
      const int i = i0 + (tid & (kM - 1));
      const int Ei = i < n ? hexp[i] : 0;
#pragma unroll
      for (int l = 0; l < SH; ++l) {
        const int w = g * S + lb + l;
        if (w >= cnt) continue;
        const int sh = list[w];
        double e2 = 0.0, x2 = 0.0;
        if (i < n) {
          const cd sigma = shifts[sh];
          const int* Ec = xexp + (size_t)g * kN + cb + l * CL;
          const cd* Xh = X + (size_t)sh * m * ldx;
#pragma unroll
          for (int u = 0; u < CL / 2; ++u) {
            const int q = cz / 2 + u;
            if (q < m) {
              const int c = l * CL + 2 * u;
              const int er_ = Ec[2 * u], ei_ = Ec[2 * u + 1];
              const bool bad = Ei == kBadExp || er_ == kBadExp || ei_ == kBadExp;
              const double hxr = ldexp((double)ah[c] + (double)al[c], Ei + er_);
              const double hxi = ldexp((double)ah[c + 1] + (double)al[c + 1], Ei + ei_);
              const cd x = Xh[i + (size_t)q * ldx];
              double vr = -hxr + (sigma.x * x.x - sigma.y * x.y);
              const double vi = -hxi + (sigma.x * x.y + sigma.y * x.x);
              if (i <= q) vr += R[i + (size_t)q * n];
              if (bad) vr = __longlong_as_double(0x7ff8000000000000LL);
              e2 += vr * vr + vi * vi;
              x2 += x.x * x.x + x.y * x.y;
              if (E != nullptr) E[(size_t)sh * n * m + i + (size_t)q * n] = make_float2((float)vr, (float)vi);
            }
          }
        }
        for (int o = 16; o > 0; o >>= 1) {
          e2 += __shfl_xor_sync(0xffffffffu, e2, o);
          x2 += __shfl_xor_sync(0xffffffffu, x2, o);
        }
        if (lane == 0) {
          atomicAdd(acc + 2 * (size_t)sh, e2);
          atomicAdd(acc + 2 * (size_t)sh + 1, x2);
        }
      }
    }
  }
  __syncwarp();
  __syncthreads();
  if (fail != 0 && tid == 0) {
    // a completion never arrived: record it (every shift then fails
    // certification) and give the copies and products in flight one more
    // bounded wait
    atomicExch(err, 1);
    const unsigned nl = (unsigned)issued[0], nm = (unsigned)issued[1];
    for (unsigned i = nl > 2 ? nl - 2 : 0; i < nl; ++i) mbar_wait(full + 8u * (i & 1u), (i >> 1) & 1u);
    for (unsigned i = nm > 2 ? nm - 2 : 0; i < nm; ++i) mbar_wait(empty + 8u * (i & 1u), (i >> 1) & 1u);
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

__global__ void tc_identity_list_kernel(int s, int* __restrict__ list, int* __restrict__ count,
                                        double* __restrict__ acc) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < s; i += gridDim.x * blockDim.x) {
    list[i] = i;
    acc[2 * (size_t)i] = 0.0;
    acc[2 * (size_t)i + 1] = 0.0;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *count = s;
}

__global__ void tc_eta_kernel(int n, int m, int s, const double* __restrict__ hn,
                              const double* __restrict__ R, const cd* __restrict__ shifts,
                              const double* __restrict__ acc, const int* __restrict__ err,
                              double* __restrict__ eta) {
  const int sh = blockIdx.x * blockDim.x + threadIdx.x;
  if (sh >= s) return;
  double r2 = 0.0;
  for (int q = 0; q < m; ++q)
    for (int i = 0; i <= q && i < n; ++i) r2 = fma(R[i + (size_t)q * n], R[i + (size_t)q * n], r2);
  const cd sg = shifts[sh];
  const double m2 = fmax(hn[0] - 2.0 * sg.x * hn[1] + (double)n * (sg.x * sg.x + sg.y * sg.y), 0.0);
  const double den = sqrt(m2) * sqrt(acc[2 * (size_t)sh + 1]) + sqrt(r2);
  double e = den > 0.0 ? sqrt(acc[2 * (size_t)sh]) / den : (den == den ? 0.0 : den);
  if (*err != 0) e = __longlong_as_double(0x7ff8000000000000LL);
  eta[sh] = e;
}

}  // namespace

int resid_tc_npad(int n) { return (n + kM - 1) / kM * kM; }

int resid_tc_ktile() { return kKS; }

size_t resid_tc_hbytes(int n) {
  const size_t np = (size_t)resid_tc_npad(n);
  return ((size_t)kSl * np * np * 2 + 255) / 256 * 256 + (np * sizeof(int) + 255) / 256 * 256;
}

// bytes of the digit tiles of s shifts in whole groups
static size_t x_tile_bytes(int n, int m, int s) {
  const int S = kN / group_cols(m);
  const size_t G = (size_t)((s + S - 1) / S);
  return (G * kSl * kN * (size_t)resid_tc_npad(n) * 2 + 255) / 256 * 256;
}

size_t resid_tc_xbytes(int n, int m, int s) {
  const int S = kN / group_cols(m);
  const size_t G = (size_t)((s + S - 1) / S);
  return x_tile_bytes(n, m, s) + (G * kN * sizeof(int) + 255) / 256 * 256 + 256;
}

int resid_tc_split_h(const Handle* h, void* hbuf, cudaStream_t st) {
  const int n = h->n, m = h->m, np = resid_tc_npad(n);
  unsigned char* b = static_cast<unsigned char*>(hbuf);
  uint4* Hs = reinterpret_cast<uint4*>(b);
  int* hexp = reinterpret_cast<int*>(b + ((size_t)kSl * np * np * 2 + 255) / 256 * 256);
  SSV_CUDA_TRY(cudaMemsetAsync(hexp, 0x80, sizeof(int) * (size_t)np, st));
  tc_hrow_kernel<<<dim3((unsigned)(np / 128), (unsigned)((n + kHChunk - 1) / kHChunk)), 256, 0, st>>>(n, m, h->H,
                                                                                                     hexp);
  count_launch();
  const long long items = (long long)np * (np / 8);
  const int grid = (int)std::min<long long>((items + 255) / 256, (long long)num_sms() * 16);
  tc_hsplit_kernel<<<grid, 256, 0, st>>>(n, m, np, h->H, hexp, Hs);
  count_launch();
  SSV_CUDA_TRY(cudaGetLastError());
  return SSV_OK;
}

int resid_tc_run(const Handle* h, const void* hbuf, void* xbuf, int s, const double* shifts,
                 const int* list, const int* count, const double* Xhat, long long ldx, void* E,
                 double* acc, int* err, cudaStream_t st) {
  const int n = h->n, m = h->m, np = resid_tc_npad(n);
  if (m > kN / 2) return SSV_ENOTSUP;
  if (s == 0) return SSV_OK;
  const unsigned char* hb = static_cast<const unsigned char*>(hbuf);
  const uint4* Hs = reinterpret_cast<const uint4*>(hb);
  const int* hexp = reinterpret_cast<const int*>(hb + ((size_t)kSl * np * np * 2 + 255) / 256 * 256);
  unsigned char* xb = static_cast<unsigned char*>(xbuf);
  uint4* Xs = reinterpret_cast<uint4*>(xb);
  int* xexp = reinterpret_cast<int*>(xb + x_tile_bytes(n, m, s));
  const cd* X = reinterpret_cast<const cd*>(Xhat);
  const int cs = group_cols(m), S = kN / cs;
  const int xr = cluster_for(s);
  SSV_CUDA_TRY(launch_cluster(tc_xsplit_kernel, s * xr, 256, xr, 0, st, n, m, np, cs, xr, list, count, X, ldx, Xs,
                              xexp));
  auto kern = cs <= 2    ? tc_residual_kernel<2>
              : cs <= 4  ? tc_residual_kernel<4>
              : cs <= 8  ? tc_residual_kernel<8>
              : cs <= 16 ? tc_residual_kernel<16>
                         : tc_residual_kernel<32>;
  SSV_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem));
  const long long tasks = (long long)((s + S - 1) / S) * (np / kM);
  const int grid = (int)std::max<long long>(1, std::min<long long>(tasks, (long long)num_sms()));
  kern<<<grid, kT, kSmem, st>>>(n, m, np, Hs, hexp, Xs, xexp, h->R, reinterpret_cast<const cd*>(shifts), list, count,
                                X, ldx, reinterpret_cast<float2*>(E), acc, err);
  count_launch();
  SSV_CUDA_TRY(cudaGetLastError());
  return SSV_OK;
}

int backward_error_tc(const Handle* h, int s, const double* shifts, const double* Xhat,
                      long long ldx, double* eta, cudaStream_t st) {
  if (s == 0) return SSV_OK;
  if (h->m > kN / 2) return SSV_ENOTSUP;
  const size_t hb = resid_tc_hbytes(h->n), xb = resid_tc_xbytes(h->n, h->m, s);
  const size_t lb = ((size_t)s * sizeof(int) + 255) / 256 * 256;
  const size_t ab = ((size_t)2 * s * sizeof(double) + 255) / 256 * 256;
  unsigned char* buf = nullptr;
  SSV_CUDA_TRY(pool_alloc((void**)&buf, hb + xb + lb + ab + 256, st));
  int* list = reinterpret_cast<int*>(buf + hb + xb);
  double* acc = reinterpret_cast<double*>(buf + hb + xb + lb);
  int* misc = reinterpret_cast<int*>(buf + hb + xb + lb + ab);  // count, err
  int rc = SSV_OK;
  cudaError_t e = cudaMemsetAsync(misc, 0, 2 * sizeof(int), st);
  if (e == cudaSuccess) {
    tc_identity_list_kernel<<<std::min(1024, (s + 255) / 256), 256, 0, st>>>(s, list, misc, acc);
    count_launch();
    rc = resid_tc_split_h(h, buf, st);
    if (rc == SSV_OK)
      rc = resid_tc_run(h, buf, buf + hb, s, shifts, list, misc, Xhat, ldx, nullptr, acc, misc + 1, st);
    if (rc == SSV_OK) {
      tc_eta_kernel<<<(s + 255) / 256, 256, 0, st>>>(h->n, h->m, s, h->hnorm2, h->R,
                                                    reinterpret_cast<const cd*>(shifts), acc,
                                                    misc + 1, eta);
      count_launch();
      e = cudaGetLastError();
    }
  }
  if (e != cudaSuccess) {
    set_cuda_error(e);
    rc = SSV_ECUDA;
  }
  cudaError_t e2 = cudaFreeAsync(buf, st);
  if (e2 != cudaSuccess && rc == SSV_OK) {
    set_cuda_error(e2);
    rc = SSV_ECUDA;
  }
  return rc;
}

}  // namespace ssv
