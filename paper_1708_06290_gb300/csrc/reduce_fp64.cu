// Controller-Hessenberg reduction in FP64 on the GPU (Algorithm 1, Sec. 2).
//
// Step 1  QR of B with Householder reflectors (one per column of B).
// Step 2  each B-reflector applied to A from both sides and to C from the right.
// Step 3  for column j, a reflector acting on rows j+m .. n-1 annihilates
//         A(j+m+1 : n-1, j); applied from the left to the trailing columns,
//         from the right to all rows of A and to C (Step 4, C <- C Q_A).
//
// The reflector H = I - tau v v^T with v(0) = 1 is generated in the
// annihilated column itself: beta is stored at the top and v(1:) below it,
// as LAPACK stores reflectors, so Q can be applied later (ssv_apply_q).
// The solver reads only the structural part of H (rows <= column + m).
//
// Every kernel is stream-ordered; tau never leaves the device.
#include <algorithm>

#include "cluster.cuh"
#include "ssv_internal.cuh"

namespace ssv {

namespace {

// Frobenius norm^2 and trace of the structural part of H.
__global__ void hnorm_kernel(const double* __restrict__ H, int n, int m, double* __restrict__ out) {
  __shared__ double red[2][8];
  double s2 = 0.0, tr = 0.0;
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < (long long)n * n;
       idx += (long long)gridDim.x * blockDim.x) {
    int i = (int)(idx % n), j = (int)(idx / n);
    if (i <= j + m) {
      double v = H[idx];
      s2 = fma(v, v, s2);
      if (i == j) tr += v;
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    s2 += __shfl_down_sync(0xffffffffu, s2, o);
    tr += __shfl_down_sync(0xffffffffu, tr, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = s2;
    red[1][threadIdx.x >> 5] = tr;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0, b = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { a += red[0][w]; b += red[1][w]; }
    atomicAdd(out, a);
    atomicAdd(out + 1, b);
  }
}

// ---------------------------------------------------------------------------
// Back-transform X = Q Xhat, Q = HB_0 .. HB_{kb-1} HA_0 .. HA_{ka-1}, in blocks
// of kQB reflectors in compact WY form (Schreiber and Van Loan 1989):
// H_0 .. H_{k-1} = I - V T V^T with T upper triangular.
//
// What bounds it: 4 real multiply-adds per (row, reflector, complex column) on
// the FP64 pipe (2 per clock and SM), so everything else only has to keep that
// pipe fed.  Columns are independent, so a cluster of CTAs owns a few columns
// for the whole back-transform: no launch per reflector, no grid barrier.  The
// rows are dealt to the cluster's warps in groups of 32 that stay with their
// warp, so X needs no synchronisation at all; the only exchange is the sum of
// W = V^T X over the cluster (32 x 2 CC doubles per block of reflectors,
// through distributed shared memory).  One launch per reflector took 39.0 ms
// for 450 columns at n = 1999 (m = 3) and 18.4 ms for 24 columns at n = 1500;
// this takes 6.6 and 1.2 ms (the multiply-adds alone 5.8 and, on 96 SMs, 0.5).
// ---------------------------------------------------------------------------
constexpr int kQB = 32;    // reflectors per block
constexpr int kQT = 256;   // threads
constexpr int kQW = kQT / 32;
constexpr int kQLd = kQB + 1;

struct QSrc {
  const double* A;    // reflectors of Q_A below the m-th subdiagonal of H (n x n)
  const double* B;    // reflectors of Q_B below the diagonal of R (n x m)
  const double* tauA;
  const double* tauB;
  int n, m, ka, kb;
};

// block b of the product, first to last: the Q_B blocks, then the Q_A blocks
struct QBlock {
  const double* v;    // v[row + k * n]: reflector k of the block
  const double* tau;
  int pv, cnt;        // pivot row of reflector 0; reflectors
};
__host__ __device__ __forceinline__ int q_blocks(int k) { return (k + kQB - 1) / kQB; }
__device__ __forceinline__ QBlock q_block(const QSrc& q, int b) {
  const int nb = q_blocks(q.kb);
  QBlock r;
  if (b < nb) {
    r.v = q.B + (size_t)b * kQB * q.n;
    r.tau = q.tauB + b * kQB;
    r.pv = b * kQB;
    r.cnt = min(kQB, q.kb - b * kQB);
  } else {
    const int j = (b - nb) * kQB;
    r.v = q.A + (size_t)j * q.n;
    r.tau = q.tauA + j;
    r.pv = q.m + j;
    r.cnt = min(kQB, q.ka - j);
  }
  return r;
}
// V(row, k): unit pivot, zeros above it
__device__ __forceinline__ double q_entry(const QBlock& q, int n, int row, int k) {
  const int d = row - q.pv - k;
  if (k >= q.cnt || row >= n || d < 0) return 0.0;
  return d == 0 ? 1.0 : q.v[row + (size_t)k * n];
}

// the 32 x 32 tile of V of one row group, staged by its warp (lane = row, so
// every load is coalesced); read back with lane = reflector
__device__ __forceinline__ void q_stage(const QBlock& q, int n, int row0, double* Vs) {
  const int lane = threadIdx.x & 31;
#pragma unroll 8
  for (int k = 0; k < kQB; ++k) Vs[lane * kQLd + k] = q_entry(q, n, row0 + lane, k);
}

// T of every block: S = V^T V by a cluster of CTAs, then column by column
// T(0:j, j) = -tau_j T(0:j, 0:j) S(0:j, j)
__global__ void __launch_bounds__(kQT) q_t_kernel(QSrc q, int R, double* __restrict__ T) {
  extern __shared__ double qsm[];
  double* Vs = qsm;                                    // kQW tiles
  double* Sp = Vs + kQW * kQB * kQLd;                  // this CTA's S
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = cluster_rank();
  const int b = blockIdx.x / R;
  const QBlock qb = q_block(q, b);
  // The tiles of kQW row groups are staged at a time, each by its warp; every warp then
  // adds up its kQB / kQW columns of S over all of them, a tile at a time (a warp that
  // kept a tile to itself had 1024 multiply-adds of 64 clocks on its scheduler, 30 us,
  // where a small system has one tile).
  constexpr int NJ = kQB / kQW;
  double acc[NJ];
#pragma unroll
  for (int u = 0; u < NJ; ++u) acc[u] = 0.0;
  for (int g0 = qb.pv / 32 + rank; g0 * 32 < q.n; g0 += kQW * R) {
    __syncthreads();
    if ((g0 + warp * R) * 32 < q.n) q_stage(qb, q.n, (g0 + warp * R) * 32, Vs + warp * kQB * kQLd);
    __syncthreads();
    for (int t = 0; t < kQW && (g0 + t * R) * 32 < q.n; ++t) {
      const double* Vt = Vs + t * kQB * kQLd;
      double s[NJ];
#pragma unroll
      for (int u = 0; u < NJ; ++u) s[u] = 0.0;
#pragma unroll 8
      for (int rr = 0; rr < 32; ++rr) {
        const double v = Vt[rr * kQLd + lane];
#pragma unroll
        for (int u = 0; u < NJ; ++u) s[u] = fma(v, Vt[rr * kQLd + warp * NJ + u], s[u]);
      }
#pragma unroll
      for (int u = 0; u < NJ; ++u) acc[u] += s[u];
    }
  }
#pragma unroll
  for (int u = 0; u < NJ; ++u) Sp[(warp * NJ + u) * kQB + lane] = acc[u];
  cluster_sync_all();
  if (rank == 0) {
    double* S = Vs;                  // summed over the cluster
    double* Ts = Vs + kQB * kQLd;
    for (int e = tid; e < kQB * kQB; e += kQT) {
      double v = 0.0;
      for (int r = 0; r < R; ++r) v += cluster_ld(Sp + e, r);
      S[(e / kQB) * kQLd + e % kQB] = v;
      Ts[(e / kQB) * kQLd + e % kQB] = 0.0;
    }
    __syncthreads();
    if (warp == 0) {
      for (int j = 0; j < qb.cnt; ++j) {
        const double tau = qb.tau[j];
        double v = 0.0;
        for (int k = lane; k < j; ++k) v = fma(Ts[lane * kQLd + k], S[k * kQLd + j], v);
        __syncwarp();
        if (lane < j) Ts[lane * kQLd + j] = -tau * v;
        if (lane == j) Ts[lane * kQLd + j] = tau;
        __syncwarp();
      }
    }
    __syncthreads();
    for (int e = tid; e < kQB * kQB; e += kQT) T[(size_t)b * kQB * kQB + e] = Ts[(e / kQB) * kQLd + e % kQB];
  }
  cluster_sync_all();  // no CTA leaves while its S may still be read
}

// X <- Q X for CC complex columns per cluster of R CTAs
template <int CC>
__global__ void __launch_bounds__(kQT) apply_q_kernel(QSrc q, int R, const double* __restrict__ T,
                                                      cd* __restrict__ X, long long ldx, int ncols) {
  constexpr int C2 = 2 * CC;
  extern __shared__ double qsm[];
  double* Vs = qsm;                                    // kQW tiles of V
  double* xs = Vs + kQW * kQB * kQLd;                  // kQW tiles of 32 x C2 of X
  double* wred = xs + kQW * 32 * C2;                   // kQW x 32 x C2
  double* wsum = wred + kQW * kQB * C2;                // 2 x 32 x C2 (by parity of the block)
  double* Wt = wsum + 2 * kQB * C2;                    // 32 x C2
  double* Zs = Wt + kQB * C2;                          // 32 x C2
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = cluster_rank();
  const int c0 = (int)(blockIdx.x / R) * CC;
  const int n = q.n, step = kQW * R;
  double* Vw = Vs + warp * kQB * kQLd;
  double* xw = xs + warp * 32 * C2;
  const int nblk = q_blocks(q.kb) + q_blocks(q.ka);
  for (int b = nblk - 1; b >= 0; --b) {
    const QBlock qb = q_block(q, b);
    // groups of 32 rows; group g belongs to warp (g / R) mod kQW of rank g mod R
    const int gs = qb.pv / 32;
    const int own = warp * R + rank;
    const int g0 = gs + ((own - gs) % step + step) % step;
    // ---- W = V^T X
    double acc[C2];
#pragma unroll
    for (int c = 0; c < C2; ++c) acc[c] = 0.0;
    for (int g = g0; g * 32 < n; g += step) {
      const int row = g * 32 + lane;
      __syncwarp();
#pragma unroll
      for (int c = 0; c < CC; ++c) {
        cd v = mkcd(0.0, 0.0);
        if (row < n && c0 + c < ncols) v = X[row + (size_t)(c0 + c) * ldx];
        xw[lane * C2 + 2 * c] = v.x;
        xw[lane * C2 + 2 * c + 1] = v.y;
      }
      q_stage(qb, n, g * 32, Vw);
      __syncwarp();
#pragma unroll 4
      for (int rr = 0; rr < 32; ++rr) {
        const double v = Vw[rr * kQLd + lane];
#pragma unroll
        for (int c = 0; c < C2; ++c) acc[c] = fma(v, xw[rr * C2 + c], acc[c]);
      }
    }
#pragma unroll
    for (int c = 0; c < C2; ++c) wred[(warp * kQB + lane) * C2 + c] = acc[c];
    __syncthreads();
    double* ws = wsum + (b & 1) * kQB * C2;
    for (int e = tid; e < kQB * C2; e += kQT) {
      double v = 0.0;
#pragma unroll
      for (int w = 0; w < kQW; ++w) v += wred[w * kQB * C2 + e];
      ws[e] = v;
      if (R == 1) Wt[e] = v;
    }
    if (R > 1) {
      // a buffer is written again two blocks later, after the next block's
      // barrier, which every reader of it has passed by then
      cluster_sync_all();
      for (int e = tid; e < kQB * C2; e += kQT) {
        double v = 0.0;
        for (int r = 0; r < R; ++r) v += cluster_ld(ws + e, r);
        Wt[e] = v;
      }
    }
    __syncthreads();
    // ---- Z = T W
    for (int e = tid; e < kQB * C2; e += kQT) {
      const int k = e / C2, c = e % C2;
      const double* Tb = T + (size_t)b * kQB * kQB + k * kQB;
      double v = 0.0;
#pragma unroll 8
      for (int j = 0; j < kQB; ++j) v = fma(__ldg(Tb + j), Wt[j * C2 + c], v);
      Zs[e] = v;
    }
    __syncthreads();
    // ---- X -= V Z: lane = row
    for (int g = g0; g * 32 < n; g += step) {
      const int row = g * 32 + lane;
      double x[C2];
#pragma unroll
      for (int c = 0; c < CC; ++c) {
        cd v = mkcd(0.0, 0.0);
        if (row < n && c0 + c < ncols) v = X[row + (size_t)(c0 + c) * ldx];
        x[2 * c] = v.x;
        x[2 * c + 1] = v.y;
      }
#pragma unroll 16
      for (int k = 0; k < kQB; ++k) {
        const double v = q_entry(qb, n, row, k);
#pragma unroll
        for (int c = 0; c < C2; ++c) x[c] = fma(-v, Zs[k * C2 + c], x[c]);
      }
#pragma unroll
      for (int c = 0; c < CC; ++c)
        if (row < n && c0 + c < ncols) X[row + (size_t)(c0 + c) * ldx] = mkcd(x[2 * c], x[2 * c + 1]);
    }
  }
  if (R > 1) cluster_sync_all();  // no CTA leaves while its sums may still be read
}

// n <= 32 NR: a warp per column, lane l the rows l, l + 32, .., one reflector after
// another.  Bound by the FP64 pipe (10 + 4 NR instructions of 64 clocks a column and
// reflector).
constexpr int kQSmall = 64;
constexpr int kQTiny = 16;  // up to here this kernel alone (no T factors)
template <int NR>
__global__ void __launch_bounds__(256) apply_q_small_kernel(QSrc q, cd* __restrict__ X, long long ldx, int ncols) {
  const int lane = threadIdx.x & 31, c = (int)((blockIdx.x * 256ll + threadIdx.x) >> 5);
  if (c >= ncols) return;  // the whole warp
  cd x[NR];
#pragma unroll
  for (int u = 0; u < NR; ++u) {
    const int r = lane + 32 * u;
    x[u] = r < q.n ? X[r + (size_t)c * ldx] : mkcd(0.0, 0.0);
  }
  auto reflect = [&](const double* v, double tau, int pv) {
    double vr[NR], wr = 0.0, wi = 0.0;
#pragma unroll
    for (int u = 0; u < NR; ++u) {
      const int r = lane + 32 * u;
      vr[u] = r < pv || r >= q.n ? 0.0 : r == pv ? 1.0 : v[r];
      wr = fma(vr[u], x[u].x, wr);
      wi = fma(vr[u], x[u].y, wi);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      wr += __shfl_xor_sync(0xffffffffu, wr, o);
      wi += __shfl_xor_sync(0xffffffffu, wi, o);
    }
    wr *= -tau;
    wi *= -tau;
#pragma unroll
    for (int u = 0; u < NR; ++u) x[u] = mkcd(fma(wr, vr[u], x[u].x), fma(wi, vr[u], x[u].y));
  };
  for (int j = q.ka - 1; j >= 0; --j) reflect(q.A + (size_t)j * q.n, __ldg(q.tauA + j), q.m + j);
  for (int j = q.kb - 1; j >= 0; --j) reflect(q.B + (size_t)j * q.n, __ldg(q.tauB + j), j);
#pragma unroll
  for (int u = 0; u < NR; ++u) {
    const int r = lane + 32 * u;
    if (r < q.n) X[r + (size_t)c * ldx] = x[u];
  }
}

constexpr size_t kQTSmem = sizeof(double) * (size_t)(kQW * kQB * kQLd + kQB * kQB);
template <int CC>
constexpr size_t q_apply_smem() {
  return sizeof(double) * (size_t)(kQW * kQB * kQLd + 2 * kQW * 32 * 2 * CC + 4 * kQB * 2 * CC);
}

template <int CC>
cudaError_t launch_apply_q(const QSrc& q, int R, const double* T, cd* X, long long ldx, int ncols,
                           cudaStream_t st) {
  const int grid = (ncols + CC - 1) / CC * R;
  const cudaError_t e = allow_smem(apply_q_kernel<CC>, q_apply_smem<CC>());
  return e != cudaSuccess ? e : launch_cluster(apply_q_kernel<CC>, grid, kQT, R, q_apply_smem<CC>(), st, q, R, T, X, ldx, ncols);
}

__global__ void copy_masked_kernel(const double* __restrict__ src, long long lds, int rows, int cols,
                                   int band, double* __restrict__ dst, long long ldd) {
  // dst(i, j) = src(i, j) if i <= j + band else 0
  long long total = (long long)rows * cols;
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x) {
    int i = (int)(idx % rows), j = (int)(idx / rows);
    dst[i + (size_t)j * ldd] = (i <= j + band) ? src[i + (size_t)j * lds] : 0.0;
  }
}

__global__ void copy_cd_kernel(const cd* __restrict__ src, long long lds, int rows, int cols,
                               cd* __restrict__ dst, long long ldd) {
  long long total = (long long)rows * cols;
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x) {
    int i = (int)(idx % rows), j = (int)(idx / rows);
    dst[i + (size_t)j * ldd] = src[i + (size_t)j * lds];
  }
}

// Hhi = fl32(H), Hlo = fl32(H - Hhi) on and above the m-th subdiagonal; 0 below.
__global__ void split_h_kernel(const double* __restrict__ H, int n, int m, float* __restrict__ hi,
                               float* __restrict__ lo) {
  long long total = (long long)n * n;
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x) {
    int i = (int)(idx % n), j = (int)(idx / n);
    float a = 0.0f, b = 0.0f;
    if (i <= j + m) {
      double v = H[idx];
      a = (float)v;
      b = (float)(v - (double)a);
    }
    hi[idx] = a;
    lo[idx] = b;
  }
}

QSrc q_src(const Handle* h) {
  QSrc q;
  q.A = h->H;
  q.B = h->R;
  q.tauA = h->tauA;
  q.tauB = h->tauB;
  q.n = h->n;
  q.m = h->m;
  q.ka = h->ka;
  q.kb = h->kb;
  return q;
}

}  // namespace

size_t q_t_count(int n, int m) { return (size_t)(q_blocks(n) + q_blocks(m)) * kQB * kQB; }

// the T factors of Q's blocks, kept in the handle; none where apply_q needs none (with
// that, and S spread over all warps, reductions of n = 2, 8 and 30 take 0.27, 0.38 and
// 1.22 ms instead of 0.34, 0.45 and 1.29)
static int make_q_t(Handle* h, cudaStream_t st) {
  const int nblk = q_blocks(h->kb) + q_blocks(h->ka);
  if (nblk == 0 || h->n <= kQTiny) return SSV_OK;
  constexpr int kR = 4;
  SSV_CUDA_TRY(allow_smem(q_t_kernel, kQTSmem));
  SSV_CUDA_TRY(launch_cluster(q_t_kernel, nblk * kR, kQT, kR, kQTSmem, st, q_src(h), kR, h->Tq));
  return SSV_OK;
}

int reduce_fp64(Handle* h, const double* A, long long lda, const double* B, long long ldb,
                const double* C, long long ldc, int arith, cudaStream_t st) {
  const int n = h->n, m = h->m, p = h->p;
  const int ldct = p > 0 ? p : 1;
  SSV_CUDA_TRY(cudaMemcpy2DAsync(h->H, sizeof(double) * n, A, sizeof(double) * lda,
                                 sizeof(double) * n, n, cudaMemcpyDeviceToDevice, st));
  SSV_CUDA_TRY(cudaMemcpy2DAsync(h->R, sizeof(double) * n, B, sizeof(double) * ldb,
                                 sizeof(double) * n, m, cudaMemcpyDeviceToDevice, st));
  if (p > 0)
    SSV_CUDA_TRY(cudaMemcpy2DAsync(h->Ct, sizeof(double) * ldct, C, sizeof(double) * ldc,
                                   sizeof(double) * p, n, cudaMemcpyDeviceToDevice, st));
  // Steps 1-4 of Algorithm 1: one persistent cooperative kernel on the FP64
  // pipe, or the two-level blocked form with its products on the tensor cores
  int rc = arith == SSV_REDUCE_TENSOR ? reduce_tc(h, st) : reduce_persistent(h, st);
  if (rc != SSV_OK) return rc;
  rc = make_q_t(h, st);
  if (rc != SSV_OK) return rc;
  h->has_q = 1;
  SSV_CUDA_TRY(cudaMemsetAsync(h->hnorm2, 0, 2 * sizeof(double), st));
  hnorm_kernel<<<std::max(1, std::min(1024, (n * n + 255) / 256)), 256, 0, st>>>(h->H, n, m,
                                                                                h->hnorm2);
  count_launch();
  SSV_CUDA_TRY(cudaGetLastError());
  return SSV_OK;
}

int apply_q(const Handle* h, int ncols, const double* Xhat, long long ldx, double* X, long long ldX,
            bool digits, cudaStream_t st, int* status, double* resid) {
  const int n = h->n;
  if (ncols == 0) return SSV_OK;
  cd* Xc = reinterpret_cast<cd*>(X);
  if (X != Xhat) {
    int blocks = (int)std::min<long long>(4096, ((long long)n * ncols + 255) / 256);
    copy_cd_kernel<<<blocks, 256, 0, st>>>(reinterpret_cast<const cd*>(Xhat), ldx, n, ncols, Xc,
                                           ldX);
    count_launch();
    SSV_CUDA_TRY(cudaGetLastError());
  }
  const int nblk = q_blocks(h->kb) + q_blocks(h->ka);
  if (nblk == 0) return SSV_OK;
  if (digits && apply_q_tc_supported(h->n, ncols)) {
    const int rc = apply_q_tc(h, ncols, Xc, ldX, st, status, resid);
    if (rc != SSV_ENOMEM) return rc;
    cudaGetLastError();  // no room for its scratch (nothing written yet): the FP64 path needs none
  }
  const QSrc q = q_src(h);
  // Small systems: the blocked kernel spends 20 us a wave of CTAs whatever n is, this
  // one 1.3 us a reflector and wave.  One launch per reflector / blocks / this, us: n =
  // 8, 700 columns 41 / 71 / 24; n = 32, 8000 columns 394 / 560 / 269; n = 64, 700
  // columns 337 / 118 / 113 and 8000 859 / 882 / 646.  With fewer columns the blocks
  // are the faster ones from n = 17 on (n = 33, 64 columns 40 / 63; n = 64 55 / 114).
  if (n <= kQTiny || (n <= kQSmall && ncols >= 512)) {
    auto kern = n <= 32 ? apply_q_small_kernel<1> : apply_q_small_kernel<2>;
    kern<<<(unsigned)((ncols + 7) / 8), 256, 0, st>>>(q, Xc, ldX, ncols);
    count_launch();
    SSV_CUDA_TRY(cudaGetLastError());
    return SSV_OK;
  }
  const double* T = h->Tq;
  // Columns per cluster: the widest (V is read once per cluster) with at most a tenth
  // more columns on the busiest SM than the best width gives (8000 columns: four
  // rather than one, whose SM has 56 instead of 53: n = 200, 3.67 -> 2.50 ms); CTAs per
  // cluster: as many as the SMs allow when there are fewer columns than SMs.
  const int sms = num_sms();
  auto load = [&](int c) { return ((ncols + c - 1) / c + sms - 1) / sms * (long long)c; };
  const long long best = std::min({load(1), load(2), load(3), load(4)});
  int cc = 4;
  while (10 * load(cc) > 11 * best) --cc;
  const int groups = (ncols + cc - 1) / cc;
  int R = 1;
  while (R < 8 && (long long)groups * R * 2 <= sms && n > 32 * kQW * R) R *= 2;
  if (cc == 1) SSV_CUDA_TRY(launch_apply_q<1>(q, R, T, Xc, ldX, ncols, st));
  else if (cc == 2) SSV_CUDA_TRY(launch_apply_q<2>(q, R, T, Xc, ldX, ncols, st));
  else if (cc == 3) SSV_CUDA_TRY(launch_apply_q<3>(q, R, T, Xc, ldX, ncols, st));
  else SSV_CUDA_TRY(launch_apply_q<4>(q, R, T, Xc, ldX, ncols, st));
  return SSV_OK;
}

int load_reduced(Handle* h, const double* H, long long ldh, const double* R, long long ldr,
                 const double* Ct, long long ldc, cudaStream_t st) {
  const int n = h->n, m = h->m, p = h->p;
  int blocks = (int)std::min<long long>(4096, ((long long)n * n + 255) / 256);
  copy_masked_kernel<<<blocks, 256, 0, st>>>(H, ldh, n, n, m, h->H, n);
  count_launch();
  SSV_CUDA_TRY(cudaGetLastError());
  blocks = (int)std::min<long long>(4096, ((long long)n * m + 255) / 256);
  copy_masked_kernel<<<blocks, 256, 0, st>>>(R, ldr, n, m, 0, h->R, n);
  count_launch();
  SSV_CUDA_TRY(cudaGetLastError());
  if (p > 0)
    SSV_CUDA_TRY(cudaMemcpy2DAsync(h->Ct, sizeof(double) * p, Ct, sizeof(double) * ldc,
                                   sizeof(double) * p, n, cudaMemcpyDeviceToDevice, st));
  h->kb = 0;
  h->ka = 0;
  h->has_q = 0;
  SSV_CUDA_TRY(cudaMemsetAsync(h->hnorm2, 0, 2 * sizeof(double), st));
  hnorm_kernel<<<std::max(1, std::min(1024, (n * n + 255) / 256)), 256, 0, st>>>(h->H, n, m,
                                                                                h->hnorm2);
  count_launch();
  SSV_CUDA_TRY(cudaGetLastError());
  return SSV_OK;
}

int split_h(Handle* h, cudaStream_t st) {
  const int n = h->n;
  int blocks = (int)std::min<long long>(8192, ((long long)n * n + 255) / 256);
  split_h_kernel<<<blocks, 256, 0, st>>>(h->H, n, h->m, h->Hhi, h->Hlo);
  count_launch();
  SSV_CUDA_TRY(cudaGetLastError());
  return SSV_OK;
}

int get_reduced(const Handle* h, double* H, long long ldh, double* R, long long ldr, double* Ct,
                long long ldc, cudaStream_t st) {
  const int n = h->n, m = h->m, p = h->p;
  if (H) {
    int blocks = (int)std::min<long long>(4096, ((long long)n * n + 255) / 256);
    copy_masked_kernel<<<blocks, 256, 0, st>>>(h->H, n, n, n, m, H, ldh);
    count_launch();
    SSV_CUDA_TRY(cudaGetLastError());
  }
  if (R) {
    int blocks = (int)std::min<long long>(4096, ((long long)n * m + 255) / 256);
    copy_masked_kernel<<<blocks, 256, 0, st>>>(h->R, n, n, m, 0, R, ldr);
    count_launch();
    SSV_CUDA_TRY(cudaGetLastError());
  }
  if (Ct && p > 0) {
    SSV_CUDA_TRY(cudaMemcpy2DAsync(Ct, sizeof(double) * ldc, h->Ct, sizeof(double) * p,
                                   sizeof(double) * p, n, cudaMemcpyDeviceToDevice, st));
  }
  return SSV_OK;
}

}  // namespace ssv
