// Shift-batched sweep with the trailing update on the tensor cores.
//
// The sweep of Sec. 3.1 / Algorithm 8 for every shift, run as the paper runs
// it on a GPU: one phase per block step k for all shifts at once, so that the
// update of the rows above the block ("Step 2, revisited": one GEMM with the
// shared operand Z1 = [Ct; H](1:r, fresh columns) and every shift's block
// transform, Z2 <- Z1 P1 + Z2 P2 - sigma E P1) multiplies a tile of H that is
// staged once for a group of shifts.  Per block step:
//
//   1. panel (one thread block per shift; five, three, two or one per SM by m and
//      the number of shifts): the n_b x (n_b + m) window block is triangularised
//      bottom-up by one complex Householder reflector per row
//      over the m + 1 candidate columns (double-word reflector scalars,
//      double-float application, as in the double-float sweep), giving the
//      coefficients P1 (n_b x m) and P2 (m x m).  The panel also updates the p
//      rows of Ct (small), writes P1 as BF16 digit tiles, and keeps the P1
//      rows and P2 that the X-hat back pass needs;
//   2. update (persistent, one thread block per SM): work items of 128 rows
//      of H x one group of shifts (N = 32 real columns: each shift's m complex
//      columns as 2m real ones, padded to a power of two).  Z1 P1 is formed
//      exactly as in the tensor-core residual (error-free splitting after
//      Ozaki, Ogita, Oishi and Rump): H's rows and P1's real columns are
//      written as 7-bit digits relative to a power-of-two scale (eight for a
//      row of H, seven for a column of P1), each digit exact in BF16, and the
//      35 digit products H_k P_l with k + l <= 7 run as tcgen05.mma (BF16 x
//      BF16 -> FP32, M = 128, K = 16, seven digits of P1 per product) into eight TMEM accumulators, one
//      per level k + l, where every partial sum is an integer below
//      128 * 127 * (128 + 6 * 80) < 2^24 and therefore exact (H's digits are up to
//      127, a column's first up to 128 and the others up to 80 in modulus).  The
//      digit tiles reach shared memory by 1-D TMA bulk copies on an mbarrier,
//      two stages in flight.  The epilogue reads the levels back (tcgen05.ld),
//      adds them scaled by 2^{-7 t} into double-float sums, scales by the row
//      and column exponents, and adds Z2 P2 (m >= 5: digit products too) and the
//      shifted-diagonal correction in double-float on the FP32 pipe;
//   3. after the last block: the final m x m block, G = Ct Xhat or X-hat by the
//      backward pass over the stored block transforms.
//
// Accuracy: the digits beyond the eighth of H and the seventh of P1 and the
// products of level > 7 are dropped, about 2^-49 of the row scale times the
// column scale (the double-float class of the SSV_DFLOAT sweep).  H's rows get
// all eight digits because a dominant diagonal sets the row scale: the
// off-diagonal entries of a row can be 2^7 below it.  The first block holds
// (n - m) mod n_b rows (n_b when that is 0), so that every later block starts
// at a column that is a multiple of n_b and the H digit tiles (32 columns
// deep) line up with the fresh columns.
#include <algorithm>

#include "dfloat.cuh"
#include "panel.cuh"
#include "ssv_internal.cuh"
#include "tc_common.cuh"

namespace ssv {

namespace {

using namespace tcg;

// Debug builds (-DSSV_BOUNDS_CHECK): the indices into the sweep's scratch, its
// digit tiles, the panels' H and X-hat are checked against their buffers; an
// index out of range sets bit 2 of the solve's error word (every shift of the
// solve then reports a non-finite result) and is replaced by 0, so the access
// stays inside the buffer.  In normal builds BCK(i, n) is i.
#ifdef SSV_BOUNDS_CHECK
__device__ __forceinline__ size_t bck(long long i, size_t n, int* err) {
  if (i < 0 || (size_t)i >= n) {
    atomicOr(err, 2);
    return 0;
  }
  return (size_t)i;
}
#define BCK(i, n) bck((long long)(i), (size_t)(n), a.err)
#else
#define BCK(i, n) ((size_t)(i))
#endif

constexpr int kPT = 256;             // threads of the setup and final kernels
constexpr int kNBT = 128;            // n_b of the tensor-core sweep (K of the update)
constexpr int kMaxM = kTcMaxM;       // m <= 16
constexpr int kUM = 128;             // H rows per update item = TMEM lanes
constexpr int kUN = 32;              // real columns per update item (a group of shifts)
constexpr int kKS = 32;              // K per shared-memory stage
constexpr int kKG = kKS / 8;         // core matrices along K in a tile
constexpr int kSDH = 8;              // digits of H (all eight slices of its digit tiles)
constexpr int kSD = 7;               // digits of the block transforms' columns
constexpr int kLev = 8;              // levels k + l = 0 .. 7
constexpr int kStages = kNBT / kKS;  // stages per block step
constexpr int kAT = kUM * kKS;       // BF16 elements of one H digit tile
constexpr int kBT = kUN * kKS;       // BF16 elements of one P1 digit tile
constexpr uint32_t kStageBytes = (uint32_t)(kSDH * kAT + kSD * kBT) * 2;  // H and P1 digit tiles
constexpr int kWinCols = kLev * kUN;  // TMEM columns of a window; there are two
// polls of one mbarrier wait before the update gives up (a stage's copies and
// products complete within microseconds)
constexpr long long kUpdWait = 1LL << 22;
static_assert(2 * kWinCols == 512, "TMEM columns of the two windows");
// shared memory of the update: two stage buffers, then the Z2 and P2 digit tiles
// of one item (S shifts: 7 digits of 128 x cs and of cs x cs; S cs = kUN)
constexpr size_t kOffZ = 2 * (size_t)kStageBytes;
constexpr size_t kUpdSmem = kOffZ + (size_t)7 * (128 * kUN + kUN * 32) * 2;
static_assert(kUpdSmem + 1024 <= 227 * 1024, "shared memory of the update");

// element offset in a K-major core-matrix tile (8 rows x 8 K per 128 bytes;
// byte strides 128 along K, kKG * 128 along rows): the layout of the residual's
// H digit tiles
__host__ __device__ __forceinline__ int tile_off(int row, int k) {
  return (((row >> 3) * kKG + (k >> 3)) * 8 + (row & 7)) * 8 + (k & 7);
}

// column stride of one shift in a group: 2m real columns rounded up to a power of two
__host__ __device__ inline int shift_cols(int m) {
  int c = 2;
  while (c < 2 * m) c <<= 1;
  return c;
}

struct TcsArgs {
  int n, m, p, s, cs, S, ngroups, mode;
  const double* H;       // n x n
  const float* Hhi;      // double-float split of H
  const float* Hlo;
  const double* Ct;      // p x n (ld ldct)
  int ldct;
  const double* R;       // n x m
  const cd* shifts;
  const double* hnorm;   // ||H||_F^2, trace(H)
  float4* Z2;            // per shift: (p + n) x m double-float window columns, ld p + n
  cd* ZT;                // per shift: n x m rows P1 of every step (X-hat mode), or null
  size_t z2_stride;      // float4 per shift slot
  uint16_t* Pd;          // P1 digit tiles: [group][digit][stage][kBT]
  int* pexp;             // per shift: 2m column exponents (stride 2 kMaxM)
  float4* pc;            // per shift: P2 (m x m) then sigma rows P1(0:min(m,nbe), :) (m x m)
  cd* out;
  long long ldo;
  int* flags;            // per shift: 1 = singular to working precision
  int* status;
  const uint4* Hs;       // H digit tiles (residual layout) and row exponents
  const int* hexp;
  int RB, KT;            // row blocks / K blocks of the H digit tiles
  int* err;              // an update wait gave up
  // Z2 P2 on the tensor cores (cs >= 16, m >= 5): the H rows of every shift's
  // window columns as digit tiles (row-scaled, K = cs real entries interleaved
  // Re, Im) and the real form of each step's P2 (column-scaled, cs x cs)
  int tcz;
  int npad;
  uint16_t* Zd;          // [shift][row block][digit][128 x cs]
  int* zexp;             // [shift][npad] row exponents
  uint16_t* P2d;         // [shift][digit][cs x cs]
  int* p2exp;            // [shift][2 kMaxM] column exponents
  // buffer sizes (elements) for the debug build's index checks
  size_t n_z2, n_zt, n_pd, n_zd, n_p2d, n_pc, n_hs, n_out;
};

// exponent 0 for a zero (or denormal) row or column: its digits are zero at any
// scale, and the update's fast path takes moderate exponents only
__device__ __forceinline__ int col_exp(int E) { return E <= -126 ? 0 : E; }

// digit tiles of window row p + i (H row i) of shift sh, from the double-float
// values Z2f(p + i, q): the row exponent over the 2m real entries, seven
// digits of each entry at K = 2q (Re), 2q + 1 (Im), zero up to cs
__device__ void write_z2_digits(const TcsArgs& a, int sh, int i, const float4* Z2f, int ldz) {
  const int m = a.m, cs = a.cs, kg = cs / 8;
  float mx = 0.f;
  for (int q = 0; q < m; ++q) {
    const float4 z = Z2f[BCK((a.p + i) + (size_t)q * ldz, a.z2_stride)];
    mx = fmaxf(mx, fmaxf(fabsf(z.x), fabsf(z.z)));
    if (!(fabsf(z.x) <= 3.4e38f) || !(fabsf(z.z) <= 3.4e38f)) mx = __int_as_float(0x7f800000);
  }
  const int E = col_exp(scale_exp_f(mx));
  a.zexp[BCK((size_t)sh * a.npad + i, (size_t)a.s * a.npad)] = E;
  const float inv = digit_scale(E);
  const size_t T0 = ((size_t)sh * a.RB + i / 128) * 7 * (128 * cs);
  for (int k8 = 0; k8 < cs; k8 += 8) {
    float hi[8], lo[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int kk = k8 + e, q = kk >> 1;
      hi[e] = lo[e] = 0.f;
      if (q < m) {
        const float4 z = Z2f[BCK((a.p + i) + (size_t)q * ldz, a.z2_stride)];
        hi[e] = (kk & 1) ? z.z : z.x;
        lo[e] = (kk & 1) ? z.w : z.y;
      }
    }
    const int off = tile_off_kg(i % 128, k8, kg);
    uint4 dg[7];
    digits7_oct(hi, lo, inv, dg);
#pragma unroll
    for (int l = 0; l < 7; ++l)
      *reinterpret_cast<uint4*>(a.Zd + BCK(T0 + (size_t)l * (128 * cs) + off, a.n_zd)) = dg[l];
  }
}

__device__ __forceinline__ double shifted_norm2(const double* hnorm, int n, cd sg) {
  return fmax(hnorm[0] - 2.0 * sg.x * hnorm[1] + (double)n * (sg.x * sg.x + sg.y * sg.y), 0.0);
}

// ---- setup: Z2 = last m columns of [Ct; H] - sigma on the diagonal ---------
__global__ void __launch_bounds__(kPT) tcs_setup_kernel(TcsArgs a) {
  const int sh = blockIdx.x;
  const int n = a.n, m = a.m, p = a.p, ldz = p + n;
  const cd sigma = a.shifts[sh];
  float4* Z2 = a.Z2 + (size_t)sh * a.z2_stride;
  for (long long idx = threadIdx.x; idx < (long long)ldz * m; idx += kPT) {
    const int i = (int)(idx % ldz), q = (int)(idx / ldz);
    const int j = n - m + q;
    const double v = i < p ? a.Ct[i + (size_t)j * a.ldct] : a.H[(i - p) + (size_t)j * n];
    cd z = mkcd(v, 0.0);
    if (i - p == j) z = csub(z, sigma);
    Z2[BCK(idx, a.z2_stride)] = df_split(z);
  }
  if (threadIdx.x == 0) a.flags[sh] = 0;
  if (a.tcz) {
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += kPT) write_z2_digits(a, sh, i, Z2, ldz);
  }
}

// ---- panel of block step `step` (1-based), rows k - nbe .. k - 1 ------------
constexpr int kCtRows = 16;  // rows of Ct staged at a time
template <int MAXM>
struct PanelSmem {
  using Panel = pan::Smem<pan::DF32, MAXM, kNBT>;
  static constexpr int S = Panel::S;
  Panel p;  // p.W: the coefficients; p.F: later a chunk of Ct rows as FP32 pairs
  int fexp[2 * kMaxM];
  int f2exp[2 * kMaxM];
  int sing;
};
// Threads and resident panels per SM.  FEW (no more shifts than SMs, m > 8): one
// panel per SM with twice the threads for the update of the sub-block's other
// rows (m = 16: 180 us per block of 128 rows against 188); else two with 256.
template <int MAXM, bool FEW>
constexpr int panel_threads() { return MAXM <= 4 ? 128 : MAXM <= 8 || !FEW ? 256 : 512; }
template <int MAXM, bool FEW>
constexpr int panel_per_sm() { return MAXM <= 4 ? 5 : MAXM <= 8 ? 3 : FEW ? 1 : 2; }

template <int MAXM, bool FEW>
__global__ void __launch_bounds__(panel_threads<MAXM, FEW>(), panel_per_sm<MAXM, FEW>())
    tcs_panel_kernel(TcsArgs a, int k, int nbe, int step) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  using PS = PanelSmem<MAXM>;
  PS& sm = *reinterpret_cast<PS*>(smem_raw);
  constexpr int S = PS::S;
  constexpr int T = panel_threads<MAXM, FEW>();
  const int sh = blockIdx.x;
  const int tid = threadIdx.x;
  const int n = a.n, m = a.m, p = a.p, ldz = p + n;
  const int r = p + k - nbe;       // rows of [Ct; M] above the block
  const int j0 = k - m - nbe;      // first fresh column
  const cd sigma = a.shifts[sh];
  float4* Z2f = a.Z2 + (size_t)sh * a.z2_stride;
  const double sing_tol = (double)n * 7.105427357601002e-15 * sqrt(shifted_norm2(a.hnorm, n, sigma));
  float4* coef4 = sm.p.W;
  float2* ct = &sm.p.F[0][0];   // kCtRows x (kNBT + 1), after the panel
  static_assert(sizeof(sm.p.F) >= sizeof(float2) * kCtRows * (kNBT + 1), "staged Ct rows");
  if (tid == 0) sm.sing = 0;
  for (int e = tid; e < nbe * m; e += T) {
    const int row = e % nbe, q = e / nbe;
    coef4[row * S + q] = Z2f[BCK((r + row) + (size_t)q * ldz, a.z2_stride)];
  }
  pan::DF32::H hm{a.Hhi, a.Hlo, n, {}};
#ifdef SSV_BOUNDS_CHECK
  hm.bound.count = (size_t)n * n;
  hm.bound.err = a.err;
#endif
  pan::run<pan::DF32, MAXM, kNBT, T, false>(hm, k - nbe, j0, sigma, nbe, m, sm.p,
                                            (pan::SmemR<pan::DF32, MAXM, kNBT>*)nullptr, sing_tol, &sm.sing);
  // coef rows c < nbe hold P1(c, :), rows kNBT + qq hold P2(qq, :) (slots 0..m-1)

  // ---- P1 as BF16 digit tiles: column exponents first (one warp per complex column)
  const int warp = tid >> 5, lane = tid & 31;
  for (int q = warp; q < m; q += T / 32) {
    float mr = 0.f, mi = 0.f;
    bool br = false, bi = false;
    for (int c = lane; c < nbe; c += 32) {
      const float4 w = coef4[c * S + q];
      mr = fmaxf(mr, fabsf(w.x));
      mi = fmaxf(mi, fabsf(w.z));
      br = br || !(fabsf(w.x) <= 3.4e38f);
      bi = bi || !(fabsf(w.z) <= 3.4e38f);
    }
    const int er = __reduce_max_sync(0xffffffffu, br ? kBadExp : scale_exp_f(mr));
    const int ei = __reduce_max_sync(0xffffffffu, bi ? kBadExp : scale_exp_f(mi));
    if (lane < 2) {
      const int E = col_exp(lane ? ei : er);
      sm.fexp[2 * q + lane] = E;
      a.pexp[BCK((size_t)sh * 2 * kMaxM + 2 * q + lane, (size_t)a.s * 2 * kMaxM)] = E;
    }
  }
  __syncthreads();
  {
    // item = (real column cr, 8 consecutive K rows): seven uint4 stores
    const int g = sh / a.S, slot_row = (sh % a.S) * a.cs;
    const size_t Pg0 = (size_t)g * kSD * kStages * kBT;
    for (int it = tid; it < 2 * m * (kNBT / 8); it += T) {
      const int cr = it / (kNBT / 8), c8 = (it % (kNBT / 8)) * 8;
      const int q = cr >> 1;
      float hi[8], lo[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int c = c8 + e;
        hi[e] = lo[e] = 0.f;
        if (c < nbe) {
          const float4 w = coef4[c * S + q];
          hi[e] = (cr & 1) ? w.z : w.x;
          lo[e] = (cr & 1) ? w.w : w.y;
        }
      }
      uint4 dg[7];
      digits7_oct(hi, lo, digit_scale(sm.fexp[cr]), dg);
      const int J = c8 / kKS;
      const int off = tile_off(slot_row + cr, c8 % kKS);
#pragma unroll
      for (int l = 0; l < kSD; ++l)
        *reinterpret_cast<uint4*>(a.Pd + BCK(Pg0 + ((size_t)l * kStages + J) * kBT + off, a.n_pd)) = dg[l];
    }
  }
  // ---- P2 and the sigma rows for the update's epilogue
  {
    float4* pc = a.pc + (size_t)sh * 2 * kMaxM * kMaxM;
    const int nsig = min(m, nbe);
    for (int e = tid; e < 2 * m * m; e += T) {
      const int row = e / m, q = e % m;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (row < m) v = coef4[(kNBT + row) * S + q];
      else if (row - m < nsig) v = coef4[(row - m) * S + q];
      pc[e] = v;
    }
  }
  // ---- Z2 P2 on the tensor cores: P2's real form (cs x cs, entry (K = 2qq + ri,
  //      N = 2q + ro) from P2(qq, q): Re for ri = ro, -Im for (1, 0), Im for
  //      (0, 1)) as seven-digit tiles, column-scaled
  if (a.tcz) {
    const int cs = a.cs, kg = cs / 8;
    for (int c = tid; c < cs; c += T) {
      const int q = c >> 1;
      float mx = 0.f;
      if (q < m) {
        for (int qq = 0; qq < m; ++qq) {
          const float4 w = coef4[(kNBT + qq) * S + q];
          mx = fmaxf(mx, fmaxf(fabsf(w.x), fabsf(w.z)));
          if (!(fabsf(w.x) <= 3.4e38f) || !(fabsf(w.z) <= 3.4e38f)) mx = __int_as_float(0x7f800000);
        }
      }
      const int E = col_exp(scale_exp_f(mx));
      sm.f2exp[c] = E;
      a.p2exp[BCK((size_t)sh * 2 * kMaxM + c, (size_t)a.s * 2 * kMaxM)] = E;
    }
    __syncthreads();
    const size_t T0 = (size_t)sh * 7 * cs * cs;
    for (int it = tid; it < cs * (cs / 8); it += T) {
      const int c = it / (cs / 8), k8 = (it % (cs / 8)) * 8;
      const int q = c >> 1, ro = c & 1, E = sm.f2exp[c];
      float hi[8], lo[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int kk = k8 + e, qq = kk >> 1, ri = kk & 1;
        hi[e] = lo[e] = 0.f;
        if (q < m && qq < m) {
          const float4 w = coef4[(kNBT + qq) * S + q];
          if (ri == ro) { hi[e] = w.x; lo[e] = w.y; }
          else if (ri == 1) { hi[e] = -w.z; lo[e] = -w.w; }
          else { hi[e] = w.z; lo[e] = w.w; }
        }
      }
      const int off = tile_off_kg(c, k8, kg);
      uint4 dg[7];
      digits7_oct(hi, lo, digit_scale(E), dg);
#pragma unroll
      for (int l = 0; l < 7; ++l)
        *reinterpret_cast<uint4*>(a.P2d + BCK(T0 + (size_t)l * cs * cs + off, a.n_p2d)) = dg[l];
    }
  }
  // ---- X-hat mode: P1 rows into ZT, P2 parked in this shift's output rows
  //      n - step m .. n - (step - 1) m - 1 (read back before the back pass
  //      writes them, since every later block is at least m rows high)
  if (a.mode == SSV_XHAT) {
    cd* ZT = a.ZT + (size_t)sh * (size_t)n * m;
    for (int idx = tid; idx < nbe * m; idx += T) {
      const int c = idx % nbe, q = idx / nbe;
      ZT[BCK((j0 + c) + (size_t)q * n, (size_t)n * m)] = df_join(coef4[c * S + q]);
    }
    cd* tout = a.out + (size_t)sh * m * a.ldo;
    for (int idx = tid; idx < m * m; idx += T) {
      const int qq = idx % m, q = idx / m;
      tout[BCK(n - step * m + qq, n) + (size_t)q * a.ldo] = df_join(coef4[(kNBT + qq) * S + q]);
    }
  }
  // ---- the p rows of Ct: Z2(i, :) = Ct(i, fresh) P1 + Z2(i, :) P2, double-float,
  //      in chunks of whole rows (each entry reads its row's old values); the
  //      chunk of Ct is staged once, ks neighbouring lanes share the sum of one
  //      entry
  const int rows_per_chunk = min(kCtRows, max(1, T / m));
  for (int i0 = 0; i0 < p; i0 += rows_per_chunk) {
    const int ic = min(rows_per_chunk, p - i0);
    for (int e = tid; e < ic * nbe; e += T) {
      const int i = e % ic, c = e / ic;
      const double z = a.Ct[(i0 + i) + (size_t)(j0 + c) * a.ldct];
      const float zh = (float)z;
      ct[i * (kNBT + 1) + c] = make_float2(zh, (float)(z - (double)zh));
    }
    __syncthreads();
    int ks = 1;
    while (ks < 32 && 2 * ks * ic * m <= T) ks <<= 1;
    const int e = tid / ks, sub = tid % ks;
    const bool act = e < ic * m;
    const int i = act ? e / m : 0, q = act ? e % m : 0;
    float rh = 0.f, rl = 0.f, ih = 0.f, il = 0.f;
    if (act) {
#pragma unroll 4
      for (int c = sub; c < nbe; c += ks) {
        const float2 z = ct[i * (kNBT + 1) + c];
        const float4 w = coef4[c * S + q];
        df_mac(rh, rl, z.x, z.y, w.x, w.y);
        df_mac(ih, il, z.x, z.y, w.z, w.w);
      }
      for (int qq = sub; qq < m; qq += ks) {
        const float4 zz = Z2f[BCK((i0 + i) + (size_t)qq * ldz, a.z2_stride)];
        const float4 w = coef4[(kNBT + qq) * S + q];
        df_mac(rh, rl, zz.x, zz.y, w.x, w.y);
        df_mac(rh, rl, -zz.z, -zz.w, w.z, w.w);
        df_mac(ih, il, zz.x, zz.y, w.z, w.w);
        df_mac(ih, il, zz.z, zz.w, w.x, w.y);
      }
    }
    for (int o = ks >> 1; o > 0; o >>= 1) {
      const dw x = dw_add(dw{rh, rl}, dw{__shfl_xor_sync(0xffffffffu, rh, o), __shfl_xor_sync(0xffffffffu, rl, o)});
      const dw y = dw_add(dw{ih, il}, dw{__shfl_xor_sync(0xffffffffu, ih, o), __shfl_xor_sync(0xffffffffu, il, o)});
      rh = x.hi; rl = x.lo; ih = y.hi; il = y.lo;
    }
    __syncthreads();  // every old entry of these rows is read before any is written
    if (act && sub == 0) {
      const float sr = rh + rl, si = ih + il;
      Z2f[BCK((i0 + i) + (size_t)q * ldz, a.z2_stride)] = make_float4(sr, rl - (sr - rh), si, il - (si - ih));
    }
  }
  if (tid == 0 && sm.sing) a.flags[sh] = 1;
}

// ---- update of the H rows above the block: Z2 <- Z1 P1 + Z2 P2 - sigma E P1 --
// a += b for double-float a and FP32 b (two-sum)
static __device__ __forceinline__ void add_f(float& hi, float& lo, float b) {
  const float s = hi + b;
  const float bp = s - hi;
  lo += (hi - (s - bp)) + (b - bp);
  hi = s;
}
// 2^e as FP32 for e in [-126, 127]
static __device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }
// exponents whose pairwise sums, less the levels' 2^-63, stay in FP32's normal
// range: rows and columns outside take the ldexpf path
constexpr int kFastExp = 30;
static __device__ __forceinline__ bool fast_exp(int e) { return e >= -kFastExp && e <= kFastExp; }

constexpr int kUH = 16;              // columns of an epilogue thread
constexpr int kUG = kUM * kUN / kUH;  // threads of an epilogue group
constexpr int kUT = 2 * kUG + 64;    // update threads: two epilogue groups, the producer's and the issuer's warp

// a bounded wait of one role: gives up at the poll limit or when another role
// has (the block then leaves together)
static __device__ __forceinline__ bool role_wait(uint32_t mbar, uint32_t parity, volatile int* fail) {
  for (long long it = 0; it < kUpdWait / 64; ++it) {
    if (mbar_wait(mbar, parity, 64)) return true;
    if (*fail) return false;
  }
  *fail = 1;
  return false;
}

// Item -> row block I of RT and group g of G.  All groups per row block, so that
// the blocks running together share H's digit tiles; but where the groups' P1
// digits (57 KB each) do not stay in L2, only as many groups at a time as blocks
// run: theirs then stay while the rows go by.  2000 groups of 32 columns at n =
// 5000: 93.3 ms in all one row block at a time, 87.8 in chunks (before each product
// had a window of its own); 250 groups at n =
// 1000: a call of 7.97 ms one row block at a time, 8.25 in chunks.
constexpr size_t kPGroupBytes = (size_t)kSD * kStages * kBT * 2;
constexpr size_t kPKeep = (size_t)64 << 20;
static __device__ __forceinline__ void item_of(long long item, int RT, int G, int& I, int& g) {
  const int gb = (size_t)G * kPGroupBytes > kPKeep ? (int)gridDim.x : G;
  const int q = (int)(item / ((long long)RT * gb));
  const int rem = (int)(item - (long long)q * RT * gb), w = min(gb, G - q * gb);
  I = rem / w;
  g = q * gb + rem % w;
}

// The update of block step (k, nbe) for shifts of CS real columns (2m rounded
// up to a power of two).  An item is 128 rows of H x one group of S = 32 / CS
// shifts; a persistent block works on two at a time, in roles that only meet at
// mbarriers:
//   * a producer thread copies the K stages of Z1 P1 (H digit tiles x P1 digit
//     tiles) into two stage buffers and, CS >= 16, the group's Z2 and P2 digit
//     tiles into a third;
//   * an issuing thread multiplies: Z1 P1 into the eight levels of the first TMEM
//     window, Z2 P2 into the seven of the second, so that each window is read
//     under the other's products (CS < 16: item v's Z1 P1 into window v mod 2);
//   * two groups of eight warps take alternate items (thread = row, 16 columns):
//     levels into double-float sums, scaling, the shifted-diagonal correction,
//     and the new rows: as FP32 pairs the 128 that the next panel (or the final
//     block) reads, all others as the digit tiles of the next block step (CS <
//     16: Z2 P2 in double-float here, and every row as pairs).
//
// What bounds it, per item at CS = 32: the products with their shared-memory
// traffic (about 10 k clocks), the epilogue's instructions (8.4 k issue slots a
// scheduler) and the copies from L2 (392 KB, 6.5 k clocks), which run side by side;
// DRAM 28 % busy.  Measured steps, the sweep of 2000 shifts at n = 5000, m = 16 (39
// launches) and of 600 at n = 2500, m = 8 (20): one item at a time, each phase after
// the other 114 ms; roles, and the two products of an item in one window, which the
// issuer waited 5 k of 18 k clocks an item to have read 93 and 4.7; sixteen epilogue
// warps (eight left a scheduler idle for 58 % of the clocks) and the order of items
// 87.8 and 4.29; a window for each product 79.5 and 3.55.
template <int CS>
__global__ void __launch_bounds__(kUT, 1) tcs_update_kernel(TcsArgs a, int k, int nbe) {
  constexpr bool TCZ = CS >= 16;
  constexpr int S = kUN / CS;             // shifts of a group
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) unsigned long long mbar[22];
  __shared__ uint32_t tslot;
  __shared__ volatile int fail;
  // stages copied / multiplied, Z2 tiles copied / multiplied (read when a wait gave up)
  __shared__ int issued[4];
  __shared__ unsigned char rowmax[2][2][kUM];  // CS = 32: FP32 exponent fields of the halves of a row
  const int n = a.n, m = a.m, p = a.p, ldz = p + n;
  const int hrows = k - nbe;              // H rows above the block
  const int j0 = k - m - nbe;             // first fresh column (a multiple of 32)
  const int nsig = min(m, nbe);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int G = a.ngroups;
  // an earlier launch of this solve gave up a wait: its results are void, skip
  // (the flag is read by every thread and combined, so the whole block agrees)
  if (__syncthreads_or(*(volatile int*)a.err != 0)) return;
  const int RT = (hrows + kUM - 1) / kUM;
  const long long items = (long long)RT * G;
  const int nst = (nbe + kKS - 1) / kKS;
  const int JH0 = j0 / kKS;
  // full / empty[2]: a stage buffer copied / multiplied; zfull / zempty: the Z2
  // buffer; pfull / pread[2]: the Z1 P1 levels of group h's item complete / read;
  // qfull / qread[2]: its Z2 P2 levels
  const uint32_t full = smem_addr(mbar), empty = full + 16, zfull = full + 32, zempty = full + 40;
  const uint32_t pfull = full + 48, pread = full + 64, qfull = full + 80, qread = full + 96;
  const uint32_t sBase = smem_addr(smem), sZ = sBase + (uint32_t)kOffZ;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tslot)),
                 "r"(2 * kWinCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    // pread and qread: one arrival per warp of the group; from 14 on: the warp
    // pairs that share rows
    for (int q = 0; q < 22; ++q)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(full + 8u * q),
                   "r"(q >= 14 ? 2 : q == 8 || q == 9 || q >= 12 ? kUG / 32 : 1));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fail = 0;
    for (int q = 0; q < 4; ++q) issued[q] = 0;
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tslot;
  // Z2 / P2 digit bytes of one shift
  constexpr uint32_t zbytes = 7u * 128u * (uint32_t)CS * 2u;
  constexpr uint32_t pbytes = 7u * (uint32_t)(CS * CS) * 2u;
  constexpr int kgz = CS >= 8 ? CS / 8 : 1;
  const long long mine = blockIdx.x < items ? (items - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;

  if (warp == 2 * kUG / 32) {
    if (lane == 0) {
      // ---- producer
      unsigned i = 0;
      bool ok = true;
      auto stages = [&](long long v, int s0, int s1) {
        const long long item = blockIdx.x + v * gridDim.x;
        int I, g;
        item_of(item, RT, G, I, g);
        const size_t Pg0 = (size_t)g * kSD * kStages * kBT;
        for (int st = s0; st < s1 && ok; ++st, ++i) {
          const uint32_t b = i & 1u;
          if (!role_wait(empty + 8u * b, ((i >> 1) & 1u) ^ 1u, &fail)) {
            ok = false;
            return;
          }
          const uint32_t dst = sBase + b * kStageBytes, lb = full + 8u * b;
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(lb), "r"(kStageBytes)
                       : "memory");
          for (int l = 0; l < kSDH; ++l)
            bulk_copy(dst + (uint32_t)(l * kAT * 2),
                      a.Hs + BCK(((size_t)(l * a.RB + I) * a.KT + (JH0 + st)) * (kAT / 8), a.n_hs),
                      (uint32_t)(kAT * 2), lb);
          for (int l = 0; l < kSD; ++l)
            bulk_copy(dst + (uint32_t)(kSDH * kAT * 2 + l * kBT * 2),
                      a.Pd + BCK(Pg0 + ((size_t)l * kStages + st) * kBT, a.n_pd), (uint32_t)(kBT * 2), lb);
          issued[0] = (int)(i + 1);
        }
      };
      auto ztiles = [&](long long v) {
        const long long item = blockIdx.x + v * gridDim.x;
        int I, g;
        item_of(item, RT, G, I, g);
        if (!role_wait(zempty, ((unsigned)v & 1u) ^ 1u, &fail)) {
          ok = false;
          return;
        }
        const int nsh = min(S, a.s - g * S);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(zfull),
                     "r"((uint32_t)nsh * (zbytes + pbytes))
                     : "memory");
        for (int l = 0; l < nsh; ++l) {
          const int sh = g * S + l;
          bulk_copy(sZ + (uint32_t)l * zbytes, a.Zd + BCK(((size_t)sh * a.RB + I) * 7 * (128 * CS), a.n_zd), zbytes,
                    zfull);
          bulk_copy(sZ + (uint32_t)S * zbytes + (uint32_t)l * pbytes, a.P2d + BCK((size_t)sh * 7 * CS * CS, a.n_p2d),
                    pbytes, zfull);
        }
        issued[2] = (int)(v + 1);
      };
      // both stage buffers first: they fill under the last item's Z2 P2
      const int first = min(2, nst);
      for (long long v = 0; v < mine && ok; ++v) {
        stages(v, 0, first);
        if (TCZ && ok) ztiles(v);
        stages(v, first, nst);
      }
    }
  } else if (warp == 2 * kUG / 32 + 1) {
    if (lane == 0) {
      // ---- issuer
      unsigned i = 0;
      bool ok = true;
      // the group of item v has read its window
      auto read_of = [&](uint32_t bars, long long v) {
        return role_wait(bars + 8u * ((unsigned)v & 1u), (unsigned)(v >> 1) & 1u, &fail);
      };
      // fused levels: the P1 digit tiles sit side by side (kUN rows each), so one
      // product of H digit kd against P1 digits 0 .. c - 1 (N = kUN c) lands digit
      // b in level kd + b.  The first products of an item open the levels: those
      // of kd = 0 levels 0 .. 6, digit 6 of kd = 1 level 7.
      auto z1p1 = [&](long long v) {
        const uint32_t h = (unsigned)v & 1u, u = (unsigned)(v >> 1);
        const uint32_t d = tmem + (TCZ ? 0u : h * (uint32_t)kWinCols);
        if (TCZ ? v > 0 && !read_of(pread, v - 1) : !role_wait(pread + 8u * h, (u & 1u) ^ 1u, &fail)) ok = false;
        for (int st = 0; st < nst && ok; ++st, ++i) {
          const uint32_t b = i & 1u;
          if (!role_wait(full + 8u * b, (i >> 1) & 1u, &fail)) {
            ok = false;
            return;
          }
          fence_after();
          const uint32_t aBase = sBase + b * kStageBytes;
          const uint32_t bBase = aBase + (uint32_t)(kSDH * kAT * 2);
          constexpr uint32_t kSbo = (uint32_t)kKG * 128u;
#pragma unroll
          for (int ks = 0; ks < kKS / 16; ++ks) {
            const bool first = st == 0 && ks == 0;
#pragma unroll
            for (int kd = 0; kd < kSDH; ++kd) {
              const uint64_t ad = mat_desc(aBase + (uint32_t)(kd * kAT * 2 + ks * 256), 128u, kSbo);
              const uint64_t bd = mat_desc(bBase + (uint32_t)(ks * 256), 128u, kSbo);
              constexpr int kOpen = kSD - 1;  // the digit of kd = 1 that opens the last level
              if (kd == 1 && first) {
                mma_bf16(d + (uint32_t)kUN, ad, bd, idesc_bf16(kUM, kUN * kOpen), 1u);
                const uint64_t b6 = mat_desc(bBase + (uint32_t)(kOpen * kBT * 2 + ks * 256), 128u, kSbo);
                mma_bf16(d + (uint32_t)((kOpen + 1) * kUN), ad, b6, idesc_bf16(kUM, kUN), 0u);
              } else {
                const int c = kd == 0 ? kSD : kLev - kd;
                mma_bf16(d + (uint32_t)(kd * kUN), ad, bd, idesc_bf16(kUM, kUN * c), (first && kd == 0) ? 0u : 1u);
              }
            }
          }
          mma_commit(empty + 8u * b);
          issued[1] = (int)(i + 1);
        }
        if (ok) mma_commit(pfull + 8u * h);
      };
      // shift l's seven levels sit side by side (columns 7 CS l + CS lv) and its
      // P2 digit tiles (CS rows each) are stacked: one product of Z2 digit kd
      // against P2 digits 0 .. 6 - kd lands digit ld in level kd + ld
      auto z2p2 = [&](long long v) {
        const uint32_t h = (unsigned)v & 1u;
        const uint32_t d = tmem + (uint32_t)kWinCols;
        int I, g;
        item_of(blockIdx.x + v * gridDim.x, RT, G, I, g);
        const int nsh = min(S, a.s - g * S);
        if ((v > 0 && !read_of(qread, v - 1)) || !role_wait(zfull, (unsigned)v & 1u, &fail)) {
          ok = false;
          return;
        }
        fence_after();
        constexpr uint32_t sboz = (uint32_t)kgz * 128u;
        for (int l = 0; l < nsh; ++l) {
          const uint32_t zb = sZ + (uint32_t)l * zbytes;
          const uint32_t pb = sZ + (uint32_t)S * zbytes + (uint32_t)l * pbytes;
#pragma unroll
          for (int ks = 0; ks < CS / 16; ++ks) {
#pragma unroll
            for (int kd = 0; kd < 7; ++kd) {
              const uint64_t ad = mat_desc(zb + (uint32_t)(kd * 128 * CS * 2 + ks * 256), 128u, sboz);
              const uint64_t bd = mat_desc(pb + (uint32_t)(ks * 256), 128u, sboz);
              mma_bf16(d + (uint32_t)(7 * CS * l + kd * CS), ad, bd, idesc_bf16(kUM, CS * (7 - kd)),
                       (kd == 0 && ks == 0) ? 0u : 1u);
            }
          }
        }
        mma_commit(zempty);
        mma_commit(qfull + 8u * h);
        issued[3] = (int)(v + 1);
      };
      for (long long v = 0; v < mine && ok; ++v) {
        z1p1(v);
        if (TCZ && ok) z2p2(v);
      }
    }
  } else {
    // ---- epilogue: group h takes items v = h, h + 2, ..; thread = (row, half of
    // the columns): eight warps to a scheduler's two hide each other's latency
    const uint32_t h = (uint32_t)(warp / (kUG / 32));
    const int hf = (warp >> 2) & 1, cb = kUH * hf;  // its first column
    const int row = tid & (kUM - 1);
    const uint32_t tl = tmem + (TCZ ? 0u : h * (uint32_t)kWinCols) + ((uint32_t)((warp & 3) * 32) << 16);
    // shifts of this half: lb .. lb + SH - 1 of the group
    constexpr int SH = CS >= kUH ? 1 : kUH / CS, CL = CS < kUH ? CS : kUH;  // CL: columns of a shift here
    const int lb = cb / CS, cz = cb % CS;  // cz: the first one's first column within its shift
    auto arrive = [&](uint32_t b) {
      fence_before();
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(b) : "memory");
    };
    [[maybe_unused]] int xn = 0;  // exchanges of row maxima so far
    for (long long v = h; v < mine; v += 2) {
      const uint32_t par = (unsigned)(v >> 1) & 1u;
      const long long item = blockIdx.x + v * gridDim.x;
      int I, g;
      item_of(item, RT, G, I, g);
      const int ih = I * kUM + row;
      const bool live = ih < hrows;
      // exponents: of the row, of this lane's column (P1's, P2's), of the row's Z2
      const int Ei = live ? a.hexp[BCK(ih, a.npad)] : 0;
      int E1 = 0, E2 = 0;
      {
        const int cg = cb + (lane & (kUH - 1)), sh = g * S + cg / CS, c = cg % CS;
        if (sh < a.s && c < 2 * m) {
          E1 = a.pexp[(size_t)sh * 2 * kMaxM + c];
          if (TCZ) E2 = a.p2exp[(size_t)sh * 2 * kMaxM + c];
        }
      }
      int ez = 0;
      if constexpr (TCZ)
        if (live && g * S + lb < a.s) ez = a.zexp[BCK((size_t)(g * S + lb) * a.npad + ih, (size_t)a.s * a.npad)];
      // the row exponents of a warp and the column exponents: one path per warp
      const bool fast =
          __all_sync(0xffffffffu, fast_exp(Ei) && fast_exp(ez) && fast_exp(E1) && fast_exp(E2));
      if (!__all_sync(0xffffffffu, role_wait(pfull + 8u * h, par, &fail))) break;
      fence_after();
      // the new entries, 16 real columns of the row (Re, Im interleaved), as pairs
      float ah[kUH], al[kUH];
#pragma unroll
      for (int c = 0; c < kUH; ++c) { ah[c] = 0.f; al[c] = 0.f; }
      {
        float sc = 0.0078125f * 0.0078125f;  // 2^{-7 (t + 2)}, t = 0
#pragma unroll 1
        for (int lv = 0; lv < kLev; ++lv) {
          uint32_t rr[kUH];
          tmem_ld16(tl + (uint32_t)(lv * kUN + cb), rr);
#pragma unroll
          for (int c = 0; c < kUH; ++c) add_f(ah[c], al[c], __uint_as_float(rr[c]) * sc);
          sc *= 0.0078125f;
        }
      }
      arrive(pread + 8u * h);
#pragma unroll
      for (int c = 0; c < kUH; ++c) {
        const int Ec = __shfl_sync(0xffffffffu, E1, c);
        if (fast) {
          const float f = pow2f(Ei + Ec);
          ah[c] *= f;
          al[c] *= f;
        } else if (Ei == kBadExp || Ec == kBadExp) {
          ah[c] = __int_as_float(0x7fc00000);
          al[c] = 0.f;
        } else {
          ah[c] = ldexpf(ah[c], Ei + Ec);
          al[c] = ldexpf(al[c], Ei + Ec);
        }
      }
      if constexpr (TCZ) {
        if (!__all_sync(0xffffffffu, role_wait(qfull + 8u * h, par, &fail))) break;
        fence_after();
        // shift l's levels start at column 7 CS l
        const uint32_t tz = tl + (uint32_t)(kWinCols + 7 * CS * lb + cz);
        if (fast) {
          float f[kUH];
#pragma unroll
          for (int c = 0; c < kUH; ++c) f[c] = pow2f(ez + __shfl_sync(0xffffffffu, E2, c) - 14);
#pragma unroll 1
          for (int lv = 0; lv < 7; ++lv) {
            uint32_t rr[kUH];
            tmem_ld16(tz + (uint32_t)(lv * CS), rr);
#pragma unroll
            for (int c = 0; c < kUH; ++c) {
              add_f(ah[c], al[c], __uint_as_float(rr[c]) * f[c]);
              f[c] *= 0.0078125f;
            }
          }
        } else {
          float bh[kUH], bl[kUH];
#pragma unroll
          for (int c = 0; c < kUH; ++c) { bh[c] = 0.f; bl[c] = 0.f; }
          float sc = 0.0078125f * 0.0078125f;
#pragma unroll 1
          for (int lv = 0; lv < 7; ++lv) {
            uint32_t rr[kUH];
            tmem_ld16(tz + (uint32_t)(lv * CS), rr);
#pragma unroll
            for (int c = 0; c < kUH; ++c) add_f(bh[c], bl[c], __uint_as_float(rr[c]) * sc);
            sc *= 0.0078125f;
          }
#pragma unroll
          for (int c = 0; c < kUH; ++c) {
            const int Ec = __shfl_sync(0xffffffffu, E2, c);
            if (ez == kBadExp || Ec == kBadExp) {
              ah[c] = __int_as_float(0x7fc00000);
              al[c] = 0.f;
            } else {
              add_f(ah[c], al[c], ldexpf(bh[c], ez + Ec));
              al[c] += ldexpf(bl[c], ez + Ec);
            }
          }
        }
        arrive(qread + 8u * h);
      } else if (live) {
        // several shifts (m <= 4): + Z2(row, :) P2(:, q) in double-float from the
        // old row of each shift
        constexpr int CC = CS / 2;  // complex columns of a shift
#pragma unroll
        for (int l = 0; l < SH; ++l) {
          if (g * S + lb + l < a.s) {
            const float4* z = a.Z2 + BCK((size_t)(g * S + lb + l) * a.z2_stride + (p + ih), a.n_z2);
            const float4* pc = a.pc + BCK((size_t)(g * S + lb + l) * 2 * kMaxM * kMaxM, a.n_pc);
            float4 zz[CC];
#pragma unroll
            for (int qq = 0; qq < CC; ++qq) zz[qq] = qq < m ? z[(size_t)qq * ldz] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int q = 0; q < CC; ++q) {
              if (q >= m) continue;
              const int c = l * CS + 2 * q;
#pragma unroll
              for (int qq = 0; qq < CC; ++qq) {
                if (qq >= m) continue;
                const float4 w = pc[qq * m + q];
                df_mac(ah[c], al[c], zz[qq].x, zz[qq].y, w.x, w.y);
                df_mac(ah[c], al[c], -zz[qq].z, -zz[qq].w, w.z, w.w);
                df_mac(ah[c + 1], al[c + 1], zz[qq].x, zz[qq].y, w.z, w.w);
                df_mac(ah[c + 1], al[c + 1], zz[qq].z, zz[qq].w, w.x, w.y);
              }
            }
          }
        }
      }
      const int cdr = ih - j0;  // shifted-diagonal correction row of fresh column cdr
      if (live && cdr >= 0 && cdr < nsig) {
        // - sigma P1(cdr, q)
#pragma unroll
        for (int c = 0; c < kUH; c += 2) {
          const int l = lb + c / CL, q = (cz + c % CL) >> 1, sh = g * S + l;
          if (q >= m || sh >= a.s) continue;
          const float4 sgf = df_split(a.shifts[sh]);
          const float4 w = a.pc[BCK((size_t)sh * 2 * kMaxM * kMaxM + m * m + cdr * m + q, a.n_pc)];
          df_mac(ah[c], al[c], -sgf.x, -sgf.y, w.x, w.y);
          df_mac(ah[c], al[c], sgf.z, sgf.w, w.z, w.w);
          df_mac(ah[c + 1], al[c + 1], -sgf.x, -sgf.y, w.z, w.w);
          df_mac(ah[c + 1], al[c + 1], -sgf.z, -sgf.w, w.x, w.y);
        }
      }
      // normalised pairs
#pragma unroll
      for (int c = 0; c < kUH; ++c) {
        const float s = ah[c] + al[c];
        al[c] = al[c] - (s - ah[c]);
        ah[c] = s;
      }
      // as pairs: the rows of the next panel or the final block
      if (live && (!TCZ || ih >= hrows - kNBT)) {
#pragma unroll
        for (int c = 0; c < kUH; c += 2) {
          const int l = lb + c / CL, q = (cz + c % CL) >> 1;
          if (q >= m || g * S + l >= a.s) continue;
          a.Z2[BCK((size_t)(g * S + l) * a.z2_stride + (p + ih) + (size_t)q * ldz, a.n_z2)] =
              make_float4(ah[c], al[c], ah[c + 1], al[c + 1]);
        }
      }
      // as digits: the rows above them (none of a tile that lies within the last 128 rows)
      if constexpr (TCZ) {
        if (I * kUM < hrows - kNBT) {
          const int sh = g * S + lb;
          // the row's digit exponent: the maximum over the shift's 2m entries, by
          // FP32 exponent field (255: not finite)
          int fe = 0;
#pragma unroll
          for (int c = 0; c < kUH; ++c) {
            if (cz + c >= 2 * m) { ah[c] = 0.f; al[c] = 0.f; }
            fe = max(fe, __float_as_int(ah[c]) & 0x7fffffff);
          }
          fe >>= 23;
          if constexpr (CS > kUH) {
            // the other half of the row is in the warp with the same rows: written
            // in even phases of the pair's barrier, read in odd ones
            const uint32_t xb = full + 8u * (14u + h * 4u + (uint32_t)(warp & 3));
            if (xn > 0 && !__all_sync(0xffffffffu, role_wait(xb, 1u, &fail))) break;
            rowmax[h][hf][row] = (unsigned char)fe;
            arrive(xb);
            if (!__all_sync(0xffffffffu, role_wait(xb, 0u, &fail))) break;
            fe = max(fe, (int)rowmax[h][hf ^ 1][row]);
            arrive(xb);
            ++xn;
          }
          if (live && sh < a.s) {
            const int E = col_exp(scale_exp_f(__int_as_float(fe << 23)));
            if (cz == 0) a.zexp[BCK((size_t)sh * a.npad + ih, (size_t)a.s * a.npad)] = E;
            const float inv = digit_scale(E);
            const size_t T0 = ((size_t)sh * a.RB + I) * 7 * (128 * CS);
#pragma unroll
            for (int k8 = 0; k8 < kUH; k8 += 8) {
              float hi[8], lo[8];
#pragma unroll
              for (int e = 0; e < 8; ++e) { hi[e] = ah[k8 + e]; lo[e] = al[k8 + e]; }
              uint4 dg[7];
              digits7_oct(hi, lo, inv, dg);
              const int off = tile_off_kg(row, cz + k8, kgz);
#pragma unroll
              for (int l2 = 0; l2 < 7; ++l2)
                *reinterpret_cast<uint4*>(a.Zd + BCK(T0 + (size_t)l2 * (128 * CS) + off, a.n_zd)) = dg[l2];
            }
          }
        }
      }
    }
  }
  __syncwarp();
  __syncthreads();
  if (fail != 0 && tid == 0) {
    // a completion never arrived: record it and give the copies and products in
    // flight one more bounded wait
    atomicExch(a.err, 1);
    const unsigned nl = (unsigned)issued[0], nm = (unsigned)issued[1];
    for (unsigned i = nl > 2 ? nl - 2 : 0; i < nl; ++i) mbar_wait(full + 8u * (i & 1u), (i >> 1) & 1u, kUpdWait);
    for (unsigned i = nm > 2 ? nm - 2 : 0; i < nm; ++i) mbar_wait(empty + 8u * (i & 1u), (i >> 1) & 1u, kUpdWait);
    if (issued[2] > 0) mbar_wait(zfull, (unsigned)(issued[2] - 1) & 1u, kUpdWait);
    if (issued[3] > 0) mbar_wait(zempty, (unsigned)(issued[3] - 1) & 1u, kUpdWait);
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * kWinCols));
}

#ifdef SSV_BOUNDS_CHECK
// bit 2 of the error word when a byte of the canary after the scratch changed
__global__ void tcs_canary_kernel(const unsigned char* c, size_t nbytes, int* err) {
  for (size_t i = threadIdx.x; i < nbytes; i += blockDim.x)
    if (c[i] != 0xA5) atomicOr(err, 4);
}
#endif

// ---- final m x m block, G or the X-hat back pass ----------------------------
__global__ void __launch_bounds__(kPT) tcs_final_kernel(TcsArgs a, int nsteps) {
  __shared__ cd Wm[kMaxM * 2 * kMaxM];
  __shared__ cd lmul[kMaxM];
  __shared__ cd Yb[kMaxM * kMaxM];
  __shared__ cd zs[kMaxM * kMaxM], p2s[kMaxM * kMaxM], zn[kMaxM * kMaxM];
  __shared__ int s_piv, s_sing;
  const int sh = blockIdx.x, tid = threadIdx.x;
  const int n = a.n, m = a.m, p = a.p, ldz = p + n;
  const cd sigma = a.shifts[sh];
  const double sing_tol = (double)n * 7.105427357601002e-15 * sqrt(shifted_norm2(a.hnorm, n, sigma));
  const float4* Z2f = a.Z2 + (size_t)sh * a.z2_stride;
  const bool failed = *a.err != 0;
  if (tid == 0) s_sing = a.flags[sh];
  for (int idx = tid; idx < m * 2 * m; idx += kPT) {
    const int i = idx % m, j = idx / m;
    cd v;
    if (j < m) v = df_join(Z2f[BCK((p + i) + (size_t)j * ldz, a.z2_stride)]);
    else v = mkcd(i <= j - m ? a.R[i + (size_t)(j - m) * n] : 0.0, 0.0);
    Wm[i + j * kMaxM] = v;
  }
  __syncthreads();
  // Gauss-Jordan with partial pivoting on [Wm | R(0:m, 0:m)]
  for (int kk = 0; kk < m; ++kk) {
    if (tid < 32) {
      double best = -1.0;
      int brow = kk;
      for (int i = kk + tid; i < m; i += 32) {
        const double v = cabs1(Wm[i + kk * kMaxM]);
        if (v > best) { best = v; brow = i; }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const double ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int orow = __shfl_xor_sync(0xffffffffu, brow, o);
        if (ob > best || (ob == best && orow < brow)) { best = ob; brow = orow; }
      }
      if (tid == 0) {
        s_piv = brow;
        const cd pv = Wm[brow + kk * kMaxM];
        if (best == 0.0 || sqrt(pv.x * pv.x + pv.y * pv.y) <= sing_tol) s_sing = 1;
      }
    }
    __syncthreads();
    const int pr = s_piv;
    if (pr != kk) {
      for (int j = tid; j < 2 * m; j += kPT) {
        const cd t = Wm[kk + j * kMaxM];
        Wm[kk + j * kMaxM] = Wm[pr + j * kMaxM];
        Wm[pr + j * kMaxM] = t;
      }
    }
    __syncthreads();
    const cd d = Wm[kk + kk * kMaxM];
    const bool dz = (d.x == 0.0 && d.y == 0.0);
    if (tid < m) lmul[tid] = (tid == kk || dz) ? mkcd(0.0, 0.0) : cdiv(Wm[tid + kk * kMaxM], d);
    __syncthreads();
    for (int idx = tid; idx < m * 2 * m; idx += kPT) {
      const int i = idx % m, j = idx / m;
      if (i != kk && j > kk) Wm[i + j * kMaxM] = cfms(lmul[i], Wm[kk + j * kMaxM], Wm[i + j * kMaxM]);
    }
    __syncthreads();
  }
  for (int idx = tid; idx < m * m; idx += kPT) {
    const int i = idx % m, q = idx / m;
    const cd d = Wm[i + i * kMaxM];
    Yb[i + q * kMaxM] = (d.x == 0.0 && d.y == 0.0) ? mkcd(0.0, 0.0) : cdiv(Wm[i + (m + q) * kMaxM], d);
  }
  __syncthreads();
  const bool sing = s_sing != 0;
  const double nanv = __longlong_as_double(0x7ff8000000000000LL);
  const bool bad = sing || failed;
  cd* tout = a.out + (size_t)sh * m * a.ldo;
  if (a.mode == SSV_G || a.mode == SSV_TF) {
    const double sgn = a.mode == SSV_TF ? -1.0 : 1.0;
    for (int idx = tid; idx < p * m; idx += kPT) {
      const int i = idx % p, q = idx / p;
      cd acc = mkcd(0.0, 0.0);
      for (int t = 0; t < m; ++t)
        acc = cfma(df_join(Z2f[BCK(i + (size_t)t * ldz, a.z2_stride)]), Yb[t + q * kMaxM], acc);
      if (bad) acc = mkcd(nanv, nanv);
      tout[BCK(i, p) + (size_t)q * a.ldo] = mkcd(sgn * acc.x, sgn * acc.y);
    }
  } else {
    // backward pass: z_B = Y; per step b = B .. 1: X-hat rows of b = P1_b z_b,
    // then z_{b-1} = P2_b z_b; the initial live rows n - m .. n - 1 take the
    // last z.  Only the chain of the z_b runs here: they go into the shift's
    // window state (dead by now; nsteps m <= n), and tcs_back_kernel forms the
    // X-hat rows of all blocks at once.
    cd* zb = reinterpret_cast<cd*>(a.Z2 + (size_t)sh * a.z2_stride);
    for (int e = tid; e < m * m; e += kPT) zs[(e % m) + (e / m) * kMaxM] = Yb[(e % m) + (e / m) * kMaxM];
    __syncthreads();
    for (int b = nsteps; b >= 1; --b) {
      for (int e = tid; e < m * m; e += kPT) {
        p2s[(e % m) + (e / m) * kMaxM] = tout[BCK(n - b * m + e % m, n) + (size_t)(e / m) * a.ldo];
        zb[BCK((size_t)(b - 1) * m * m + e, a.z2_stride)] = zs[(e % m) + (e / m) * kMaxM];
      }
      __syncthreads();
      for (int e = tid; e < m * m; e += kPT) {
        const int rr = e % m, q = e / m;
        cd acc = mkcd(0.0, 0.0);
        for (int t = 0; t < m; ++t) acc = cfma(p2s[rr + t * kMaxM], zs[t + q * kMaxM], acc);
        zn[rr + q * kMaxM] = acc;
      }
      __syncthreads();
      for (int e = tid; e < m * m; e += kPT) zs[(e % m) + (e / m) * kMaxM] = zn[(e % m) + (e / m) * kMaxM];
      __syncthreads();
    }
    for (int e = tid; e < m * m; e += kPT) {
      const int rr = e % m, q = e / m;
      tout[(n - m + rr) + (size_t)q * a.ldo] = bad ? mkcd(nanv, nanv) : zs[rr + q * kMaxM];
    }
    if (tid == 0) a.flags[sh] = bad ? 1 : 0;
  }
  if (a.status != nullptr && tid == 0) {
    bool fin = true;
    for (int e = 0; e < m * m; ++e) {
      const cd y = Yb[(e % m) + (e / m) * kMaxM];
      fin = fin && isfinite(y.x) && isfinite(y.y);
    }
    a.status[sh] = sing ? SSV_SHIFT_SINGULAR : ((fin && !failed) ? SSV_SHIFT_OK : SSV_SHIFT_NONFINITE);
  }
}

// X-hat rows of block step b = blockIdx.x mod B + 1 (fresh columns j0_b = (B - b) n_b
// .. + nbe_b - 1): P1_b z_b, FP64.  One CTA per (block, shift); two threads per
// row, each half of the m columns.  Bound by the FP64 pipe (4 n m^2
// multiply-adds a shift); inside the serial chain of the z_b, on one SM per
// shift, it took 1.34 ms for 40 shifts at n = 4000, m = 16.
// QH: columns of a thread, ceil(m / 2) rounded up to a power of two (an inactive
// column costs its FP64 issue slots all the same: 0.96 ms with eight for m = 4,
// 2000 shifts at n = 1000).
template <int QH>
__global__ void __launch_bounds__(kPT) tcs_back_kernel(TcsArgs a, int nsteps, int nbe_first) {
  __shared__ cd zs[kMaxM * kMaxM];
  const int b = blockIdx.x % nsteps + 1, sh = blockIdx.x / nsteps, tid = threadIdx.x;
  const int n = a.n, m = a.m;
  const int nbe_b = b == 1 ? nbe_first : kNBT;
  const int j0b = (nsteps - b) * kNBT;
  const cd* zb = reinterpret_cast<const cd*>(a.Z2 + (size_t)sh * a.z2_stride) + (size_t)(b - 1) * m * m;
  for (int e = tid; e < m * m; e += kPT) zs[e] = zb[BCK(e, a.z2_stride)];
  const bool bad = a.flags[sh] != 0 || *a.err != 0;
  __syncthreads();
  const int i = j0b + (tid & (kNBT - 1)), half = tid / kNBT;
  if (i >= j0b + nbe_b) return;
  const cd* ZT = a.ZT + (size_t)sh * (size_t)n * m;
  cd* tout = a.out + (size_t)sh * m * a.ldo;
  const double nanv = __longlong_as_double(0x7ff8000000000000LL);
  const int qh = (m + 1) / 2, q0 = half * qh, q1 = min(m, q0 + qh);
  cd acc[QH];
#pragma unroll
  for (int u = 0; u < QH; ++u) acc[u] = mkcd(0.0, 0.0);
#pragma unroll 4
  for (int t = 0; t < m; ++t) {
    const cd x = ZT[BCK(i + (size_t)t * n, (size_t)n * m)];
#pragma unroll
    for (int u = 0; u < QH; ++u)
      if (q0 + u < q1) acc[u] = cfma(x, zs[t + (q0 + u) * m], acc[u]);
  }
#pragma unroll
  for (int u = 0; u < QH; ++u)
    if (q0 + u < q1) tout[BCK(i, n) + (size_t)(q0 + u) * a.ldo] = bad ? mkcd(nanv, nanv) : acc[u];
}

// the panel kernel for up to MAXM live columns
struct PanelLaunch {
  void (*kern)(TcsArgs, int, int, int);
  int threads;
  size_t smem;
};
template <int MAXM, bool FEW = false>
PanelLaunch panel_config(cudaError_t* e) {
  PanelLaunch l{tcs_panel_kernel<MAXM, FEW>, panel_threads<MAXM, FEW>(), sizeof(PanelSmem<MAXM>)};
  if (*e == cudaSuccess)
    *e = cudaFuncSetAttribute(l.kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)l.smem);
  if (*e == cudaSuccess)
    *e = cudaFuncSetAttribute(l.kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                              (int)cudaSharedmemCarveoutMaxShared);
  return l;
}

}  // namespace

bool solve_tc_supported(const Handle* h, int mode) {
  return h->m <= kMaxM && h->n > h->m && (mode == SSV_G || mode == SSV_TF || mode == SSV_XHAT);
}

size_t solve_tc_scratch_bytes(int n, int m, int p, int s, int mode) {
  const int cs = shift_cols(m), S = kUN / cs;
  const size_t G = (size_t)(s + S - 1) / S;
  auto al = [](size_t b) { return (b + 255) / 256 * 256; };
  size_t b = al(sizeof(float4) * (size_t)s * (size_t)(p + n) * m);
  if (mode == SSV_XHAT) b += al(sizeof(cd) * (size_t)s * (size_t)n * m);
  b += al(G * kSD * kStages * kBT * 2) + al(sizeof(int) * (size_t)s * 2 * kMaxM) +
       al(sizeof(float4) * (size_t)s * 2 * kMaxM * kMaxM) + al(sizeof(int) * ((size_t)s + 1));
  if (cs >= 16) {  // Z2 P2 on the tensor cores: window and P2 digit tiles
    const size_t np = (size_t)resid_tc_npad(n);
    b += al((size_t)s * np * 7 * cs * 2) + al(sizeof(int) * (size_t)s * np) +
         al((size_t)s * 7 * cs * cs * 2) + al(sizeof(int) * (size_t)s * 2 * kMaxM);
  }
  return b + 256;
}

int solve_tc(const Handle* h, int s, const double* shifts, int mode, double* out, long long ldo,
             int* status, const void* hdig, cudaStream_t st) {
  const int n = h->n, m = h->m, p = h->p;
  if (!solve_tc_supported(h, mode)) return SSV_ENOTSUP;
  if (resid_tc_ktile() != kKS) return SSV_ENOTSUP;
  if (s == 0) return SSV_OK;
  const int cs = shift_cols(m), S = kUN / cs;
  const int G = (s + S - 1) / S;
  auto al = [](size_t b) { return (b + 255) / 256 * 256; };
  const size_t bZ = al(sizeof(float4) * (size_t)s * (size_t)(p + n) * m);
  const size_t bT = mode == SSV_XHAT ? al(sizeof(cd) * (size_t)s * (size_t)n * m) : 0;
  const size_t bP = al((size_t)G * kSD * kStages * kBT * 2);
  const size_t bE = al(sizeof(int) * (size_t)s * 2 * kMaxM);
  const size_t bC = al(sizeof(float4) * (size_t)s * 2 * kMaxM * kMaxM);
  const size_t bF = al(sizeof(int) * ((size_t)s + 1));
  const size_t bH = hdig == nullptr ? al(resid_tc_hbytes(n)) : 0;
  const int np = resid_tc_npad(n);
  const bool tcz = cs >= 16;
  const size_t bZd = tcz ? al((size_t)s * np * 7 * cs * 2) : 0;
  const size_t bZe = tcz ? al(sizeof(int) * (size_t)s * np) : 0;
  const size_t bPd2 = tcz ? al((size_t)s * 7 * cs * cs * 2) : 0;
  const size_t bPe2 = tcz ? al(sizeof(int) * (size_t)s * 2 * kMaxM) : 0;
  const size_t total = bZ + bT + bP + bE + bC + bF + bZd + bZe + bPd2 + bPe2 + bH;
#ifdef SSV_BOUNDS_CHECK
  constexpr size_t kCanary = 256;  // checked after the last block step
#else
  constexpr size_t kCanary = 0;
#endif
  unsigned char* buf = nullptr;
  SSV_CUDA_TRY(pool_alloc((void**)&buf, total + kCanary, st));
  unsigned char* o = buf;
  TcsArgs a;
  a.n = n; a.m = m; a.p = p; a.s = s; a.cs = cs; a.S = S; a.ngroups = G; a.mode = mode;
  a.H = h->H; a.Hhi = h->Hhi; a.Hlo = h->Hlo; a.Ct = h->Ct; a.ldct = p > 0 ? p : 1; a.R = h->R;
  a.shifts = reinterpret_cast<const cd*>(shifts); a.hnorm = h->hnorm2;
  a.Z2 = reinterpret_cast<float4*>(o); o += bZ;
  a.z2_stride = (size_t)(p + n) * m;
  a.ZT = bT ? reinterpret_cast<cd*>(o) : nullptr; o += bT;
  a.Pd = reinterpret_cast<uint16_t*>(o); o += bP;
  a.pexp = reinterpret_cast<int*>(o); o += bE;
  a.pc = reinterpret_cast<float4*>(o); o += bC;
  a.flags = reinterpret_cast<int*>(o);
  a.err = a.flags + s; o += bF;
  a.tcz = tcz ? 1 : 0;
  a.npad = np;
  a.Zd = tcz ? reinterpret_cast<uint16_t*>(o) : nullptr; o += bZd;
  a.zexp = tcz ? reinterpret_cast<int*>(o) : nullptr; o += bZe;
  a.P2d = tcz ? reinterpret_cast<uint16_t*>(o) : nullptr; o += bPd2;
  a.p2exp = tcz ? reinterpret_cast<int*>(o) : nullptr; o += bPe2;
  a.out = reinterpret_cast<cd*>(out); a.ldo = ldo; a.status = status;
  a.RB = np / kUM;
  a.KT = np / kKS;
  a.n_z2 = (size_t)s * a.z2_stride;
  a.n_zt = bT ? (size_t)s * n * m : 0;
  a.n_pd = (size_t)G * kSD * kStages * kBT;
  a.n_zd = tcz ? (size_t)s * np * 7 * cs : 0;
  a.n_p2d = tcz ? (size_t)s * 7 * cs * cs : 0;
  a.n_pc = (size_t)s * 2 * kMaxM * kMaxM;
  a.n_hs = (size_t)np * np;  // uint4 of the eight H digit slices
  a.n_out = 0;
  int rc = SSV_OK;
  cudaError_t e = cudaSuccess;
#ifdef SSV_BOUNDS_CHECK
  // scratch read before it is written shows up as NaN (0xFF bytes), and the
  // canary after the scratch as a changed byte
  e = cudaMemsetAsync(buf, 0xFF, total, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(buf + total, 0xA5, kCanary, st);
#endif
  if (e == cudaSuccess) e = cudaMemsetAsync(a.Pd, 0, bP, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(a.err, 0, sizeof(int), st);
  if (e == cudaSuccess && hdig == nullptr) {
    rc = resid_tc_split_h(h, o, st);
    hdig = o;
  }
  if (e == cudaSuccess && rc == SSV_OK) {
    const unsigned char* hb = static_cast<const unsigned char*>(hdig);
    a.Hs = reinterpret_cast<const uint4*>(hb);
    a.hexp = reinterpret_cast<const int*>(hb + ((size_t)kDigits * np * np * 2 + 255) / 256 * 256);
    PanelLaunch panel = m <= 1   ? panel_config<1>(&e)
                        : m <= 2 ? panel_config<2>(&e)
                        : m <= 4 ? panel_config<4>(&e)
                        : m <= 8 ? panel_config<8>(&e)
                        : s <= num_sms() ? panel_config<16, true>(&e)
                                         : panel_config<16>(&e);
    void (*upd)(TcsArgs, int, int) = cs <= 2    ? tcs_update_kernel<2>
                                     : cs <= 4  ? tcs_update_kernel<4>
                                     : cs <= 8  ? tcs_update_kernel<8>
                                     : cs <= 16 ? tcs_update_kernel<16>
                                                : tcs_update_kernel<32>;
    if (e == cudaSuccess) e = cudaFuncSetAttribute(upd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kUpdSmem);
    if (e == cudaSuccess) {
      tcs_setup_kernel<<<s, kPT, 0, st>>>(a);
      count_launch();
      int nbe_first = (n - m) % kNBT;
      if (nbe_first == 0) nbe_first = kNBT;
      int k = n, step = 0;
      while (k > m) {
        const int nbe = step == 0 ? nbe_first : kNBT;
        ++step;
        panel.kern<<<s, panel.threads, panel.smem, st>>>(a, k, nbe, step);
        count_launch();
        const int hrows = k - nbe;
        if (hrows > 0) {
          const long long items = (long long)((hrows + kUM - 1) / kUM) * G;
          const int grid =
              (int)std::max<long long>(1, std::min<long long>(items, (long long)num_sms()));
          void* tru = trace_begin("tcs_update", st);  // per-launch span when tracing is on
          upd<<<grid, kUT, kUpdSmem, st>>>(a, k, nbe);
          count_launch();
          trace_end(tru, st);
        }
        k -= nbe;
      }
#ifdef SSV_BOUNDS_CHECK
      tcs_canary_kernel<<<1, 256, 0, st>>>(buf + total, kCanary, a.err);
      count_launch();
#endif
      tcs_final_kernel<<<s, kPT, 0, st>>>(a, step);
      count_launch();
      if (mode == SSV_XHAT) {
        auto back = m <= 2 ? tcs_back_kernel<1> : m <= 4 ? tcs_back_kernel<2> : m <= 8 ? tcs_back_kernel<4>
                                                                              : tcs_back_kernel<8>;
        back<<<(unsigned)((long long)s * step), kPT, 0, st>>>(a, step, nbe_first);
        count_launch();
      }
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
