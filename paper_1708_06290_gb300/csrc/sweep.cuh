// The persistent sweep of one shift, shared by the solves of one system
// (solve_fp64.cu), of many systems (solve_batch.cu) and of the transposed systems
// and the Givens panel (solve_trans.cu).
//
// Persistent shift-batched solver for (H - sigma I) Xhat = R, FP64.
//
// The method is the blocked bottom-up elimination of Sec. 3.1 / Algorithm 8:
// a sliding window of the columns of [Ct; H - sigma I] moves from the last
// column to the first.  Its "live" part Z2 (m columns, specific to the shift)
// is combined with n_b fresh columns Z1 of the original [Ct; H] (shared by all
// shifts) on each block of n_b rows:
//   1. the n_b x (n_b + m) window block is triangularised from its bottom row
//      up.  Row c has m + 1 candidate entries (m live columns and the fresh
//      column that enters at this row); one complex Householder reflector
//      acting on those m + 1 columns from the right maps the row onto the
//      fresh column's slot (an RQ step, as in Sec. 3.1).  The reflector is
//      applied to the rows of the block above c and accumulated into the
//      coefficients P ((n_b + m) x m) that express the m surviving columns in
//      terms of [Z1 | Z2]; the rest of the block transform is never formed,
//      the economy of Sec. 3.1;
//   2. the rows above the block are updated once:
//      Z2 <- Z1 P(1:n_b, :) + Z2 P(n_b+1:, :) - sigma E P(1:min(m,n_b), :),
//      the last term being the shifted diagonal of the fresh columns that
//      lies above the block (Algorithm 8, diagonal correction);
//   3. the window slides up by n_b rows.
// When m rows remain, the live block W = [Wc; Wm] (p + m rows) gives
// Y = Wm^{-1} R(1:m, 1:m) (Gauss-Jordan with partial pivoting) and G = Wc Y
// (Algorithm 8, final loop; here on the GPU).  For Xhat the window also
// carries the rows of the accumulated column transformation T (the "Q*" rows
// of Sec. 3.3), Xhat = T(:, live) Y.  With one right-hand side R bhat_l per
// shift (Sec. 3.3) Y is the m-vector Wm^{-1} R(1:m, 1:m) bhat_l.
//
// Differences from the paper: one Householder reflector per row instead of
// the Givens schedule (unitary either way, so the one-shot update of the rows
// above stays stable); each thread block owns one shift at a time for the
// whole sweep (no grid-wide phases); the final m x m solve runs on the GPU.
#pragma once
#include <algorithm>
#include <map>
#include <tuple>
#include <type_traits>
#include <mutex>
#include <new>
#include <utility>
#include <vector>

#include "cluster.cuh"
#include "dfloat.cuh"
#include "panel.cuh"
#include "ssv_internal.cuh"

namespace ssv {

namespace {

constexpr int kThreads = 256;  // of the Givens sweep
constexpr int kNB = 128;  // maximum rows per block (runtime nb <= kNB)

// Shared memory per thread block:
//   the panel (pan::Smem); its rows W[c * (MAXM + 1) + q] are the coefficients
//   of window column c (fresh c < kNB, old live kNB + q) in surviving column q
//   Wm, lmul, Yb   final m x m solve
//   coefr          the dense right-hand side's block rows and coefficients (RHS)
template <int MAXM>
struct Layout {
  static constexpr int kSlots = MAXM + 1;
  static constexpr int kCoefRows = kNB + MAXM;
  static constexpr size_t coef_elems = (size_t)kCoefRows * kSlots;
  // both arithmetics have 16-byte entries and the same layout
  static constexpr size_t panel = (sizeof(pan::Smem<pan::F64, MAXM, kNB>) + 15) / 16 * 16;
  static constexpr size_t panel_df = (sizeof(pan::Smem<pan::DF32, MAXM, kNB>) + 15) / 16 * 16;
  static constexpr size_t panel_bytes = panel > panel_df ? panel : panel_df;
  static constexpr size_t bytes = panel_bytes + (3 * MAXM * MAXM + MAXM + 4) * sizeof(cd) +
                                  sizeof(pan::SmemR<pan::F64, MAXM, kNB>) + 64;
};
// Threads of a sweep's blocks and blocks per SM.  FP64: two blocks fill the
// FP64 pipe (one's panel chain under the other's updates); double-float panels
// of few columns leave more of the chain exposed.
template <int MAXM>
constexpr int sweep_threads() {
  return MAXM <= 16 ? 256 : 512;
}
constexpr int sweep_per_sm(int maxm, bool df) { return maxm > 16 ? 1 : df && maxm <= 8 ? 3 : 2; }
// CTAs that share a shift: a power of two up to 8 while every team's CTAs have SMs
// of their own (clusters of four and eight do not tile all SMs of the chip: 19
// teams of eight took 17.7 ms where 24 of four take 14.7), for windows with enough
// rows to share (n = 256, m = 2: 0.54 ms either way).  FP64, n = 3000, m = 8: up to
// 10 shifts 28.4 -> 12.4 ms, 24 shifts 14.7, 64 shifts 19.2; n = 600, m = 4, 64 shifts
// 1.73 -> 1.60; double-float, n = 1500, m = 16, 24 shifts 9.1 -> 5.2.
[[maybe_unused]] static int team_for(int s, int n, int m) {
  if ((long long)n * m < 1024) return 1;
  const long long sms = num_sms();
  if (s * 8LL <= sms * 5 / 6) return 8;
  if (s * 4LL <= sms * 5 / 6) return 4;
  return s * 2LL <= sms ? 2 : 1;
}
constexpr int m_class(int m) { return m <= 1 ? 1 : m <= 2 ? 2 : m <= 4 ? 4 : m <= 8 ? 8 : m <= 16 ? 16 : 32; }

// Givens-panel variant (Sec. 3.2, Algorithms 9/10): the whole window block
// Zb (n_b x (n_b + m), column-major, ld kNBG) and its column transform P
// ((n_b + m) x (n_b + m), ld kNBG + MAXM) live in shared memory, so
// n_b <= kNBG; coefficient rows: fresh c < kNBG, old live kNBG + q.
constexpr int kNBG = 32;
template <int MAXM>
struct GivensLayout {
  static constexpr int kSlots = MAXM + 2;
  static constexpr int kCols = kNBG + MAXM;
  static constexpr int kCoefRows = kNBG + MAXM;
  static constexpr size_t zb_elems = (size_t)kNBG * kCols;
  static constexpr size_t p_elems = (size_t)kCols * kCols;
  static constexpr size_t coef_elems = (size_t)kCoefRows * kSlots;
  static constexpr size_t bytes =
      (zb_elems + p_elems + coef_elems + 3 * MAXM * MAXM + 2 * MAXM + 4 + 2 * kNBG) * sizeof(cd) +
      kNBG * sizeof(int) + 64;
};

}  // namespace

// Greedy annihilation schedule of one block shape (n_b rows, n_b + m columns):
// rotation j zeroes (r, c1) of the block with (r, c2), packed r | c1 << 8 |
// c2 << 16 (0-based); step t holds rotations off[t] .. off[t+1]-1.
struct GivensSched {
  const int* rot;
  const int* off;
  int nsteps;
};

// One system as the FP64 solve sees it.
struct FpSys {
  int n, m, p, nb, mode;
  const double* H;
  const double* Ct;
  int ldct;
  const double* R;
  const cd* shifts;
  cd* out;
  long long ldo;
  int* status;
  cd* xhat_copy;
  long long ldxc;
  const double* hnorm;
  const cd* bhat;    // per-shift right-hand side coefficients (m x s, ld ldb), or null
  long long ldb;
  const cd* rhs;     // dense right-hand sides (n x s, ld ldr) of an RHS sweep (p == 0)
  long long ldr;
  int flip_out;      // write output row i to row n-1-i (transposed systems)
  const float* Hhi;   // double-float split of H (SSV_DFLOAT updates)
  const float* Hlo;
  GivensSched gfull;  // Givens panel: schedule of full blocks (n_b rows)
  GivensSched gtail;  // and of the last, shorter block
};

namespace {

// Solve shift sh of system d with the window state in Z2 (and ZT).  With RHS,
// the dense right-hand side d.rhs(:, sh) is carried through the sweep: each
// finalised column F_c (diagonal beta_c) removes f_c = rhs_c / beta_c times
// itself from the rows above (back substitution against the triangular factor
// as it is produced, bottom-up), the rows above the block through the
// accumulated coefficients `coefr`; the solution is T(:, live) y - Tr with Tr
// the T rows of sum_c (-f_c) F_c and y from the final m x m block.
//
// team > 1: the CTAs of a cluster share the shift and its window state.  Each runs
// the panels (the same bits in all of them, so nothing is exchanged) and takes
// its share of the other rows.
template <int MAXM, int NT, bool RHS = false, bool GIVENS = false, bool DF = false>
__device__ void fp64_shift(const FpSys& d, const int sh, cd* Z2,
                           unsigned char* smem_raw, int* s_piv_p, int* s_sing_p, const int team = 1,
                           const int rank = 0) {
  using L = Layout<MAXM>;
  using GL = GivensLayout<MAXM>;
  constexpr int S = GIVENS ? GL::kSlots : L::kSlots;
  // update of the rows above: lanes per row, columns per lane
  constexpr int G = MAXM <= 4 ? 1 : MAXM <= 8 ? 2 : 4, NS = (MAXM + G - 1) / G;
  constexpr int RPP = NT / G;               // rows the block takes at a time
  constexpr int LB = GIVENS ? kNBG : kNB;   // coefficient row of old live column 0
  constexpr int CR = GIVENS ? GL::kCoefRows : L::kCoefRows;
  cd* Zb = reinterpret_cast<cd*>(smem_raw);  // Givens: window block
  cd* Pg = Zb + GL::zb_elems;                // Givens: column transform
  cd* coef = GIVENS ? Pg + GL::p_elems : reinterpret_cast<cd*>(smem_raw);
  // MAXM x (2 MAXM) augmented [Wm | R1]
  cd* Wm = GIVENS ? coef + GL::coef_elems : reinterpret_cast<cd*>(smem_raw + L::panel_bytes);
  cd* lmul = Wm + 2 * MAXM * MAXM;           // multipliers of the final solve
  cd* Yb = lmul + (MAXM + 4);                // MAXM x MAXM solution
  cd* coefr = Yb + MAXM * MAXM;              // RHS coefficients (kCoefRows)
  const pan::Lane<G> ln(threadIdx.x);
  cd* grot = Yb + MAXM * MAXM;               // Givens: (g0, g1) of the step's rotations
  int* grc = reinterpret_cast<int*>(grot + 2 * kNBG);  // Givens: packed (r, c1, c2)
  int& s_piv = *s_piv_p;
  int& s_sing = *s_sing_p;
  const int n = d.n, m = d.m, p = d.p, nb = d.nb, mode = d.mode, ldct = d.ldct;
  const double* __restrict__ H = d.H;
  const double* __restrict__ Ct = d.Ct;
  const double* __restrict__ R = d.R;
  const cd* __restrict__ shifts = d.shifts;
  cd* __restrict__ out = d.out;
  const long long ldo = d.ldo, ldxc = d.ldxc;
  int* __restrict__ status = d.status;
  cd* __restrict__ xhat_copy = d.xhat_copy;
  const double* __restrict__ hnorm = d.hnorm;
  const int tid = threadIdx.x;
  const int gt = tid + rank * NT, GT = team * NT;  // thread of the team
  auto team_sync = [&] {
    if (!GIVENS && team > 1) cluster_sync_all();
    else __syncthreads();
  };
  const int ldz = p + n;
  const bool track_t = RHS || (mode == SSV_XHAT || mode == SSV_X || xhat_copy != nullptr);
  cd* ZT = Z2 + (size_t)ldz * m;  // n x m, valid when track_t
  cd* Zr = ZT + (size_t)n * m;    // RHS rows in progress (n), when RHS
  cd* Tr = Zr + n;                // T rows of the removed finalised columns (n), when RHS
  // With double-float updates the window state Z2 is kept as FP32 pairs
  // (one float4 per complex entry, the size of a complex128), so the bulk
  // update reads and writes it without FP64 conversions.
  float4* const Z2f = reinterpret_cast<float4*>(Z2);
  auto z2ld = [&](size_t idx) -> cd {
    if constexpr (DF) return df_join(Z2f[idx]);
    else return Z2[idx];
  };
  auto z2st = [&](size_t idx, cd v) {
    if constexpr (DF) Z2f[idx] = df_split(v);
    else Z2[idx] = v;
  };
  const cd sigma = shifts[sh];
  // ||H - sigma I||_F from ||H||_F^2 and trace(H); a finalized diagonal entry
  // of magnitude <= n eps ||H - sigma I||_F marks the shift singular.
  const double mnorm2 = fmax(hnorm[0] - 2.0 * sigma.x * hnorm[1] +
                                 (double)n * (sigma.x * sigma.x + sigma.y * sigma.y), 0.0);
  // (with double-float bulk updates the working precision is 2^-47)
  const double sing_tol = (double)n * (DF ? 7.105427357601002e-15 : 2.220446049250313e-16) * sqrt(mnorm2);
  // ---- shift setup: Z2 = last m columns of [Ct; H] - sigma on the diagonal
  for (long long idx = gt; idx < (long long)ldz * m; idx += GT) {
    int i = (int)(idx % ldz), q = (int)(idx / ldz);
    int j = n - m + q;
    double v = i < p ? Ct[i + (size_t)j * ldct] : H[(i - p) + (size_t)j * n];
    cd z = mkcd(v, 0.0);
    if (i - p == j) z = csub(z, sigma);
    z2st(idx, z);
  }
  if (track_t) {
    for (long long idx = gt; idx < (long long)n * m; idx += GT) {
      int i = (int)(idx % n), q = (int)(idx / n);
      ZT[idx] = mkcd(i == n - m + q ? 1.0 : 0.0, 0.0);
    }
  }
  if (RHS) {
    const cd* rin = d.rhs + (size_t)sh * d.ldr;
    for (int i = gt; i < n; i += GT) {
      Zr[i] = rin[i];
      Tr[i] = mkcd(0.0, 0.0);
    }
  }
  if (tid == 0) s_sing = 0;
  team_sync();

  // Deferred T rows (X-hat output without per-step T updates).  The rows of
  // the accumulated column transform T set at block step b are P1_b, and
  // every later step multiplies all rows set before it by its P2, so
  //   X-hat(rows of step b) = P1_b P2_{b+1} ... P2_B Y,
  // which a backward pass z_B = Y, X-hat_b = P1_b z_b, z_{b-1} = P2_b z_b
  // forms in O(n m^2) instead of O(n^2 m^2 / n_b) updates.  P1_b stays in ZT;
  // P2_b (m x m) is parked in this shift's own output rows n - b m ..
  // n - (b - 1) m - 1, which the backward pass reaches only after reading it
  // when n_b >= m.
  const bool defer_t = track_t && !RHS && d.bhat == nullptr && !d.flip_out && nb >= m;
  cd* const tout = (mode == SSV_XHAT || mode == SSV_X) ? out + (size_t)sh * m * ldo
                                                        : (xhat_copy != nullptr ? xhat_copy + (size_t)sh * m * ldxc : nullptr);
  const long long tld = (mode == SSV_XHAT || mode == SSV_X) ? ldo : ldxc;
  int nsteps = 0;

  int k = n;
  while (k > m) {
    ++nsteps;
    const int nbe = min(nb, k - m);
    const int r = p + k - nbe;        // rows of [Ct; M] above the block
    const int j0 = k - m - nbe;       // first fresh column
    if constexpr (GIVENS) {
      // ---- RQ of the window block with the greedy Givens schedule
      const int nc = nbe + m;
      constexpr int ldp = GL::kCols;
      for (int idx = tid; idx < nc * nbe; idx += NT) {
        const int t = idx % nbe, col = idx / nbe;
        cd z;
        if (col < nbe) {  // fresh column j0 + col: nonzero in block rows t <= col
          z = mkcd(t <= col ? H[(k - nbe + t) + (size_t)(j0 + col) * n] : 0.0, 0.0);
          if (t == col - m) z = csub(z, sigma);
        } else {
          z = Z2[(r + t) + (size_t)(col - nbe) * ldz];
        }
        Zb[col * kNBG + t] = z;
      }
      for (int idx = tid; idx < nc * nc; idx += NT) {
        const int row = idx % nc, col = idx / nc;
        Pg[col * ldp + row] = mkcd(row == col ? 1.0 : 0.0, 0.0);
      }
      __syncthreads();
      const GivensSched& gs = (nbe == nb) ? d.gfull : d.gtail;
      for (int step = 0; step < gs.nsteps; ++step) {
        const int j0r = gs.off[step], cnt = gs.off[step + 1] - j0r;
        // rotation j maps [a, b] = Zb(r, (c1, c2)) to [0, rho]:
        // G = [[g0, conj(g1)], [-g1, conj(g0)]], g0 = b / rho, g1 = a / rho
        for (int j = tid; j < cnt; j += NT) {
          const int pk = gs.rot[j0r + j];
          const int rr = pk & 255, c1 = (pk >> 8) & 255, c2 = (pk >> 16) & 255;
          const cd a = Zb[c1 * kNBG + rr], b = Zb[c2 * kNBG + rr];
          const double rho = hypot(hypot(a.x, a.y), hypot(b.x, b.y));
          cd g0 = mkcd(1.0, 0.0), g1 = mkcd(0.0, 0.0);
          if (rho > 0.0) {
            g0 = mkcd(b.x / rho, b.y / rho);
            g1 = mkcd(a.x / rho, a.y / rho);
          }
          grot[2 * j] = g0;
          grot[2 * j + 1] = g1;
          grc[j] = pk;
        }
        __syncthreads();
        // [x1, x2] <- [x1 g0 - x2 g1, x1 conj(g1) + x2 conj(g0)] on the block rows
        // 0 .. r and on every row of P
        const int span = nbe + nc;
        for (int e = tid; e < cnt * span; e += NT) {
          const int j = e / span, w = e % span;
          const int pk = grc[j];
          const int rr = pk & 255, c1 = (pk >> 8) & 255, c2 = (pk >> 16) & 255;
          cd *x1, *x2;
          if (w < nbe) {
            if (w > rr) continue;
            x1 = Zb + c1 * kNBG + w;
            x2 = Zb + c2 * kNBG + w;
          } else {
            x1 = Pg + c1 * ldp + (w - nbe);
            x2 = Pg + c2 * ldp + (w - nbe);
          }
          const cd g0 = grot[2 * j], g1 = grot[2 * j + 1];
          const cd u = *x1, v = *x2;
          const cd nu = csub(cmul(u, g0), cmul(v, g1));
          const cd nv = cfma(u, mkcd(g1.x, -g1.y), cmul(v, mkcd(g0.x, -g0.y)));
          *x1 = (w == rr) ? mkcd(0.0, 0.0) : nu;
          *x2 = nv;
        }
        __syncthreads();
      }
      // R(t, t + m) is the finalised diagonal of block row t
      for (int t = tid; t < nbe; t += NT) {
        const cd dgl = Zb[(t + m) * kNBG + t];
        if (sqrt(dgl.x * dgl.x + dgl.y * dgl.y) <= sing_tol) s_sing = 1;
      }
      // the first m columns of P express the surviving (new live) columns:
      // coefficient rows fresh c -> P(c, q), old live qq -> P(nbe + qq, q)
      for (int idx = tid; idx < CR * S; idx += NT) {
        const int crow = idx / S, q = idx % S;
        cd v = mkcd(0.0, 0.0);
        if (q < m) {
          if (crow < nbe) v = Pg[q * ldp + crow];
          else if (crow >= LB && crow - LB < m) v = Pg[q * ldp + nbe + (crow - LB)];
        }
        coef[idx] = v;
      }
      __syncthreads();
    } else {
      // ---- panel (panel.cuh): with DF in double-float on the FP32 pipe, the
      // coefficients left in `coef` as FP32 pairs
      using A = typename std::conditional<DF, pan::DF32, pan::F64>::type;
      using V = typename A::V;
      auto& psm = *reinterpret_cast<pan::Smem<A, MAXM, kNB>*>(smem_raw);
      static_assert(pan::Smem<A, MAXM, kNB>::S == S, "coefficient rows");
      auto* psr = reinterpret_cast<pan::SmemR<A, MAXM, kNB>*>(coefr);
      for (int e = tid; e < nbe * m; e += NT) {
        const int row = e % nbe, q = e / nbe;
        psm.W[row * S + q] = reinterpret_cast<const V*>(Z2)[(r + row) + (size_t)q * ldz];
      }
      if constexpr (RHS) {
        for (int t = tid; t < nbe; t += NT) psr->r[t] = Zr[r + t];
      }
      typename A::H hm;
      if constexpr (DF) hm = {d.Hhi, d.Hlo, n, {}};
      else hm = {H, n, {}};
      pan::run<A, MAXM, kNB, NT, RHS>(hm, k - nbe, j0, sigma, nbe, m, psm, psr, sing_tol, &s_sing);
    }

    // ---- update the rows above the block (and the T rows)
    auto coefd = [&](int crow, int q) -> cd {
      if constexpr (DF) {
        const float4 w = reinterpret_cast<const float4*>(coef)[crow * S + q];
        return mkcd((double)w.x + (double)w.y, (double)w.z + (double)w.w);
      } else {
        return coef[crow * S + q];
      }
    };
    // Row i takes G lanes, lane g the columns q = g, g + G, ..: the row's old
    // entries are read by all of them before any is written (__syncwarp).
    for (int i0 = rank * RPP; i0 < r; i0 += team * RPP) {
      const int i = i0 + ln.row;
      const int cd_ = i - (r - m);  // diagonal correction of fresh column cd_
      const bool live = i < r, diag = live && cd_ >= 0 && cd_ < min(m, nbe);
      typename std::conditional<DF, float4, cd>::type res[NS];  // the new entries, as Z2 holds them
      cd racc = mkcd(0.0, 0.0);
      if (DF && live && i >= p) {
        // double-float (SSV_DFLOAT): H as (Hhi, Hlo), exact FMA products,
        // two-sum accumulation (48-bit class); the Ct rows and the diagonal
        // correction stay in FP64
        if constexpr (DF) {
          float rh[NS], rl[NS], ih[NS], il[NS];
          const float4* cf4 = reinterpret_cast<const float4*>(coef);
#pragma unroll
          for (int u = 0; u < NS; ++u) { rh[u] = 0.f; rl[u] = 0.f; ih[u] = 0.f; il[u] = 0.f; }
          const float* __restrict__ hh = d.Hhi + (i - p) + (size_t)j0 * n;
          const float* __restrict__ hl = d.Hlo + (i - p) + (size_t)j0 * n;
#pragma unroll 4
          for (int c = 0; c < nbe; ++c) {
            const float zh = hh[(size_t)c * n], zl = hl[(size_t)c * n];
            const float4* cr = cf4 + c * S + ln.g;
#pragma unroll
            for (int u = 0; u < NS; ++u) {
              if (u * G + ln.g < m) {
                const float4 w = cr[u * G];
                df_mac(rh[u], rl[u], zh, zl, w.x, w.y);
                df_mac(ih[u], il[u], zh, zl, w.z, w.w);
              }
            }
          }
          for (int qq = 0; qq < m; ++qq) {
            const float4 zz = Z2f[i + (size_t)qq * ldz];
            const float4* cr = cf4 + (LB + qq) * S + ln.g;
#pragma unroll
            for (int u = 0; u < NS; ++u) {
              if (u * G + ln.g < m) {
                const float4 w = cr[u * G];
                // (zr + i zi)(wr + i wi) = (zr wr - zi wi) + i (zr wi + zi wr)
                df_mac(rh[u], rl[u], zz.x, zz.y, w.x, w.y);
                df_mac(rh[u], rl[u], -zz.z, -zz.w, w.z, w.w);
                df_mac(ih[u], il[u], zz.x, zz.y, w.z, w.w);
                df_mac(ih[u], il[u], zz.z, zz.w, w.x, w.y);
              }
            }
          }
#pragma unroll
          for (int u = 0; u < NS; ++u) {
            if (diag && u * G + ln.g < m) {
              const cd z = mkcd((double)rh[u] + (double)rl[u], (double)ih[u] + (double)il[u]);
              res[u] = df_split(cfms(sigma, coefd(cd_, u * G + ln.g), z));
            } else {  // normalised pairs
              const float sr = rh[u] + rl[u], si = ih[u] + il[u];
              res[u] = make_float4(sr, rl[u] - (sr - rh[u]), si, il[u] - (si - ih[u]));
            }
          }
        }
      } else if (live) {
        cd acc[NS];
#pragma unroll
        for (int u = 0; u < NS; ++u) acc[u] = mkcd(0.0, 0.0);
        if (RHS && ln.g == 0) racc = Zr[i];
        const double* __restrict__ hc = i < p ? Ct + i + (size_t)j0 * ldct : H + (i - p) + (size_t)j0 * n;
        const size_t hld = i < p ? (size_t)ldct : (size_t)n;
#pragma unroll 4
        for (int c = 0; c < nbe; ++c) {
          const double z = hc[(size_t)c * hld];
#pragma unroll
          for (int u = 0; u < NS; ++u) {
            if (u * G + ln.g < m) {
              const cd w = coefd(c, u * G + ln.g);
              acc[u].x = fma(z, w.x, acc[u].x);
              acc[u].y = fma(z, w.y, acc[u].y);
            }
          }
          if (RHS && ln.g == 0) racc = mkcd(fma(z, coefr[c].x, racc.x), fma(z, coefr[c].y, racc.y));
        }
        for (int qq = 0; qq < m; ++qq) {
          const cd zz = z2ld(i + (size_t)qq * ldz);
#pragma unroll
          for (int u = 0; u < NS; ++u)
            if (u * G + ln.g < m) acc[u] = cfma(zz, coefd(LB + qq, u * G + ln.g), acc[u]);
          if (RHS && ln.g == 0) racc = cfma(zz, coefr[kNB + qq], racc);
        }
        if (diag) {
#pragma unroll
          for (int u = 0; u < NS; ++u)
            if (u * G + ln.g < m) acc[u] = cfms(sigma, coefd(cd_, u * G + ln.g), acc[u]);
          if (RHS && ln.g == 0) racc = cfms(sigma, coefr[cd_], racc);
        }
#pragma unroll
        for (int u = 0; u < NS; ++u) {
          if constexpr (DF) res[u] = df_split(acc[u]);
          else res[u] = acc[u];
        }
      }
      __syncwarp();
      if (live) {
        if (RHS && ln.g == 0) Zr[i] = racc;
#pragma unroll
        for (int u = 0; u < NS; ++u) {
          const int q = u * G + ln.g;
          if (q < m) {
            if constexpr (DF) Z2f[i + (size_t)q * ldz] = res[u];
            else Z2[i + (size_t)q * ldz] = res[u];
          }
        }
      }
    }
    if (defer_t && rank == 0) {
      // rows j0 .. j0+nbe-1: ZT = P1; P2 parked in the output (see above)
      for (int idx = tid; idx < nbe * m; idx += NT) {
        const int i = j0 + idx % nbe, q = idx / nbe;
        ZT[i + (size_t)q * n] = coefd(i - j0, q);
      }
      for (int idx = tid; idx < m * m; idx += NT) {
        const int qq = idx % m, q = idx / m;
        tout[(n - nsteps * m + qq) + (size_t)q * tld] = coefd(LB + qq, q);
      }
    } else if (track_t && !defer_t) {
      // rows k-m .. n-1: ZT <- ZT P2 ; rows j0 .. j0+nbe-1: ZT = P1
      const int lo = k - m;
      for (int i0 = j0 + rank * RPP; i0 < n; i0 += team * RPP) {
        const int i = i0 + ln.row;
        const bool live = i < n;
        cd acc[NS];
#pragma unroll
        for (int u = 0; u < NS; ++u) acc[u] = mkcd(0.0, 0.0);
        cd tr = mkcd(0.0, 0.0);
        if (live && i < lo) {
          if (RHS) tr = coefr[i - j0];
#pragma unroll
          for (int u = 0; u < NS; ++u)
            if (u * G + ln.g < m) acc[u] = coefd(i - j0, u * G + ln.g);
        } else if (live) {
          if (RHS && ln.g == 0) tr = Tr[i];
          float rh[DF ? NS : 1], rl[DF ? NS : 1], ih[DF ? NS : 1], il[DF ? NS : 1];
          if constexpr (DF) {
#pragma unroll
            for (int u = 0; u < NS; ++u) { rh[u] = 0.f; rl[u] = 0.f; ih[u] = 0.f; il[u] = 0.f; }
          }
          for (int qq = 0; qq < m; ++qq) {
            const cd zz = ZT[i + (size_t)qq * n];
            if constexpr (DF) {
              const float4 z = df_split(zz);
              const float4* cr = reinterpret_cast<const float4*>(coef) + (LB + qq) * S + ln.g;
#pragma unroll
              for (int u = 0; u < NS; ++u) {
                if (u * G + ln.g < m) {
                  const float4 w = cr[u * G];
                  df_mac(rh[u], rl[u], z.x, z.y, w.x, w.y);
                  df_mac(rh[u], rl[u], -z.z, -z.w, w.z, w.w);
                  df_mac(ih[u], il[u], z.x, z.y, w.z, w.w);
                  df_mac(ih[u], il[u], z.z, z.w, w.x, w.y);
                }
              }
            } else {
#pragma unroll
              for (int u = 0; u < NS; ++u)
                if (u * G + ln.g < m) acc[u] = cfma(zz, coefd(LB + qq, u * G + ln.g), acc[u]);
              if (RHS && ln.g == 0) tr = cfma(zz, coefr[kNB + qq], tr);
            }
          }
          if constexpr (DF) {
#pragma unroll
            for (int u = 0; u < NS; ++u)
              acc[u] = mkcd((double)rh[u] + (double)rl[u], (double)ih[u] + (double)il[u]);
          }
        }
        __syncwarp();
        if (live) {
          if (RHS && ln.g == 0) Tr[i] = tr;
#pragma unroll
          for (int u = 0; u < NS; ++u)
            if (u * G + ln.g < m) ZT[i + (size_t)(u * G + ln.g) * n] = acc[u];
        }
      }
    }
    team_sync();
    k -= nbe;
  }

  // ---- final m x m block: solve Wm Y = R(0:m, 0:m) by Gauss-Jordan with
  // partial pivoting on the augmented [Wm | R1] (2m columns).  With a
  // right-hand side per shift (Sec. 3.3) the augmented part is the single
  // column R1 bhat, and Y is m x 1.
  const cd* __restrict__ bh = d.bhat != nullptr ? d.bhat + (size_t)sh * d.ldb : nullptr;
  const int nr = (RHS || bh != nullptr) ? 1 : m;
  const int w2 = m + nr;
  for (int idx = tid; idx < m * w2; idx += NT) {
    int i = idx % m, j = idx / m;
    cd v;
    if (j < m) v = z2ld((p + i) + (size_t)j * ldz);
    else if (RHS) {
      v = Zr[i];
    } else if (bh != nullptr) {
      v = mkcd(0.0, 0.0);
      for (int t = i; t < m; ++t) {
        const double rv = R[i + (size_t)t * n];
        v = mkcd(fma(rv, bh[t].x, v.x), fma(rv, bh[t].y, v.y));
      }
    } else {
      int jj = j - m;
      v = mkcd(i <= jj ? R[i + (size_t)jj * n] : 0.0, 0.0);
    }
    Wm[i + j * MAXM] = v;
  }
  __syncthreads();
  for (int kk = 0; kk < m; ++kk) {
    if (tid < 32) {
      double best = -1.0;
      int brow = kk;
      for (int i = kk + tid; i < m; i += 32) {
        double v = cabs1(Wm[i + kk * MAXM]);
        if (v > best) { best = v; brow = i; }
      }
      for (int o = 16; o > 0; o >>= 1) {
        double ob = __shfl_xor_sync(0xffffffffu, best, o);
        int orow = __shfl_xor_sync(0xffffffffu, brow, o);
        if (ob > best || (ob == best && orow < brow)) { best = ob; brow = orow; }
      }
      if (tid == 0) {
        s_piv = brow;
        const cd pv = Wm[brow + kk * MAXM];
        if (best == 0.0 || sqrt(pv.x * pv.x + pv.y * pv.y) <= sing_tol) s_sing = 1;
      }
    }
    __syncthreads();
    const int pr = s_piv;
    if (pr != kk) {
      for (int j = tid; j < w2; j += NT) {
        cd a = Wm[kk + j * MAXM];
        Wm[kk + j * MAXM] = Wm[pr + j * MAXM];
        Wm[pr + j * MAXM] = a;
      }
    }
    __syncthreads();
    const cd d = Wm[kk + kk * MAXM];
    const bool dz = (d.x == 0.0 && d.y == 0.0);
    if (tid < m) lmul[tid] = (tid == kk || dz) ? mkcd(0.0, 0.0) : cdiv(Wm[tid + kk * MAXM], d);
    __syncthreads();
    for (int idx = tid; idx < m * w2; idx += NT) {
      int i = idx % m, j = idx / m;
      if (i != kk && j > kk) Wm[i + j * MAXM] = cfms(lmul[i], Wm[kk + j * MAXM], Wm[i + j * MAXM]);
    }
    __syncthreads();
  }
  // Y(i, q) = Wm(i, m+q) / Wm(i, i)
  for (int idx = tid; idx < m * nr; idx += NT) {
    int i = idx % m, q = idx / m;
    cd d = Wm[i + i * MAXM];
    Yb[i + q * MAXM] = (d.x == 0.0 && d.y == 0.0) ? mkcd(0.0, 0.0) : cdiv(Wm[i + (m + q) * MAXM], d);
  }
  __syncthreads();
  const bool sing = s_sing != 0;
  const double nanv = __longlong_as_double(0x7ff8000000000000LL);
  // ---- outputs
  if ((mode == SSV_G || mode == SSV_TF) && rank == 0) {
    const double sg = mode == SSV_TF ? -1.0 : 1.0;
    cd* o = out + (size_t)sh * nr * ldo;
    for (int idx = tid; idx < p * nr; idx += NT) {
      int i = idx % p, q = idx / p;
      cd acc = mkcd(0.0, 0.0);
      for (int t = 0; t < m; ++t) acc = cfma(z2ld(i + (size_t)t * ldz), Yb[t + q * MAXM], acc);
      if (sing) acc = mkcd(nanv, nanv);
      o[i + (size_t)q * ldo] = mkcd(sg * acc.x, sg * acc.y);
    }
  }
  if (defer_t && rank == 0) {
    // backward pass: z = Y; per step b = B .. 1: X-hat rows of b = P1_b z,
    // then z = P2_b z; finally the initial live rows n-m .. n-1 take z
    cd* zs = reinterpret_cast<cd*>(smem_raw);  // m x m (ld MAXM); the panel's arrays are done with
    cd* p2s = zs + MAXM * MAXM;   // P2_b
    cd* zn = p2s + MAXM * MAXM;   // P2_b z
    static_assert((GIVENS ? GL::zb_elems + GL::p_elems : L::coef_elems) >= 3 * MAXM * MAXM, "backward-pass scratch");
    for (int e = tid; e < m * m; e += NT) zs[(e % m) + (e / m) * MAXM] = Yb[(e % m) + (e / m) * MAXM];
    __syncthreads();
    for (int b = nsteps; b >= 1; --b) {
      const int kb = n - (b - 1) * nb;  // every step before the last takes nb rows
      const int nbe_b = min(nb, kb - m);
      const int j0b = kb - m - nbe_b;
      for (int e = tid; e < m * m; e += NT)
        p2s[(e % m) + (e / m) * MAXM] = tout[(n - b * m + e % m) + (size_t)(e / m) * tld];
      __syncthreads();
      for (int idx = tid; idx < nbe_b * m; idx += NT) {
        const int i = j0b + idx % nbe_b, q = idx / nbe_b;
        cd acc = mkcd(0.0, 0.0);
        for (int t = 0; t < m; ++t) acc = cfma(ZT[i + (size_t)t * n], zs[t + q * MAXM], acc);
        tout[i + (size_t)q * tld] = sing ? mkcd(nanv, nanv) : acc;
      }
      for (int e = tid; e < m * m; e += NT) {
        const int rr = e % m, q = e / m;
        cd acc = mkcd(0.0, 0.0);
        for (int t = 0; t < m; ++t) acc = cfma(p2s[rr + t * MAXM], zs[t + q * MAXM], acc);
        zn[rr + q * MAXM] = acc;
      }
      __syncthreads();
      for (int e = tid; e < m * m; e += NT) zs[(e % m) + (e / m) * MAXM] = zn[(e % m) + (e / m) * MAXM];
      __syncthreads();
    }
    for (int e = tid; e < m * m; e += NT) {
      const int rr = e % m, q = e / m;
      tout[(n - m + rr) + (size_t)q * tld] = sing ? mkcd(nanv, nanv) : zs[rr + q * MAXM];
    }
  } else if (track_t && !defer_t) {
    cd* o;
    long long ld;
    if (mode == SSV_XHAT || mode == SSV_X) {
      o = out + (size_t)sh * nr * ldo;
      ld = ldo;
    } else {
      o = xhat_copy + (size_t)sh * nr * ldxc;
      ld = ldxc;
    }
    for (int idx = gt; idx < n * nr; idx += GT) {
      int i = idx % n, q = idx / n;
      cd acc = mkcd(0.0, 0.0);
      if (RHS) acc = mkcd(-Tr[i].x, -Tr[i].y);
      for (int t = 0; t < m; ++t) acc = cfma(ZT[i + (size_t)t * n], Yb[t + q * MAXM], acc);
      if (sing) acc = mkcd(nanv, nanv);
      o[(d.flip_out ? n - 1 - i : i) + (size_t)q * ld] = acc;
    }
  }
  if (status != nullptr && tid == 0 && rank == 0) {
    // a non-finite solution (NaN / Inf in the inputs or an overflow) is reported
    // as such, also when no separate scan of the outputs follows
    bool fin = true;
    for (int e = 0; e < m * nr; ++e) {
      const cd y = Yb[(e % m) + (e / m) * MAXM];
      fin = fin && isfinite(y.x) && isfinite(y.y);
    }
    status[sh] = sing ? SSV_SHIFT_SINGULAR : (fin ? SSV_SHIFT_OK : SSV_SHIFT_NONFINITE);
  }
  team_sync();
}

// Non-finite scan: status[sh] = NONFINITE if an output of an OK shift is not finite.
[[maybe_unused]] __global__ void nonfinite_kernel(const cd* __restrict__ out, long long ldo, int rows, int m, int s,
                                 int* __restrict__ status) {
  int sh = blockIdx.x;
  if (sh >= s) return;
  __shared__ int bad;
  if (threadIdx.x == 0) bad = 0;
  __syncthreads();
  const cd* o = out + (size_t)sh * m * ldo;
  for (int idx = threadIdx.x; idx < rows * m; idx += blockDim.x) {
    int i = idx % rows, q = idx / rows;
    cd v = o[i + (size_t)q * ldo];
    if (!isfinite(v.x) || !isfinite(v.y)) bad = 1;
  }
  __syncthreads();
  if (threadIdx.x == 0 && bad && status[sh] == SSV_SHIFT_OK) status[sh] = SSV_SHIFT_NONFINITE;
}

}  // namespace

}  // namespace ssv
