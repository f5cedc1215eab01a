// Controller-Hessenberg reduction (Algorithm 1, Sec. 2) with two levels of
// blocking (Sec. 2.1: blocks of b columns, each split into mini-blocks of m
// columns; Algorithms 2 and 3, Eqs. for V, T and Y), where every product of
// O(n^3) total work runs on the tensor cores as an FP64-accurate product of
// error-free BF16 digits, and the panels stay in FP64.
//
// Arithmetic of the products.  An operand row (or column) is scaled by the
// power of two 2^E above its largest magnitude and cut into eight 7-bit
// digits (56 bits, more than FP64's 53).  The product of digit pair (a, b)
// over one K = 16 slice is a tcgen05.mma of kind::f16 into FP32 TMEM; pairs
// with a + b = t accumulate in level t.  The rank-b updates keep t = 0..7 (36 pairs; the
// dropped pairs weigh below 2^-53 of the product's scale, the row maximum
// times the column maximum); the long-K products A V_s and V^T A keep
// t = 0..8 (43 pairs, dropped part below 2^-60): their terms mostly sit far
// below that scale, and with eight levels their error grew to about ten
// times an FP64 product's.  One instruction serves several pairs: the B digit
// tiles of a stage sit side by side, so A digit a against B digits b0 .. b0+c-1
// (N c <= 256 columns) lands digit b in level a + b (fused levels).  A level's
// sums are integers below 2^24 for K <= 128 (8 pairs x 128 x 127^2 < 2^24),
// hence exact in FP32; after each window of 128 the levels are added exactly into 64-bit
// fixed-point words (levels 0-3, 4-7 and 8; a window adds below 2^46 to a
// word), kept across the whole K range and turned into FP64 once per output.
//
// A column of the V factor of a block's reflectors has entries of magnitude
// <= 1 with a unit pivot (|v_r| <= 1 because |alpha - beta| >= |beta| >=
// |x_r|), so V by columns uses the fixed exponent 1 and the QR kernel
// writes those digits as the reflectors appear; V by rows (mostly far below
// 1) is split with per-row exponents at the end of the block.
//
// Per block of jb reflectors (rows r0 = z + m .. n-1, trailing columns
// z + b ..):
//   per mini-block (FP64):
//     P <- P - Y V(cols, :)^T  (from the right),  P <- P - V T^T V^T P  (left),
//     one cooperative launch; Householder QR of the mini-block, one cluster;
//   then A V_s and V^T V_s in one product on the tensor cores (A = the matrix at
//     the start of the block), and the new columns of Y (Eq. for Y),
//     Y_s = (A V_s - Y V^T V_s) T_s, and of T (Eq. for T);
//   block end (Algorithm 3, all on the tensor cores but the T^T product):
//     A(:, z+m:) -= Y V^T  (rows above r0 and C: from column z + m; rows r0..:
//                           from column z + b),
//     W = V^T A(r0:, z+b:),  Z = T^T W,  A(r0:, z+b:) -= V Z.
// Step 1 of Algorithm 1 (the QR of B, applied to A from both sides and to C
// from the right) is one more block with r0 = 0 and no block columns.
//
// The working matrix E stacks C (rows 0..p-1) above A (rows p..p+n-1),
// column-major, so that every right update of A and C is one product.
//
// Every wait (grid barrier, mbarrier) is bounded and raises an error flag;
// the host then reports SSV_ETIMEOUT.
#include <algorithm>
#include <climits>

#include "cluster.cuh"
#include "tc_common.cuh"

namespace ssv {

namespace {

using namespace tcg;

constexpr int kTR = 64;                  // rows of a digit tile
constexpr int kTK = 32;                  // K of a digit tile
constexpr int kTileEl = kTR * kTK;       // 2048 BF16 values (4 KB) in the core-matrix layout
constexpr int kD = kDigits;              // digits per operand value
constexpr int kBmax = 128;               // reflectors per block at most
constexpr int kMaxW = 64;                // mini-block width (m) at most
constexpr int kWinTiles = 4;             // K tiles per exact window (4 x 32 = 128)
constexpr int kDrainT = 256;             // readout and epilogue threads of the product kernel
constexpr int kGT = kDrainT + 64;        // + the producer's and the issuer's warp
constexpr unsigned long long kSpin = 1ull << 26;  // grid barrier naps before giving up

// Debug builds (-DSSV_BOUNDS_CHECK): every global index of these kernels is
// checked against its buffer's extent; one out of range is clamped to 0 (a
// bulk copy then stays inside its buffer) and sets bit 2 of the error word,
// so the reduction fails (the back-transform reports NaN).  The scratch is filled with NaN before use and a
// canary after it is verified at the end.  In normal builds RBCK(i, n, e) is i.
#ifdef SSV_BOUNDS_CHECK
__device__ __forceinline__ size_t rbck(long long i, size_t n, int* err) {
  if (i < 0 || (size_t)i >= n) {
    if (err) atomicOr(err, 2);
    return 0;
  }
  return (size_t)i;
}
// [i, i + len) inside [0, n)
__device__ __forceinline__ size_t rbcr(long long i, long long len, size_t n, int* err) {
  if (i < 0 || (size_t)(i + len) > n) {
    if (err) atomicOr(err, 2);
    return 0;
  }
  return (size_t)i;
}
#define RBCK(i, n, e) rbck((long long)(i), (size_t)(n), (e))
#define RBCR(i, len, n, e) rbcr((long long)(i), (long long)(len), (size_t)(n), (e))
#else
#define RBCK(i, n, e) ((size_t)(i))
#define RBCR(i, len, n, e) ((size_t)(i))
#endif

// Digit tiles of an R x K operand (R rows, each scaled by 2^ex[r]): tile
// (digit, J, I) holds rows 64 I .. 64 I + 63 and K 32 J .. 32 J + 31, the
// tiles of one (digit, J) consecutive in I, so that two neighbours are the
// 128-row A operand of one product.
struct DigitMat {
  unsigned short* d;
  int* ex;    // per row; null: the fixed exponent 1
  int RT;     // 64-row tiles (even)
  int KT;     // 32-wide K tiles
  size_t nd;  // BF16 values in d (the extent the debug build checks)
};

__host__ __device__ __forceinline__ size_t tile_index(const DigitMat& M, int dig, int J, int I) {
  return (((size_t)dig * M.KT + J) * M.RT + I) * kTileEl;
}

// bit pattern of the BF16 digit `l` of x at exponent E
__device__ __forceinline__ void digits_of(double x, int E, unsigned short (&d)[kD]) { digits8(x, E, d); }

// ---------------------------------------------------------------------------
// Splitting.  Element (r, k) of the source is src[off(r) + k * sk]; rows
// [r_lo, r_hi) and K [k_lo, k_hi) are taken, everything else of a tile is 0.
// off(r) = r * sr, and for r >= wrap the imaginary part of row r - wrap: the
// real form of a complex operand (sr and sk counted in doubles).
// ---------------------------------------------------------------------------
__device__ __forceinline__ long long row_off(int r, long long sr, int wrap) {
  return r < wrap ? (long long)r * sr : 1 + (long long)(r - wrap) * sr;
}


// exponent pass: ex[r] = max over the K range of scale_exp(|x|) (ex preset to
// INT_MIN), from the high words as integers: a maximum of doubles holds the FP64
// pipe for 64 clocks a warp (the reduction of n = 3000: 2.64 -> 0.64 ms in all)
__global__ void __launch_bounds__(256) split_exp_kernel(const double* __restrict__ src, long long sr,
                                                        long long sk, int r_lo, int r_hi, int k_lo,
                                                        int k_hi, int kchunk, int wrap, int* __restrict__ ex,
                                                        size_t nsrc, size_t nex, int* err) {
  const int tid = threadIdx.x;
  const int rb = r_lo + blockIdx.x * 64;
  const int kb = k_lo + blockIdx.y * kchunk;
  const int ke = min(k_hi, kb + kchunk);
  auto bits = [&](int r, int k) {
    return abs_hi(src[RBCK(row_off(r, sr, wrap) + (long long)k * sk, nsrc, err)]);
  };
  if (sk <= 2) {
    // K (nearly) contiguous: a warp per row, lanes along K
    const int lane = tid & 31, wp = tid >> 5;
#pragma unroll 2
    for (int rr = wp; rr < 64; rr += 8) {
      const int r = rb + rr;
      if (r >= r_hi) break;
      int mx = 0;
#pragma unroll 4
      for (int k = kb + lane; k < ke; k += 32) mx = max(mx, bits(r, k));
      mx = __reduce_max_sync(0xffffffffu, mx);
      if (lane == 0) atomicMax(ex + RBCK(r, nex, err), scale_exp_hi(mx));
    }
  } else {
    // rows contiguous (sr == 1 in every use): threads along rows, four K groups
    __shared__ int part[4][64];
    const int rr = tid & 63, g = tid >> 6;
    const int r = rb + rr;
    int mx = 0;
    if (r < r_hi)
#pragma unroll 8
      for (int k = kb + g; k < ke; k += 4) mx = max(mx, bits(r, k));
    part[g][rr] = mx;
    __syncthreads();
    if (g == 0 && r < r_hi) {
      mx = max(max(part[0][rr], part[1][rr]), max(part[2][rr], part[3][rr]));
      atomicMax(ex + RBCK(r, nex, err), scale_exp_hi(mx));
    }
  }
}

// digit pass: one CTA per tile (I, J) of [I0, I0 + gridDim.x) x [J0, J0 + gridDim.y)
__global__ void __launch_bounds__(256) split_dig_kernel(const double* __restrict__ src, long long sr,
                                                        long long sk, int r_lo, int r_hi, int k_lo,
                                                        int k_hi, int wrap, DigitMat M, int I0, int J0,
                                                        size_t nsrc, size_t nex, int* err) {
  __shared__ double t[kTR][kTK + 1];
  const int tid = threadIdx.x;
  const int I = I0 + blockIdx.x, J = J0 + blockIdx.y;
  const int rb = I * kTR, kb = J * kTK;
  for (int e = tid; e < kTileEl; e += 256) {
    int rr, kk;
    if (sk <= 2) { rr = e / kTK; kk = e % kTK; }
    else { rr = e % kTR; kk = e / kTR; }
    const int r = rb + rr, k = kb + kk;
    double v = 0.0;
    if (r >= r_lo && r < r_hi && k >= k_lo && k < k_hi) v = src[RBCK(row_off(r, sr, wrap) + (long long)k * sk, nsrc, err)];
    t[rr][kk] = v;
  }
  __syncthreads();
  const int rr = tid >> 2, kq = (tid & 3) * 8;
  const int r = rb + rr;
  int E = (r >= r_lo && r < r_hi) ? (M.ex ? M.ex[RBCK(r, nex, err)] : 1) : 0;
  if (E < -4000) E = 0;  // a row with an empty K range (all of its values are 0)
  unsigned short dg[8][kD];
#pragma unroll
  for (int q = 0; q < 8; ++q) digits_of(t[rr][kq + q], E, dg[q]);
  const size_t off = (size_t)tile_off_kg(rr, kq, kTK / 8);
#pragma unroll
  for (int l = 0; l < kD; ++l) {
    uint4 v;
    v.x = (unsigned)dg[0][l] | ((unsigned)dg[1][l] << 16);
    v.y = (unsigned)dg[2][l] | ((unsigned)dg[3][l] << 16);
    v.z = (unsigned)dg[4][l] | ((unsigned)dg[5][l] << 16);
    v.w = (unsigned)dg[6][l] | ((unsigned)dg[7][l] << 16);
    *reinterpret_cast<uint4*>(M.d + RBCR(tile_index(M, l, J, I) + off, 8, M.nd, err)) = v;
  }
}


// ---------------------------------------------------------------------------
// The digit product: output (r + roff, c + coff) for A rows r in [M0, M1)
// and B rows c in [N0, N1) (column-major C, leading dimension ldc) receives
// x = sum_k A(r, k) B(c, k), k over the K tiles [J0, J1).  sub: C -= x, else
// C = x; with ksplit > 1 chunk s of the K range writes C + s * kstride.
// ---------------------------------------------------------------------------
struct GSeg {
  DigitMat A, B;
  int J0, J1;
};
struct GArgs {
  GSeg seg;
  int M0, M1, N0, N1;
  int roff, coff;
  double* C;
  size_t nc;  // doubles from C on (the extent the debug build checks)
  long long ldc;
  int sub;
  int ksplit;
  long long kstride;
  int rs = 1;          // row stride of C in doubles (2: one part of a complex matrix)
  int wrap = INT_MAX;  // columns from here on: the imaginary parts of columns 0 ..
  // with C2: one more row tile, B's first 128 rows in A's place, rows < N1 written
  // to C2 (leading dimension kBmax, partial sums kstride2 apart): V^T V_s beside A V_s
  double* C2 = nullptr;
  size_t nc2 = 0;
  long long kstride2 = 0;
  int* err;
};

template <int NT, int LV>
struct GCfg {
  static constexpr uint32_t kABytes = 2u * kTileEl * 2u;        // 128 rows x 32 K of one digit
  static constexpr uint32_t kBBytes = (uint32_t)NT * kTK * 2u;  // NT rows x 32 K of one digit
  // A digit planes, B digit planes, then one B plane of zeros (written once)
  // so that the first fused product of a window covers every level
  static constexpr uint32_t kStage = (uint32_t)kD * (kABytes + kBBytes) + kBBytes;
  // stage buffers: three when they fit (N = 16: two loads in flight), else two
  static constexpr int kNS = 3 * (size_t)kStage + 256 <= 227 * 1024 ? 3 : 2;
  static constexpr size_t kSmem = kNS * (size_t)kStage + 256;
  static constexpr uint32_t kUsed = (uint32_t)LV * NT;
  // TMEM windows: two when they fit (N = 16), so that one is read back while the
  // next one multiplies
  static constexpr int kTW = 2 * kUsed <= 512 ? 2 : 1;
  static constexpr uint32_t kNeed = (uint32_t)kTW * kUsed;
  static constexpr uint32_t kCols = kNeed <= 32 ? 32 : kNeed <= 64 ? 64 : kNeed <= 128 ? 128 : kNeed <= 256 ? 256 : 512;
  static_assert(kSmem <= 227 * 1024, "shared memory of the digit product");
  static_assert(kUsed <= 512, "TMEM columns");
  static_assert(LV == 8 || LV == 9, "levels");
};

template <int CPT>
__device__ __forceinline__ void tmem_ld_cols(uint32_t taddr, uint32_t (&r)[CPT]) {
  if constexpr (CPT == 8) tmem_ld8(taddr, r);
  else if constexpr (CPT == 16) tmem_ld16(taddr, r);
  else tmem_ld32(taddr, r);
}

// (w[0] 2^56 + w[1] 2^28 + w[2]) 2^(e - 56), or with two words (w[0] 2^28 + w[1])
// 2^(e - 28), rounded once to nearest even, in integer arithmetic: about 45
// integer instructions of 2 clocks a warp, where a conversion and a multiply-add
// per word hold the FP64 pipe for 64 clocks each (n = 2000, 900 real columns, K = 128 by
// 64 columns: 58 -> 44 us a launch; nine levels, K = 2000: 33 -> 24 us).
template <int NW>
__device__ __forceinline__ double words_to_double(const long long* w, int e) {
  __int128 t = w[0];
#pragma unroll
  for (int q = 1; q < NW; ++q) t = (t << 28) + w[q];
  const bool neg = t < 0;
  unsigned __int128 a = neg ? -(unsigned __int128)t : (unsigned __int128)t;
  unsigned long long hi = (unsigned long long)(a >> 64), lo = (unsigned long long)a;
  int top = 127;  // weight of the leading bit of hi after the shift
  if (hi == 0) {
    hi = lo;
    lo = 0;
    top = 63;
  }
  if (hi == 0) return 0.0;
  const int z = __clzll((long long)hi);
  if (z > 0) {
    hi = (hi << z) | (lo >> (64 - z));
    lo <<= z;
  }
  const int ex = top - z + e - 28 * (NW - 1);  // the value is in [2^ex, 2^(ex + 1))
  unsigned long long r = hi >> 11;
  const bool half = (hi & 0x400ull) != 0, rest = (hi & 0x3ffull) != 0 || lo != 0;
  if (half && (rest || (r & 1))) ++r;
  const unsigned long long sg = neg ? 0x8000000000000000ull : 0ull;
  if (ex > -1022 && ex < 1022) return __longlong_as_double((long long)(sg | (((unsigned long long)(ex + 1022) << 52) + r)));
  return ldexp(neg ? -(double)r : (double)r, ex - 52);
}

// a bounded wait of one role: gives up at the poll limit or when another role
// has (the CTA then leaves together)
__device__ __forceinline__ bool role_wait(uint32_t mbar, uint32_t parity, volatile int* fail) {
  for (long long it = 0; it < kWaitLimit / 64; ++it) {
    if (mbar_wait(mbar, parity, 64)) return true;
    if (*fail) return false;
  }
  *fail = 1;
  return false;
}

// Three roles that only meet at mbarriers: a producer thread copies K stages
// into the stage buffers, an issuing thread multiplies them into a TMEM window,
// eight warps read finished windows back and write the tile.  So the next
// stages' copies and products run under the readout and the FP64 epilogue, which
// had alternated with them (one stage in flight, block barriers around each).
template <int NT, int LV>
__global__ void __launch_bounds__(kGT, 1) tc_gemm_kernel(GArgs g) {
  using Cfg = GCfg<NT, LV>;
  constexpr int CPT = NT / 2;
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr int NS = Cfg::kNS, TW = Cfg::kTW;
  // full[NS], empty[NS]: stage buffer copied / multiplied; tfull[TW], tempty[TW]:
  // TMEM window complete / read back
  __shared__ __align__(8) unsigned long long mbar[2 * NS + 2 * TW];
  __shared__ uint32_t tslot;
  __shared__ volatile int fail;
  __shared__ int issued[2];  // stages copied, stages multiplied (read when a wait gave up)
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int quarter = warp & 3, half = warp >> 2;
  const uint32_t full = smem_addr(mbar), empty = full + 8u * NS, tfull = empty + 8u * NS, tempty = tfull + 8u * TW;
  const uint32_t sBase = smem_addr(smem);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tslot)),
                 "r"(Cfg::kCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int q = 0; q < 2 * NS + 2 * TW; ++q)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(full + 8u * q),
                   "r"(q >= 2 * NS + TW ? kDrainT / 32 : 1));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fail = 0;
    issued[0] = 0;
    issued[1] = 0;
  }
  for (int bq = 0; bq < NS; ++bq) {
    uint4* zp = reinterpret_cast<uint4*>(smem + (size_t)bq * Cfg::kStage + kD * (Cfg::kABytes + Cfg::kBBytes));
    for (int e = tid; e < (int)(Cfg::kBBytes / 16); e += kGT) zp[e] = make_uint4(0u, 0u, 0u, 0u);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the zeros, seen by the tensor cores
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tslot;
  const int iI0 = g.M0 / 128, iI1 = (g.M1 + 127) / 128;
  const int iN0 = g.N0 / NT, iN1 = (g.N1 + NT - 1) / NT;
  const int nA = max(0, iI1 - iI0), nN = max(0, iN1 - iN0);
  const int nI = nA + (LV == 9 && g.C2 != nullptr ? 1 : 0);
  const long long ntile = (long long)nI * nN * g.ksplit;
  const DigitMat& B = g.seg.B;
  constexpr int NW = (LV + 3) / 4;  // 64-bit words of the level sums
  struct Tile {
    int iI, n0, ks, jlo, nst;
    bool vv;  // B against itself
  };
  auto tile_of = [&](long long tt) {
    Tile t;
    t.n0 = (iN0 + (int)(tt % nN)) * NT;
    const int it = (int)((tt / nN) % nI);
    t.vv = LV == 9 && it >= nA;
    t.iI = t.vv ? 0 : iI0 + it;
    t.ks = (int)(tt / ((long long)nN * nI));
    int jlo = g.seg.J0, jhi = g.seg.J1;
    if (g.ksplit > 1) {
      int chunk = (jhi - jlo + g.ksplit - 1) / g.ksplit;
      chunk = (chunk + kWinTiles - 1) / kWinTiles * kWinTiles;
      jlo = jlo + t.ks * chunk;
      jhi = min(jhi, jlo + chunk);
    }
    t.jlo = jlo;
    t.nst = max(0, jhi - jlo);
    return t;
  };
  if (warp == kDrainT / 32) {
    if (lane == 0) {
      // ---- producer: stage i (counted over all tiles) into buffer i mod NS
      unsigned i = 0;
      bool ok = true;
      for (long long tt = blockIdx.x; tt < ntile && ok; tt += gridDim.x) {
        const Tile t = tile_of(tt);
        const DigitMat& A = LV == 9 && t.vv ? g.seg.B : g.seg.A;
        for (int st = 0; st < t.nst; ++st, ++i) {
          const uint32_t b = i % NS;
          if (!role_wait(empty + 8u * b, ((i / NS) & 1u) ^ 1u, &fail)) {
            ok = false;
            break;
          }
          const int J = t.jlo + st;
          const uint32_t dst = sBase + b * Cfg::kStage, lb = full + 8u * b;
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(lb),
                       "r"(Cfg::kStage - Cfg::kBBytes)
                       : "memory");
          for (int d = 0; d < kD; ++d)
            bulk_copy(dst + (uint32_t)d * Cfg::kABytes,
                      A.d + RBCR(tile_index(A, d, J, 2 * t.iI), 2 * kTileEl, A.nd, g.err), Cfg::kABytes, lb);
          for (int d = 0; d < kD; ++d)
            bulk_copy(dst + kD * Cfg::kABytes + (uint32_t)d * Cfg::kBBytes,
                      B.d + RBCR(tile_index(B, d, J, t.n0 / kTR) + (size_t)(t.n0 % kTR) * kTK, NT * kTK, B.nd, g.err),
                      Cfg::kBBytes, lb);
          issued[0] = (int)(i + 1);
        }
      }
    }
  } else if (warp == kDrainT / 32 + 1) {
    if (lane == 0) {
      // ---- issuer: window v (counted over all tiles) into TMEM window v mod TW
      unsigned i = 0, v = 0;
      bool ok = true;
      for (long long tt = blockIdx.x; tt < ntile && ok; tt += gridDim.x) {
        const int nst = tile_of(tt).nst;
        for (int st = 0; st < nst; ++st, ++i) {
          const uint32_t b = i % NS, h = v % TW;
          const bool fresh = (st % kWinTiles) == 0;
          if (fresh && !role_wait(tempty + 8u * h, ((v / TW) & 1u) ^ 1u, &fail)) ok = false;
          if (ok && !role_wait(full + 8u * b, (i / NS) & 1u, &fail)) ok = false;
          if (!ok) break;
          // fused levels: the B digit planes of a stage sit side by side (NT rows
          // each, then the zero plane), so one product of A digit a against B
          // digits b0 .. b0 + c - 1 (N = NT c <= 256) lands digit b in TMEM level
          // a + b; the products of a = 0 reach every level (the zero plane stands
          // for B digit 8) and open the window, so one thread issues them all
          fence_after();
          const uint32_t aBase = sBase + b * Cfg::kStage;
          const uint32_t bBase = aBase + kD * Cfg::kABytes;
          const uint32_t dt = tmem + h * Cfg::kUsed;
          constexpr int kMaxC = 256 / NT;
#pragma unroll
          for (int kk = 0; kk < kTK / 16; ++kk) {
#pragma unroll
            for (int a = 0; a < kD; ++a) {
              const int nb = a == 0 ? LV : LV - a;  // B digits 0 .. nb - 1 (digit 8: the zero plane)
#pragma unroll
              for (int b0 = 0; b0 < nb; b0 += kMaxC) {
                const int c = min(kMaxC, nb - b0);
                const uint64_t ad = mat_desc(aBase + (uint32_t)a * Cfg::kABytes + (uint32_t)kk * 256u, 128u, 512u);
                const uint64_t bd = mat_desc(bBase + (uint32_t)b0 * Cfg::kBBytes + (uint32_t)kk * 256u, 128u, 512u);
                mma_bf16(dt + (uint32_t)((a + b0) * NT), ad, bd, idesc_bf16(128, NT * c),
                         (fresh && kk == 0 && a == 0) ? 0u : 1u);
              }
            }
          }
          mma_commit(empty + 8u * b);
          issued[1] = (int)(i + 1);
          if ((st % kWinTiles) == kWinTiles - 1 || st == nst - 1) {
            mma_commit(tfull + 8u * h);
            ++v;
          }
        }
      }
    }
  } else {
    // ---- readout and epilogue: thread = (row, half of the columns)
    unsigned v = 0;
    bool ok = true;
    for (long long tt = blockIdx.x; tt < ntile && ok; tt += gridDim.x) {
      const Tile cur = tile_of(tt);
      const int i0 = cur.iI * 128, n0 = cur.n0, ks = cur.ks;
      // exact level sums of every window, in 64-bit words: word w holds levels
      // 4w .. 4w + 3, level L at bit 21 - 7 (L - 4 w); a window adds less than
      // 2^46 to a word, so 2^17 windows (K up to 16 M) cannot overflow it
      long long wacc[NW][CPT];
#pragma unroll
      for (int w = 0; w < NW; ++w)
#pragma unroll
        for (int c = 0; c < CPT; ++c) wacc[w][c] = 0;
      for (int st = 0; st < cur.nst; st += kWinTiles, ++v) {
        const uint32_t h = v % TW;
        ok = __all_sync(0xffffffffu, role_wait(tfull + 8u * h, (v / TW) & 1u, &fail));
        if (!ok) break;
        fence_after();
#pragma unroll
        for (int w = 0; w < NW; ++w) {
#pragma unroll 1
          for (int L = 4 * w; L < min(LV, 4 * w + 4); ++L) {
            uint32_t rv[CPT];
            tmem_ld_cols<CPT>(tmem + h * Cfg::kUsed + ((uint32_t)(quarter * 32) << 16) +
                                  (uint32_t)(L * NT + half * CPT),
                              rv);
            const int sh = 21 - 7 * (L - 4 * w);
#pragma unroll
            for (int c = 0; c < CPT; ++c) wacc[w][c] += (long long)__float2int_rn(__uint_as_float(rv[c])) << sh;
          }
        }
        fence_before();
        __syncwarp();
        if (lane == 0)
          asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tempty + 8u * h) : "memory");
      }
      if (!ok) break;
      // word w weighs 2^{Ea + Eb - 35 - 28 w}
      const int r = i0 + quarter * 32 + lane;
      if (LV == 9 && cur.vv ? r < g.N1 : (r >= g.M0 && r < g.M1)) {
        const DigitMat& A = LV == 9 && cur.vv ? g.seg.B : g.seg.A;
        double* const C = LV == 9 && cur.vv ? g.C2 : g.C;
        const int Ea = A.ex ? A.ex[RBCK(r, (size_t)A.RT * kTR, g.err)] : 1;
        const long long ldc = LV == 9 && cur.vv ? kBmax : g.ldc;
        // C offset of column 0
        const size_t c0 = LV == 9 && cur.vv ? (size_t)ks * g.kstride2 + r : (size_t)ks * g.kstride + (size_t)(r + g.roff) * g.rs;
        auto cidx = [&](int col) {
          return RBCK(c0 + row_off(col + g.coff, ldc, g.wrap), LV == 9 && cur.vv ? g.nc2 : g.nc, g.err);
        };
        // eight columns at a time, their loads of C in flight together
#pragma unroll
        for (int cb = 0; cb < CPT; cb += 8) {
          double x[8], old[8];
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            const int col = n0 + half * CPT + cb + c;
            old[c] = (g.sub && col >= g.N0 && col < g.N1) ? C[cidx(col)] : 0.0;
          }
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            const int col = n0 + half * CPT + cb + c;
            const int Eb = (col >= g.N0 && col < g.N1) ? (B.ex ? B.ex[RBCK(col, (size_t)B.RT * kTR, g.err)] : 1) : 0;
            double xv = 0.0;
            if (Ea == kBadExp || Eb == kBadExp) {
              xv = __longlong_as_double(0x7ff8000000000000LL);
            } else if (Ea > -4000 && Eb > -4000) {
              long long wv[NW];
#pragma unroll
              for (int w = 0; w < NW; ++w) wv[w] = wacc[w][cb + c];
              xv = words_to_double<NW>(wv, Ea + Eb - 35);
            }
            x[c] = xv;
          }
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            const int col = n0 + half * CPT + cb + c;
            if (col >= g.N0 && col < g.N1) C[cidx(col)] = g.sub ? old[c] - x[c] : x[c];
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
    atomicExch(g.err, 1);
    const unsigned nl = (unsigned)issued[0], nm = (unsigned)issued[1];
    for (unsigned i = nl > NS ? nl - NS : 0; i < nl; ++i) mbar_wait(full + 8u * (i % NS), (i / NS) & 1u);
    for (unsigned i = nm > NS ? nm - NS : 0; i < nm; ++i) mbar_wait(empty + 8u * (i % NS), (i / NS) & 1u);
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(Cfg::kCols));
}

// ---------------------------------------------------------------------------
// Panel of one mini-block (Algorithm 2 between two updates of Y).  First its
// columns receive the block's reflectors so far (panel_update_kernel, one
// cooperative launch): CTA g owns a contiguous range of the panel rows r0 .. n-1,
// kept in shared memory (column-major per CTA); cross-CTA sums go through
// per-CTA partial slots and a bounded grid barrier.  Then one cluster factors
// them (panel_qr_kernel).
// ---------------------------------------------------------------------------
constexpr int kPT = 256;
constexpr int kPartW = 4096;             // partial-sum slot per CTA (doubles)
constexpr int kPanRowsW = 8192;          // rows x columns of the panel per CTA at most
constexpr int kRedW = 0;                 // W = V^T P (j x w)
constexpr int kRedZ = 4096;              // Z = T^T W
constexpr int kRedTotal = 8192;
constexpr size_t kPanFixed = 4096 + 4096;  // doubles besides the panel
constexpr size_t kPanSmem = 200 * 1024;  // with the staged rows of V and Y at most
static_assert(sizeof(double) * (kPanRowsW + kPanFixed) <= kPanSmem, "a panel without the staged rows");

struct PanArgs {
  double* P;          // panel column t, matrix row r: P[r + t * ldp]
  long long ldp;
  int r0, n;          // panel rows [r0, n)
  int w;              // panel columns
  int j;              // reflectors of the block before this mini-block
  int c0;             // matrix column of panel column 0 (rows c0.. of V: the right update)
  const double* V;    // V(r, i) = V[r + i * ldv], explicit zeros and unit pivots
  long long ldv;
  const double* T;    // T(i, k) = T[i + k * kBmax], upper triangular
  const double* Y;    // Y(matrix row r, i) = Y[yoff + r + i * ldy]
  long long ldy;
  int yoff;
  int staged;         // the CTA's rows of V and Y (j columns) go to shared memory
  double* part;       // [G][kPartW]
  double* red;        // kRedTotal
  unsigned* bar;      // this launch's arrival counter (zero at its start)
  int* err;
  // extents (doubles from each pointer on) the debug build checks
  size_t np, nv, ny, npart;
};

// Grid-wide barrier with a bounded wait: false once any CTA has given up.
// *bar counts this launch's arrivals (every panel launch has a counter of its
// own, zeroed at the start of the reduction); the k-th barrier (k from 1) of
// the launch completes when it reaches k * gridDim.x.  The arrival returns
// nothing: it and the first poll are on their way together.
__device__ bool grid_sync(unsigned* bar, int* err, unsigned k) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned target = k * gridDim.x;
    asm volatile("fence.acq_rel.gpu;\n\tred.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    unsigned long long spins = 0;
    for (;;) {
      unsigned now;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(now) : "l"(bar) : "memory");
      if ((int)(now - target) >= 0) break;
      if ((spins & 15) == 15 && *(volatile int*)err != 0) break;
      if (++spins > kSpin) {
        atomicExch(err, 1);
        break;
      }
      if (spins > 4096) __nanosleep(32);
    }
    __threadfence();
    s_ok = (*(volatile int*)err == 0);
  }
  __syncthreads();
  return s_ok != 0;
}

// Sums with every thread of the CTA: out(e) = sum_k term(e, k) for e in
// [e0, e1), k < count(e); tpe threads (a power of two <= 32, the largest with
// tpe (e1 - e0) <= kPT) share an output, each taking every tpe-th k sixteen at
// a time (all loads of a panel's cross-CTA sums in flight at once), then a
// shuffle tree.  The order is fixed, so every CTA that forms the
// same sums gets the same bits.
template <typename Count, typename Term, typename Store>
__device__ __forceinline__ void block_sums(int e0, int e1, Count count, Term term, Store store) {
  const int nE = e1 - e0;
  if (nE <= 0) return;
  int tpe = 32;
  while (tpe > 1 && tpe * nE > kPT) tpe >>= 1;
  const int per = kPT / tpe;
  const int t = threadIdx.x, sub = t % tpe;
  for (int c0 = 0; c0 < nE; c0 += per) {
    const int el = c0 + t / tpe;
    const bool act = el < nE;
    const int e = e0 + el;
    double acc = 0.0;
    if (act) {
      const int K = count(e);
      for (int k = sub; k < K; k += 16 * tpe) {
        double v[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) v[q] = k + q * tpe < K ? term(e, k + q * tpe) : 0.0;
#pragma unroll
        for (int h = 8; h > 0; h >>= 1)
#pragma unroll
          for (int q = 0; q < 8; ++q)
            if (q < h) v[q] += v[q + h];
        acc += v[0];
      }
    }
    for (int o = tpe >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (act && sub == 0) store(e, acc);
  }
}

__device__ __forceinline__ void put_digits_v(const DigitMat& M, int row, int k, double v, int* err) {
  unsigned short d[kD];
  digits_of(v, 1, d);
  const size_t off = (size_t)tile_off_kg(row % kTR, k % kTK, kTK / 8);
#pragma unroll
  for (int l = 0; l < kD; ++l) M.d[RBCK(tile_index(M, l, k / kTK, row / kTR) + off, M.nd, err)] = d[l];
  (void)err;
}

__global__ void __launch_bounds__(kPT, 1) panel_update_kernel(PanArgs a) {
  extern __shared__ double psm[];
  const int G = gridDim.x, g = blockIdx.x, tid = threadIdx.x;
  const int w = a.w, j = a.j;
  const int L = a.n - a.r0;
  const int rpc = (L + G - 1) / G;
  const int ra = a.r0 + g * rpc;
  const int nr = max(0, min(a.n, ra + rpc) - ra);
  double* Ps = psm;                      // Ps[t * rpc + rl]
  double* Vc = Ps + (size_t)rpc * w;     // Vc[t * j + i] = V(c0 + t, i)
  double* Zs = Vc + 4096;                // Zs[i * w + t]
  double* Vb = Zs + 4096;                // staged: V(ra + rl, i) at Vb[i * rpc + rl]
  double* Yb = Vb + (size_t)rpc * j;     // staged: Y of the same rows
  unsigned nbar = 0;                     // grid barriers so far
  // checked element accesses (plain indexing in normal builds)
  auto Pi = [&](long long i) -> double& { return a.P[RBCK(i, a.np, a.err)]; };
  auto Vi = [&](long long i) -> const double& { return a.V[RBCK(i, a.nv, a.err)]; };
  auto Ti = [&](long long i) -> const double& { return a.T[RBCK(i, (size_t)kBmax * kBmax, a.err)]; };
  auto Ri = [&](long long i) { return a.red + RBCK(i, (size_t)kRedTotal, a.err); };
  // partial e of CTA gg
  auto Pt = [&](int gg, int e) { return a.part + RBCK((size_t)gg * kPartW + e, a.npart, a.err); };

  // Everything the panel reads of earlier results starts at once: its columns,
  // the rows of V that carry the right update's coefficients, and (staged) this
  // CTA's rows of V and Y.  Read in the loops that use them they cost an L2
  // round trip every few multiply-adds.
  auto cp8 = [](double* dst, const double* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
  };
  for (int e = tid; e < nr * w; e += kPT) {
    const int rl = e % nr, t = e / nr;
    cp8(Ps + t * rpc + rl, &Pi((size_t)(ra + rl) + (size_t)t * a.ldp));
  }
  for (int e = tid; e < w * j; e += kPT) {
    const int t = e % w, i = e / w;
    cp8(Vc + t * j + i, &Vi((size_t)(a.c0 + t) + (size_t)i * a.ldv));
  }
  if (a.staged) {
    for (int e = tid; e < nr * j; e += kPT) {
      const int rl = e % nr, i = e / nr;
      cp8(Vb + i * rpc + rl, &Vi((size_t)(ra + rl) + (size_t)i * a.ldv));
      cp8(Yb + i * rpc + rl, a.Y + RBCK((size_t)a.yoff + ra + rl + (size_t)i * a.ldy, a.ny, a.err));
    }
  }
  asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  // V and Y of this CTA's rows (reflector i < j)
  auto vr = [&](int rl, int i) -> double {
    return a.staged ? Vb[i * rpc + rl] : Vi((size_t)(ra + rl) + (size_t)i * a.ldv);
  };
  auto yr = [&](int rl, int i) -> double {
    return a.staged ? Yb[i * rpc + rl] : a.Y[RBCK((size_t)a.yoff + ra + rl + (size_t)i * a.ldy, a.ny, a.err)];
  };
  // P(rl, t) -= sum_{i < j} f(rl, i) g(i, t): tpe lanes share an entry
  auto rank_update = [&](auto f, auto gq) {
    const int nE = nr * w;
    int tpe = 8;
    while (tpe > 1 && tpe * nE > kPT) tpe >>= 1;
    const int per = kPT / tpe, sub = tid % tpe;
    for (int c0 = 0; c0 < nE; c0 += per) {
      const int e = c0 + tid / tpe;
      const bool act = e < nE;
      const int rl = act ? e % nr : 0, t = act ? e / nr : 0;
      double acc = 0.0;
      if (act) {
#pragma unroll 8
        for (int i = sub; i < j; i += tpe) acc = fma(f(rl, i), gq(i, t), acc);
      }
      for (int o = tpe >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (act && sub == 0) Ps[t * rpc + rl] -= acc;
    }
    __syncthreads();
  };
  // from the right: P -= Y(rows, 0:j) V(c0:c0+w, 0:j)^T
  rank_update(yr, [&](int i, int t) { return Vc[t * j + i]; });
  // from the left: W = V^T P, Z = T^T W, P -= V Z
  for (int e = tid; e < j * w; e += kPT) {
    const int i = e / w, t = e % w;
    double acc = 0.0;
#pragma unroll 8
    for (int rl = 0; rl < nr; ++rl) acc = fma(vr(rl, i), Ps[t * rpc + rl], acc);
    *Pt(g, RBCK(e, kPartW, a.err)) = acc;
  }
  if (!grid_sync(a.bar, a.err, ++nbar)) return;
  const int ch = (j * w + G - 1) / G;
  const int e0 = min(j * w, g * ch), e1 = min(j * w, (g + 1) * ch);
  block_sums(
      e0, e1, [&](int) { return G; }, [&](int e, int gg) { return __ldcg(Pt(gg, e)); },
      [&](int e, double v) { *Ri(kRedW + e) = v; });
  if (!grid_sync(a.bar, a.err, ++nbar)) return;
  block_sums(
      e0, e1, [&](int e) { return e / w + 1; },
      [&](int e, int k) { return Ti(k + (size_t)(e / w) * kBmax) * __ldcg(Ri(kRedW + k * w + e % w)); },
      [&](int e, double v) { *Ri(kRedZ + e) = v; });
  if (!grid_sync(a.bar, a.err, ++nbar)) return;
  for (int e = tid; e < j * w; e += kPT) Zs[e] = __ldcg(Ri(kRedZ + e));
  __syncthreads();
  rank_update(vr, [&](int i, int t) { return Zs[i * w + t]; });
  for (int e = tid; e < nr * w; e += kPT) {
    const int rl = e % nr, t = e / nr;
    Pi((size_t)(ra + rl) + (size_t)t * a.ldp) = Ps[t * rpc + rl];
  }
}

// ---------------------------------------------------------------------------
// Householder QR of the updated mini-block by one cluster: CTA c owns a
// contiguous range of the rows (in shared memory where they fit).  Bound by the
// chain of a reflector: one exchange of partial dot products (v^T P follows from
// the raw column's), a root, a division, one pass over the rows.  Among 16 CTAs
// the exchange is a store to distributed shared memory and a cluster barrier;
// over the whole chip it was a grid barrier and a read of 152 partials, and took
// more than the arithmetic.  A mini-block of n = 3000, m = 4: 53 us in one launch
// with V^T V_s and T, now 18 (update) + 19 (QR), V^T V_s a tile of the next product.
// ---------------------------------------------------------------------------
constexpr int kQrT = 512;                // threads: 16 warps over the columns
constexpr int kQrC = 16;                 // CTAs of the cluster at most
constexpr int kQrW = kQrT / 32;
constexpr int kQrX = kQrC * kMaxW;       // an exchange buffer (sources x columns)
// exchange buffers, pivot rows, coefficients, scales, pivots (doubles)
constexpr size_t kQrFixed = 2 * kQrX + 2 * kMaxW + 3 * kMaxW;
constexpr size_t kQrSmem = 216 * 1024;

struct QrArgs {
  double* P;          // panel column t, matrix row r: P[r + t * ldp]
  long long ldp;
  int r0, n;          // panel rows [r0, n)
  int w, wp;          // panel columns; reflectors generated (wp <= w)
  int pv0;            // pivot row of reflector t: pv0 + t
  int j;              // reflectors of the block before this mini-block
  int cs;             // CTAs of the cluster
  int insm;           // the rows fit the CTAs' shared memory
  double* V;          // V(r, i) = V[r + i * ldv], explicit zeros and unit pivots
  long long ldv;
  double* tau;        // tau of reflector t at tau[t]
  DigitMat vcol;      // V's digits, operand row = reflector, K = r (exponent 1: the unit pivot is
                      // every reflector's largest entry)
  int* err;
  size_t np, nv, ntau;  // extents the debug build checks
};

__global__ void __launch_bounds__(kQrT, 1) panel_qr_kernel(QrArgs a) {
  extern __shared__ double qsm[];
  double* xch = qsm;                     // [2][source][column]
  double* piv = xch + 2 * kQrX;          // [2][kMaxW]
  double* cf = piv + 2 * kMaxW;          // coefficients of the update
  double* scl = cf + kMaxW;              // v = scl * column below the pivot
  double* bet = scl + kMaxW;             // R's diagonal
  double* Psm = bet + kMaxW;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int c = cluster_rank(), C = a.cs, w = a.w;
  const int rpc = (a.n - a.r0 + C - 1) / C;
  const int ra = a.r0 + c * rpc;
  const int nr = max(0, min(a.n, ra + rpc) - ra);
  const long long ld = a.insm ? rpc : a.ldp;
  double* Pg = a.P + ra;
  double* Ps = a.insm ? Psm : Pg;
  auto Gi = [&](long long i) { return (long long)RBCK(ra + i, a.np, a.err) - ra; };
  if (a.insm)
    for (int t = warp; t < w; t += kQrW)
#pragma unroll 4
      for (int rl = lane; rl < nr; rl += 32) Psm[t * ld + rl] = Pg[Gi(rl + (long long)t * a.ldp)];
  // the cluster has started (its shared memory can be written) and the rows are in
  cluster_sync_all();
  for (int t = 0; t < a.wp; ++t) {
    const int q = t & 1, pr = a.pv0 + t, prl = pr - ra;  // the pivot's row here (or outside [0, nr))
    const int rb = max(0, prl + 1);
    const int nk = w - t;  // columns t .. w-1 (k = t: the squared norm below the pivot)
    int pw = 1;            // columns rounded up to a power of two; wps warps share one
    while (pw < nk) pw <<= 1;
    const int wps = max(1, kQrW / pw), sub = warp % wps;
    const double* ct = Ps + t * ld;
    for (int k = warp / wps; k < nk; k += kQrW / wps) {
      const double* ck = ct + k * ld;
      double acc = 0.0;
#pragma unroll 4
      for (int rl = rb + sub * 32 + lane; rl < nr; rl += 32 * wps) acc = fma(ck[rl], ct[rl], acc);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (lane < C) {
        cluster_st(xch + q * kQrX + (c * wps + sub) * pw + k, lane, acc);
        if (sub == 0 && prl >= 0 && prl < nr) cluster_st(piv + q * kMaxW + k, lane, ck[prl]);
      }
    }
    __syncwarp();
    cluster_sync_all();
    if (warp == 0) {
      // sums over the sources in a fixed order: the same bits in every CTA
      const double* x = xch + q * kQrX;
      const int pl = min(pw, 32), parts = 32 / pl;
      double d[kMaxW / 32];
#pragma unroll
      for (int u = 0; u < kMaxW / 32; ++u) {
        d[u] = 0.0;
        const int k = (lane & (pl - 1)) + 32 * u;
        if (32 * u >= nk) continue;
        if (k < nk)
#pragma unroll 4
          for (int sq = lane / pl; sq < C * wps; sq += parts) d[u] += x[sq * pw + k];
        for (int o = 16; o >= pl; o >>= 1) d[u] += __shfl_xor_sync(0xffffffffu, d[u], o);
      }
      const double sig = __shfl_sync(0xffffffffu, d[0], 0), alpha = piv[q * kMaxW];
      double tk = 0.0, scal = 0.0, beta = alpha;
      if (sig != 0.0) {
        const double nrm = sqrt(fma(alpha, alpha, sig));
        beta = alpha >= 0.0 ? -nrm : nrm;
        // both quotients in one division: lane parity
        const double qt = (lane & 1) ? 1.0 / (alpha - beta) : (beta - alpha) / beta;
        tk = __shfl_sync(0xffffffffu, qt, 0);
        scal = __shfl_sync(0xffffffffu, qt, 1);
      }
      // P(:, k) -= tau v (v^T P(:, k)), v^T P(:, k) = P(pr, k) + scal d_k
#pragma unroll
      for (int u = 0; u < kMaxW / 32; ++u) {
        const int k = lane + 32 * u;
        if (lane < pl && k < nk) cf[k] = tk != 0.0 ? -tk * fma(scal, d[u], piv[q * kMaxW + k]) : 0.0;
      }
      if (lane == 0) {
        scl[t] = scal;
        bet[t] = beta;
        if (c == 0) a.tau[RBCK(t, a.ntau, a.err)] = tk;
      }
    }
    __syncthreads();
    const double sc = scl[t];
    for (int k = 1 + warp / wps; k < nk; k += kQrW / wps) {
      double* pk = Ps + (t + k) * ld;
      const double g = cf[k], gs = g * sc;
#pragma unroll 4
      for (int rl = rb + sub * 32 + lane; rl < nr; rl += 32 * wps) pk[rl] = fma(gs, ct[rl], pk[rl]);
      if (sub == 0 && lane == 0 && prl >= 0 && prl < nr) pk[prl] += g;
    }
    __syncthreads();
  }
  // the factored panel (unscaled columns and pivots until here), the new columns
  // of V (values and digits)
  for (int t = warp; t < w; t += kQrW) {
    const int pr = a.pv0 + t;
    const bool ref = t < a.wp;
    const double sc = ref ? scl[t] : 1.0;
    for (int rl = lane; rl < nr; rl += 32) {
      const int r = ra + rl;
      double x = Ps[t * ld + rl];
      if (ref && r > pr) x = sc != 0.0 ? x * sc : x;
      if (ref && r == pr) x = bet[t];
      Pg[Gi(rl + (long long)t * a.ldp)] = x;
      if (!ref) continue;
      const double v = r < pr ? 0.0 : (r == pr ? 1.0 : x);
      a.V[RBCK((size_t)r + (size_t)(a.j + t) * a.ldv, a.nv, a.err)] = v;
      if (v != 0.0) put_digits_v(a.vcol, a.j + t, r, v, a.err);
    }
  }
}

// New columns of Y and T after a mini-block with reflectors j .. j + wp - 1,
// V_s.  T's recursion, T^{-1} = striu(V^T V) + diag(1 / tau), makes both the same
// forward substitution by rows: with S = V^T V_s,
//   u_t = x_t - sum_{i < j} F(e, i) S(i, t),  f_t = tau_t (u_t - sum_{q < t} f_q S(j + q, t)),
// F = Y and x = A V_s for a row of Y, F = T and x_t = (t == e - j) for row e of T.
// A V_s and S arrive as `ks` partial sums.  Bound by a thread's latency over the
// j <= 128 columns: 16 rows to a CTA (1 / 16 of wp > 16's share), the threads left
// over split the sum.
struct YfixArgs {
  const double* AV;   // partial q of row e, column t: AV[q * avstride + e + t * ldav]
  long long avstride, ldav;
  const double* S;    // partial q of S(i, t): S[q * sstride + i + t * kBmax]
  long long sstride;
  int ks, rows, j, wp;
  double* Y;
  long long ldy;
  double* T;
  const double* tau;
  size_t nav, ns, ny;
  int* err;
};
__host__ __device__ constexpr int yfix_rows(int wp) { return wp <= 16 ? 16 : 256 / wp; }
constexpr size_t kYfixSmem = sizeof(double) * ((size_t)kBmax * kMaxW + 256);

__global__ void __launch_bounds__(256) yfix_kernel(YfixArgs a) {
  extern __shared__ double ysm[];
  const int tid = threadIdx.x, j = a.j, wp = a.wp, ns = j + wp;
  const int R = yfix_rows(wp), KS = 256 / (R * wp);
  double* Ss = ysm;              // S(i, t) at Ss[i * wp + t], i < j + wp
  double* us = Ss + ns * wp;     // us[(kq * wp + t) * R + rl]
  const int nby = (a.rows + R - 1) / R;
  const bool isT = (int)blockIdx.x >= nby;  // T's rows come after Y's
  const int rl = tid % R, tq = tid / R, tp = tq % wp, kq = tq / wp;
  const int e = ((int)blockIdx.x - (isT ? nby : 0)) * R + rl;
  const bool act = kq < KS && e < (isT ? ns : a.rows);
  double* F = isT ? a.T : a.Y;
  const long long ldf = isT ? kBmax : a.ldy;
  [[maybe_unused]] const size_t nf = isT ? (size_t)kBmax * kBmax : a.ny;
  double u = 0.0;
  if (act) {
    if (isT) u = (kq == 0 && e - j == tp) ? 1.0 : 0.0;
    else
      for (int q = kq; q < a.ks; q += KS) u += a.AV[RBCK((size_t)q * a.avstride + e + (size_t)tp * a.ldav, a.nav, a.err)];
  }
  for (int x = tid; x < ns * wp; x += 256) {
    const int i = x % ns, t = x / ns;
    double v = 0.0;
#pragma unroll 4
    for (int q = 0; q < a.ks; ++q) v += a.S[RBCK((size_t)q * a.sstride + i + (size_t)t * kBmax, a.ns, a.err)];
    Ss[i * wp + t] = v;
  }
  __syncthreads();
  if (act) {
#pragma unroll 8
    for (int i = kq; i < j; i += KS) u = fma(-F[RBCK(e + (size_t)i * ldf, nf, a.err)], Ss[i * wp + tp], u);
    us[tq * R + rl] = u;
  }
  __syncthreads();
  if (act && kq == 0) {
    for (int k = 1; k < KS; ++k) u += us[(k * wp + tp) * R + rl];
  }
  // column q of the row is final after step q; every column after it takes its part
  for (int q = 0; q < wp; ++q) {
    if (act && kq == 0 && tp == q) {
      u *= a.tau[q];
      us[q * R + rl] = u;
    }
    __syncthreads();
    if (act && kq == 0 && tp > q) u = fma(-us[q * R + rl], Ss[(j + q) * wp + tp], u);
  }
  if (act && kq == 0) F[RBCK(e + (size_t)(j + tp) * ldf, nf, a.err)] = u;
}

// Z = T^T W for the trailing columns (W in `ks` partial sums, W(i, c) at
// Wp[i + c * kBmax]) straight into Z's digits: operand row c, K = i, with
// the exponent of column c.
__global__ void __launch_bounds__(256) zmake_kernel(const double* __restrict__ Wp, int ks, long long kstride,
                                                    int jb, int cs, int n, const double* __restrict__ T,
                                                    DigitMat Z, size_t nw, int* err) {
  __shared__ double Ws[kBmax][33];
  __shared__ int Es[32];
  const int tid = threadIdx.x;
  const int cb = cs + blockIdx.x * 32;
  for (int e = tid; e < kBmax * 32; e += 256) {
    const int i = e % kBmax, cl = e / kBmax;
    const int c = cb + cl;
    double v = 0.0;
    if (i < jb && c < n)
      for (int q = 0; q < ks; ++q) v += Wp[RBCK((size_t)q * kstride + i + (size_t)c * kBmax, nw, err)];
    Ws[i][cl] = v;
  }
  __syncthreads();
  const int cl = tid & 31, ig = tid >> 5;
  double zv[kBmax / 8];
#pragma unroll
  for (int q = 0; q < kBmax / 8; ++q) {
    const int i = ig + 8 * q;
    double acc = 0.0;
    if (i < jb)
      for (int k = 0; k <= i; ++k) acc = fma(T[RBCK(k + (size_t)i * kBmax, (size_t)kBmax * kBmax, err)], Ws[k][cl], acc);
    zv[q] = acc;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < kBmax / 8; ++q) Ws[ig + 8 * q][cl] = zv[q];
  __syncthreads();
  if (tid < 32) {
    int mx = 0;
#pragma unroll 8
    for (int i = 0; i < jb; ++i) mx = max(mx, abs_hi(Ws[i][tid]));
    const int E = scale_exp_hi(mx);
    Es[tid] = E;
    if (cb + tid < n) Z.ex[RBCK(cb + tid, (size_t)Z.RT * kTR, err)] = E;
  }
  __syncthreads();
  const int kmax = ((jb + kTK - 1) / kTK) * kTK;
  for (int u = tid; u < 32 * (kBmax / 8); u += 256) {
    const int c2 = u & 31, kg = u >> 5;
    const int c = cb + c2, i0 = kg * 8;
    if (c >= n || i0 >= kmax) continue;
    unsigned short dg[8][kD];
#pragma unroll
    for (int q = 0; q < 8; ++q) digits_of(Ws[i0 + q][c2], Es[c2], dg[q]);
    const size_t off = (size_t)tile_off_kg(c % kTR, i0 % kTK, kTK / 8);
#pragma unroll
    for (int l = 0; l < kD; ++l) {
      uint4 v;
      v.x = (unsigned)dg[0][l] | ((unsigned)dg[1][l] << 16);
      v.y = (unsigned)dg[2][l] | ((unsigned)dg[3][l] << 16);
      v.z = (unsigned)dg[4][l] | ((unsigned)dg[5][l] << 16);
      v.w = (unsigned)dg[6][l] | ((unsigned)dg[7][l] << 16);
      *reinterpret_cast<uint4*>(Z.d + RBCR(tile_index(Z, l, i0 / kTK, c / kTR) + off, 8, Z.nd, err)) = v;
    }
  }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
struct RtcScratch {
  double* E;        // (p + n) x n, leading dimension ldE: C above A
  long long ldE;
  double* V;        // ldv x kBmax
  long long ldv;
  double* T;        // kBmax x kBmax
  double* Y;        // ldE x kBmax
  double* W;        // ksW x (kBmax x n)
  double* AV;       // ksY x (ldE x kMaxW)
  double* Sp;       // ksY x (kBmax x kMaxW): V^T V_s
  double* part;     // G x kPartW
  double* red;      // kRedTotal
  int qrC;          // CTAs of the cluster that factors a panel
  unsigned* bar;    // [0..3]: [2] the error flag; then one arrival counter per panel launch
  int nbar;         // panel-launch counters available
  int panels;       // panel launches so far
  DigitMat erow, ecol, yrow, vrow, vcol, zcol;
  int G;
  size_t nE, nV, nY, nW, nAV, nSp, npart;  // extents in doubles
};

inline long long rup(long long x, long long a) { return (x + a - 1) / a * a; }

size_t digit_bytes(int RT, int KT) { return (size_t)kD * KT * RT * kTileEl * sizeof(unsigned short); }

// Carve (or size, with base == nullptr) the scratch of an n x n reduction.
size_t rtc_layout(int n, int p, unsigned char* base, RtcScratch* S) {
  const int G = std::max(1, num_sms());
  const long long rowsE = (long long)p + n;
  const long long ldE = rup(rowsE, 32), ldv = rup(n, 32);
  const int RTe = 2 * (int)((rowsE + 127) / 128), RTn = 2 * ((n + 127) / 128);
  const int KTn = (n + kTK - 1) / kTK, KTb = kBmax / kTK;
  const int ksW = 8, ksY = 8;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    unsigned char* q = base ? base + off : nullptr;
    off += rup((long long)bytes, 256);
    return q;
  };
  RtcScratch s;
  s.ldE = ldE;
  s.ldv = ldv;
  s.G = G;
  s.nE = (size_t)ldE * n;
  s.nV = (size_t)ldv * kBmax;
  s.nY = (size_t)ldE * kBmax;
  s.nW = (size_t)ksW * kBmax * (size_t)n;
  s.nAV = (size_t)ksY * ldE * kMaxW;
  s.nSp = (size_t)ksY * kBmax * kMaxW;
  s.npart = (size_t)G * kPartW;
  s.E = (double*)take(sizeof(double) * s.nE);
  s.V = (double*)take(sizeof(double) * s.nV);
  s.T = (double*)take(sizeof(double) * kBmax * kBmax);
  s.Y = (double*)take(sizeof(double) * s.nY);
  s.W = (double*)take(sizeof(double) * s.nW);
  s.AV = (double*)take(sizeof(double) * s.nAV);
  s.Sp = (double*)take(sizeof(double) * s.nSp);
  s.part = (double*)take(sizeof(double) * s.npart);
  s.red = (double*)take(sizeof(double) * kRedTotal);
  s.nbar = n + 16;
  s.panels = 0;
  s.bar = (unsigned*)take(16 + sizeof(unsigned) * (size_t)s.nbar);
  auto dm = [&](int RT, int KT, bool ex) {
    DigitMat M;
    M.RT = RT;
    M.KT = KT;
    M.d = (unsigned short*)take(digit_bytes(RT, KT));
    M.nd = digit_bytes(RT, KT) / sizeof(unsigned short);
    M.ex = ex ? (int*)take(sizeof(int) * (size_t)RT * kTR) : nullptr;
    return M;
  };
  s.erow = dm(RTe, KTn, true);
  s.ecol = dm(RTn, KTn, true);
  s.yrow = dm(RTe, KTb, true);
  s.vrow = dm(RTn, KTb, true);
  s.vcol = dm(2, KTn, false);
  s.zcol = dm(RTn, KTb, true);
  if (S) *S = s;
  return off;
}

// rows [r_lo, r_hi) x K [k_lo, k_hi) of src into M (tiles of whole 128-row pairs)
int split_into(const double* src, long long sr, long long sk, int r_lo, int r_hi, int k_lo, int k_hi,
               const DigitMat& M, size_t nsrc, int* err, cudaStream_t st, int wrap = INT_MAX) {
  const size_t nex = (size_t)M.RT * kTR;
  if (r_hi <= r_lo || k_hi <= k_lo) return SSV_OK;
  if (M.ex) {
    SSV_CUDA_TRY(cudaMemsetAsync(M.ex, 0x80, sizeof(int) * (size_t)M.RT * kTR, st));
    // K range of a block: 512, less where the chip would stay idle
    int kchunk = 512;
    const int rblk = (r_hi - r_lo + 63) / 64;
    while (kchunk > 64 && (long long)rblk * ((k_hi - k_lo + kchunk - 1) / kchunk) < 4 * std::max(1, num_sms())) kchunk /= 2;
    dim3 grid((unsigned)rblk, (unsigned)((k_hi - k_lo + kchunk - 1) / kchunk));
    split_exp_kernel<<<grid, 256, 0, st>>>(src, sr, sk, r_lo, r_hi, k_lo, k_hi, kchunk, wrap, M.ex, nsrc, nex, err);
    count_launch();
    SSV_CUDA_TRY(cudaGetLastError());
  }
  const int I0 = 2 * (r_lo / 128), I1 = 2 * ((r_hi + 127) / 128);
  const int J0 = k_lo / kTK, J1 = (k_hi + kTK - 1) / kTK;
  split_dig_kernel<<<dim3((unsigned)(I1 - I0), (unsigned)(J1 - J0)), 256, 0, st>>>(src, sr, sk, r_lo, r_hi, k_lo, k_hi,
                                                                                 wrap, M, I0, J0, nsrc, nex, err);
  count_launch();
  SSV_CUDA_TRY(cudaGetLastError());
  return SSV_OK;
}

template <int NT, int LV>
int gemm_launch(const GArgs& g, cudaStream_t st) {
  using Cfg = GCfg<NT, LV>;
  const int nI = (g.M1 + 127) / 128 - g.M0 / 128 + (g.C2 != nullptr ? 1 : 0);
  const int nN = (g.N1 + NT - 1) / NT - g.N0 / NT;
  if (g.M1 <= g.M0 || g.N1 <= g.N0 || nI <= 0 || nN <= 0) return SSV_OK;
  const long long tiles = (long long)nI * nN * g.ksplit;
  const int grid = (int)std::min<long long>(tiles, std::max(1, num_sms()));
  SSV_CUDA_TRY(cudaFuncSetAttribute(tc_gemm_kernel<NT, LV>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)Cfg::kSmem));
  tc_gemm_kernel<NT, LV><<<grid, kGT, Cfg::kSmem, st>>>(g);
  count_launch();
  SSV_CUDA_TRY(cudaGetLastError());
  return SSV_OK;
}

// the long-K products (A V_s, V^T A): nine levels, N <= 32
int gemm_long(int width, const GArgs& g, cudaStream_t st) {
  if (width <= 16) return gemm_launch<16, 9>(g, st);
  return gemm_launch<32, 9>(g, st);
}

GArgs gemm_args(const DigitMat& A, const DigitMat& B, int J0, int J1, int M0, int M1, int N0, int N1, double* C,
                size_t nc, long long ldc, int sub, const RtcScratch& S) {
  GArgs g;
  g.seg.A = A;
  g.seg.B = B;
  g.seg.J0 = J0;
  g.seg.J1 = J1;
  g.M0 = M0;
  g.M1 = M1;
  g.N0 = N0;
  g.N1 = N1;
  g.roff = 0;
  g.coff = 0;
  g.C = C;
  g.nc = nc;
  g.ldc = ldc;
  g.sub = sub;
  g.ksplit = 1;
  g.kstride = 0;
  g.err = reinterpret_cast<int*>(S.bar + 2);
  return g;
}

// One mini-block: update and QR of the panel, A V_s and V^T V_s on the tensor
// cores, Y's and T's new columns.
int run_panel(RtcScratch& S, int n, int p, double* P, size_t np, long long ldp, int r0, int w, int wp, int pv0,
              int j, int c0, double* tau, size_t ntau, cudaStream_t st) {
  const int L = n - r0;
  int* err = reinterpret_cast<int*>(S.bar + 2);
  if (j > 0) {
    if (S.panels >= S.nbar) return SSV_EINVAL;
    const int G = std::min(S.G, std::max(1, (L + 15) / 16));
    const int rpc = (L + G - 1) / G;
    if ((long long)rpc * w > kPanRowsW) return SSV_ENOTSUP;
    PanArgs a;
    a.P = P;
    a.ldp = ldp;
    a.r0 = r0;
    a.n = n;
    a.w = w;
    a.j = j;
    a.c0 = c0;
    a.V = S.V;
    a.ldv = S.ldv;
    a.T = S.T;
    a.Y = S.Y;
    a.ldy = S.ldE;
    a.yoff = p;
    a.part = S.part;
    a.red = S.red;
    a.bar = S.bar + 4 + S.panels++;
    a.err = err;
    a.np = np;
    a.nv = S.nV;
    a.ny = S.nY;
    a.npart = S.npart;
    size_t smem = sizeof(double) * ((size_t)rpc * w + kPanFixed);
    const size_t rows = sizeof(double) * 2 * (size_t)rpc * j;
    a.staged = smem + rows <= kPanSmem ? 1 : 0;
    if (a.staged) smem += rows;
    SSV_CUDA_TRY(allow_smem(panel_update_kernel, kPanSmem));
    void* args[] = {&a};
    SSV_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)panel_update_kernel, dim3(G), dim3(kPT), args, smem, st));
    count_launch();
  }
  {
    QrArgs a;
    a.P = P;
    a.ldp = ldp;
    a.r0 = r0;
    a.n = n;
    a.w = w;
    a.wp = wp;
    a.pv0 = pv0;
    a.j = j;
    // fewer CTAs where each would have 16 rows or less
    a.cs = S.qrC;
    while (a.cs > 1 && L <= 16 * a.cs) a.cs /= 2;
    const size_t rows = sizeof(double) * (size_t)((L + a.cs - 1) / a.cs) * w;
    a.insm = sizeof(double) * kQrFixed + rows <= kQrSmem ? 1 : 0;
    a.V = S.V;
    a.ldv = S.ldv;
    a.tau = tau;
    a.vcol = S.vcol;
    a.err = err;
    a.np = np;
    a.nv = S.nV;
    a.ntau = ntau;
    SSV_CUDA_TRY(allow_smem(panel_qr_kernel, kQrSmem));
    SSV_CUDA_TRY(launch_cluster(panel_qr_kernel, a.cs, kQrT, a.cs, sizeof(double) * kQrFixed + (a.insm ? rows : 0),
                                st, a));
  }
  // A V_s: every row of E against the new reflectors (rows pv0.. of V_s are nonzero)
  const int KTn = (n + kTK - 1) / kTK;
  const int rowsE = p + n;
  GArgs g = gemm_args(S.erow, S.vcol, pv0 / kTK, KTn, 0, rowsE, j, j + wp, S.AV, S.nAV, S.ldE, 0, S);
  g.coff = -j;
  const int NT = wp <= 16 ? 16 : 32;
  const int nI = (rowsE + 127) / 128 + 1, nN = (j + wp + NT - 1) / NT - j / NT;
  g.ksplit = std::max(1, std::min(8, S.G / std::max(1, nI * nN)));
  g.kstride = S.ldE * kMaxW;
  g.C2 = S.Sp;
  g.nc2 = S.nSp;
  g.kstride2 = (long long)kBmax * kMaxW;
  int rc = gemm_long(wp, g, st);
  if (rc != SSV_OK) return rc;
  YfixArgs y;
  y.AV = S.AV;
  y.avstride = g.kstride;
  y.ldav = S.ldE;
  y.S = S.Sp;
  y.sstride = g.kstride2;
  y.ks = g.ksplit;
  y.rows = rowsE;
  y.j = j;
  y.wp = wp;
  y.Y = S.Y;
  y.ldy = S.ldE;
  y.T = S.T;
  y.tau = tau;
  y.nav = S.nAV;
  y.ns = S.nSp;
  y.ny = S.nY;
  y.err = err;
  const int R = yfix_rows(wp);
  const size_t ysm = sizeof(double) * ((size_t)(j + wp) * wp + 256);
  SSV_CUDA_TRY(allow_smem(yfix_kernel, kYfixSmem));
  yfix_kernel<<<(rowsE + R - 1) / R + (j + wp + R - 1) / R, 256, ysm, st>>>(y);
  count_launch();
  SSV_CUDA_TRY(cudaGetLastError());
  return SSV_OK;
}

// Block end (Algorithm 3): right update, W = V^T A, Z = T^T W, left update.
// Rows [0, p + r0) take the right update from column tc0, rows [p + r0, p + n)
// from column cs; the left update covers rows r0.. and columns cs...
int run_block_end(const RtcScratch& S, int n, int p, int r0, int tc0, int cs, int jb, cudaStream_t st) {
  const int rowsE = p + n;
  const int KTn = (n + kTK - 1) / kTK, KTj = (jb + kTK - 1) / kTK;
  int* err = reinterpret_cast<int*>(S.bar + 2);
  int rc = split_into(S.Y, 1, S.ldE, 0, rowsE, 0, jb, S.yrow, S.nY, err, st);
  // V by rows, each with its own exponent (a row of V across the block's
  // reflectors is mostly far below the unit pivots)
  if (rc == SSV_OK) rc = split_into(S.V, 1, S.ldv, 0, n, 0, jb, S.vrow, S.nV, err, st);
  if (rc != SSV_OK) return rc;
  if (tc0 == cs) {
    rc = gemm_launch<64, 8>(gemm_args(S.yrow, S.vrow, 0, KTj, 0, rowsE, cs, n, S.E, S.nE, S.ldE, 1, S), st);
  } else {
    rc = gemm_launch<64, 8>(gemm_args(S.yrow, S.vrow, 0, KTj, 0, p + r0, tc0, n, S.E, S.nE, S.ldE, 1, S), st);
    if (rc == SSV_OK)
      rc = gemm_launch<64, 8>(gemm_args(S.yrow, S.vrow, 0, KTj, p + r0, rowsE, cs, n, S.E, S.nE, S.ldE, 1, S), st);
  }
  if (rc != SSV_OK || cs >= n) return rc;
  rc = split_into(S.E + p, S.ldE, 1, cs, n, r0, n, S.ecol, S.nE - p, err, st);
  if (rc != SSV_OK) return rc;
  GArgs g = gemm_args(S.vcol, S.ecol, r0 / kTK, KTn, 0, jb, cs, n, S.W, S.nW, kBmax, 0, S);
  const int nN = (n + 31) / 32 - cs / 32;
  g.ksplit = std::max(1, std::min(8, S.G / std::max(1, nN)));
  g.kstride = (long long)kBmax * n;
  rc = gemm_launch<32, 9>(g, st);
  if (rc != SSV_OK) return rc;
  zmake_kernel<<<(n - cs + 31) / 32, 256, 0, st>>>(S.W, g.ksplit, g.kstride, jb, cs, n, S.T, S.zcol, S.nW, err);
  count_launch();
  SSV_CUDA_TRY(cudaGetLastError());
  GArgs gl = gemm_args(S.vrow, S.zcol, 0, KTj, r0, n, cs, n, S.E, S.nE, S.ldE, 1, S);
  gl.roff = p;
  return gemm_launch<64, 8>(gl, st);
}

#ifdef SSV_BOUNDS_CHECK
// bit 4 of the error word when a byte of the canary after the scratch changed
__global__ void rtc_canary_kernel(const unsigned char* c, size_t nbytes, int* err) {
  for (size_t i = threadIdx.x; i < nbytes; i += blockDim.x)
    if (c[i] != 0xA5) atomicOr(err, 4);
}
#endif

// CTAs of the panel's cluster: 16 where the chip can hold such a cluster, else the
// portable 8
int qr_cluster() {
  int nc = 0;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kQrC;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(kQrC);
  cfg.blockDim = dim3(kQrT);
  cfg.dynamicSmemBytes = kQrSmem;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (allow_smem(panel_qr_kernel, kQrSmem) == cudaSuccess &&
      cudaFuncSetAttribute(panel_qr_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
      cudaOccupancyMaxActiveClusters(&nc, panel_qr_kernel, &cfg) == cudaSuccess && nc > 0)
    return kQrC;
  (void)cudaGetLastError();
  return 8;
}

int clear_block(const RtcScratch& S, int n, cudaStream_t st) {
  SSV_CUDA_TRY(cudaMemsetAsync(S.V, 0, sizeof(double) * S.ldv * kBmax, st));
  SSV_CUDA_TRY(cudaMemsetAsync(S.T, 0, sizeof(double) * kBmax * kBmax, st));
  SSV_CUDA_TRY(cudaMemsetAsync(S.vcol.d, 0, digit_bytes(S.vcol.RT, S.vcol.KT), st));
  (void)n;
  return SSV_OK;
}

}  // namespace

bool reduce_tc_supported(int n, int m) {
  if (m < 1 || m > kMaxW || n < 2) return false;
  const int G = std::max(1, num_sms());
  return (long long)((n + G - 1) / G) * m <= kPanRowsW;
}

size_t reduce_tc_scratch_bytes(int n, int p) { return rtc_layout(n, p, nullptr, nullptr); }

int reduce_tc(Handle* h, cudaStream_t st) {
  const int n = h->n, m = h->m, p = h->p;
  h->kb = std::min(m, n - 1);
  h->ka = std::max(0, n - m - 1);
  if (h->kb <= 0 && h->ka <= 0) return SSV_OK;
  if (!reduce_tc_supported(n, m)) return SSV_ENOTSUP;
  const int ldct = p > 0 ? p : 1;
  const size_t bytes = rtc_layout(n, p, nullptr, nullptr);
#ifdef SSV_BOUNDS_CHECK
  constexpr size_t kCanary = 256;  // checked at the end
#else
  constexpr size_t kCanary = 0;
#endif
  unsigned char* base = nullptr;
  SSV_CUDA_TRY(pool_alloc((void**)&base, bytes + kCanary, st));
  RtcScratch S;
  rtc_layout(n, p, base, &S);
  S.qrC = qr_cluster();
  int* err = reinterpret_cast<int*>(S.bar + 2);
  int rc = SSV_OK;
  auto step = [&](int r) {
    if (rc == SSV_OK) rc = r;
  };
  auto cu = [&](cudaError_t e) {
    if (rc == SSV_OK && e != cudaSuccess) {
      set_cuda_error(e);
      rc = e == cudaErrorMemoryAllocation ? SSV_ENOMEM : SSV_ECUDA;
    }
  };
#ifdef SSV_BOUNDS_CHECK
  // scratch read before it is written shows up as NaN (0xFF bytes), the canary
  // after the scratch as a changed byte
  cu(cudaMemsetAsync(base, 0xFF, bytes, st));
  cu(cudaMemsetAsync(base + bytes, 0xA5, kCanary, st));
#endif
  cu(cudaMemsetAsync(S.bar, 0, 16 + sizeof(unsigned) * (size_t)S.nbar, st));
  if (p > 0)
    cu(cudaMemcpy2DAsync(S.E, sizeof(double) * S.ldE, h->Ct, sizeof(double) * ldct, sizeof(double) * p, n,
                         cudaMemcpyDeviceToDevice, st));
  cu(cudaMemcpy2DAsync(S.E + p, sizeof(double) * S.ldE, h->H, sizeof(double) * n, sizeof(double) * n, n,
                       cudaMemcpyDeviceToDevice, st));
  // Step 1: the QR of B, applied to A from both sides and to C from the right
  if (h->kb > 0) {
    step(clear_block(S, n, st));
    step(split_into(S.E, 1, S.ldE, 0, p + n, 0, n, S.erow, S.nE, err, st));
    if (rc == SSV_OK)
      step(run_panel(S, n, p, h->R, (size_t)n * m, n, 0, m, h->kb, 0, 0, 0, h->tauB, (size_t)h->kb, st));
    if (rc == SSV_OK) step(run_block_end(S, n, p, 0, 0, 0, h->kb, st));
  }
  // Steps 2-3: the m-Hessenberg reduction of A, blocks of b = floor(128 / m) m columns
  const int b = (kBmax / m) * m;
  for (int z = 0; z < h->ka && rc == SSV_OK; z += b) {
    const int jb = std::min(b, h->ka - z);
    const int r0 = z + m;
    step(clear_block(S, n, st));
    step(split_into(S.E, 1, S.ldE, 0, p + n, r0, n, S.erow, S.nE, err, st));
    for (int j = 0; j < jb && rc == SSV_OK; j += m) {
      const int w = std::min(m, jb - j);
      const int c0 = z + j;
      const size_t off = (size_t)p + (size_t)c0 * S.ldE;
      step(run_panel(S, n, p, S.E + off, S.nE - off, S.ldE, r0, w, w, c0 + m, j, c0, h->tauA + c0,
                     (size_t)(h->ka - c0), st));
    }
    if (rc == SSV_OK) step(run_block_end(S, n, p, r0, r0, z + jb, jb, st));
  }
  cu(cudaMemcpy2DAsync(h->H, sizeof(double) * n, S.E + p, sizeof(double) * S.ldE, sizeof(double) * n, n,
                       cudaMemcpyDeviceToDevice, st));
  if (p > 0)
    cu(cudaMemcpy2DAsync(h->Ct, sizeof(double) * ldct, S.E, sizeof(double) * S.ldE, sizeof(double) * p, n,
                         cudaMemcpyDeviceToDevice, st));
#ifdef SSV_BOUNDS_CHECK
  if (rc == SSV_OK) {
    rtc_canary_kernel<<<1, 256, 0, st>>>(base + bytes, kCanary, err);
    count_launch();
    cu(cudaGetLastError());
  }
#endif
  int herr = 0;
  cu(cudaMemcpyAsync(&herr, S.bar + 2, sizeof(int), cudaMemcpyDeviceToHost, st));
  cu(cudaStreamSynchronize(st));
  // bit 1: a wait gave up; bits 2 and 4 (debug builds): an index out of range,
  // a changed canary
  if (rc == SSV_OK && (herr & 1)) rc = SSV_ETIMEOUT;
  else if (rc == SSV_OK && herr != 0) rc = SSV_ECUDA;
  cudaError_t e2 = cudaFreeAsync(base, st);
  if (e2 != cudaSuccess && rc == SSV_OK) {
    set_cuda_error(e2);
    rc = SSV_ECUDA;
  }
  return rc;
}


// ---------------------------------------------------------------------------
// X <- Q X for many columns: the reflectors in blocks of kBmax, Q_b = I - V T V^T,
// with W = V^T X and X -= V Z as digit products.  Z = T W is a triangular solve,
// T^{-1} = striu(V^T V) + diag(1 / tau) (Joffrain, Low, Quintana-Orti, van de
// Geijn and Van Zee 2006), so no T is formed.  X enters as its real form, the
// real parts of all columns, then the imaginary parts.
// ---------------------------------------------------------------------------
namespace {

// V(r, k), explicit zeros and unit pivots, of reflectors 0 .. cnt - 1 with pivot
// rows pv + k, from their packed storage; rows r0 .. n - 1, columns 0 .. kBmax - 1
__global__ void __launch_bounds__(256) qv_kernel(const double* __restrict__ src, int n, int r0, int pv, int cnt,
                                                 double* __restrict__ V, long long ldv, size_t nsrc, size_t nv,
                                                 int* err) {
  const int r = r0 + blockIdx.x * 256 + threadIdx.x, k = blockIdx.y;
  if (r >= n) return;
  const int d = r - pv - k;
  V[RBCK(r + (size_t)k * ldv, nv, err)] = (k >= cnt || d < 0) ? 0.0
                                          : d == 0            ? 1.0
                                                              : src[RBCK(r + (size_t)k * n, nsrc, err)];
}

constexpr int kQCols = 1024;  // complex columns at a time (bounds the digit scratch)
constexpr int kQSplit = 7;    // partial sums of V^T V at most

// S = V^T V from its partial sums, row i scaled by tau_i: a step of the back
// substitution is then a broadcast and a multiply-add
__global__ void __launch_bounds__(256) qs_kernel(const double* __restrict__ Sp, int kss, int cnt,
                                                 const double* __restrict__ tau, double* __restrict__ S, size_t ns,
                                                 size_t ntau, int* err) {
  const int e = blockIdx.x * 256 + threadIdx.x, i = e % kBmax;
  double v[kQSplit];
#pragma unroll
  for (int q = 0; q < kQSplit; ++q) v[q] = q < kss ? Sp[RBCK((size_t)q * kBmax * kBmax + e, ns, err)] : 0.0;
#pragma unroll
  for (int q = 1; q < kQSplit; ++q) v[0] += v[q];
  S[RBCK(e, (size_t)kBmax * kBmax, err)] = i < cnt ? v[0] * __ldg(tau + RBCK(i, ntau, err)) : 0.0;
}

// Z = T W for 8 real columns per CTA, a warp each: lane l holds the rows l, l +
// 32, ..; back substitution from the last reflector, then Z's digits with the
// column's exponent.  W arrives as partial sums.  Bound by the FP64 pipe: 2.5
// instructions of 64 clocks a step on average, two warps to a scheduler (900
// columns: 27 us; with every CTA adding S's partial sums itself 69).
__global__ void __launch_bounds__(256) qz_kernel(const double* __restrict__ Wp, int ksw, long long wstride,
                                                 const double* __restrict__ Sg, int cnt, int ncol,
                                                 const double* __restrict__ tau, DigitMat Z, size_t nw, size_t ntau,
                                                 int* err) {
  extern __shared__ double S[];  // kBmax x kBmax
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
#pragma unroll 8
  for (int e = 2 * tid; e < kBmax * kBmax; e += 512)
    *reinterpret_cast<double2*>(S + e) = *reinterpret_cast<const double2*>(Sg + e);
  __syncthreads();
  const int c = blockIdx.x * 8 + warp;
  if (c >= ncol) return;
  double w[kBmax / 32];
#pragma unroll
  for (int u = 0; u < kBmax / 32; ++u) {
    const int i = lane + 32 * u;
    double v = 0.0;
    if (i < cnt) {
      for (int q = 0; q < ksw; ++q) v += Wp[RBCK((size_t)q * wstride + i + (size_t)c * kBmax, nw, err)];
      v *= __ldg(tau + RBCK(i, ntau, err));
    }
    w[u] = v;
  }
  // z_k = w_k, final once the steps after it have taken their part
#pragma unroll
  for (int uk = kBmax / 32 - 1; uk >= 0; --uk) {
    for (int lk = 31; lk >= 0; --lk) {
      const int k = 32 * uk + lk;
      if (k >= cnt) continue;
      const double z = __shfl_sync(0xffffffffu, w[uk], lk);
#pragma unroll
      for (int u = 0; u <= uk; ++u) {
        const double f = fma(-S[lane + 32 * u + k * kBmax], z, w[u]);
        if (u < uk || lane < lk) w[u] = f;
      }
    }
  }
  int mx = 0;
#pragma unroll
  for (int u = 0; u < kBmax / 32; ++u) mx = max(mx, abs_hi(w[u]));
  mx = __reduce_max_sync(0xffffffffu, mx);
  const int E = scale_exp_hi(mx);
  if (lane == 0) Z.ex[RBCK(c, (size_t)Z.RT * kTR, err)] = E;
#pragma unroll
  for (int u = 0; u < kBmax / 32; ++u) {
    unsigned short d[kD];
    digits_of(w[u], E, d);
    const size_t off = (size_t)tile_off_kg(c % kTR, lane, kTK / 8);
#pragma unroll
    for (int l = 0; l < kD; ++l) Z.d[RBCK(tile_index(Z, l, u, c / kTR) + off, Z.nd, err)] = d[l];
  }
}

// when a wait gave up: every entry NaN, and the shifts (m columns each) so reported
__global__ void q_fail_kernel(const int* err, cd* X, long long ldx, int n, int ncols, int m, int* status,
                              double* resid) {
  if (*err == 0) return;
  const double nanv = __longlong_as_double(0x7ff8000000000000LL);
  for (int sh = blockIdx.x * blockDim.x + threadIdx.x; sh < ncols / m; sh += gridDim.x * blockDim.x) {
    if (status != nullptr && status[sh] == SSV_SHIFT_OK) status[sh] = SSV_SHIFT_NONFINITE;
    if (resid != nullptr) resid[sh] = nanv;
  }
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < (long long)n * ncols;
       e += (long long)gridDim.x * blockDim.x)
    X[e % n + (size_t)(e / n) * ldx] = mkcd(nanv, nanv);
}


struct QtcScratch {
  double *V, *W, *S;
  long long ldv;
  DigitMat vrow, vcol, xcol, zcol;
  int* err;
  size_t nV, nW;
};

size_t qtc_layout(int n, int nc, unsigned char* base, QtcScratch* Q) {
  size_t off = 0;
  auto take = [&](size_t bytes) {
    unsigned char* q = base ? base + off : nullptr;
    off += rup((long long)bytes, 256);
    return q;
  };
  QtcScratch s;
  const int RTn = 2 * ((n + 127) / 128), KTn = (n + kTK - 1) / kTK, KTb = kBmax / kTK;
  const int RTc = 2 * ((2 * nc + 127) / 128);
  s.ldv = rup(n, 32);
  s.nV = (size_t)s.ldv * kBmax;
  s.nW = (size_t)8 * kBmax * 2 * nc;
  s.V = (double*)take(sizeof(double) * s.nV);
  s.W = (double*)take(sizeof(double) * s.nW);
  s.S = (double*)take(sizeof(double) * 8 * kBmax * kBmax);
  s.err = (int*)take(sizeof(int));
  auto dm = [&](int RT, int KT, bool ex) {
    DigitMat M;
    M.RT = RT;
    M.KT = KT;
    M.nd = digit_bytes(RT, KT) / sizeof(unsigned short);
    M.d = (unsigned short*)take(digit_bytes(RT, KT));
    M.ex = ex ? (int*)take(sizeof(int) * (size_t)RT * kTR) : nullptr;
    return M;
  };
  s.vrow = dm(RTn, KTb, true);
  s.vcol = dm(2, KTn, false);
  s.xcol = dm(RTc, KTn, true);
  s.zcol = dm(RTc, KTb, true);
  if (Q) *Q = s;
  return off;
}

}  // namespace

// Where the digit products take over from the FP64 pipe (mode X of the precisions
// below FP64): that path grows with n^2 ncols, this one up to some 256 columns with
// the number of blocks alone (150 us each).  FP64 / digit products in ms, along the
// line (n ncols = 180000): n = 256 0.50 / 0.44, 384 0.61 / 0.52, 768 1.20 / 0.92, 1200
// 2.00 / 1.58, 2048 5.09 / 2.44, 4096 12.5 / 5.12; far above it: n = 4096, 640 columns
// 80.7 / 8.9.  Below it the sides cross: n = 512, 256 columns 0.62 / 0.65 and n = 256,
// 450 columns 0.28 / 0.39, but n = 2048, 64 columns 2.98 / 2.42, so the product of the
// two does not part them there; such X stays on the FP64 pipe, which keeps every
// entry's accuracy.
bool apply_q_tc_supported(int n, int ncols) { return n >= 256 && (long long)n * ncols >= 180000; }

size_t apply_q_tc_scratch_bytes(int n, int ncols) {
  return apply_q_tc_supported(n, ncols) ? qtc_layout(n, std::min(ncols, kQCols), nullptr, nullptr) : 0;
}

int apply_q_tc(const Handle* h, int ncols, cd* X, long long ldX, cudaStream_t st, int* status, double* resid,
               int err0) {
  const int n = h->n, m = h->m, sms = std::max(1, num_sms());
  const int ncm = std::min(ncols, kQCols);
  unsigned char* base = nullptr;
  const size_t bytes = qtc_layout(n, ncm, nullptr, nullptr);
#ifdef SSV_BOUNDS_CHECK
  constexpr size_t kCanary = 256;  // checked at the end
#else
  constexpr size_t kCanary = 0;
#endif
  SSV_CUDA_TRY(pool_alloc((void**)&base, bytes + kCanary, st));
  QtcScratch Q;
  qtc_layout(n, ncm, base, &Q);
  int rc = SSV_OK;
  auto step = [&](int r) {
    if (rc == SSV_OK) rc = r;
  };
  auto cu = [&](cudaError_t e) {
    if (rc == SSV_OK && e != cudaSuccess) {
      set_cuda_error(e);
      rc = SSV_ECUDA;
    }
  };
#ifdef SSV_BOUNDS_CHECK
  cu(cudaMemsetAsync(base, 0xFF, bytes, st));
  cu(cudaMemsetAsync(base + bytes, 0xA5, kCanary, st));
#endif
  cu(cudaMemsetAsync(Q.err, err0, sizeof(int), st));
  cu(cudaFuncSetAttribute(qz_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                          (int)(sizeof(double) * kBmax * kBmax)));
  const int nbA = (h->ka + kBmax - 1) / kBmax, nbB = (h->kb + kBmax - 1) / kBmax;
  const int KTn = (n + kTK - 1) / kTK;
  auto args = [&](const DigitMat& A, const DigitMat& B, int J0, int J1, int M0, int M1, int N1, double* C, size_t nc,
                  long long ldc) {
    GArgs g;
    g.seg = GSeg{A, B, J0, J1};
    g.M0 = M0; g.M1 = M1; g.N0 = 0; g.N1 = N1;
    g.roff = 0; g.coff = 0;
    g.C = C; g.nc = nc; g.ldc = ldc;
    g.sub = 0; g.ksplit = 1; g.kstride = 0;
    g.err = Q.err;
    return g;
  };
  for (int b = nbA + nbB - 1; b >= 0 && rc == SSV_OK; --b) {
    const bool isA = b >= nbB;
    const int j = (isA ? b - nbB : b) * kBmax;
    const int cnt = std::min(kBmax, (isA ? h->ka : h->kb) - j), pv = isA ? m + j : j;
    const double* src = isA ? h->H + (size_t)j * n : h->R + (size_t)j * n;
    const double* tau = isA ? h->tauA + j : h->tauB + j;
    const size_t nsrc = (size_t)n * ((isA ? n : m) - j), ntau = (size_t)(isA ? n : m) - j;
    qv_kernel<<<dim3((unsigned)((n - pv + 255) / 256), kBmax), 256, 0, st>>>(src, n, pv, pv, cnt, Q.V, Q.ldv,
                                                                                      nsrc, Q.nV, Q.err);
    count_launch();
    cu(cudaGetLastError());
    step(split_into(Q.V, 1, Q.ldv, pv, n, 0, cnt, Q.vrow, Q.nV, Q.err, st));
    step(split_into(Q.V, Q.ldv, 1, 0, cnt, pv, n, Q.vcol, Q.nV, Q.err, st));
    // S = V^T V
    const int J0 = pv / kTK, nst = KTn - J0;
    GArgs gs = args(Q.vcol, Q.vcol, J0, KTn, 0, cnt, cnt, Q.S, (size_t)8 * kBmax * kBmax, kBmax);
    gs.ksplit = std::max(1, std::min(kQSplit, nst / 4));
    gs.kstride = (long long)kBmax * kBmax;
    if (rc == SSV_OK) step(gemm_launch<32, 9>(gs, st));
    double* S1 = Q.S + (size_t)kQSplit * kBmax * kBmax;
    qs_kernel<<<kBmax * kBmax / 256, 256, 0, st>>>(Q.S, gs.ksplit, cnt, tau, S1, (size_t)8 * kBmax * kBmax,
                                                         ntau, Q.err);
    count_launch();
    cu(cudaGetLastError());
    for (int c0 = 0; c0 < ncols && rc == SSV_OK; c0 += ncm) {
      const int nc = std::min(ncm, ncols - c0);
      double* Xd = reinterpret_cast<double*>(X + (size_t)c0 * ldX);
      const size_t nX = 2 * ((size_t)ldX * (nc - 1) + n);
      step(split_into(Xd, 2 * ldX, 2, 0, 2 * nc, pv, n, Q.xcol, nX, Q.err, st, nc));
      GArgs gw = args(Q.vcol, Q.xcol, J0, KTn, 0, cnt, 2 * nc, Q.W, Q.nW, kBmax);
      const int nN = (2 * nc + 31) / 32;
      gw.ksplit = std::max(1, std::min({8, sms / nN, std::max(1, nst / 4)}));
      gw.kstride = (long long)kBmax * 2 * nc;
      if (rc == SSV_OK) step(gemm_launch<32, 9>(gw, st));
      qz_kernel<<<(2 * nc + 7) / 8, 256, sizeof(double) * kBmax * kBmax, st>>>(
          Q.W, gw.ksplit, gw.kstride, S1, cnt, 2 * nc, tau, Q.zcol, Q.nW, ntau, Q.err);
      count_launch();
      cu(cudaGetLastError());
      GArgs gx = args(Q.vrow, Q.zcol, 0, (cnt + kTK - 1) / kTK, pv, n, 2 * nc, Xd, nX, 2 * ldX);
      gx.sub = 1;
      gx.rs = 2;
      gx.wrap = nc;
      // nine levels: the pairs eight leave out all have the sign of the product,
      // and X lost 1e-15 of its norm over 1000 reflectors (2e-16 with nine)
      if (rc == SSV_OK) step(gemm_launch<32, 9>(gx, st));
    }
  }
#ifdef SSV_BOUNDS_CHECK
  if (rc == SSV_OK) {
    rtc_canary_kernel<<<1, 256, 0, st>>>(base + bytes, kCanary, Q.err);
    count_launch();
    cu(cudaGetLastError());
  }
#endif
  if (rc == SSV_OK) {
    q_fail_kernel<<<256, 256, 0, st>>>(Q.err, X, ldX, n, ncols, m, status, resid);
    count_launch();
    cu(cudaGetLastError());
  }
  if (rc == SSV_ENOMEM) rc = SSV_ECUDA;  // X may have changed: not for another path to redo
  cudaError_t e2 = cudaFreeAsync(base, st);
  if (e2 != cudaSuccess && rc == SSV_OK) {
    set_cuda_error(e2);
    rc = SSV_ECUDA;
  }
  return rc;
}

}  // namespace ssv
