// FP64 and double-float solves of one system (ssv_solve, ssv_solve_rhs, the
// masked re-solve of the mixed path, ssv_solve_noalloc) and the n_b autotuner.
#include "sweep.cuh"

namespace ssv {

namespace {

template <int MAXM, bool DF = false>
__global__ void __launch_bounds__(sweep_threads<MAXM>(), sweep_per_sm(MAXM, DF)) solve_fp64_kernel(
    int n, int m, int p, int nb, const double* __restrict__ H, const double* __restrict__ Ct,
    int ldct, const double* __restrict__ R, int s, const cd* __restrict__ shifts, int mode,
    cd* scratch, size_t slot_stride, cd* __restrict__ out, long long ldo,
    int* __restrict__ status, cd* __restrict__ xhat_copy, long long ldxc,
    const double* __restrict__ hnorm, const int* __restrict__ list,
    const int* __restrict__ count, const cd* __restrict__ bhat, long long ldb,
    const float* __restrict__ Hhi, const float* __restrict__ Hlo, int team) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_piv;
  __shared__ int s_sing;
  FpSys d;
  d.n = n; d.m = m; d.p = p; d.nb = nb; d.mode = mode; d.H = H; d.Ct = Ct; d.ldct = ldct;
  d.R = R; d.shifts = shifts; d.out = out; d.ldo = ldo; d.status = status;
  d.xhat_copy = xhat_copy; d.ldxc = ldxc; d.hnorm = hnorm; d.bhat = bhat; d.ldb = ldb;
  d.rhs = nullptr; d.ldr = 0; d.flip_out = 0;
  d.Hhi = Hhi; d.Hlo = Hlo;
  d.gfull = GivensSched{nullptr, nullptr, 0};
  d.gtail = d.gfull;
  // team: CTAs of a cluster per shift (fp64_shift)
  const int rank = team > 1 ? cluster_rank() : 0, g = blockIdx.x / team, G = gridDim.x / team;
  cd* Z2 = scratch + (size_t)g * slot_stride;
  // With a work list, the team takes list entries g, g + G, ...
  const int nwork = list != nullptr ? *count : s;
  for (int w = g; w < nwork; w += G) {
    const int sh = list != nullptr ? list[w] : w;
    fp64_shift<MAXM, sweep_threads<MAXM>(), false, false, DF>(d, sh, Z2, smem_raw, &s_piv, &s_sing, team, rank);
  }
}

template <int MAXM, bool DF = false>
int launch_solve(const Handle* h, int s, const double* shifts, int nb, int mode, double* out,
                 long long ldo, int* status, cd* xhat_copy, long long ldxc, cudaStream_t st,
                 const int* list = nullptr, const int* count = nullptr,
                 const cd* bhat = nullptr, long long ldb = 0) {
  using L = Layout<MAXM>;
  const int n = h->n, m = h->m, p = h->p;
  const bool track_t = (mode == SSV_XHAT || mode == SSV_X || xhat_copy != nullptr);
  const size_t slot = (size_t)(p + n) * m + (track_t ? (size_t)n * m : 0);
  int dev = 0;
  SSV_CUDA_TRY(cudaGetDevice(&dev));
  auto kern = solve_fp64_kernel<MAXM, DF>;
  SSV_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::bytes));
  constexpr int NT = sweep_threads<MAXM>();
  int per_sm = 0;
  SSV_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NT, L::bytes));
  per_sm = std::max(1, std::min(per_sm, sweep_per_sm(MAXM, DF)));
  int grid = std::min(s, num_sms() * per_sm);
  cd* scratch = nullptr;
  SSV_CUDA_TRY(pool_alloc((void**)&scratch, sizeof(cd) * slot * grid, st));
  const int team = team_for(s, n, m);
  cudaError_t e = launch_cluster(kern, grid * team, NT, team, L::bytes, st, n, m, p, nb, h->H, h->Ct, p > 0 ? p : 1,
                                 h->R, s, reinterpret_cast<const cd*>(shifts), mode, scratch, slot,
                                 reinterpret_cast<cd*>(out), ldo, status, xhat_copy, ldxc, h->hnorm2, list, count,
                                 bhat, ldb, h->Hhi, h->Hlo, team);
  cudaError_t e2 = cudaFreeAsync(scratch, st);
  if (e == cudaSuccess) e = e2;
  if (e != cudaSuccess) {
    set_cuda_error(e);
    return SSV_ECUDA;
  }
  if (status != nullptr && list == nullptr) {
    int rows = (mode == SSV_G || mode == SSV_TF) ? p : n;
    if (rows > 0) {
      nonfinite_kernel<<<s, 256, 0, st>>>(reinterpret_cast<const cd*>(out), ldo, rows,
                                          bhat != nullptr ? 1 : m, s, status);
      count_launch();
      SSV_CUDA_TRY(cudaGetLastError());
    }
  }
  return SSV_OK;
}

}  // namespace

// Default block width of the FP64 sweep: n_b = 128 halves the per-shift
// Z2 P2 work of n_b = 64 at the price of a longer panel (measured 9 % faster
// at n = 5000, m = 16); small problems keep 64 (n = 1000, FP64, 64 / 128: m = 4 8.67
// / 8.65 ms, m = 16 17.7 / 17.7).  Double-float sweeps keep it too: 128 rows are 3 to
// 8 % faster at n = 256 .. 1000, but sum twice as many products per update, and the
// error of Xhat grows from 1.9e-14 to 3.4e-14 at n = 600, m = 4 and from 2.4e-14 to
// 4.0e-14 at m = 8 (geometric mean over 120 shifts).
int default_nb(int n, int m) {
  (void)m;
  return n >= 1024 ? 128 : 64;
}

// Work list of the shifts with mask[j] != 0 (single block, order preserved).
__global__ void __launch_bounds__(1024) mask_to_list_kernel(int s, const int* __restrict__ mask,
                                                            int* __restrict__ list,
                                                            int* __restrict__ count) {
  __shared__ int part[1024];
  const int tid = threadIdx.x;
  const int chunk = (s + 1023) / 1024;
  const int b = tid * chunk, e = min(s, b + chunk);
  int c = 0;
  for (int j = b; j < e; ++j) c += mask[j] != 0;
  part[tid] = c;
  __syncthreads();
  for (int o = 1; o < 1024; o <<= 1) {
    int v = tid >= o ? part[tid - o] : 0;
    __syncthreads();
    part[tid] += v;
    __syncthreads();
  }
  int pos = part[tid] - c;
  for (int j = b; j < e; ++j)
    if (mask[j] != 0) list[pos++] = j;
  if (tid == 1023) *count = part[1023];
}

int solve_fp64_masked(const Handle* h, int s, const double* shifts, int mode, int nb,
                      double* out, long long ldo, int* status, const int* mask, void* xhat_copy,
                      long long ldxc, cudaStream_t st) {
  const int m = h->m;
  if (nb <= 0) nb = default_nb(h->n, m);
  if (nb > kNB) return SSV_ENOTSUP;
  if (s == 0) return SSV_OK;
  int* list = nullptr;
  SSV_CUDA_TRY(pool_alloc((void**)&list, sizeof(int) * ((size_t)s + 1), st));
  int* count = list + s;
  mask_to_list_kernel<<<1, 1024, 0, st>>>(s, mask, list, count);
  count_launch();
  cd* xc = reinterpret_cast<cd*>(xhat_copy);
  int rc;
  if (m <= 1) rc = launch_solve<1>(h, s, shifts, nb, mode, out, ldo, status, xc, ldxc, st, list, count);
  else if (m <= 2) rc = launch_solve<2>(h, s, shifts, nb, mode, out, ldo, status, xc, ldxc, st, list, count);
  else if (m <= 4) rc = launch_solve<4>(h, s, shifts, nb, mode, out, ldo, status, xc, ldxc, st, list, count);
  else if (m <= 8) rc = launch_solve<8>(h, s, shifts, nb, mode, out, ldo, status, xc, ldxc, st, list, count);
  else if (m <= 16) rc = launch_solve<16>(h, s, shifts, nb, mode, out, ldo, status, xc, ldxc, st, list, count);
  else if (m <= 32) rc = launch_solve<32>(h, s, shifts, nb, mode, out, ldo, status, xc, ldxc, st, list, count);
  else rc = SSV_ENOTSUP;
  cudaError_t e = cudaFreeAsync(list, st);
  if (e != cudaSuccess && rc == SSV_OK) {
    set_cuda_error(e);
    rc = SSV_ECUDA;
  }
  return rc;
}

size_t solve_fp64_scratch_bytes(int n, int m, int p, int s, const ssv_opts* o) {
  const bool track_t = (o->mode == SSV_XHAT || o->mode == SSV_X);
  size_t slot = (size_t)(p + n) * m + (track_t ? (size_t)n * m : 0);
  const size_t grid = (size_t)std::min(s, num_sms() * sweep_per_sm(m_class(m), o->precision == SSV_DFLOAT));
  return sizeof(cd) * slot * grid + 256;
}

int solve_fp64(const Handle* h, int s, const double* shifts, const ssv_opts* o, double* out,
               long long ldo, int* status, double* resid, cudaStream_t st) {
  const int m = h->m;
  int nb = o->nb > 0 ? o->nb : tuned_nb(h->n, m, h->p, o->precision, o->mode);
  if (nb > kNB) return SSV_ENOTSUP;
  if (s == 0) return SSV_OK;
  cd* xcopy = nullptr;
  long long ldxc = 0;
  if (resid != nullptr && (o->mode == SSV_G || o->mode == SSV_TF)) {
    ldxc = h->n;
    SSV_CUDA_TRY(pool_alloc((void**)&xcopy, sizeof(cd) * (size_t)h->n * m * s, st));
  }
  int rc;
  if (o->precision == SSV_DFLOAT) {
    if (m <= 1) rc = launch_solve<1, true>(h, s, shifts, nb, o->mode, out, ldo, status, xcopy, ldxc, st);
    else if (m <= 2) rc = launch_solve<2, true>(h, s, shifts, nb, o->mode, out, ldo, status, xcopy, ldxc, st);
    else if (m <= 4) rc = launch_solve<4, true>(h, s, shifts, nb, o->mode, out, ldo, status, xcopy, ldxc, st);
    else if (m <= 8) rc = launch_solve<8, true>(h, s, shifts, nb, o->mode, out, ldo, status, xcopy, ldxc, st);
    else if (m <= 16) rc = launch_solve<16, true>(h, s, shifts, nb, o->mode, out, ldo, status, xcopy, ldxc, st);
    else if (m <= 32) rc = launch_solve<32, true>(h, s, shifts, nb, o->mode, out, ldo, status, xcopy, ldxc, st);
    else rc = SSV_ENOTSUP;
  } else {
    if (m <= 1) rc = launch_solve<1>(h, s, shifts, nb, o->mode, out, ldo, status, xcopy, ldxc, st);
    else if (m <= 2) rc = launch_solve<2>(h, s, shifts, nb, o->mode, out, ldo, status, xcopy, ldxc, st);
    else if (m <= 4) rc = launch_solve<4>(h, s, shifts, nb, o->mode, out, ldo, status, xcopy, ldxc, st);
    else if (m <= 8) rc = launch_solve<8>(h, s, shifts, nb, o->mode, out, ldo, status, xcopy, ldxc, st);
    else if (m <= 16) rc = launch_solve<16>(h, s, shifts, nb, o->mode, out, ldo, status, xcopy, ldxc, st);
    else if (m <= 32) rc = launch_solve<32>(h, s, shifts, nb, o->mode, out, ldo, status, xcopy, ldxc, st);
    else rc = SSV_ENOTSUP;
  }
  if (rc == SSV_OK && resid != nullptr) {
    const double* xh = xcopy ? reinterpret_cast<const double*>(xcopy) : out;
    long long ldx = xcopy ? ldxc : ldo;
    rc = backward_error_fp64(h, s, shifts, xh, ldx, resid, st);
  }
  if (xcopy) {
    cudaError_t e = cudaFreeAsync(xcopy, st);
    if (e != cudaSuccess && rc == SSV_OK) {
      set_cuda_error(e);
      rc = SSV_ECUDA;
    }
  }
  return rc;
}

// One right-hand side B bhat_l per shift (Sec. 3.3): out column l holds
// Xhat_l bhat_l (SSV_XHAT / SSV_X before the back-transform) or
// +-Ct Xhat_l bhat_l (SSV_G / SSV_TF).
int solve_fp64_rhs(const Handle* h, int s, const double* shifts, const double* bhat,
                   long long ldb, const ssv_opts* o, double* out, long long ldo, int* status,
                   cudaStream_t st) {
  const int m = h->m;
  const int nb = o->nb > 0 ? o->nb : tuned_nb(h->n, m, h->p, SSV_FP64, o->mode);
  if (nb > kNB) return SSV_ENOTSUP;
  if (s == 0) return SSV_OK;
  const int mode = o->mode == SSV_X ? SSV_XHAT : o->mode;
  const cd* b = reinterpret_cast<const cd*>(bhat);
  if (m <= 1) return launch_solve<1>(h, s, shifts, nb, mode, out, ldo, status, nullptr, 0, st, nullptr, nullptr, b, ldb);
  if (m <= 2) return launch_solve<2>(h, s, shifts, nb, mode, out, ldo, status, nullptr, 0, st, nullptr, nullptr, b, ldb);
  if (m <= 4) return launch_solve<4>(h, s, shifts, nb, mode, out, ldo, status, nullptr, 0, st, nullptr, nullptr, b, ldb);
  if (m <= 8) return launch_solve<8>(h, s, shifts, nb, mode, out, ldo, status, nullptr, 0, st, nullptr, nullptr, b, ldb);
  if (m <= 16) return launch_solve<16>(h, s, shifts, nb, mode, out, ldo, status, nullptr, 0, st, nullptr, nullptr, b, ldb);
  if (m <= 32) return launch_solve<32>(h, s, shifts, nb, mode, out, ldo, status, nullptr, 0, st, nullptr, nullptr, b, ldb);
  return SSV_ENOTSUP;
}

// ---------------------------------------------------------------------------
// Allocation-free variant of the FP64 solve (ssv_solve_noalloc).
//
// Some callers cannot allocate device memory at the point where they need a
// solve: code that runs while another component owns the allocator (a custom
// pool or a framework that forbids cudaMalloc / cudaMallocAsync inside its
// step), processes with a hard device-memory budget that was fixed up front,
// or real-time loops where an allocation's latency or failure is not
// acceptable.  For them the per-thread-block window state lives in one
// fixed array that is part of the loaded library image, so the call itself
// allocates nothing: no cudaMalloc / cudaMallocAsync / cudaFree and no
// allocating library routine.
//
// The array below holds kNoAllocScratchBytes (64 MiB) on every GPU where this
// translation unit's module is loaded, for as long as the process lives: any
// FP64 or double-float solve loads the module, so the 64 MiB is taken by
// those callers too, not only by callers of ssv_solve_noalloc.  In host code
// the array's name is only a host-side stand-in, so the device address is
// looked up once per device with cudaGetSymbolAddress (with that device
// current) and cached; the first call on each device performs that lookup,
// which under lazy module loading may itself load the module (an implicit
// device allocation).
// ---------------------------------------------------------------------------
constexpr size_t kNoAllocScratchBytes = size_t(64) << 20;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

namespace {
constexpr int kMaxDevices = 64;
void* g_noalloc_addr[kMaxDevices] = {nullptr};

int noalloc_scratch_address(void** out) {
  int dev = 0;
  SSV_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return SSV_ENOTSUP;
  if (g_noalloc_addr[dev] == nullptr) {
    void* ptr = nullptr;
    SSV_CUDA_TRY(cudaGetSymbolAddress(&ptr, g_noalloc_scratch));
    g_noalloc_addr[dev] = ptr;
  }
  *out = g_noalloc_addr[dev];
  return SSV_OK;
}

template <int MAXM>
int launch_solve_noalloc(const Handle* h, int s, const double* shifts, int nb, int mode,
                         double* out, long long ldo, int* status, cudaStream_t st) {
  using L = Layout<MAXM>;
  const int n = h->n, m = h->m, p = h->p;
  const bool track_t = (mode == SSV_XHAT);
  const size_t slot = (size_t)(p + n) * m + (track_t ? (size_t)n * m : 0);
  const size_t max_slots = kNoAllocScratchBytes / (sizeof(cd) * slot);
  if (max_slots < 1) return SSV_ESCRATCH;
  void* base = nullptr;
  int rc = noalloc_scratch_address(&base);
  if (rc != SSV_OK) return rc;
  auto kern = solve_fp64_kernel<MAXM>;
  SSV_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::bytes));
  int per_sm = 0;
  constexpr int NT = sweep_threads<MAXM>();
  SSV_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NT, L::bytes));
  per_sm = std::max(1, std::min(per_sm, sweep_per_sm(MAXM, false)));
  const int grid = (int)std::min<size_t>((size_t)std::min(s, num_sms() * per_sm), max_slots);
  // Every window entry the kernel reads is written earlier in the same call
  // (the shift setup overwrites the whole slot), so nothing left in the array
  // by a previous call needs clearing.
  kern<<<grid, NT, L::bytes, st>>>(n, m, p, nb, h->H, h->Ct, p > 0 ? p : 1, h->R, s,
                                         reinterpret_cast<const cd*>(shifts), mode,
                                         reinterpret_cast<cd*>(base), slot,
                                         reinterpret_cast<cd*>(out), ldo, status, nullptr, 0,
                                         h->hnorm2, nullptr, nullptr, nullptr, 0, nullptr, nullptr, 1);
  count_launch();
  SSV_CUDA_TRY(cudaGetLastError());
  if (status != nullptr) {
    const int rows = (mode == SSV_G || mode == SSV_TF) ? p : n;
    if (rows > 0) {
      nonfinite_kernel<<<s, 256, 0, st>>>(reinterpret_cast<const cd*>(out), ldo, rows,
                                          m, s, status);
      count_launch();
      SSV_CUDA_TRY(cudaGetLastError());
    }
  }
  return SSV_OK;
}
}  // namespace

size_t noalloc_scratch_bytes() { return kNoAllocScratchBytes; }

int solve_fp64_noalloc(const Handle* h, int s, const double* shifts, const ssv_opts* o,
                       double* out, long long ldo, int* status, cudaStream_t st) {
  const int m = h->m;
  // the same block width as ssv_solve (an autotuned choice included), so the
  // two entry points give the same results
  const int nb = o->nb > 0 ? o->nb : tuned_nb(h->n, m, h->p, SSV_FP64, o->mode);
  if (nb > kNB) return SSV_ENOTSUP;
  if (s == 0) return SSV_OK;
  if (m <= 1) return launch_solve_noalloc<1>(h, s, shifts, nb, o->mode, out, ldo, status, st);
  if (m <= 2) return launch_solve_noalloc<2>(h, s, shifts, nb, o->mode, out, ldo, status, st);
  if (m <= 4) return launch_solve_noalloc<4>(h, s, shifts, nb, o->mode, out, ldo, status, st);
  if (m <= 8) return launch_solve_noalloc<8>(h, s, shifts, nb, o->mode, out, ldo, status, st);
  if (m <= 16) return launch_solve_noalloc<16>(h, s, shifts, nb, o->mode, out, ldo, status, st);
  if (m <= 32) return launch_solve_noalloc<32>(h, s, shifts, nb, o->mode, out, ldo, status, st);
  return SSV_ENOTSUP;
}

// ---------------------------------------------------------------------------
// Autotuner for the elimination block width n_b: times each candidate on the
// caller's shifts with CUDA events and caches the fastest per
// (n, m, p, precision, mode) for the life of the process.
// ---------------------------------------------------------------------------
namespace {
struct TuneKey {
  int n, m, p, prec, mode;
  bool operator<(const TuneKey& o) const {
    if (n != o.n) return n < o.n;
    if (m != o.m) return m < o.m;
    if (p != o.p) return p < o.p;
    if (prec != o.prec) return prec < o.prec;
    return mode < o.mode;
  }
};
std::mutex g_tune_mu;
std::map<TuneKey, int> g_tune;
}  // namespace

int tuned_nb(int n, int m, int p, int prec, int mode) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  auto it = g_tune.find(TuneKey{n, m, p, prec, mode});
  return it == g_tune.end() ? default_nb(n, m) : it->second;
}

int autotune_nb(const Handle* h, int s, const double* shifts, const ssv_opts* o, double* out,
                long long ldo, cudaStream_t st, int* best_nb, float* best_ms) {
  static const int cand_fp64[] = {32, 48, 64, 96, 128};
  static const int cand_mixed[] = {16, 24, 32, 48, 64};
  const int* cand = o->precision == SSV_MIXED ? cand_mixed : cand_fp64;
  cudaEvent_t e0, e1;
  SSV_CUDA_TRY(cudaEventCreate(&e0));
  SSV_CUDA_TRY(cudaEventCreate(&e1));
  int best = default_nb(h->n, h->m);
  float bms = 1e30f;
  int rc = SSV_OK;
  for (int ci = 0; ci < 5; ++ci) {
    const int c = cand[ci];
    ssv_opts oo = *o;
    oo.nb = c;
    for (int rep = 0; rep < 2 && rc == SSV_OK; ++rep) {  // first run warms up
      cudaEventRecord(e0, st);
      rc = oo.precision == SSV_MIXED ? solve_mixed(h, s, shifts, &oo, out, ldo, nullptr, nullptr, st)
                                     : solve_fp64(h, s, shifts, &oo, out, ldo, nullptr, nullptr, st);
      cudaEventRecord(e1, st);
      if (rc == SSV_OK && cudaEventSynchronize(e1) == cudaSuccess && rep == 1) {
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (ms < bms) { bms = ms; best = c; }
      }
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc != SSV_OK) return rc;
  {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    g_tune[TuneKey{h->n, h->m, h->p, o->precision, o->mode}] = best;
  }
  *best_nb = best;
  if (best_ms) *best_ms = bms;
  return SSV_OK;
}

}  // namespace ssv
