// Transposed systems (Sec. 3.3) and the Givens panel (Sec. 3.2), FP64.
#include "sweep.cuh"

namespace ssv {

namespace {

// Givens-panel sweep (Sec. 3.2): the same work list as solve_fp64_kernel.
template <int MAXM>
__global__ void __launch_bounds__(kThreads) solve_fp64_givens_kernel(FpSys d, int s,
                                                                     cd* __restrict__ scratch,
                                                                     size_t slot_stride) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_piv;
  __shared__ int s_sing;
  cd* Z2 = scratch + (size_t)blockIdx.x * slot_stride;
  for (int w = blockIdx.x; w < s; w += gridDim.x)
    fp64_shift<MAXM, kThreads, false, true>(d, w, Z2, smem_raw, &s_piv, &s_sing);
}

// Dense right-hand side per shift (the transposed systems of Sec. 3.3, in the
// flipped form built by solve_fp64_trans); d.p == 0.
template <int MAXM>
__global__ void __launch_bounds__(sweep_threads<MAXM>(), sweep_per_sm(MAXM, false))
    solve_fp64_rhs_kernel(FpSys d, int s, cd* scratch, size_t slot_stride, int team) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_piv;
  __shared__ int s_sing;
  // team: CTAs of a cluster per shift (fp64_shift)
  const int rank = team > 1 ? cluster_rank() : 0, g = blockIdx.x / team, G = gridDim.x / team;
  cd* Z2 = scratch + (size_t)g * slot_stride;
  for (int w = g; w < s; w += G)
    fp64_shift<MAXM, sweep_threads<MAXM>(), true>(d, w, Z2, smem_raw, &s_piv, &s_sing, team, rank);
}

// Ht(i, j) = H(n-1-j, n-1-i) on the structural part i <= j + m, zero below:
// J (H - sigma I)^T J = Ht - sigma I is upper m-Hessenberg again.  32 x 32
// tiles through shared memory, coalesced on both sides.
__global__ void flip_transpose_kernel(const double* __restrict__ H, int n, int m,
                                      double* __restrict__ Ht) {
  __shared__ double tile[32][33];
  const int a0 = blockIdx.x * 32, b0 = blockIdx.y * 32;  // rows / columns of H
  const int tx = threadIdx.x, ty = threadIdx.y;
  for (int k = 0; k < 32; k += 8) {
    const int a = a0 + tx, b = b0 + ty + k;
    tile[ty + k][tx] = (a < n && b < n) ? H[a + (size_t)b * n] : 0.0;
  }
  __syncthreads();
  for (int k = 0; k < 32; k += 8) {
    const int b = b0 + tx, a = a0 + ty + k;
    if (a < n && b < n) {
      const int i = n - 1 - b, j = n - 1 - a;
      Ht[i + (size_t)j * n] = (i <= j + m) ? tile[tx][ty + k] : 0.0;
    }
  }
}

// d(i, l) = (Ct^T chat_l)(n-1-i): the flipped reduced right-hand side C~^T chat_l.
__global__ void flipped_rhs_kernel(const double* __restrict__ Ct, int ldct, int p, int n,
                                   const cd* __restrict__ chat, long long ldc, int s,
                                   cd* __restrict__ dvec) {
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < (long long)n * s;
       idx += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(idx % n), l = (int)(idx / n);
    const int col = n - 1 - i;
    const cd* c = chat + (size_t)l * ldc;
    double re = 0.0, im = 0.0;
    for (int k = 0; k < p; ++k) {
      const double v = Ct[k + (size_t)col * ldct];
      re = fma(v, c[k].x, re);
      im = fma(v, c[k].y, im);
    }
    dvec[idx] = mkcd(re, im);
  }
}

}  // namespace

namespace {
template <int MAXM>
int launch_rhs(const FpSys& d, int s, cudaStream_t st) {
  using L = Layout<MAXM>;
  const size_t slot = (size_t)d.n * d.m * 2 + 2 * (size_t)d.n;
  auto kern = solve_fp64_rhs_kernel<MAXM>;
  SSV_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::bytes));
  constexpr int NT = sweep_threads<MAXM>();
  int per_sm = 0;
  SSV_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NT, L::bytes));
  per_sm = std::max(1, std::min(per_sm, sweep_per_sm(MAXM, false)));
  const int grid = std::min(s, num_sms() * per_sm);
  cd* scratch = nullptr;
  SSV_CUDA_TRY(pool_alloc((void**)&scratch, sizeof(cd) * slot * grid, st));
  const int team = team_for(s, d.n, d.m);
  cudaError_t e = launch_cluster(kern, grid * team, NT, team, L::bytes, st, d, s, scratch, slot, team);
  cudaError_t e2 = cudaFreeAsync(scratch, st);
  if (e == cudaSuccess) e = e2;
  if (e != cudaSuccess) {
    set_cuda_error(e);
    return SSV_ECUDA;
  }
  return SSV_OK;
}
}  // namespace

// Transposed systems (A - sigma_l I)^T x_l = C^T chat_l (Sec. 3.3) in reduced
// coordinates: (H - sigma I)^T xt = C~^T chat with x = Q xt.  With J the
// reversal, J (H - sigma I)^T J = Ht - sigma I is upper m-Hessenberg, so the
// same bottom-up sweep solves it for the dense right-hand side J C~^T chat;
// the solution is flipped back on output (out = Q^T x_l).
int solve_fp64_trans(const Handle* h, int s, const double* shifts, const double* chat,
                     long long ldc, const ssv_opts* o, double* out, long long ldo, int* status,
                     cudaStream_t st) {
  const int n = h->n, m = h->m, p = h->p;
  const int nb = o->nb > 0 ? o->nb : tuned_nb(n, m, 0, SSV_FP64, SSV_XHAT);
  if (nb > kNB) return SSV_ENOTSUP;
  if (s == 0) return SSV_OK;
  double* Ht = nullptr;
  cd* dvec = nullptr;
  SSV_CUDA_TRY(pool_alloc((void**)&Ht, sizeof(double) * (size_t)n * n, st));
  cudaError_t e = pool_alloc((void**)&dvec, sizeof(cd) * (size_t)n * s, st);
  int rc = SSV_OK;
  if (e == cudaSuccess) {
    const dim3 tg((n + 31) / 32, (n + 31) / 32);
    flip_transpose_kernel<<<tg, dim3(32, 8), 0, st>>>(h->H, n, m, Ht);
    count_launch();
    const long long tot = (long long)n * s;
    flipped_rhs_kernel<<<(int)std::min<long long>(4096, (tot + 255) / 256), 256, 0, st>>>(
        h->Ct, p > 0 ? p : 1, p, n, reinterpret_cast<const cd*>(chat), ldc, s, dvec);
    count_launch();
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) {
    set_cuda_error(e);
    rc = e == cudaErrorMemoryAllocation ? SSV_ENOMEM : SSV_ECUDA;
  }
  if (rc == SSV_OK) {
    FpSys d;
    d.n = n; d.m = m; d.p = 0; d.nb = nb; d.mode = SSV_XHAT; d.H = Ht; d.Ct = nullptr; d.ldct = 1;
    d.R = h->R; d.shifts = reinterpret_cast<const cd*>(shifts);
    d.out = reinterpret_cast<cd*>(out); d.ldo = ldo; d.status = status;
    d.xhat_copy = nullptr; d.ldxc = 0; d.hnorm = h->hnorm2; d.bhat = nullptr; d.ldb = 0;
    d.rhs = dvec; d.ldr = n; d.flip_out = 1;
    d.gfull = GivensSched{nullptr, nullptr, 0};
    d.gtail = d.gfull;
    if (m <= 1) rc = launch_rhs<1>(d, s, st);
    else if (m <= 2) rc = launch_rhs<2>(d, s, st);
    else if (m <= 4) rc = launch_rhs<4>(d, s, st);
    else if (m <= 8) rc = launch_rhs<8>(d, s, st);
    else if (m <= 16) rc = launch_rhs<16>(d, s, st);
    else if (m <= 32) rc = launch_rhs<32>(d, s, st);
    else rc = SSV_ENOTSUP;
  }
  if (rc == SSV_OK && status != nullptr) {
    nonfinite_kernel<<<s, 256, 0, st>>>(reinterpret_cast<const cd*>(out), ldo, n, 1, s, status);
    count_launch();
    e = cudaGetLastError();
    if (e != cudaSuccess) {
      set_cuda_error(e);
      rc = SSV_ECUDA;
    }
  }
  if (dvec) cudaFreeAsync(dvec, st);
  if (Ht) cudaFreeAsync(Ht, st);
  return rc;
}
// ---------------------------------------------------------------------------
// Givens panel (Sec. 3.2): the greedy annihilation schedule for a block of
// `rows` rows and rows + m columns, computed on the host once per shape and
// device and kept in device memory.
//
// Row r (0-based) of the block holds nonzeros in columns r .. r + m; every
// entry but the last of a row is zeroed by a rotation with another entry of
// the same row, rotations of one step touching disjoint columns.  Seen per
// column, the entries that may be rotated form a frontier moving up: column c
// starts at its lowest band entry (row min(c, rows - 1)), and once the
// frontier entry of c is zeroed the entry above it joins in the next step;
// column c never rises above row c - m, where it survives as the diagonal of
// the triangular factor.  A step therefore looks at each row's frontier
// columns c_1 < ... < c_k and zeroes as many as the greedy choice allows:
// c_1 with the partner c_k, c_2 with c_(k-1), and so on, the middle one of an
// odd count waiting.  Steps are emitted rows from the bottom, zeroed columns
// ascending within a row, until a step finds no pair.
// ---------------------------------------------------------------------------
void greedy_rows(int rows, int m, std::vector<int>* rot, std::vector<int>* off) {
  const int cols = rows + m;
  // front[c]: row of column c's frontier entry; -1 once the column is empty
  std::vector<int> front(cols);
  for (int c = 0; c < cols; ++c) front[c] = std::min(c, rows - 1);
  std::vector<std::vector<int>> at_row(rows);
  std::vector<int> zeroed;
  rot->clear();
  off->assign(1, 0);
  for (;;) {
    for (auto& v : at_row) v.clear();
    for (int c = 0; c < cols; ++c)
      if (front[c] >= 0) at_row[front[c]].push_back(c);  // ascending in c
    zeroed.clear();
    for (int r = rows - 1; r >= 0; --r) {
      const std::vector<int>& e = at_row[r];
      const int k = (int)e.size();
      for (int i = 0; i < k / 2; ++i) {
        rot->push_back(r | (e[i] << 8) | (e[k - 1 - i] << 16));
        zeroed.push_back(e[i]);
      }
    }
    if (zeroed.empty()) break;
    for (int c : zeroed) front[c] -= 1;  // the entry above joins next step
    off->push_back((int)rot->size());
  }
}

namespace {

struct SchedEntry {
  int* rot = nullptr;
  int* off = nullptr;
  int nsteps = 0;
};
std::mutex g_sched_mu;
std::map<std::tuple<int, int, int>, SchedEntry> g_sched;  // (device, rows, m)

int givens_schedule(int rows, int m, GivensSched* out) {
  int dev = 0;
  SSV_CUDA_TRY(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lk(g_sched_mu);
  auto key = std::make_tuple(dev, rows, m);
  auto it = g_sched.find(key);
  if (it == g_sched.end()) {
    std::vector<int> rot, off;
    greedy_rows(rows, m, &rot, &off);
    SchedEntry e;
    e.nsteps = (int)off.size() - 1;
    SSV_CUDA_TRY(cudaMalloc((void**)&e.rot, sizeof(int) * std::max<size_t>(1, rot.size())));
    SSV_CUDA_TRY(cudaMalloc((void**)&e.off, sizeof(int) * off.size()));
    SSV_CUDA_TRY(cudaMemcpy(e.rot, rot.data(), sizeof(int) * rot.size(), cudaMemcpyHostToDevice));
    SSV_CUDA_TRY(cudaMemcpy(e.off, off.data(), sizeof(int) * off.size(), cudaMemcpyHostToDevice));
    it = g_sched.emplace(key, e).first;
  }
  *out = GivensSched{it->second.rot, it->second.off, it->second.nsteps};
  return SSV_OK;
}

template <int MAXM>
int launch_givens(const FpSys& d, int s, cudaStream_t st) {
  using GL = GivensLayout<MAXM>;
  const bool track_t = (d.mode == SSV_XHAT || d.mode == SSV_X || d.xhat_copy != nullptr);
  const size_t slot = (size_t)(d.p + d.n) * d.m + (track_t ? (size_t)d.n * d.m : 0);
  auto kern = solve_fp64_givens_kernel<MAXM>;
  SSV_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GL::bytes));
  int per_sm = 0;
  SSV_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThreads, GL::bytes));
  per_sm = std::max(1, std::min(per_sm, 2));
  const int grid = std::min(s, num_sms() * per_sm);
  cd* scratch = nullptr;
  SSV_CUDA_TRY(pool_alloc((void**)&scratch, sizeof(cd) * slot * grid, st));
  kern<<<grid, kThreads, GL::bytes, st>>>(d, s, scratch, slot);
  count_launch();
  cudaError_t e = cudaGetLastError();
  cudaError_t e2 = cudaFreeAsync(scratch, st);
  if (e == cudaSuccess) e = e2;
  if (e != cudaSuccess) {
    set_cuda_error(e);
    return SSV_ECUDA;
  }
  return SSV_OK;
}

}  // namespace

int solve_fp64_givens(const Handle* h, int s, const double* shifts, const ssv_opts* o, double* out,
                      long long ldo, int* status, double* resid, cudaStream_t st) {
  const int n = h->n, m = h->m, p = h->p;
  const int nb = o->nb > 0 ? o->nb : kNBG;
  if (nb > kNBG || m > 32) return SSV_ENOTSUP;
  if (s == 0) return SSV_OK;
  const int mode = o->mode == SSV_X ? SSV_XHAT : o->mode;
  FpSys d;
  d.n = n; d.m = m; d.p = p; d.nb = nb; d.mode = mode; d.H = h->H; d.Ct = h->Ct;
  d.ldct = p > 0 ? p : 1; d.R = h->R; d.shifts = reinterpret_cast<const cd*>(shifts);
  d.out = reinterpret_cast<cd*>(out); d.ldo = ldo; d.status = status;
  d.xhat_copy = nullptr; d.ldxc = 0; d.hnorm = h->hnorm2; d.bhat = nullptr; d.ldb = 0;
  d.rhs = nullptr; d.ldr = 0; d.flip_out = 0;
  d.gfull = GivensSched{nullptr, nullptr, 0};
  d.gtail = d.gfull;
  const int tail = (n - m) % nb;
  int rc = SSV_OK;
  if (n > m) {
    rc = givens_schedule(std::min(nb, n - m), m, &d.gfull);
    if (rc == SSV_OK && tail != 0 && n - m > nb) rc = givens_schedule(tail, m, &d.gtail);
    if (rc == SSV_OK && n - m <= nb) d.gtail = d.gfull;
  }
  if (rc != SSV_OK) return rc;
  cd* xcopy = nullptr;
  if (resid != nullptr && (mode == SSV_G || mode == SSV_TF)) {
    SSV_CUDA_TRY(pool_alloc((void**)&xcopy, sizeof(cd) * (size_t)n * m * s, st));
    d.xhat_copy = xcopy;
    d.ldxc = n;
  }
  if (m <= 1) rc = launch_givens<1>(d, s, st);
  else if (m <= 2) rc = launch_givens<2>(d, s, st);
  else if (m <= 4) rc = launch_givens<4>(d, s, st);
  else if (m <= 8) rc = launch_givens<8>(d, s, st);
  else if (m <= 16) rc = launch_givens<16>(d, s, st);
  else rc = launch_givens<32>(d, s, st);
  if (rc == SSV_OK && status != nullptr) {
    const int rows = (mode == SSV_G || mode == SSV_TF) ? p : n;
    if (rows > 0) {
      nonfinite_kernel<<<s, 256, 0, st>>>(reinterpret_cast<const cd*>(out), ldo, rows, m, s, status);
      count_launch();
      cudaError_t e = cudaGetLastError();
      if (e != cudaSuccess) {
        set_cuda_error(e);
        rc = SSV_ECUDA;
      }
    }
  }
  if (rc == SSV_OK && resid != nullptr) {
    const double* xh = xcopy ? reinterpret_cast<const double*>(xcopy) : out;
    rc = backward_error_fp64(h, s, shifts, xh, xcopy ? n : ldo, resid, st);
  }
  if (xcopy) cudaFreeAsync(xcopy, st);
  return rc;
}

}  // namespace ssv
