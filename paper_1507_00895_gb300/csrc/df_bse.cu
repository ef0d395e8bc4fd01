// Ladder (Bethe-Salpeter) solves of Eq. lin_alg_inv, FP64 path, and the ladder
// term of the susceptibilities.
//
// For every (q, W) and channel: D = 1 - gamma_W diag(chi~_W(q)), solve
// D Gamma = gamma_W, keep only diag Gamma, and write the Eq. sd bracket
//     kc = c (Gamma_ww - Gamma^(2)_ww / 2),  Gamma^(2)_ww = sum_x gamma_wx chi~_x gamma_xw,
// with c = 1 (density) or 3 (magnetic).
//
// Design: one CTA per system (persistent grid, systems strided by
// gridDim.x), D factorised in place by right-looking LU with partial
// pivoting (pivot = largest |re|+|im| in the column, first on ties), the
// right-hand sides P gamma processed in column chunks.  Because only the
// diagonal of Gamma is needed, the back substitution for column j stops at
// row j: LU (n^3/3) + forward (n^3/2) + truncated back substitution (n^3/6)
// = n^3 complex multiply-adds per system instead of 4n^3/3.  U's columns are
// pre-scaled by 1/U_kk so that neither substitution divides.
#include "df_bse_dev.cuh"

namespace df {

// gg[c][a][i][j] = gamma[c][a][i][j] * gamma[c][a][j][i]  (for Gamma^(2))
__global__ void gamma_gt_kernel(int n, int count, const double2* __restrict__ gam, double2* __restrict__ gg) {
  const size_t total = (size_t)count * n * n;
  for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total; idx += (size_t)gridDim.x * blockDim.x) {
    const size_t mat = idx / ((size_t)n * n);
    const int rem = (int)(idx - mat * n * n);
    const int i = rem / n, j = rem - i * n;
    const double2* G = gam + mat * n * n;
    gg[idx] = cmul(G[i * n + j], G[j * n + i]);
  }
}

// The hand-back list of a launch (list NULL: every system of the planes), whose length only the
// device knows: the launch takes lists of above < length <= up_to, in ranges of nc right-hand sides up
// to a length of short_up_to and of nc_long beyond it.
struct LadderList {
  const int* list = nullptr;
  int spread = 0;
  int above = -1, up_to = 0x7FFFFFFF, short_up_to = 0x7FFFFFFF, nc_long = 0;
};

template <bool LU_SMEM>
__global__ void __launch_bounds__(kBseThreads)
bse_f64_kernel(Dims dm, int ch0, int nch, int nc, const double2* __restrict__ gam,
               const double2* __restrict__ gg, const double2* __restrict__ chi,
               double2* __restrict__ kc, double2* __restrict__ ws, int* __restrict__ flags, int radius_K,
               const double2* __restrict__ lam, LadderList ll) {
  extern __shared__ double2 sm[];
  __shared__ BseF64Shared sh;
  const int n = dm.n_w, N = dm.N, nb = dm.nb, na = dm.na;
  const int* __restrict__ list = ll.list;
  const int spread = ll.spread;
  if (list && (list[0] <= ll.above || list[0] > ll.up_to)) return;
  if (list && list[0] > ll.short_up_to) nc = ll.nc_long;
  const BseSmem L = bse_layout(n, nc, LU_SMEM);
  double2* LU = LU_SMEM ? sm + L.lu : ws + (size_t)blockIdx.x * n * n;
  // the handle's planes of channels ch0 .. ch0 + nch - 1, or with a list its
  // list[0] systems (c N_W + a) N + q that follow it (ladders the mixed-precision
  // kernels handed back).  A short list is spread over up to `spread` blocks:
  // each ladder's right-hand-side chunks are split into `parts` column ranges,
  // one block per range, each factorising the ladder itself (the FP64 pipe of
  // one SM bounds a lone ladder's latency)
  const int chunks = (n + nc - 1) / nc;
  long count = list ? (long)list[0] : 0;
  int parts = 1;
  if (list && count > 0 && spread > count) {
    const long p = spread / count;
    parts = (int)(p < chunks ? p : chunks);
  }
  const int cpp = (chunks + parts - 1) / parts;      // chunks per part
  const long systems = list ? count * parts : (long)nch * na * N;
  for (long s = blockIdx.x; s < systems; s += gridDim.x) {
    int c, a, q, jb = 0, je = n;
    if (list) {
      const int part = (int)(s % parts);
      jb = part * cpp * nc;
      je = jb + cpp * nc < n ? jb + cpp * nc : n;
      if (jb >= je) continue;                         // the same in the whole block
      const long sys = list[1 + s / parts];
      c = (int)(sys / ((long)nb * N));
      const int rem = (int)(sys - (long)c * nb * N);
      a = rem / N;
      q = rem - a * N;
    } else {
      c = ch0 + (int)(s / ((long)na * N));
      const int rem = (int)(s - (long)(c - ch0) * na * N);
      a = dm.a0 + rem / N;
      q = rem - (a - dm.a0) * N;
    }
    bse_f64_system(dm, c, a, q, nc, gam, gg, chi, kc, LU, sm + L.y, sm + L.xs, sm + L.invu, sh, flags, radius_K,
                   lam, jb, je);
  }
}

// The ladder term of the susceptibilities (section "Resulting observables"):
// for one (q, W, channel), sum_{w,w'} L_w Gamma_{w,w'} L_w' with
// Gamma = D^-1 gamma (Eq. lin_alg_inv) = L . x, D x = gamma L, D in LU
// (bse_f64_factor, FP64); out = chi0 + L . x.  Y holds [n][2]: the permuted
// right-hand side, then L.
__device__ __forceinline__ void chi_ladder_system(const Dims& dm, int c, int a, int q,
                                                  const double2* __restrict__ gam, const double2* __restrict__ chi,
                                                  const double2* __restrict__ Lb, const double2* __restrict__ chi0,
                                                  double2* __restrict__ out, double2* LU, double2* Y, double2* xs,
                                                  double2* invu, BseF64Shared& sh, int* __restrict__ flags) {
  const int n = dm.n_w, N = dm.N, nb = dm.nb;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const double2* G = gam + ((size_t)c * nb + a) * n * n;
  double2* y = Y;
  double2* lv = Y + n;
  bse_f64_factor(dm, c, a, q, gam, chi, LU, xs, invu, sh, flags);
  for (int i = tid; i < n; i += blockDim.x) lv[i] = Lb[((size_t)a * n + i) * N + q];
  __syncthreads();
  for (int r = tid; r < n; r += blockDim.x) {      // y = P (gamma L)
    const double2* gr = G + (size_t)sh.perm[r] * n;
    double2 b = mk(0.0, 0.0);
    for (int j = 0; j < n; ++j) b = cfma(gr[j], lv[j], b);
    y[r] = b;
  }
  __syncthreads();
  if (warp == 0) {
    for (int k = 0; k < n - 1; ++k) {              // unit-lower forward substitution
      const double2 yk = y[k];
      for (int r = k + 1 + lane; r < n; r += 32) y[r] = cfms(LU[r * n + k], yk, y[r]);
      __syncwarp();
    }
    for (int k = n - 1; k > 0; --k) {              // unit-upper back substitution (V = U diag(1/U_kk))
      const double2 yk = y[k];
      for (int r = lane; r < k; r += 32) y[r] = cfms(LU[r * n + k], yk, y[r]);
      __syncwarp();
    }
    double2 s2 = mk(0.0, 0.0);                     // L . x, x = y / U_kk
    for (int i = lane; i < n; i += 32) s2 = cfma(lv[i], cmul(y[i], invu[i]), s2);
    for (int o = 16; o > 0; o >>= 1) {
      s2.x += __shfl_xor_sync(0xffffffffu, s2.x, o);
      s2.y += __shfl_xor_sync(0xffffffffu, s2.y, o);
    }
    if (lane == 0) {
      const double2 c0 = chi0[(size_t)a * N + q];
      out[((size_t)c * nb + a) * N + q] = mk(c0.x + s2.x, c0.y + s2.y);
    }
  }
  __syncthreads();
}

// All 2 nb N systems, or with `list` non-null the list[0] systems whose
// indices follow it (the ones the refinement kernel below handed back).
template <bool LU_SMEM>
__global__ void __launch_bounds__(kBseThreads)
chi_ladder_kernel(Dims dm, const double2* __restrict__ gam, const double2* __restrict__ chi,
                  const double2* __restrict__ Lb, const double2* __restrict__ chi0, double2* __restrict__ out,
                  double2* __restrict__ ws, int* __restrict__ flags, const int* __restrict__ list) {
  extern __shared__ double2 sm[];
  __shared__ BseF64Shared sh;
  const int n = dm.n_w, N = dm.N, nb = dm.nb;
  const BseSmem L = bse_layout(n, 2, LU_SMEM);
  double2* LU = LU_SMEM ? sm + L.lu : ws + (size_t)blockIdx.x * n * n;
  const long systems = list ? (long)list[0] : 2L * nb * N;
  for (long s = blockIdx.x; s < systems; s += gridDim.x) {
    const long sys = list ? (long)list[1 + s] : s;
    const int c = (int)(sys / ((long)nb * N));
    const int rem = (int)(sys - (long)c * nb * N);
    const int a = rem / N, q = rem - a * N;
    chi_ladder_system(dm, c, a, q, gam, chi, Lb, chi0, out, LU, sm + L.y, sm + L.xs, sm + L.invu, sh, flags);
  }
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------

static int bse_chunk(int n) { return n <= 32 ? n : (n <= 64 ? 32 : 16); }
static bool bse_lu_in_smem(int n) { return n <= kLuSmemOrder; }
static bool bse_lu_fits_smem(int n) { return n <= 96; }   // the allocation-free entry point's limit

size_t bse_workspace_bytes(const Dims& dm, int grid) {
  size_t b = (size_t)2 * dm.nb * dm.n_w * dm.n_w * sizeof(double2);      // gamma o gamma^T
  if (!bse_lu_in_smem(dm.n_w)) b += (size_t)grid * dm.n_w * dm.n_w * sizeof(double2);
  return b;
}

static size_t bse_smem_bytes(int n) {
  return sizeof(double2) * (size_t)bse_layout(n, bse_chunk(n), bse_lu_in_smem(n)).total;
}

int bse_default_grid(const Dims& dm, int device) {
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  const size_t smem = bse_smem_bytes(dm.n_w);
  const void* fn = bse_lu_in_smem(dm.n_w) ? (const void*)bse_f64_kernel<true> : (const void*)bse_f64_kernel<false>;
  cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kBseThreads, smem);
  if (per_sm < 1) per_sm = 1;
  return sms * per_sm;
}

static double2* gg_ptr(df_ctx* c) { return (double2*)c->bse_ws; }
const double2* gamma_gt_ptr(df_ctx* c) { return gg_ptr(c); }
static int* flag_ptr(df_ctx* c) { return bse_flags(c); }
static double2* lu_ws_ptr(df_ctx* c) {
  return (double2*)((char*)c->bse_ws + (size_t)2 * c->dm.nb * c->dm.n_w * c->dm.n_w * sizeof(double2));
}

cudaError_t launch_gamma_gt(df_ctx* c) {
  const Dims& dm = c->dm;
  gamma_gt_kernel<<<2 * dm.nb * 8, 256, 0, c->stream>>>(dm.n_w, 2 * dm.nb, c->gam, gg_ptr(c));
  return cudaGetLastError();
}

cudaError_t launch_bse(df_ctx* c, int channel_mask) {
  const Dims& dm = c->dm;
  const int n = dm.n_w;
  const int nc = bse_chunk(n);
  const size_t smem = bse_smem_bytes(n);
  cudaError_t e = cudaSuccess;
  if (c->opts.precision == DF_FP32_IR) return launch_bse_mixed(c, channel_mask, flag_ptr(c));
  const int K = c->opts.radius_order;
  const double2* lam = K > 0 ? c->lam : nullptr;
  // both channels in one launch of the grid-stride kernel when both are asked
  // for (one partial wave instead of two)
  const bool both = (channel_mask & 3) == 3;
  for (int ch = 0; ch < 2; ++ch) {
    if (!(channel_mask & (1 << ch))) continue;
    const int nch = both ? 2 : 1;
    const long systems = (long)nch * dm.na * dm.N;
    const int grid = (int)(systems < c->bse_grid ? systems : c->bse_grid);
    if (bse_lu_in_smem(n)) {
      bse_f64_kernel<true><<<grid, kBseThreads, smem, c->stream>>>(dm, ch, nch, nc, c->gam, gg_ptr(c), c->chi,
                                                                   c->kc, nullptr, flag_ptr(c), K, lam, LadderList{});
    } else {
      bse_f64_kernel<false><<<grid, kBseThreads, smem, c->stream>>>(dm, ch, nch, nc, c->gam, gg_ptr(c), c->chi,
                                                                    c->kc, lu_ws_ptr(c), flag_ptr(c), K, lam,
                                                                    LadderList{});
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (both) break;
  }
  return cudaSuccess;
}

template <bool LU_SMEM>
static cudaError_t launch_list(df_ctx* c, int nc, int nc_smem, int max_grid, LadderList ll) {
  const size_t smem = sizeof(double2) * (size_t)bse_layout(c->dm.n_w, nc_smem, LU_SMEM).total;
  const void* fn = (const void*)bse_f64_kernel<LU_SMEM>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int grid = max_grid < ll.up_to ? max_grid : ll.up_to;
  ll.spread = grid;
  bse_f64_kernel<LU_SMEM><<<grid, kBseThreads, smem, c->stream>>>(c->dm, 0, 2, nc, c->gam, gg_ptr(c), c->chi, c->kc,
                                                                  LU_SMEM ? nullptr : lu_ws_ptr(c), flag_ptr(c), 0,
                                                                  nullptr, ll);
  return cudaGetLastError();
}

// blocks of a shared-memory list launch that run at once (asked once per handle)
static int list_wave(df_ctx* c, int nc) {
  if (c->list_wave > 0) return c->list_wave;
  const size_t smem = sizeof(double2) * (size_t)bse_layout(c->dm.n_w, nc, true).total;
  int sms = 0, per_sm = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
  cudaFuncSetAttribute((const void*)bse_f64_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, bse_f64_kernel<true>, kBseThreads, smem);
  return c->list_wave = sms * (per_sm < 1 ? 1 : per_sm);
}

// the FP64 LU over the ladders the mixed-precision kernels handed back: list[0]
// (read on the device) systems (c N_W + a) N + q, on the persistent grid; a
// list shorter than the grid is spread over it by right-hand-side ranges.  How the list is solved
// follows from its length (kListSmemOrder): of the two launches of orders 41-96 one returns at once.
cudaError_t launch_bse_f64_list(df_ctx* c, const int* list) {
  const int n = c->dm.n_w, nc = n < kListChunk ? n : kListChunk, nc_long = bse_chunk(n);
  LadderList ll;
  ll.list = list;
  ll.nc_long = nc_long;
  if (n > kListSmemOrder) return launch_list<false>(c, nc_long, nc_long, c->bse_grid, ll);   // (the scratch has bse_grid slices)
  const int wave = list_wave(c, n <= kLuSmemOrder ? nc_long : nc);
  if (n <= kLuSmemOrder) {
    ll.short_up_to = kListShort;
    return launch_list<true>(c, nc, nc_long, wave, ll);
  }
  ll.up_to = wave;
  const cudaError_t e = launch_list<true>(c, nc, nc, wave, ll);
  if (e != cudaSuccess) return e;
  ll.above = wave;
  ll.up_to = 0x7FFFFFFF;
  return launch_list<false>(c, nc_long, nc_long, c->bse_grid, ll);
}

// the ladder term of the susceptibilities for both channels: FP64 LU on the
// persistent grid and LU scratch of the FP64 ladder kernel, or under
// DF_FP32_IR (n_w <= 64) the refinement kernel of df_chi.cu first and the FP64 LU
// only for the systems it hands back (redo: 1 + 2 nb N ints)
cudaError_t launch_chi_ladder(df_ctx* c, const double2* Lb, const double2* chi0, double2* out, int* redo) {
  const Dims& dm = c->dm;
  const int n = dm.n_w;
  const bool in_smem = bse_lu_in_smem(n);
  const size_t smem = sizeof(double2) * (size_t)bse_layout(n, 2, in_smem).total;
  const void* fn = in_smem ? (const void*)chi_ladder_kernel<true> : (const void*)chi_ladder_kernel<false>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const long systems = 2L * dm.nb * dm.N;
  const int* list = nullptr;
  if (c->opts.precision == DF_FP32_IR && n <= 64 && c->mixed_ws) {
    if ((e = cudaMemsetAsync(redo, 0, sizeof(int), c->stream)) != cudaSuccess) return e;
    if ((e = launch_chi_ladder_ir(c, Lb, chi0, out, redo)) != cudaSuccess) return e;
    list = redo;
  }
  const int grid = (int)(systems < c->bse_grid ? systems : c->bse_grid);
  if (in_smem)
    chi_ladder_kernel<true><<<grid, kBseThreads, smem, c->stream>>>(dm, c->gam, c->chi, Lb, chi0, out, nullptr,
                                                                    flag_ptr(c), list);
  else
    chi_ladder_kernel<false><<<grid, kBseThreads, smem, c->stream>>>(dm, c->gam, c->chi, Lb, chi0, out,
                                                                     lu_ws_ptr(c), flag_ptr(c), list);
  return cudaGetLastError();
}

}  // namespace df

// ---------------------------------------------------------------------------
// launchers on caller-given buffers (no handle), used by the allocation-free
// entry point; the kernels are the ones above
// ---------------------------------------------------------------------------
namespace df {

cudaError_t launch_gamma_gt_raw(int n, int count, const double2* gam, double2* gg, cudaStream_t stream) {
  gamma_gt_kernel<<<count * 8, 256, 0, stream>>>(n, count, gam, gg);
  return cudaGetLastError();
}

cudaError_t launch_bse_both_raw(const Dims& dm, const double2* gam, const double2* gg, const double2* chi,
                                double2* kc, int* flags, int device, cudaStream_t stream) {
  if (!bse_lu_fits_smem(dm.n_w)) return cudaErrorInvalidValue;
  const int nc = bse_chunk(dm.n_w);
  const size_t smem = sizeof(double2) * (size_t)bse_layout(dm.n_w, nc, true).total;
  int sms = 0, per_sm = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  cudaError_t e = cudaFuncSetAttribute((const void*)bse_f64_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, bse_f64_kernel<true>, kBseThreads, smem);
  const int grid_max = sms * (per_sm < 1 ? 1 : per_sm);
  const long systems = 2L * dm.nb * dm.N;
  const int grid = (int)(systems < grid_max ? systems : grid_max);
  bse_f64_kernel<true><<<grid, kBseThreads, smem, stream>>>(dm, 0, 2, nc, gam, gg, chi, kc, nullptr, flags, 0,
                                                            nullptr, LadderList{});
  return cudaGetLastError();
}

}  // namespace df
