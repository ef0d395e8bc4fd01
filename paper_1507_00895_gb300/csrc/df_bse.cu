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

template <bool LU_SMEM>
__global__ void __launch_bounds__(kBseThreads)
bse_f64_kernel(Dims dm, int ch0, int nch, int nc, const double2* __restrict__ gam,
               const double2* __restrict__ gg, const double2* __restrict__ chi,
               double2* __restrict__ kc, double2* __restrict__ ws, int* __restrict__ flags, int radius_K,
               const double2* __restrict__ lam, const int* __restrict__ list, int spread) {
  extern __shared__ double2 sm[];
  __shared__ BseF64Shared sh;
  const int n = dm.n_w, N = dm.N, nb = dm.nb, na = dm.na;
  const BseSmem L = bse_layout(n, nc, LU_SMEM);
  double2* LU = LU_SMEM ? sm + L.lu : ws + (size_t)blockIdx.x * n * n;
  // the handle's planes of channels ch0 .. ch0 + nch - 1, or with `list` the
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
// The same ladder term under DF_FP32_IR (n_w <= 64): x = D^-1 gamma L by
// mixed-precision iterative refinement.  D = 1 - gamma_W diag(chi~_W(q)) is
// factorised once in FP32 (complex64 in shared memory, row stride n + 1,
// partial pivoting on |re| + |im|); then, from x = 0 and r = gamma L,
//     D d = r / |r|   (the FP32 factors),   x += |r| d,   r = gamma L - D x
// with x, r and the products gamma v in FP64 (D x = x - gamma (chi~ o x)).
// Each step shrinks the error by about cond(D) 2^-24.  A system stops when
// its correction d is below ir_tol |x| (max norms of |re| + |im|), or when
// d times its ratio to the previous correction is (the error left after a
// contracting step); it is handed back to the FP64 LU kernel (appended to
// `redo`, count in redo[0], output not written here) on an exactly zero FP32
// pivot, a non-finite value, a correction that did not halve, or after
// max_steps solves.  128 threads: all of them run the rank-1 updates (one
// column each, rows split in 128 / n groups; the owners of the next column
// leave per-group pivot candidates, so that a column step takes two
// barriers) and the FP64 row products (128 / n rounded down to a power of
// two lanes per row; those of gamma L interleaved with the column steps);
// warp 0 runs the FP32 triangular solves (two rows per lane in registers).
// ---------------------------------------------------------------------------
constexpr int kChiIrThreads = 128;
constexpr int kChiIrMaxN = 64;

struct ChiIrShared {
  int perm[kChiIrMaxN];
  double2 xs[kChiIrMaxN], lv[kChiIrMaxN], b[kChiIrMaxN], x[kChiIrMaxN], v[kChiIrMaxN], r[kChiIrMaxN];
  float2 invd[kChiIrMaxN];
  // per row group: the largest |re| + |im| of the next pivot column among the
  // group's rows, its row (n when the group has none) and its value
  float pabs[kChiIrThreads];
  int prow[kChiIrThreads];
  float2 pval[kChiIrThreads];
  int bad, state;
};

// sum_j gamma_ij v_j for row i by `tpr` adjacent lanes (lane part of them
// takes j = part mod tpr); every lane of the warp must call it, rows i >= n
// contribute nothing.  The sum is complete in every lane of the group.
__device__ __forceinline__ double2 chi_ir_rowdot(const double2* __restrict__ G, const double2* v, int n, int i,
                                                 int part, int tpr) {
  double2 s0 = mk(0.0, 0.0), s1 = mk(0.0, 0.0);
  if (i < n) {
    const double2* g = G + (size_t)i * n;
    int j = part;
    for (; j + tpr < n; j += 2 * tpr) {
      s0 = cfma(__ldg(g + j), v[j], s0);
      s1 = cfma(__ldg(g + j + tpr), v[j + tpr], s1);
    }
    if (j < n) s0 = cfma(__ldg(g + j), v[j], s0);
  }
  s0 = s0 + s1;
  for (int o = tpr >> 1; o > 0; o >>= 1) {
    s0.x += __shfl_xor_sync(0xffffffffu, s0.x, o);
    s0.y += __shfl_xor_sync(0xffffffffu, s0.y, o);
  }
  return s0;
}

// 1/z in FP32 for the FP32 factorisation (a reciprocal of |z|^2: outside
// ~1e-19 < |z| < 1e19 it gives 0 or non-finite values, and the system is
// handed back by the refinement's checks)
__device__ __forceinline__ float2 cinv_f32(float2 z) {
  const float d = __frcp_rn(z.x * z.x + z.y * z.y);
  return make_float2(z.x * d, -z.y * d);
}

__device__ __forceinline__ double warp_max(double v) {
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

__global__ void __launch_bounds__(kChiIrThreads, 5)
chi_ladder_ir_kernel(Dims dm, const double2* __restrict__ gam, const float2* __restrict__ gam32,
                     const double2* __restrict__ chi, const double2* __restrict__ Lb,
                     const double2* __restrict__ chi0, double2* __restrict__ out, int* __restrict__ redo,
                     int max_steps, double tol) {
  extern __shared__ float2 A[];        // [n][n + 1]
  __shared__ ChiIrShared sh;
  const int n = dm.n_w, N = dm.N, nb = dm.nb, ld = n + 1;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // rank-1 update / build map: column j, row group i0 of rpp
  const int rpp = kChiIrThreads / n, j = tid % n, i0 = tid / n;
  // row-product map: tpr lanes per row
  int tpr = 1;
  while (tpr < 32 && 2 * tpr * n <= kChiIrThreads) tpr *= 2;
  const int ri = tid / tpr, rpart = tid % tpr;
  const long systems = 2L * nb * N;
  for (long sys = blockIdx.x; sys < systems; sys += gridDim.x) {
    const int c = (int)(sys / ((long)nb * N));
    const int rem = (int)(sys - (long)c * nb * N);
    const int a = rem / N, q = rem - a * N;
    const double2* G = gam + ((size_t)c * nb + a) * n * n;
    const float2* G32 = gam32 + ((size_t)c * nb + a) * n * n;
    for (int i = tid; i < n; i += kChiIrThreads) {
      sh.xs[i] = chi[((size_t)a * n + i) * N + q];
      sh.lv[i] = Lb[((size_t)a * n + i) * N + q];
      sh.perm[i] = i;
    }
    if (tid == 0) sh.bad = 0;
    __syncthreads();
    // D in FP32 from gamma's leading FP32 words and FP32-rounded chi~ (only
    // the factorisation uses it; the residuals take D from FP64 gamma); the
    // threads of column 0 leave their row group's pivot candidate
    if (i0 < rpp) {
      const float2 xj = make_float2((float)sh.xs[j].x, (float)sh.xs[j].y);
      float best = -1.f;
      int brow = n;
      float2 bval = make_float2(0.f, 0.f);
      for (int i = i0; i < n; i += rpp) {
        float2 t = cmul(__ldg(G32 + (size_t)i * n + j), xj);
        t = make_float2((i == j ? 1.f : 0.f) - t.x, -t.y);
        A[i * ld + j] = t;
        if (j == 0 && cabs1(t) > best) { best = cabs1(t); brow = i; bval = t; }
      }
      if (j == 0) { sh.pabs[i0] = best; sh.prow[i0] = brow; sh.pval[i0] = bval; }
    }
    __syncthreads();
    // ---- FP32 LU with partial pivoting, two barriers per column; the FP64
    // row products b = gamma L run alongside, one term per column step, their
    // loads issued a step ahead ----
    double2 bacc = mk(0.0, 0.0), gnext = mk(0.0, 0.0);
    if (ri < n && rpart < n) gnext = __ldg(G + (size_t)ri * n + rpart);
    int npart = rpp < n ? rpp : n;         // row groups holding pivot candidates
    for (int k = 0; k < n; ++k) {
      // the pivot of column k from the row groups' candidates (every thread
      // takes the same one: largest, then lowest row)
      float best = -1.f;
      int p = n;
      float2 pv = make_float2(0.f, 0.f);
      for (int g = 0; g < npart; ++g) {
        const float v = sh.pabs[g];
        const int rr = sh.prow[g];
        if (v > best || (v == best && rr < p)) { best = v; p = rr; pv = sh.pval[g]; }
      }
      if (p >= n) { p = k; pv = make_float2(0.f, 0.f); }   // no candidate (NaN column): a zero pivot
      const bool zero = (pv.x == 0.f && pv.y == 0.f);
      const float2 inv = zero ? make_float2(0.f, 0.f) : cinv_f32(pv);
      if (tid == 0) {
        if (zero) sh.bad = 1;
        sh.invd[k] = inv;
        if (p != k) { const int t = sh.perm[k]; sh.perm[k] = sh.perm[p]; sh.perm[p] = t; }
      }
      // rows k and p exchanged (column k: the pivot on the diagonal, the old
      // A_kk scaled into row p), the other multipliers of column k scaled
      if (p != k && tid < n) {
        if (tid == k) {
          const float2 okk = A[k * ld + k];
          A[k * ld + k] = pv;
          A[p * ld + k] = cmul(okk, inv);
        } else {
          const float2 t = A[k * ld + tid];
          A[k * ld + tid] = A[p * ld + tid];
          A[p * ld + tid] = t;
        }
      }
      if (tid > k && tid < n && tid != p) A[tid * ld + k] = cmul(A[tid * ld + k], inv);
      __syncthreads();
      // rank-1 update of the trailing m x m block, spread over all threads:
      // thread = g m + jc takes column k + 1 + jc, rows k + 1 + g + ng t with
      // ng = floor(128 / m) groups (the quotients in FP32: exact here, every
      // true quotient is at least 0.5 / m from an integer); the threads of
      // column k + 1 leave the next pivot candidates
      const int m = n - k - 1;
      if (m > 0) {
        const float rcp = __frcp_rn((float)m);
        const int ng = __float2int_rz(128.f * rcp + 0.5f * rcp);
        const int g = __float2int_rz(((float)tid + 0.5f) * rcp);
        npart = ng < m ? ng : m;
        if (g < ng) {
          const int jcol = k + 1 + (tid - g * m);
          const bool cand = (jcol == k + 1);
          const float2 u = A[k * ld + jcol];
          float bb = -1.f;
          int br = n;
          float2 bv = make_float2(0.f, 0.f);
          int r = k + 1 + g;
          // rows in batches of four, all loads of a batch before its stores
          // (the compiler cannot order them otherwise: columns k and jcol share A)
          for (; r + 3 * ng < n; r += 4 * ng) {
            float2 l[4], t[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              l[e] = A[(r + e * ng) * ld + k];
              t[e] = A[(r + e * ng) * ld + jcol];
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              t[e] = cfms(l[e], u, t[e]);
              A[(r + e * ng) * ld + jcol] = t[e];
            }
            if (cand) {
#pragma unroll
              for (int e = 0; e < 4; ++e)
                if (cabs1(t[e]) > bb) { bb = cabs1(t[e]); br = r + e * ng; bv = t[e]; }
            }
          }
          for (; r < n; r += ng) {
            const float2 t = cfms(A[r * ld + k], u, A[r * ld + jcol]);
            A[r * ld + jcol] = t;
            if (cand && cabs1(t) > bb) { bb = cabs1(t); br = r; bv = t; }
          }
          if (cand && g < m) {
            sh.pabs[g] = bb;
            sh.prow[g] = br;
            sh.pval[g] = bv;
          }
        }
      }
      {
        const int jj = rpart + tpr * k;
        if (ri < n && jj < n) {
          const double2 gv = gnext;
          if (jj + tpr < n) gnext = __ldg(G + (size_t)ri * n + jj + tpr);
          bacc = cfma(gv, sh.lv[jj], bacc);
        }
      }
      __syncthreads();
    }
    for (int o = tpr >> 1; o > 0; o >>= 1) {
      bacc.x += __shfl_xor_sync(0xffffffffu, bacc.x, o);
      bacc.y += __shfl_xor_sync(0xffffffffu, bacc.y, o);
    }
    if (rpart == 0 && ri < n) {
      sh.b[ri] = bacc;
      sh.r[ri] = bacc;
      sh.x[ri] = mk(0.0, 0.0);
    }
    __syncthreads();
    // ---- refinement: state 0 going on, 1 converged, 2 handed back; every
    // thread reads the state right after the barrier that follows its write,
    // and warp 0 writes it again only after the next barrier ----
    int state = sh.bad ? 2 : 0;
    double dprev = 0.0;
    for (int it = 0; state == 0; ++it) {
      if (warp == 0) {
        const bool h0 = lane < n, h1 = lane + 32 < n;
        double rm = fmax(h0 ? cabs1(sh.r[sh.perm[lane]]) : 0.0, h1 ? cabs1(sh.r[sh.perm[lane + 32]]) : 0.0);
        rm = warp_max(rm);
        const double sc = rm > 0.0 ? 1.0 / rm : 0.0;
        float2 y0 = make_float2(0.f, 0.f), y1 = y0;
        if (h0) { const double2 t = sh.r[sh.perm[lane]]; y0 = make_float2((float)(t.x * sc), (float)(t.y * sc)); }
        if (h1) { const double2 t = sh.r[sh.perm[lane + 32]]; y1 = make_float2((float)(t.x * sc), (float)(t.y * sc)); }
        for (int k = 0; k < n - 1; ++k) {          // unit-lower forward substitution
          const float2 src = k < 32 ? y0 : y1;
          const float2 yk = make_float2(__shfl_sync(0xffffffffu, src.x, k & 31), __shfl_sync(0xffffffffu, src.y, k & 31));
          if (lane > k && h0) y0 = cfms(A[lane * ld + k], yk, y0);
          if (lane + 32 > k && h1) y1 = cfms(A[(lane + 32) * ld + k], yk, y1);
        }
        for (int k = n - 1; k >= 0; --k) {         // upper back substitution
          const float2 src = k < 32 ? y0 : y1;
          const float2 yk = make_float2(__shfl_sync(0xffffffffu, src.x, k & 31), __shfl_sync(0xffffffffu, src.y, k & 31));
          const float2 xk = cmul(yk, sh.invd[k]);
          if (lane == k) y0 = xk;
          if (lane + 32 == k) y1 = xk;
          if (lane < k) y0 = cfms(A[lane * ld + k], xk, y0);
          if (lane + 32 < k) y1 = cfms(A[(lane + 32) * ld + k], xk, y1);
        }
        double dn = 0.0, xn = 0.0;
        if (h0) {
          const double2 d = mk((double)y0.x * rm, (double)y0.y * rm);
          const double2 xv = sh.x[lane] + d;
          sh.x[lane] = xv;
          sh.v[lane] = cmul(sh.xs[lane], xv);
          dn = cabs1(d);
          xn = cabs1(xv);
        }
        if (h1) {
          const double2 d = mk((double)y1.x * rm, (double)y1.y * rm);
          const double2 xv = sh.x[lane + 32] + d;
          sh.x[lane + 32] = xv;
          sh.v[lane + 32] = cmul(sh.xs[lane + 32], xv);
          dn = fmax(dn, cabs1(d));
          xn = fmax(xn, cabs1(xv));
        }
        // NaN compares false: a non-finite value hands the system back
        dn = warp_max(isfinite(dn) ? dn : INFINITY);
        xn = warp_max(isfinite(xn) ? xn : INFINITY);
        int st = 0;
        if (!(dn < INFINITY) || !(xn < INFINITY)) st = 2;
        else if (dn <= tol * xn) st = 1;
        else if (it > 0 && dn > 0.5 * dprev) st = 2;
        else if (it > 0 && dn * dn <= 0.5 * tol * xn * dprev) st = 1;
        else if (it + 1 >= max_steps) st = 2;
        dprev = dn;
        if (st == 1) {                              // out = chi0 + L . x
          double2 s2 = mk(0.0, 0.0);
          if (h0) s2 = cfma(sh.lv[lane], sh.x[lane], s2);
          if (h1) s2 = cfma(sh.lv[lane + 32], sh.x[lane + 32], s2);
          for (int o = 16; o > 0; o >>= 1) {
            s2.x += __shfl_xor_sync(0xffffffffu, s2.x, o);
            s2.y += __shfl_xor_sync(0xffffffffu, s2.y, o);
          }
          if (lane == 0) {
            const double2 c0 = chi0[(size_t)a * N + q];
            out[((size_t)c * nb + a) * N + q] = mk(c0.x + s2.x, c0.y + s2.y);
          }
        }
        if (lane == 0) sh.state = st;
      }
      __syncthreads();
      state = sh.state;
      if (state != 0) break;
      {   // r = gamma L - x + gamma (chi~ o x)
        const double2 s = chi_ir_rowdot(G, sh.v, n, ri, rpart, tpr);
        if (rpart == 0 && ri < n) sh.r[ri] = sh.b[ri] - sh.x[ri] + s;
      }
      __syncthreads();
    }
    if (tid == 0 && state == 2) {
      const int slot = atomicAdd(redo, 1);
      redo[1 + slot] = (int)sys;
    }
    __syncthreads();
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
                                                                   c->kc, nullptr, flag_ptr(c), K, lam, nullptr, 0);
    } else {
      bse_f64_kernel<false><<<grid, kBseThreads, smem, c->stream>>>(dm, ch, nch, nc, c->gam, gg_ptr(c), c->chi,
                                                                    c->kc, lu_ws_ptr(c), flag_ptr(c), K, lam,
                                                                    nullptr, 0);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (both) break;
  }
  return cudaSuccess;
}

// the FP64 LU over the ladders the mixed-precision kernels handed back: list[0]
// (read on the device) systems (c N_W + a) N + q, on the persistent grid; a
// list shorter than the SM count is spread over the SMs by right-hand-side ranges
cudaError_t launch_bse_f64_list(df_ctx* c, const int* list) {
  const Dims& dm = c->dm;
  const int n = dm.n_w;
  const int nc = bse_chunk(n) < 16 ? bse_chunk(n) : 16;   // 16-column ranges to spread (fits the default layout)
  const size_t smem = bse_smem_bytes(n);
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
  cudaError_t e = cudaFuncSetAttribute(bse_lu_in_smem(n) ? (const void*)bse_f64_kernel<true>
                                                         : (const void*)bse_f64_kernel<false>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  if (bse_lu_in_smem(n))
    bse_f64_kernel<true><<<c->bse_grid, kBseThreads, smem, c->stream>>>(dm, 0, 2, nc, c->gam, gg_ptr(c), c->chi,
                                                                        c->kc, nullptr, flag_ptr(c), 0, nullptr, list,
                                                                        sms);
  else
    bse_f64_kernel<false><<<c->bse_grid, kBseThreads, smem, c->stream>>>(dm, 0, 2, nc, c->gam, gg_ptr(c), c->chi,
                                                                         c->kc, lu_ws_ptr(c), flag_ptr(c), 0, nullptr,
                                                                         list, sms);
  return cudaGetLastError();
}

// the ladder term of the susceptibilities for both channels: FP64 LU on the
// persistent grid and LU scratch of the FP64 ladder kernel, or under
// DF_FP32_IR the refinement kernel first (D from gamma's FP32 leading words,
// the first array of the mixed-precision workspace) and the FP64 LU only for
// the systems it hands back (redo: 1 + 2 nb N ints)
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
  if (c->opts.precision == DF_FP32_IR && n <= kChiIrMaxN && c->mixed_ws) {
    const size_t ism = sizeof(float2) * (size_t)n * (n + 1);
    e = cudaFuncSetAttribute((const void*)chi_ladder_ir_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ism);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute((const void*)chi_ladder_ir_kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                             (int)cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    int sms = 0, per_sm = 0;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device)) != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (const void*)chi_ladder_ir_kernel, kChiIrThreads, ism);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    const long ig = (long)sms * per_sm;
    if ((e = cudaMemsetAsync(redo, 0, sizeof(int), c->stream)) != cudaSuccess) return e;
    chi_ladder_ir_kernel<<<(int)(systems < ig ? systems : ig), kChiIrThreads, ism, c->stream>>>(
        dm, c->gam, (const float2*)c->mixed_ws, c->chi, Lb, chi0, out, redo, c->opts.ir_max_steps, c->opts.ir_tol);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
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
                                                            nullptr, nullptr, 0);
  return cudaGetLastError();
}

}  // namespace df
