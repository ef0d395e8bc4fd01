// The ladder term of the susceptibilities under DF_FP32_IR (n_w <= 64): for one
// (q, W, channel) out = chi0 + L . x, D x = gamma L, D = 1 - gamma_W diag(chi~_W(q)),
// by mixed-precision iterative refinement with the FP32 inverse S ~ D^-1:
//     d_0 = S (gamma L),   x = sum_i d_i,   d_i = S r_i,   r_i = gamma L - D x,
// x and r in FP64.  Each step shrinks the error by about cond(D) 2^-24.  A system
// stops when its correction d is below ir_tol |x| (max norms of |re| + |im|), or when
// d times its ratio to the previous correction is (the error left after a
// contracting step); it is handed back to the FP64 LU kernel (appended to
// `redo`, count in redo[0], output not written here) on an exactly zero FP32
// pivot, a non-finite value, a correction that did not halve, or after max_steps solves.
//
//   * S by the in-place Gauss-Jordan sweep of df_mixed32_dev.cuh (unscaled rows, implicit
//     partial pivoting), one ladder by NP threads (two warps at
//     orders 33-64), 8 x 8 (4 x 8) entries of it per thread in registers, where it stays:
//     a solve is one matrix-vector product, not two serial triangular substitutions.
//   * FP64 goes where it is needed, since its pipe is slow here (1.8 FMA per cycle and SM; 64^2 complex
//     multiply-adds are 9k cycles).  d_0 only has to be an FP32 solution, so gamma L in it is a
//     double-float product (2^-46).  r_1 = gamma (L + chi~ o x) - x is one FP64 product.  From then on r_{i+1} =
//     r_i - D d_i, and d_i is below 2^-13 |x|, so that D d_i in double-float (2^-46 of
//     |d_i|) adds less than FP64's rounding of |x| does; while d_i is larger, r comes from x again.
//     L, the residuals and the corrections are scaled by powers of two and the norms compared by their upper
//     FP64 words, so that x may lie anywhere in FP64's range.
//     Error against 64 bits (geometric mean over 8 or 10 inputs), with an FP32 LU and three FP64 products per
//     step -> now: doped square lattice, order 16 2.5e-14 -> 2.4e-14, 30 6.4e-14 -> 6.4e-14, 48 7.1e-14 -> 6.2e-14,
//     64 4.1e-14 -> 4.4e-14; generic vertices, 64 1.2e-13 -> 1.2e-13; the paper's, 48 5.0e-13 -> 5.0e-13.
//   * A block keeps gamma of its (channel, W) in shared memory, FP64 and FP32 (hi, lo) words, and
//     runs six (orders up to 32: twelve) ladders at a time.
// Bound by instruction issue and the two barriers of a sweep step (two warps per ladder, 12 per SM, issue
// 52-65% busy; the step is one body, since eight unrolled ones leave the instruction cache: 7.6 ms).
// Measured, 30,720 ladders of order 64: 4.0 ms (6.3 ms with an FP32 LU in shared memory, two triangular
// substitutions per solve by one warp and three FP64 products; 3.8 with gamma L in FP32 and unscaled);
// five ladders at a time 4.3 ms, four 4.4 ms, both against 3.8.
#include "df_mixed32_dev.cuh"

namespace df {

template <int NP>
struct ChiIr {
  static constexpr int W = NP / 32;                       // warps per ladder
  static constexpr int G = NP / 8;                        // column classes: column = lcol + G r
  static constexpr int RP = NP / 8, CP = 8;               // rows, columns per thread
  static constexpr int PS = RP + 2, kCol = 8 * PS;        // a column: 8 row classes, padded against bank conflicts
  static constexpr int LD = NP + 8;                       // column stride of gamma's words (bank offset 16)
  static constexpr int oHi = NP * NP * 16, oLo = oHi + NP * LD * 8, oLad = oLo + NP * LD * 8;
  // per ladder: chi~, L, x, y (FP64); their FP32 forms / vectors; the sweep's column and row (two slots)
  static constexpr int oL = NP * 16, oX = 2 * NP * 16, oY = 3 * NP * 16, oVh = 4 * NP * 16, oVl = oVh + NP * 8,
                       oPart = oVl + NP * 8, oCol = oPart + 2 * NP * 8, oRow = oCol + 2 * kCol * 8,
                       oInv = oRow + 2 * NP * 8, oPiv = oInv + NP * 8, oStep = oPiv + NP * 4, oRed = oStep + NP * 4,
                       kLadder = oRed + 64;
  static constexpr int kLadders = NP == 64 ? 6 : 12;
  static constexpr int kThreads = NP * kLadders;
  static constexpr int kSmem = oLad + kLadders * kLadder;
};
static_assert(ChiIr<64>::kSmem <= 232448 && ChiIr<32>::kSmem <= 232448, "a block's shared memory");

template <int NP>
__device__ __forceinline__ void chi_ir_sync(int ladder) {
  if constexpr (NP == 64)
    asm volatile("bar.sync %0, 64;" ::"r"(1 + ladder) : "memory");
  else
    __syncwarp();
}

// max of |v| (|re| + |im|) over a ladder's threads, its lower word cut off (2^-20; the whole FP64 range; an
// infinity or NaN wins): the upper word; red: a slot per call of a sequence
template <int NP>
__device__ __forceinline__ unsigned chi_ir_max(double2 v, unsigned* red, int t, int ladder) {
  unsigned u = __reduce_max_sync(0xffffffffu, (unsigned)__double2hiint(cabs1(v)));
  if constexpr (NP == 64) {
    if ((t & 31) == 0) red[t >> 5] = u;
    chi_ir_sync<NP>(ladder);
    u = max(red[0], red[1]);
  }
  return u;
}
constexpr unsigned kHiInf = 0x7FF00000u;                  // upper word of an infinity
// 2^e (|e| <= 1022), e the exponent of an upper word (0 of zero, subnormal or not finite)
__device__ __forceinline__ int hi_exp(unsigned hi) {
  return hi >= 0x00100000u && hi < 0x7FE00000u ? (int)(hi >> 20) - 1023 : 0;
}
__device__ __forceinline__ double pow2d(int e) { return __hiloint2double((1023 + e) << 20, 0); }

template <int NP>
__device__ __forceinline__ void chi_ir_system(const Dims& dm, int c, int a, int q, const unsigned char* gsm,
                                              unsigned char* ws, const double2* __restrict__ chi,
                                              const double2* __restrict__ Lb, const double2* __restrict__ chi0,
                                              double2* __restrict__ out, int* __restrict__ redo, int max_steps,
                                              double tol, int ladder) {
  using C = ChiIr<NP>;
  constexpr int G = C::G, RP = C::RP, CP = C::CP, LD = C::LD, PS = C::PS;
  const int n = dm.n_w, N = dm.N, nb = dm.nb;
  const int t = threadIdx.x % NP, lane = t & 31, warp = t >> 5, lrow = t & 7, lcol = t >> 3;
  const double2* g64 = reinterpret_cast<const double2*>(gsm);           // [l][i]
  const float2* ghi = reinterpret_cast<const float2*>(gsm + C::oHi);    // [l][i], stride LD
  const float2* glo = reinterpret_cast<const float2*>(gsm + C::oLo);
  double2* xs = reinterpret_cast<double2*>(ws);
  double2* lv = reinterpret_cast<double2*>(ws + C::oL);
  double2* x = reinterpret_cast<double2*>(ws + C::oX);
  double2* y = reinterpret_cast<double2*>(ws + C::oY);
  float2* vh = reinterpret_cast<float2*>(ws + C::oVh);
  float2* vl = reinterpret_cast<float2*>(ws + C::oVl);
  float2* part = reinterpret_cast<float2*>(ws + C::oPart);              // [W][NP]
  float2* pcol = reinterpret_cast<float2*>(ws + C::oCol);               // [2][8][PS]
  float2* prow = reinterpret_cast<float2*>(ws + C::oRow);               // [2][G][CP]
  float2* pinv = reinterpret_cast<float2*>(ws + C::oInv);
  int* piv = reinterpret_cast<int*>(ws + C::oPiv);
  int* rstep = reinterpret_cast<int*>(ws + C::oStep);
  unsigned* red = reinterpret_cast<unsigned*>(ws + C::oRed);
  auto sync = [&]() { chi_ir_sync<NP>(ladder); };

  sync();                                                 // the last ladder's vectors are read
  {
    const double2 xv = t < n ? chi[((size_t)a * n + t) * N + q] : mk(0.0, 0.0);
    const double2 l = t < n ? Lb[((size_t)a * n + t) * N + q] : mk(0.0, 0.0);
    xs[t] = xv;
    lv[t] = l;
    x[t] = mk(0.0, 0.0);
    vh[t] = make_float2((float)xv.x, (float)xv.y);
    piv[t] = t;
    rstep[t] = t;
    pinv[t] = make_float2(0.f, 0.f);
  }
  sync();
  // ---- gamma L in double-float (L to [1, 2)), D in FP32 (only S uses it) ----
  {
    const int e = hi_exp(chi_ir_max<NP>(lv[t], red, t, ladder));
    const double2 l = cscale(lv[t], pow2d(-e));
    const float2 h = make_float2((float)l.x, (float)l.y);
    vl[t] = h;
    part[t] = make_float2((float)(l.x - (double)h.x), (float)(l.y - (double)h.y));
    sync();
    float sr = 0.f, lr = 0.f, si = 0.f, li = 0.f;
#pragma unroll 2
    for (int k = 0; k < n; ++k) cdf_fma(sr, lr, si, li, ghi[k * LD + t], glo[k * LD + t], vl[k], part[k]);
    y[t] = t < n ? cscale(mk((double)sr + (double)lr, (double)si + (double)li), pow2d(e)) : mk(0.0, 0.0);
  }
  float2 A[RP][CP];
#pragma unroll
  for (int r = 0; r < CP; ++r) {
    const int col = lcol + G * r;
    const float2 ch = vh[col];
#pragma unroll
    for (int i = 0; i < RP; ++i) {
      const int row = lrow + 8 * i;
      const float2 g = cmulf(ghi[col * LD + row], ch);
      A[i][r] = make_float2((row == col ? 1.f : 0.f) - g.x, -g.y);
    }
  }
  // ---- in-place Gauss-Jordan sweep ----
  unsigned used = 0u, kmin = ~0u;
#pragma unroll
  for (int i = 0; i < RP; ++i)
    if (lrow + 8 * i >= n) used |= 1u << i;
#pragma unroll 1
  for (int k = 0; k < n; ++k) {                             // (one body for all steps: unrolled it leaves the instruction cache)
    const int s = k & (G - 1);
    float2* pc = pcol + C::kCol * (k & 1);
    float2* pr = prow + NP * (k & 1);
    if (warp == s / 4) {                                    // the warp that holds column k, in register 0 of lcol = s
      unsigned key = 0u;
      if (lcol == s) {
#pragma unroll
        for (int i = 0; i < RP; ++i) {
          const unsigned w = (__float_as_uint(fabsf(A[i][0].x) + fabsf(A[i][0].y)) & ~0x3Fu) | (unsigned)(63 - lrow - 8 * i);
          key = max(key, (used >> i) & 1u ? 0u : w);
        }
#pragma unroll
        for (int i = 0; i < RP; i += 2)
          *reinterpret_cast<float4*>(pc + PS * lrow + i) = make_float4(A[i][0].x, A[i][0].y, A[i + 1][0].x, A[i + 1][0].y);
        // the column becomes the factors, added to 0 by the update
#pragma unroll
        for (int i = 0; i < RP; ++i) A[i][0] = make_float2(0.f, 0.f);
      }
      key = __reduce_max_sync(0xffffffffu, key);
      if (lane == 0) red[4 + (k & 1)] = key;
    }
    sync();
    const unsigned key = red[4 + (k & 1)];
    const int p = (int)(~key & 63u), pi = p >> 3;
    const bool mine = lrow == (p & 7);
    kmin = min(kmin, key);
    float2 f[RP];
#pragma unroll
    for (int i = 0; i < RP; i += 2) {
      const float4 v = *reinterpret_cast<const float4*>(pc + PS * lrow + i);
      f[i] = make_float2(v.x, v.y);
      f[i + 1] = make_float2(v.z, v.w);
    }
    const float2 z = pc[PS * (p & 7) + pi];
    // the pivot row, with 1 in column k, whose own new entry 1 is added in the solves: no later step reads it
#pragma unroll
    for (int i = 0; i < RP; ++i) {
      const bool is = mine && pi == i;
      st_row_if(is, smem_u32(pr + CP * lcol), A[i]);
      f[i] = make_float2(is ? 0.f : f[i].x, is ? 0.f : f[i].y);
    }
    if (mine && lcol == s) pr[CP * lcol] = make_float2(1.f, 0.f);
    if (mine) used |= 1u << pi;
    // approximate reciprocal: S is an approximate inverse
    const float d = rcp_approx(fmaf(z.x, z.x, z.y * z.y));
    const float2 ainv = make_float2(z.x * d, -z.y * d);
    if (t == 0) {
      piv[k] = p;
      rstep[p] = k;
      pinv[p] = ainv;
    }
#pragma unroll
    for (int i = 0; i < RP; ++i) f[i] = cmulf(f[i], make_float2(-ainv.x, -ainv.y));
    sync();
    const float4* u4 = reinterpret_cast<const float4*>(pr + CP * lcol);
    if (s < G - 1) {
#pragma unroll
      for (int r = 0; r < CP; r += 2) {
        const float4 v = u4[r / 2];
#pragma unroll
        for (int i = 0; i < RP; ++i) {
          A[i][r] = cfmaf2(f[i], make_float2(v.x, v.y), A[i][r]);
          A[i][r + 1] = cfmaf2(f[i], make_float2(v.z, v.w), A[i][r + 1]);
        }
      }
    } else {                                                // the columns rotate with the last of G steps
      float2 t0[RP];
#pragma unroll
      for (int r = 0; r < CP; r += 2) {
        const float4 v = u4[r / 2];
#pragma unroll
        for (int i = 0; i < RP; ++i) {
          const float2 a0 = cfmaf2(f[i], make_float2(v.x, v.y), A[i][r]);
          if (r == 0) t0[i] = a0; else A[i][r - 1] = a0;
          A[i][r] = cfmaf2(f[i], make_float2(v.z, v.w), A[i][r + 1]);
        }
      }
#pragma unroll
      for (int i = 0; i < RP; ++i) A[i][CP - 1] = t0[i];
    }
  }
  int state = (kmin & ~0x3Fu) == 0u ? 2 : 0;              // an exactly zero pivot
  sync();
  // thread t owns the solution's entry ks (the step of row t) and the residual's entry t
  const int ks = rstep[t], pt = piv[t], rot = n / G;
  const float2 rinv = pinv[t];
  double2 res = y[t];
  // ---- refinement; every thread takes the same decisions ----
  double dprev = 0.0;
  for (int it = 0; state == 0; ++it) {
    // d = S r, r scaled to [1, 2)
    const int e = hi_exp(chi_ir_max<NP>(res, red + 2 * (it & 1), t, ladder));
    const double sc = pow2d(-e), up = pow2d(e);
    vl[t] = make_float2((float)(res.x * sc), (float)(res.y * sc));
    sync();
    vh[t] = vl[pt];
    sync();
    float2 acc[RP];
#pragma unroll
    for (int i = 0; i < RP; ++i) acc[i] = make_float2(0.f, 0.f);
#pragma unroll
    for (int r = 0; r < CP; ++r) {
      const float2 v = vh[lcol + G * ((r + rot) & (CP - 1))];
#pragma unroll
      for (int i = 0; i < RP; ++i) acc[i] = cfmaf2(A[i][r], v, acc[i]);
    }
#pragma unroll
    for (int i = 0; i < RP; ++i) {
#pragma unroll
      for (int o = 8; o < 32; o <<= 1) {
        acc[i].x += __shfl_xor_sync(0xffffffffu, acc[i].x, o);
        acc[i].y += __shfl_xor_sync(0xffffffffu, acc[i].y, o);
      }
      if (lane < 8) part[NP * warp + lrow + 8 * i] = acc[i];
    }
    sync();
    float2 ys = part[t];
    if constexpr (NP == 64) ys = make_float2(ys.x + part[NP + t].x, ys.y + part[NP + t].y);
    const float2 v1 = vh[ks];                               // the pivot row's entry 1
    ys = cmulf(make_float2(ys.x + v1.x, ys.y + v1.y), rinv);
    const double2 d = t < n ? mk((double)ys.x * up, (double)ys.y * up) : mk(0.0, 0.0);
    const double2 xv = x[ks] + d;
    x[ks] = xv;
    // NaN and infinity compare false: a non-finite value hands the system back
    const unsigned dh = chi_ir_max<NP>(d, red + 6, t, ladder), xh = chi_ir_max<NP>(xv, red + 8, t, ladder);
    const double dn = __hiloint2double(dh, 0), xn = __hiloint2double(xh, 0);
    if (dh >= kHiInf || xh >= kHiInf) state = 2;
    else if (it > 0 && dn <= tol * xn) state = 1;           // (d_0 may be 0 by FP32 underflow alone)
    else if (dprev > 0.0 && dn > 0.5 * dprev) state = 2;
    else if (it > 0 && dn * dn <= 0.5 * tol * xn * dprev) state = 1;
    else if (it + 1 >= max_steps) state = 2;
    if (state != 0) break;
    dprev = dn;
    const double2 ch = xs[ks];
    if (it == 0 || dn > 1.220703125e-4 * xn) {            // r = gamma (L + chi~ o x) - x in FP64
      y[ks] = cfma(ch, xv, lv[ks]);
      sync();
      double2 s0 = mk(0.0, 0.0), s1 = mk(0.0, 0.0);
      if (t < n) {
#pragma unroll 2
        for (int l = 0; l < n; l += 2) {
          s0 = cfma(g64[l * NP + t], y[l], s0);
          s1 = cfma(g64[(l + 1) * NP + t], y[l + 1], s1);
        }
        s0 = s0 + s1;
        res = mk(s0.x - x[t].x, s0.y - x[t].y);
      }
    } else {                                              // r -= d - gamma (chi~ o d), the product in double-float
      const double2 v = cmul(ch, mk((double)ys.x, (double)ys.y));   // 2^-e d
      const float hx = (float)v.x, hy = (float)v.y;
      part[ks] = make_float2(hx, hy);                     // (part's readers are past the norms' barriers)
      vl[ks] = make_float2((float)(v.x - (double)hx), (float)(v.y - (double)hy));
      y[ks] = d;
      sync();
      if (t < n) {
        float sr = 0.f, lr = 0.f, si = 0.f, li = 0.f;
#pragma unroll 2
        for (int l = 0; l < n; ++l) cdf_fma(sr, lr, si, li, ghi[l * LD + t], glo[l * LD + t], part[l], vl[l]);
        res = mk(res.x - y[t].x + ((double)sr + (double)lr) * up, res.y - y[t].y + ((double)si + (double)li) * up);
      }
      if constexpr (NP == 32) __syncwarp();
    }
  }
  if (state == 1) {                                       // out = chi0 + L . x
    double2 s2 = cmul(lv[ks], x[ks]);
    for (int o = 16; o > 0; o >>= 1) {
      s2.x += __shfl_xor_sync(0xffffffffu, s2.x, o);
      s2.y += __shfl_xor_sync(0xffffffffu, s2.y, o);
    }
    if constexpr (NP == 64) {
      if (t == 32) y[0] = s2;
      sync();
      s2 = s2 + y[0];
    }
    if (t == 0) {
      const double2 c0 = chi0[(size_t)a * N + q];
      out[((size_t)c * nb + a) * N + q] = mk(c0.x + s2.x, c0.y + s2.y);
    }
  } else if (t == 0) {
    const int slot = atomicAdd(redo, 1);
    redo[1 + slot] = (int)(((long)c * nb + a) * N + q);
  }
}

// one contiguous range of systems per block, split where (channel, W) changes; the ladders of a
// block take its systems in turn
template <int NP>
__global__ void __launch_bounds__(ChiIr<NP>::kThreads, 1)
chi_ladder_ir_kernel(Dims dm, const double2* __restrict__ gam, const float2* __restrict__ gam_hi,
                     const float2* __restrict__ gam_lo, const double2* __restrict__ chi,
                     const double2* __restrict__ Lb, const double2* __restrict__ chi0, double2* __restrict__ out,
                     int* __restrict__ redo, int max_steps, double tol) {
  using C = ChiIr<NP>;
  extern __shared__ __align__(16) unsigned char smc[];
  const int n = dm.n_w, N = dm.N, nb = dm.nb, ladder = threadIdx.x / NP;
  unsigned char* ws = smc + C::oLad + ladder * C::kLadder;
  const int systems = 2 * nb * N;                          // (<= 2 x 63 x 4096)
  const int s1 = (int)((long)systems * (blockIdx.x + 1) / gridDim.x);
  int s = (int)((long)systems * blockIdx.x / gridDim.x);
  while (s < s1) {
    const int plane = s / N, end = min(s1, (plane + 1) * N);
    const size_t mat = (size_t)plane * n * n;
    __syncthreads();
    for (int idx = threadIdx.x; idx < NP * NP; idx += C::kThreads) {
      const int l = idx / NP, i = idx % NP;
      const bool in = l < n && i < n;
      const size_t src = mat + (size_t)i * n + l;
      reinterpret_cast<double2*>(smc)[idx] = in ? __ldg(gam + src) : mk(0.0, 0.0);
      reinterpret_cast<float2*>(smc + C::oHi)[l * C::LD + i] = in ? __ldg(gam_hi + src) : make_float2(0.f, 0.f);
      reinterpret_cast<float2*>(smc + C::oLo)[l * C::LD + i] = in ? __ldg(gam_lo + src) : make_float2(0.f, 0.f);
    }
    __syncthreads();
    for (int v = s + ladder; v < end; v += C::kLadders)
      chi_ir_system<NP>(dm, plane / nb, plane % nb, v - plane * N, smc, ws, chi, Lb, chi0, out, redo,
                        max_steps, tol, ladder);
    s = end;
  }
}

template <int NP>
static cudaError_t launch_chi_ir_np(df_ctx* c, const double2* Lb, const double2* chi0, double2* out, int* redo) {
  using C = ChiIr<NP>;
  const Dims& dm = c->dm;
  cudaError_t e = cudaFuncSetAttribute((const void*)chi_ladder_ir_kernel<NP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       C::kSmem);
  if (e != cudaSuccess) return e;
  int sms = 0;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device)) != cudaSuccess) return e;
  const size_t count = (size_t)2 * dm.nb * dm.n_w * dm.n_w;
  const float2* hi = (const float2*)c->mixed_ws;
  const long systems = 2L * dm.nb * dm.N;
  chi_ladder_ir_kernel<NP><<<(int)(systems < sms ? systems : sms), C::kThreads, C::kSmem, c->stream>>>(
      dm, c->gam, hi, hi + count, c->chi, Lb, chi0, out, redo, c->opts.ir_max_steps, c->opts.ir_tol);
  return cudaGetLastError();
}

// the systems that did not refine are listed in redo (count, then indices), which the caller clears
cudaError_t launch_chi_ladder_ir(df_ctx* c, const double2* Lb, const double2* chi0, double2* out, int* redo) {
  return c->dm.n_w <= 32 ? launch_chi_ir_np<32>(c, Lb, chi0, out, redo) : launch_chi_ir_np<64>(c, Lb, chi0, out, redo);
}

}  // namespace df
