// Leading eigenvalue of A = gamma_W diag(chi~_W(q)) for every (q, W, channel):
// the convergence-radius condition stated after Eq. lin_alg_inv.
//
// Power iteration with a Rayleigh-quotient estimate, first in FP32 (at most
// kEigIter32 steps) until the estimate changes by no more than 2e-6, then
// polished from that vector (at most kEigIter64 steps, to tol) with the
// products gamma (chi~ o v) and the vectors in double-float FP32 (~2^-46
// relative) and the quotients in FP64.  The polish runs for the systems whose FP32 phase
// settled: one that still changes by more than 2e-6 per step after 64
// steps converges at a geometric rate above 0.81, so 24 more steps cannot reach
// 1e-12; it keeps its FP32 estimate, flagged not converged.  Where two
// eigenvalues share the largest modulus (a complex-conjugate pair) one vector
// cannot settle; then the span of the last two iterates gives the pair, to FP32
// accuracy (flag 2).
//
// A block handles Q systems of one (channel, W).  gamma's leading FP32 words
// stay in registers: thread (i, jb) = (tid / 4, tid % 4) of the 4 NP iterating
// threads holds row i, columns CPL jb .. CPL jb + CPL - 1 (NP = 4 CPL >= n_w), its
// trailing words in shared memory.  One step is: u = chi~ o v of every row
// and system to shared memory (two buffers in turn), ONE barrier, y = gamma u,
// the four column blocks of a row summed by shuffles so that lane jb owns
// systems jb QL .. jb QL + QL - 1, the dot products' partial sums per warp to
// shared memory, v = S y.  Everything scalar (sums over the warps, quotients,
// stopping tests, the pair's fit, the next scale) is the work of one extra
// warp, a step behind, while the others multiply: S is a power of two (exact)
// from the growth two steps earlier, so |v| stays near 1 without waiting for
// this step's norm.
//
// Range: chi~ of a system (and gamma, where it is far from one) is scaled by the power of two that brings max|gamma|
// max|chi~| to [1/4, 1) (exact; lambda is scaled back in FP64), so that the first two steps, which
// have no growth to go by, and the squared norms stay within FP32 whatever lambda's size.
// A growth that changes by many orders of magnitude within two steps (a start vector
// that A nearly annihilates) can still carry |v| out of [2^-40, 2^40]: the
// bookkeeping warp sees it, and the block runs the phase again in `exact` mode, which
// waits for each step's own norm (two more barriers a step).  The polish starts from a settled vector,
// with the growth of its last step.  Costs 0.2-1.2 us a launch (128 systems of order 16: 38.0 -> 39.2 us).
//
// Bound by the steps' latency (64 + 24 dependent products) with few systems,
// by FP32 issue with many.  Q = 4 systems share each register of gamma; with
// fewer blocks than SMs Q = 2 spreads them (see launch_lambda).
#include "df_mixed_dev.cuh"

namespace df {

constexpr int kEigIter32 = 64;
constexpr int kEigIter64 = 24;

template <int CPL, int Q>
struct EigShape {
  static constexpr int NP = 4 * CPL;                 // padded order
  static constexpr int T = 4 * NP;                   // iterating threads
  static constexpr int NW = T / 32;                  // their warps
  static constexpr int QL = Q >= 4 ? Q / 4 : 1;      // systems per owning lane (Q = 2: lanes jb < 2 own one)
  static constexpr int US = CPL * Q + 2;             // stride of a column block of u (float2): 16 bytes off per block
  static constexpr int LS = CPL * NP + 8;            // stride of a column block of gamma's trailing words
  static constexpr size_t smem() {                   // u hi, lo (two buffers each), gamma lo, the steps' sums
    return sizeof(float2) * (size_t)(4 * 4 * US + 4 * LS) + sizeof(float) * kEigIter32 * Q * 8;
  }
};

// sum over the four column blocks of a row (lanes jb = lane & 3): on return
// y[k], k < QL, are the sums of this lane's own systems
template <int Q, int QL>
__device__ __forceinline__ void eig_fold(float2 (&y)[Q], int jb, float2 (&out)[QL]) {
  if constexpr (Q >= 4) {
    // exchange halves: after xor 2 this lane keeps systems of its jb >> 1 half, after xor 1 its own
    constexpr int H = Q / 2;
    float2 a[H];
#pragma unroll
    for (int t = 0; t < H; ++t) {
      const float2 send = (jb & 2) ? y[t] : y[H + t], keep = (jb & 2) ? y[H + t] : y[t];
      a[t] = make_float2(keep.x + __shfl_xor_sync(0xffffffffu, send.x, 2),
                         keep.y + __shfl_xor_sync(0xffffffffu, send.y, 2));
    }
#pragma unroll
    for (int t = 0; t < QL; ++t) {
      const float2 send = (jb & 1) ? a[t] : a[QL + t], keep = (jb & 1) ? a[QL + t] : a[t];
      out[t] = make_float2(keep.x + __shfl_xor_sync(0xffffffffu, send.x, 1),
                           keep.y + __shfl_xor_sync(0xffffffffu, send.y, 1));
    }
  } else {
#pragma unroll
    for (int o = 1; o < 4; o <<= 1)
#pragma unroll
      for (int t = 0; t < Q; ++t) {
        y[t].x += __shfl_xor_sync(0xffffffffu, y[t].x, o);
        y[t].y += __shfl_xor_sync(0xffffffffu, y[t].y, o);
      }
    out[0] = (jb & 1) ? y[Q - 1] : y[0];
  }
}

// the power of two next to 1 / sqrt(w), within 2^+-40 (1 for a zero or non-finite w)
__device__ __forceinline__ float eig_pow2(float w) {
  if (!(w > 0.f) || !(w < 3e38f)) return 1.f;
  int e = (int)((__float_as_uint(w) >> 23) & 0xFFu) - 127;
  e = e < -80 ? -80 : (e > 80 ? 80 : e);
  return __int_as_float((127 - (e >> 1)) << 23);
}
// S of step j + 2 from |y_j|^2 = yy, S_j and S_{j+1}: with the growth
// g^2 = |y_j|^2 / |v_j|^2 kept, |v_{j+2}|^2 = yy S_j^2 S_{j+1}^2 g^2, and S^2 = 1 / (g^2 |v_{j+2}|^2) rounded
// to a power of four brings |v_{j+3}| into [1/2, 2]
__device__ __forceinline__ float eig_scale(float yy, float g2, float sj, float sj1) {
  const float a = g2 * (sj * sj1);
  return eig_pow2((yy * a) * a);                               // g^2 |v_{j+2}|^2
}
// the squared norms the steps can work with: 2^-80 .. 2^80
constexpr float kEigMin = 8.3e-25f, kEigMax = 1.2e24f;

template <int CPL, int Q>
__global__ void __launch_bounds__(EigShape<CPL, Q>::T + 32, CPL <= 8 ? 3 : (CPL <= 16 ? 2 : 1))
lambda_kernel(Dims dm, int ch0, int a0, int na, double tol, const double2* __restrict__ gam,
              const double2* __restrict__ chi, double2* __restrict__ lam, int* __restrict__ ok,
              int* __restrict__ flags) {
  using E = EigShape<CPL, Q>;
  constexpr int NP = E::NP, NW = E::NW, QL = E::QL, US = E::US, LS = E::LS;
  extern __shared__ __align__(16) float2 sm[];
  float2* uh = sm;                                   // [2][4][US]
  float2* ul = uh + 8 * US;
  float2* glo = ul + 8 * US;                         // [4][LS]: [k][i]
  float* hist = reinterpret_cast<float*>(glo + 4 * LS);   // [kEigIter32][Q][8]: the FP32 phase's sums
  __shared__ float part[2][NW][Q][8];                // per warp: FP32 phase: v^H y, |y|^2, vprev^H y; polish: pairs of
                                                     // v^H y (re, im), |y|^2, |v|^2
  __shared__ float scal[2][Q];                       // S of a step
  __shared__ int stop_s[2], conv_s[Q], lost_s;
  const int n = dm.n_w, N = dm.N, nb = dm.nb;
  const int qtiles = (N + Q - 1) / Q;
  const int tile = blockIdx.x % qtiles;
  const int a = a0 + (blockIdx.x / qtiles) % na;
  const int c = ch0 + blockIdx.x / (qtiles * na);
  const int q0 = tile * Q;
  const int nq = min(Q, N - q0);
  const double2* Gg = gam + ((size_t)c * nb + a) * n * n;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool book = warp == NW;                      // the bookkeeping warp
  const int i = tid >> 2, jb = tid & 3;
  const bool owner = !book && (Q >= 4 || jb < Q);
  const int t0 = Q >= 4 ? jb * QL : (jb & 1);        // this lane's first system
  const int uo = (i / CPL) * US + (i % CPL) * Q + t0;

  // gamma's words, chi~, the start vector
  float2 gh[CPL];
  float2 xh[QL], xl[QL], v[QL], vp[QL];
  auto split = [](double2 z, float2& hi, float2& lo) {
    hi = make_float2((float)z.x, (float)z.y);
    lo = make_float2((float)(z.x - (double)hi.x), (float)(z.y - (double)hi.y));
  };
  auto top = [](double2 z) {
    return (unsigned)max(__double2hiint(z.x) & 0x7FFFFFFF, __double2hiint(z.y) & 0x7FFFFFFF);
  };
  if (!book) {
    unsigned gm = 0u, xm[QL];
#pragma unroll
    for (int k = 0; k < CPL; ++k) {
      const int j = CPL * jb + k;
      const double2 g = (i < n && j < n) ? Gg[(size_t)i * n + j] : mk(0.0, 0.0);
      float2 lo;
      split(g, gh[k], lo);
      glo[jb * LS + k * NP + i] = lo;
      gm = max(gm, top(g));
    }
#pragma unroll
    for (int k = 0; k < QL; ++k) {
      const double2 x = (i < n && t0 + k < nq) ? chi[((size_t)a * n + i) * N + q0 + t0 + k] : mk(0.0, 0.0);
      split(x, xh[k], xl[k]);
      xm[k] = top(x);
    }
    // the largest upper FP64 words of |gamma| in the warp's rows, of |chi~| in its systems' entries
    gm = __reduce_max_sync(0xffffffffu, gm);
    if (lane == 0) part[0][warp][0][7] = __uint_as_float(gm);
#pragma unroll
    for (int k = 0; k < QL; ++k) {
#pragma unroll
      for (int o = 4; o < 32; o <<= 1) xm[k] = max(xm[k], __shfl_xor_sync(0xffffffffu, xm[k], o));
      if (lane < 4 && owner) part[0][warp][t0 + k][6] = __uint_as_float(xm[k]);
    }
  }
  __syncthreads();
  // exponents of the block's gamma and of system t's chi~ (|value| < 2^e; 0 for an infinite or NaN one): lambda
  // of the problem with both brought to 2^0 is 2^-(eg + ex) lambda.  False for A = 0
  int eg = 0;                                        // (the block's)
  auto range_exp = [&](int t, int& ex) {
    unsigned g = 0u, x = 0u;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      g = max(g, __float_as_uint(part[0][w][0][7]));
      x = max(x, __float_as_uint(part[0][w][t][6]));
    }
    eg = g != 0u && g < 0x7FF00000u ? (int)(g >> 20) - 1022 : 0;
    ex = x < 0x7FF00000u ? (int)(x >> 20) - 1022 : 0;
    return g != 0u && x != 0u;
  };
  int lexp = 0;                                      // eg + ex of the bookkeeping lane's system
  bool alive = false;
  if (book) {
    if (lane < nq) {
      alive = range_exp(lane, lexp);
      lexp = alive ? lexp + eg : 0;
    }
  } else {
    // far from one, the words are made anew from the scaled FP64 value (their trailing ones would leave FP32's
    // range); else chi~'s alone take both powers of two
    constexpr int kFar = 40;
#pragma unroll
    for (int k = 0; k < QL; ++k) {
      int ex;
      if (!range_exp(t0 + k, ex)) continue;
      int r = ex + (eg > kFar || eg < -kFar ? 0 : eg);
      if (ex > kFar || ex < -kFar) {
        const double2 x = (i < n && t0 + k < nq) ? chi[((size_t)a * n + i) * N + q0 + t0 + k] : mk(0.0, 0.0);
        split(mk(scalbn(x.x, -ex), scalbn(x.y, -ex)), xh[k], xl[k]);
        r -= ex;
      }
      xh[k] = cscale(xh[k], pow2f(-r));
      xl[k] = cscale(xl[k], pow2f(-r));
    }
    if (eg > kFar || eg < -kFar) {
      for (int k = 0; k < CPL; ++k) {
        const int j = CPL * jb + k;
        const double2 g = (i < n && j < n) ? Gg[(size_t)i * n + j] : mk(0.0, 0.0);
        float2 hi, lo;
        split(mk(scalbn(g.x, -eg), scalbn(g.y, -eg)), hi, lo);
#pragma unroll
        for (int m = 0; m < CPL; ++m)
          if (m == k) gh[m] = hi;
        glo[jb * LS + k * NP + i] = lo;
      }
    }
  }

  // ---- FP32 phase ----
  // bookkeeping state of system `lane` (step j's data is handled during step j + 1): the iterate's
  // norm, S of the next step, the last quotient.  Kept short: it is on the steps' critical path
  // (se: the last step's S in exact mode, g2: its squared growth, wmin, wmax: the squared norms met)
  float vv = 1.f, s1 = 1.f, se = 1.f, g2 = 0.f, wmin = 1.f, wmax = 1.f;
  float2 l32 = make_float2(0.f, 0.f);
  bool done = false, pconv = false, exact = false;
  float2 pr1 = l32, pr2 = l32;
  auto book32 = [&](int j) {                         // step j of the FP32 phase
    if (lane < Q) {
      float r[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int w = 0; w < NW; ++w)
#pragma unroll
        for (int m = 0; m < 5; ++m) r[m] += part[j & 1][w][lane][m];
      const float yy = r[2], sj = exact ? se : j < 2 ? 1.f : s1;   // S used to form the iterate after step j
      const float2 ln = cscale(make_float2(r[0], r[1]), vv > 0.f ? __fdividef(1.f, vv) : 0.f), d = ln - l32;
      if (cabs2(d) <= 4e-12f * cabs2(ln)) done = true;
      l32 = ln;
      g2 = vv > 0.f ? __fdividef(yy, vv) : 0.f;
      wmin = fminf(wmin, fminf(yy, vv));
      wmax = fmaxf(wmax, fmaxf(yy, vv));
      const float sj1 = j < 1 ? 1.f : scal[(j + 1) & 1][lane];   // S of step j + 1 (published one step ago)
      scal[j & 1][lane] = eig_scale(yy, g2, sj, sj1);            // S of step j + 2
      float* h = hist + ((size_t)j * Q + lane) * 8;              // for the pair's fit
      h[0] = r[0];
      h[1] = r[1];
      h[2] = vv;
      h[3] = r[3];
      h[4] = r[4];
      h[5] = sj;
      vv = sj * sj * yy;
      s1 = sj1;
    }
    const int all = __all_sync(0xffffffffu, done || lane >= Q);
    if (lane == 0) stop_s[j & 1] = all;
  };
  auto scale_now = [&](int j) {                      // exact mode: S of step j from its own norm
    if (lane < Q) {
      float yy = 0.f;
#pragma unroll
      for (int w = 0; w < NW; ++w) yy += part[j & 1][w][lane][2];
      se = eig_pow2(yy);
      scal[j & 1][lane] = se;
    }
  };
  // The dominant pair from span{v_prev, v} of step j > 0: A v_prev = v / S_{j-1}, fit A v ~ al v +
  // be v_prev (least squares), l^2 - al l - be / S_{j-1} = 0.  For a pair the two iterates'
  // overlap oscillates; a fit counts only when the normalised Gram determinant is
  // above 0.1 (FP32 rounding amplified <= 10x).
  auto pair_fit = [&](int j, float2& l1, float2& l2) -> bool {
    const float* h = hist + ((size_t)j * Q + lane) * 8;
    const float* h0 = h - Q * 8;
    const float2 rq = make_float2(h[0], h[1]), g = make_float2(h[3], h[4]);
    const float nv = h[2], nv0 = h0[2], s0 = h0[5];
    const float2 ov = cscale(make_float2(h0[0], h0[1]), s0);     // v_prev^H v
    const float det = nv * nv0 - cabs2(ov);
    if (!(det > 0.1f * nv * nv0)) return false;
    const float id = __fdividef(1.f, det), c1 = __fdividef(1.f, s0);
    const float2 al = cscale(cscale(rq, nv0) - cmul(cconj(ov), g), id);
    const float2 be = cscale(cscale(g, nv) - cmul(ov, rq), id);
    const float2 disc = cmul(al, al) + cscale(be, 4.f * c1);
    const float dmod = sqrtf(cabs2(disc));
    float2 sq = make_float2(sqrtf(fmaxf(0.5f * (dmod + disc.x), 0.f)), sqrtf(fmaxf(0.5f * (dmod - disc.x), 0.f)));
    if (disc.y < 0.f) sq.y = -sq.y;
    l1 = cscale(al + sq, 0.5f);
    l2 = cscale(al - sq, 0.5f);
    return true;
  };
  int it;
  for (;;) {
    if (!book) {
#pragma unroll
      for (int k = 0; k < QL; ++k) {
        v[k] = make_float2(i < n ? rsqrtf((float)n) : 0.f, 0.f);
        vp[k] = make_float2(0.f, 0.f);
      }
    } else if (lane < Q) {
      scal[0][lane] = scal[1][lane] = 1.f;
      if (lane < 2) stop_s[lane] = 0;
      vv = s1 = 1.f;
      l32 = make_float2(0.f, 0.f);
      done = lane >= nq;
    }
    __syncthreads();                                 // (part's maxima are read)
    for (it = 0;; ++it) {
      if (owner) {
        float2* u = uh + (it & 1) * 4 * US + uo;
#pragma unroll
        for (int k = 0; k < QL; ++k) u[k] = cmul(xh[k], v[k]);
      }
      __syncthreads();
      // the flag of step it - 2 (written during step it - 1); the pair is for systems that never settle
      if (it == kEigIter32 || (it >= 2 && stop_s[it & 1])) break;
      float2 yo[QL];
      if (book) {
        if (it > 0) book32(it - 1);
      } else {
        float2 y[Q];
#pragma unroll
        for (int t = 0; t < Q; ++t) y[t] = make_float2(0.f, 0.f);
        const float4* ub = reinterpret_cast<const float4*>(uh + (it & 1) * 4 * US + jb * US);
#pragma unroll
        for (int k = 0; k < CPL; ++k)
#pragma unroll
          for (int tp = 0; tp < Q / 2; ++tp) {
            const float4 w = ub[k * (Q / 2) + tp];
            y[2 * tp] = cfma(gh[k], make_float2(w.x, w.y), y[2 * tp]);
            y[2 * tp + 1] = cfma(gh[k], make_float2(w.z, w.w), y[2 * tp + 1]);
          }
        eig_fold<Q, QL>(y, jb, yo);
#pragma unroll
        for (int k = 0; k < QL; ++k) {
          const float2 rq = cmul(cconj(v[k]), yo[k]), g = cmul(cconj(vp[k]), yo[k]);
          float p[5] = {rq.x, rq.y, cabs2(yo[k]), g.x, g.y};
#pragma unroll
          for (int m = 0; m < 5; ++m)
#pragma unroll
            for (int o = 4; o < 32; o <<= 1) p[m] += __shfl_xor_sync(0xffffffffu, p[m], o);
          if (lane < 4 && owner) {
#pragma unroll
            for (int m = 0; m < 5; ++m) part[it & 1][warp][t0 + k][m] = p[m];
          }
        }
      }
      if (exact) {
        __syncthreads();
        if (book) scale_now(it);
        __syncthreads();
      }
      if (!book) {
#pragma unroll
        for (int k = 0; k < QL; ++k) {
          const float s = scal[it & 1][t0 + k];
          vp[k] = v[k];
          v[k] = cscale(yo[k], s);
        }
      }
    }
    __syncthreads();                                 // every thread has read the flag
    // the last step's data (part of step it - 1 was complete at the barrier before)
    if (book) {
      book32(it - 1);
      const int again = !exact && __any_sync(0xffffffffu, alive && !(wmin > kEigMin && wmax < kEigMax));
      if (lane == 0) lost_s = again;
    }
    __syncthreads();
    if (!lost_s) break;
    exact = true;
  }
  if (book) {
    // systems that never settled: the last two fits that count, settled when both
    // roots agree within 1e-4 (their order may swap)
    if (lane < Q && !done) {
      int j = it - 1;
      while (j > 0 && !pair_fit(j, pr1, pr2)) --j;
      float2 o1, o2;
      for (--j; j > 0; --j) {
        if (!pair_fit(j, o1, o2)) continue;
        const bool sw = cabs2(pr1 - o2) + cabs2(pr2 - o1) < cabs2(pr1 - o1) + cabs2(pr2 - o2);
        const float2 d1 = (sw ? pr2 : pr1) - o1, d2 = (sw ? pr1 : pr2) - o2;
        const float sc2 = 1e-8f * fmaxf(cabs2(pr1), cabs2(pr2));
        pconv = cabs2(d1) <= sc2 && cabs2(d2) <= sc2;
        break;
      }
    }
    if (lane < Q) conv_s[lane] = lane < nq && done;
    if (lane < 2) stop_s[lane] = 0;
    if (lane < Q) {                                  // the polish goes on at the last step's growth
      scal[0][lane] = eig_pow2(g2 * vv);
      scal[1][lane] = eig_pow2(g2);
    }
  }
  __syncthreads();
  int any = 0;
#pragma unroll
  for (int t = 0; t < Q; ++t) any |= conv_s[t];

  // ---- double-float polish from the FP32 vector ----
  const bool conv = book && lane < Q && conv_s[lane];
  double2 lo = mk(0.0, 0.0);
  bool dn = !conv;
  const float sp0 = eig_pow2(g2 * vv), sp1 = eig_pow2(g2);
  auto book64 = [&](int j) {                         // step j of the polish
    if (lane < Q) {
      double r[4];
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        float h = 0.f, l = 0.f;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
          df_add(h, l, part[j & 1][w][lane][2 * m]);
          l += part[j & 1][w][lane][2 * m + 1];
        }
        r[m] = (double)h + (double)l;
      }
      if (!dn) {
        const double iv = r[3] > 0.0 ? 1.0 / r[3] : 0.0;
        const double2 ln = mk(r[0] * iv, r[1] * iv), d = ln - lo;
        if (j > 0 && cabs2(d) <= tol * tol * cabs2(ln)) dn = true;
        lo = ln;
      }
      const float sj = j == 0 ? sp0 : j == 1 ? sp1 : s1, sj1 = j < 1 ? sp1 : scal[(j + 1) & 1][lane];
      const float y2 = (float)r[2], v2 = (float)r[3];
      scal[j & 1][lane] = eig_scale(y2, v2 > 0.f ? __fdividef(y2, v2) : 0.f, sj, sj1);
      s1 = sj1;
    }
    const int all = __all_sync(0xffffffffu, dn || lane >= Q);
    if (lane == 0) stop_s[j & 1] = all;
  };
  if (any) {
    float2 vl[QL];
#pragma unroll
    for (int k = 0; k < QL; ++k) vl[k] = make_float2(0.f, 0.f);
    int ip = 0;
    for (;; ++ip) {
      if (owner) {
        float2* u = uh + (ip & 1) * 4 * US + uo;
        float2* w = ul + (ip & 1) * 4 * US + uo;
#pragma unroll
        for (int k = 0; k < QL; ++k) {               // chi~ o v in double-float
          float sr = 0.f, lr = 0.f, si = 0.f, li = 0.f;
          cdf_fma(sr, lr, si, li, xh[k], xl[k], v[k], vl[k]);
          const float hr = sr + lr, hi = si + li;
          u[k] = make_float2(hr, hi);
          w[k] = make_float2(lr - (hr - sr), li - (hi - si));
        }
      }
      __syncthreads();
      if (ip == kEigIter64 || (ip >= 2 && stop_s[ip & 1])) break;
      if (book) {
        if (ip > 0) book64(ip - 1);
        continue;
      }
      // y = gamma u in double-float, two systems at a time (register pressure); the
      // pairs whose systems both kept their FP32 estimate are left out
      float2 ys[QL], yl[QL];
#pragma unroll
      for (int k = 0; k < QL; ++k) ys[k] = yl[k] = make_float2(0.f, 0.f);
#pragma unroll
      for (int h2 = 0; h2 < Q / 2; ++h2) {
        if (!(conv_s[2 * h2] | conv_s[2 * h2 + 1])) continue;
        float sr[2], lr[2], si[2], li[2];
#pragma unroll
        for (int t = 0; t < 2; ++t) sr[t] = lr[t] = si[t] = li[t] = 0.f;
        const float4* bh = reinterpret_cast<const float4*>(uh + (ip & 1) * 4 * US + jb * US) + h2;
        const float4* bl = reinterpret_cast<const float4*>(ul + (ip & 1) * 4 * US + jb * US) + h2;
        const float2* gl = glo + jb * LS + i;
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
          const float4 h = bh[k * (Q / 2)], l = bl[k * (Q / 2)];
          const float2 gk = gl[k * NP];
          cdf_fma(sr[0], lr[0], si[0], li[0], gh[k], gk, make_float2(h.x, h.y), make_float2(l.x, l.y));
          cdf_fma(sr[1], lr[1], si[1], li[1], gh[k], gk, make_float2(h.z, h.w), make_float2(l.z, l.w));
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1)
#pragma unroll
          for (int t = 0; t < 2; ++t) {
            const float a1 = __shfl_xor_sync(0xffffffffu, sr[t], o), a2 = __shfl_xor_sync(0xffffffffu, lr[t], o);
            const float b1 = __shfl_xor_sync(0xffffffffu, si[t], o), b2 = __shfl_xor_sync(0xffffffffu, li[t], o);
            df_add(sr[t], lr[t], a1);
            lr[t] += a2;
            df_add(si[t], li[t], b1);
            li[t] += b2;
          }
        // systems 2 h2, 2 h2 + 1 to their owners
#pragma unroll
        for (int k = 0; k < QL; ++k) {
          const int t = t0 + k - 2 * h2;
          if (t == 0 || t == 1) {
            ys[k] = make_float2(t ? sr[1] : sr[0], t ? si[1] : si[0]);
            yl[k] = make_float2(t ? lr[1] : lr[0], t ? li[1] : li[0]);
          }
        }
      }
#pragma unroll
      for (int k = 0; k < QL; ++k) {
        float p[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, d1 = 0.f, d2 = 0.f;
        cdf_fma(p[0], p[1], p[2], p[3], cconj(v[k]), cconj(vl[k]), ys[k], yl[k]);
        cdf_fma(p[4], p[5], d1, d2, cconj(ys[k]), cconj(yl[k]), ys[k], yl[k]);
        cdf_fma(p[6], p[7], d1, d2, cconj(v[k]), cconj(vl[k]), v[k], vl[k]);
#pragma unroll
        for (int o = 4; o < 32; o <<= 1)
#pragma unroll
          for (int m = 0; m < 8; m += 2) {
            const float oh = __shfl_xor_sync(0xffffffffu, p[m], o), ol = __shfl_xor_sync(0xffffffffu, p[m + 1], o);
            df_add(p[m], p[m + 1], oh);
            p[m + 1] += ol;
          }
        if (lane < 4 && owner) {
#pragma unroll
          for (int m = 0; m < 8; ++m) part[ip & 1][warp][t0 + k][m] = p[m];
        }
        const float s = scal[ip & 1][t0 + k];
        // renormalise the pair, scale by the power of two (exact)
        const float hx = ys[k].x + yl[k].x, hy = ys[k].y + yl[k].y;
        vl[k] = make_float2((yl[k].x - (hx - ys[k].x)) * s, (yl[k].y - (hy - ys[k].y)) * s);
        v[k] = make_float2(hx * s, hy * s);
      }
    }
    if (book) book64(ip - 1);
  }
  if (book && lane < nq) {
    const size_t o = ((size_t)c * nb + a) * N + q0 + lane;
    double2 l = conv ? lo : mk((double)l32.x, (double)l32.y);
    int okv = conv && dn ? 1 : 0;
    if (!conv && pconv) {
      // a settled dominant pair: the root of larger modulus (of equal moduli,
      // the one with the larger imaginary part), to FP32 accuracy
      const float m1 = cabs2(pr1), m2 = cabs2(pr2);
      const bool first = m1 > m2 * (1.f + 1e-5f) || (m2 <= m1 * (1.f + 1e-5f) && pr1.y >= pr2.y);
      const float2 lp = first ? pr1 : pr2;
      l = mk((double)lp.x, (double)lp.y);
      okv = 2;
    }
    l = mk(scalbn(l.x, lexp), scalbn(l.y, lexp));
    lam[o] = l;
    ok[o] = okv;
    if (!(cabs2(l) < 1.0)) atomicOr(flags, kFlagRadius);   // (a value that is not finite counts as outside)
  }
}

template <int CPL, int Q>
static cudaError_t launch_lambda_shape(df_ctx* c, int ch0, int nch, int a0, int na) {
  using E = EigShape<CPL, Q>;
  const Dims& dm = c->dm;
  auto fn = lambda_kernel<CPL, Q>;
  const cudaError_t e =
      cudaFuncSetAttribute((const void*)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)E::smem());
  if (e != cudaSuccess) return e;
  const int blocks = nch * na * ((dm.N + Q - 1) / Q);
  fn<<<blocks, E::T + 32, E::smem(), c->stream>>>(dm, ch0, a0, na, 1e-12, c->gam, c->chi, c->lam, c->lam_ok,
                                                  bse_flags(c));
  return cudaGetLastError();
}

template <int Q>
static cudaError_t launch_lambda_q(df_ctx* c, int ch0, int nch, int a0, int na) {
  const int n = c->dm.n_w;
  if (n <= 16) return launch_lambda_shape<4, Q>(c, ch0, nch, a0, na);
  if (n <= 32) return launch_lambda_shape<8, Q>(c, ch0, nch, a0, na);
  if (n <= 48) return launch_lambda_shape<12, Q>(c, ch0, nch, a0, na);
  if (n <= 64) return launch_lambda_shape<16, Q>(c, ch0, nch, a0, na);
  if (n <= 96) return launch_lambda_shape<24, Q>(c, ch0, nch, a0, na);
  return launch_lambda_shape<32, Q>(c, ch0, nch, a0, na);
}

cudaError_t launch_lambda(df_ctx* c, int channel_mask) {
  const Dims& dm = c->dm;
  if (c->opts.eig_mode == 0 || !(channel_mask & 3)) return cudaSuccess;
  // W = 0 only (eig_mode 1) or every plane, within the handle's bosonic range
  if (c->opts.eig_mode == 1 && (dm.m_max < dm.a0 || dm.m_max >= dm.a0 + dm.na)) return cudaSuccess;
  const int a0 = (c->opts.eig_mode == 1) ? dm.m_max : dm.a0;
  const int na = (c->opts.eig_mode == 1) ? 1 : dm.na;
  const int ch0 = (channel_mask & 1) ? 0 : 1;
  const int nch = (channel_mask & 3) == 3 ? 2 : 1;   // both channels in one launch when both are asked for
  int sms = 0;
  const cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
  if (e != cudaSuccess) return e;
  // Q = 4 systems per block, or 2 when 4 leave SMs without a block.  Measured (us, Q = 2 / 4 / 8; polish in all systems):
  // 2048 systems of order 16 101 / 102 / 139, 48 420 / 324 / 434, 64 530 / 473 / 680, 96 1485 / 916 / 1267,
  // 128 1881 / 1525 / 1719; 128 systems of order 48 145 / 170 / 233, 128 413 / 656 / 1301
  const long blocks4 = (long)nch * na * ((dm.N + 3) / 4);
  return blocks4 >= sms ? launch_lambda_q<4>(c, ch0, nch, a0, na) : launch_lambda_q<2>(c, ch0, nch, a0, na);
}

}  // namespace df
