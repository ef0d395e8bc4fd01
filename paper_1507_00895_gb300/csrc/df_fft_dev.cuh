// Device bodies of the lattice-FFT stages (Eq. gd0, Eq. dyson,
// Eq. dual_bubble, Eq. sd), one (frequency, frequency) plane per CTA.  Used
// by the single-problem kernels (df_fft.cu) and by the batched ones
// (df_batch.cu).  Every function must be called by all threads of the block.
#pragma once
#include "df_internal.cuh"

namespace df {

constexpr int kFftThreads = 256;

__device__ __forceinline__ double eps_of(int r, int D, int p, double t, double tp) {
  const int mask = (1 << p) - 1;
  const double inv_nk = 1.0 / (double)(1 << p);
  double c[4] = {0, 0, 0, 0};
  double e = 0.0;
  for (int d = 0; d < D; ++d) {
    const int j = (r >> ((D - 1 - d) * p)) & mask;   // coordinate along axis d
    c[d] = cospi(2.0 * (double)j * inv_nk);
    e += c[d];
  }
  e *= -2.0 * t;
  if (D == 2) e -= 4.0 * tp * c[0] * c[1];
  return e;
}

// ---- D-dimensional DFT of one plane in shared memory ----
// These transforms are bound by the FP64 pipe (one warp instruction per 17 cycles and SM), so what
// counts is the number of FP64 instructions and that their lanes are full.  From 1024
// points on, every axis of N_k = 2^p points is one or two passes of radix 8 / 4 / 2 in registers
// (4224 warp instructions for 16^3 points, 6144 with radix 2); below, a radix-8 pass would leave
// most lanes of a block empty, and the radix-2 passes of fft_dit_smem stay (8 x 8 points:
// one warp, 48 instructions; radix 8 would take 8 lanes through 112).
// Measured, 16^3 points: bubble_kernel, 1,056 planes, 439 -> 363 us, sigma_prod_kernel 466 -> 391;
// sigma_dyson_kernel, 96 box planes, 286 -> 244, and 196 with dyson<true>;
// dyson_ifft_kernel 109 -> 96 -> 71.  32^2 points, 960 planes: 294 -> 264 us for the four kernels.
// The choice (R8) is a template argument, made on the host: both in one kernel cost the small planes
// 2-25%.  Batches, whose launches mix sizes, take radix 2.
inline bool fft_radix8(const Dims& dm) { return dm.N >= 1024; }

// the element's place: a row of 8 elements (128 bytes) is permuted by its index, so that the strides
// of a pass along the first axis meet different banks
__device__ __forceinline__ int fft_swz(int i) { return i ^ ((i >> 3) & 7); }
// where the transform's input element r goes, where its output element k is found
template <bool R8>
__device__ __forceinline__ int fft_in(const Dims& dm, int r) {
  return R8 ? fft_swz(r) : bitrev_axes(r, dm.D, dm.p);
}
template <bool R8>
__device__ __forceinline__ int fft_out(const Dims& dm, int k) {
  if constexpr (!R8) return k;
  const int p = dm.p, b = p >= 4 ? p / 2 : 0, a = p - b;   // two passes: digit (k mod 2^a, k / 2^a) is stored reversed
  if (b == 0) return fft_swz(k);
  int out = 0;
  for (int d = 0; d < dm.D; ++d) {
    const int j = k >> (d * p);
    out |= (((j & ((1 << a) - 1)) << b) | ((j >> a) & ((1 << b) - 1))) << (d * p);
  }
  return fft_swz(out);
}

// -i z (forward) or +i z (inverse)
template <bool INV>
__device__ __forceinline__ double2 fft_rot(double2 z) {
  return INV ? mk(-z.y, z.x) : mk(z.y, -z.x);
}
template <bool INV>
__device__ __forceinline__ void fft_dft(double2 (&x)[2]) {
  const double2 a = x[0], b = x[1];
  x[0] = a + b;
  x[1] = a - b;
}
template <bool INV>
__device__ __forceinline__ void fft_dft(double2 (&x)[4]) {
  const double2 a = x[0] + x[2], b = x[0] - x[2], c = x[1] + x[3], d = fft_rot<INV>(x[1] - x[3]);
  x[0] = a + c;
  x[1] = b + d;
  x[2] = a - c;
  x[3] = b - d;
}
template <bool INV>
__device__ __forceinline__ void fft_dft(double2 (&x)[8]) {
  double2 e[4] = {x[0], x[2], x[4], x[6]}, o[4] = {x[1], x[3], x[5], x[7]};
  fft_dft<INV>(e);
  fft_dft<INV>(o);
  constexpr double h = 0.70710678118654752440;
  const double2 r1 = fft_rot<INV>(o[1]), r3 = fft_rot<INV>(o[3]);
  o[1] = mk(h * (o[1].x + r1.x), h * (o[1].y + r1.y));      // (1 -+ i) / sqrt 2
  o[2] = fft_rot<INV>(o[2]);
  o[3] = mk(h * (r3.x - o[3].x), h * (r3.y - o[3].y));      // (-1 -+ i) / sqrt 2
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    x[k] = e[k] + o[k];
    x[k + 4] = e[k] - o[k];
  }
}

// One pass over the plane: the 2^LR-point transforms along the top LR of the `rem` index bits of an axis
// (from bit `base`) that are still input bits, times the twiddles w_{2^rem}^(k1 j2), j2 the
// remaining ones; in place.
template <int LR, bool INV>
__device__ __forceinline__ void fft_pass(double2* s, int N, int p, int base, int rem, const double2* tw) {
  constexpr int R = 1 << LR;
  const int lo = base + rem - LR, half = (1 << p) >> 1;
  for (int g = threadIdx.x; g < N >> LR; g += blockDim.x) {
    const int low = g & ((1 << lo) - 1), i0 = ((g >> lo) << (lo + LR)) | low;
    double2 x[R];
#pragma unroll
    for (int m = 0; m < R; ++m) x[m] = s[fft_swz(i0 + (m << lo))];
    fft_dft<INV>(x);
    if (rem > LR) {
      const int j2 = (low >> base) << (p - rem);
#pragma unroll
      for (int k = 1; k < R; ++k) {
        const int m = k * j2;                               // < N_k
        double2 w = tw[m & (half - 1)];
        if (m & half) w = mk(-w.x, -w.y);
        if (INV) w.y = -w.y;
        x[k] = cmul(x[k], w);
      }
    }
#pragma unroll
    for (int m = 0; m < R; ++m) s[fft_swz(i0 + (m << lo))] = x[m];
  }
  __syncthreads();
}

// The transform of the plane in s (input at fft_in, output at fft_out); all threads of the block, which
// have synchronised after storing the input
template <bool R8, bool INV>
__device__ __forceinline__ void fft_plane(const Dims& dm, double2* s, const double2* tw) {
  if constexpr (!R8) {
    fft_dit_smem(s, dm.D, dm.p, tw, INV);
  } else {
    for (int d = 0; d < dm.D; ++d) {
      const int p = dm.p, base = d * p;
      if (p == 3) {
        fft_pass<3, INV>(s, dm.N, p, base, 3, tw);
      } else if (p == 4) {
        fft_pass<2, INV>(s, dm.N, p, base, 4, tw);
        fft_pass<2, INV>(s, dm.N, p, base, 2, tw);
      } else if (p == 5) {
        fft_pass<3, INV>(s, dm.N, p, base, 5, tw);
        fft_pass<2, INV>(s, dm.N, p, base, 2, tw);
      } else {
        fft_pass<3, INV>(s, dm.N, p, base, 6, tw);
        fft_pass<3, INV>(s, dm.N, p, base, 3, tw);
      }
    }
  }
}

// Eq. gd0 for one element idx = e N + r of the extended grid; G~ = G0~.
__device__ __forceinline__ void init_g0_elem(const Dims& dm, int idx, const double2* __restrict__ g,
                                             const double2* __restrict__ delta, double2* __restrict__ g0,
                                             double2* __restrict__ gk) {
  const int e = idx / dm.N, r = idx - e * dm.N;
  const double2 ge = g[e];
  const double eps = eps_of(r, dm.D, dm.p, dm.t, dm.tp);
  double2 den = cinv(ge) + delta[e];
  den.x -= eps;
  const double2 v = cinv(den) - ge;
  g0[idx] = v;
  gk[idx] = v;
}

// Eq. dyson for one element: 1 / (1/G0~ - Sigma~); on the large planes, whose blocks the FP64 pipe bounds,
// as G0~ (1 - G0~ Sigma~)* / |1 - G0~ Sigma~|^2: one FP64 division instead of four.  Error
// against 64 bits over 42 FP64 loops as before (geometric means 9.8e-16 -> 8.8e-16 on 16^3, 3.0e-16 on 32^2).
template <bool R8>
__device__ __forceinline__ double2 dyson(double2 g0, double2 sigma) {
  if constexpr (R8) {
    const double2 den = cfms(g0, sigma, mk(1.0, 0.0));
    const int e = max(__double2hiint(den.x) & 0x7FF00000, __double2hiint(den.y) & 0x7FF00000);
    if (e < 0x20000000 || e > 0x5FF00000) return cmul(g0, cinv(den));   // |den|^2 would leave the range
    const double inv = 1.0 / cabs2(den);
    return cscale(cmul(g0, cconj(den)), inv);
  } else {
    return cinv(cinv(g0) - sigma);
  }
}

// Plane e: G~(k) = Dyson(G0~, Sigma~) inside the box (G0~ outside), then
// G~(r) = (1/N) sum_k exp(ik.r) G~(k).  With sigma == nullptr the plane is
// transformed as given; with gk == nullptr the k-space copy is skipped.
template <bool R8>
__device__ __forceinline__ void dyson_ifft_plane(const Dims& dm, int e, const double2* __restrict__ g0,
                                                 const double2* __restrict__ sigma, double2* __restrict__ gk,
                                                 double2* __restrict__ gr, double2* tw, double2* s) {
  const int i = e - dm.m_max;        // box index or outside
  const bool in_box = (i >= 0 && i < dm.n_w);
  load_twiddles(tw, dm.nk);
  for (int r = threadIdx.x; r < dm.N; r += blockDim.x) {
    double2 v = g0[(size_t)e * dm.N + r];
    if (in_box && sigma) v = dyson<R8>(v, sigma[(size_t)i * dm.N + r]);
    if (gk) gk[(size_t)e * dm.N + r] = v;
    s[fft_in<R8>(dm, r)] = v;
  }
  __syncthreads();
  fft_plane<R8, true>(dm, s, tw);
  const double invN = 1.0 / (double)dm.N;
  for (int r = threadIdx.x; r < dm.N; r += blockDim.x) gr[(size_t)e * dm.N + r] = cscale(s[fft_out<R8>(dm, r)], invN);
  __syncthreads();
}

// Eq. dual_bubble for plane (a, i): chi~(q) = -T FFT[G~_w(-r) G~_{w+W}(r)](q).
template <bool R8>
__device__ __forceinline__ void bubble_plane(const Dims& dm, int a, int i, const double2* __restrict__ gr,
                                             double2* __restrict__ chi, double2* tw, double2* s) {
  const double2* A = gr + (size_t)(i + dm.m_max) * dm.N;   // G~_w
  const double2* B = gr + (size_t)(i + a) * dm.N;          // G~_{w+W}
  load_twiddles(tw, dm.nk);
  for (int r = threadIdx.x; r < dm.N; r += blockDim.x)
    s[fft_in<R8>(dm, r)] = cmul(A[reflect_index(r, dm.D, dm.p)], B[r]);
  __syncthreads();
  fft_plane<R8, false>(dm, s, tw);
  double2* out = chi + ((size_t)a * dm.n_w + i) * dm.N;
  for (int q = threadIdx.x; q < dm.N; q += blockDim.x) out[q] = cscale(s[fft_out<R8>(dm, q)], -dm.T);
  __syncthreads();
}

// Eq. sd, stage 1, plane (a, i): K(r) = (1/N) sum_q exp(iq.r) K(q),
// K = kernel_d + kernel_m, then prod(r) = K(-r) G~_{w+W}(r).
template <bool R8>
__device__ __forceinline__ void sigma_prod_plane(const Dims& dm, int a, int i, const double2* __restrict__ kc,
                                                 const double2* __restrict__ gr, double2* __restrict__ prod,
                                                 double2* tw, double2* s) {
  const size_t plane = ((size_t)a * dm.n_w + i) * dm.N;
  const size_t chstride = (size_t)dm.nb * dm.n_w * dm.N;
  load_twiddles(tw, dm.nk);
  for (int q = threadIdx.x; q < dm.N; q += blockDim.x)
    s[fft_in<R8>(dm, q)] = kc[plane + q] + kc[chstride + plane + q];
  __syncthreads();
  fft_plane<R8, true>(dm, s, tw);
  const double invN = 1.0 / (double)dm.N;
  const double2* B = gr + (size_t)(i + a) * dm.N;
  for (int r = threadIdx.x; r < dm.N; r += blockDim.x)
    prod[plane + r] = cmul(cscale(s[fft_out<R8>(dm, reflect_index(r, dm.D, dm.p))], invN), B[r]);
  __syncthreads();
}

template <int NT>
__device__ __forceinline__ double block_max(double v, double* red_sm) {
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) red_sm[w] = v;
  __syncthreads();
  if (w == 0) {
    v = (l < NT / 32) ? red_sm[l] : 0.0;
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (l == 0) red_sm[0] = v;
  }
  __syncthreads();
  v = red_sm[0];
  __syncthreads();
  return v;
}

// Eq. sd, stage 2a, box frequency i: acc(r) = sum_W prod[W][i](r) over the
// problem's bosonic planes, s = FFT[acc] (at fft_out; the T/2 is applied by
// the caller).  Loads the twiddles into tw.
// With refl (the frequency reflection, full range) only the planes W >= 0 of
// prod are formed: the term of -W at w is that of W at -w, conjugated and taken
// at -r (prod_{-W,w}(r) = prod_{W,-w}(-r)*, from bracket_{-W}(w) = bracket_W(-w)*
// and G~(-w) = G~(w)*).
template <bool R8>
__device__ __forceinline__ void sigma_sum_plane(const Dims& dm, int i, const double2* __restrict__ prod, double2* tw,
                                                double2* s, int refl = 0) {
  load_twiddles(tw, dm.nk);
  const int ir = dm.n_w - 1 - i;
  for (int r = threadIdx.x; r < dm.N; r += blockDim.x) {
    double2 acc = mk(0.0, 0.0);
    if (refl) {
      const int rr = reflect_index(r, dm.D, dm.p);
      for (int a = dm.m_max; a < dm.nb; ++a) acc = acc + prod[((size_t)a * dm.n_w + i) * dm.N + r];
      for (int a = dm.m_max + 1; a < dm.nb; ++a) acc = acc + cconj(prod[((size_t)a * dm.n_w + ir) * dm.N + rr]);
    } else {
      for (int a = dm.a0; a < dm.a0 + dm.na; ++a) acc = acc + prod[((size_t)a * dm.n_w + i) * dm.N + r];
    }
    s[fft_in<R8>(dm, r)] = acc;
  }
  __syncthreads();
  fft_plane<R8, false>(dm, s, tw);
}

// Eq. sd, stage 2b, fused with mixing, the residual partials and Eq. dyson,
// for box frequency i: Sigma~_new(k) = pref s(k); Sigma~ <- mix new +
// (1-mix) old; G~ = 1/(1/G0~ - Sigma~); G~(r) = IFFT[G~(k)] / N.
// red[i], red[n_w + i] = max|dSigma~|, max|Sigma~|.  Needs the twiddles in tw.
template <bool R8>
__device__ __forceinline__ void sigma_finish_plane(const Dims& dm, int i, double mix, double pref, const double2* s,
                                                   const double2* __restrict__ g0, double2* __restrict__ sigma,
                                                   double2* __restrict__ gk, double2* __restrict__ gr,
                                                   double* __restrict__ red, const double2* tw, double2* s2,
                                                   double* red_sm) {
  const int e = i + dm.m_max;
  double dmax = 0.0, smax = 0.0;
  for (int k = threadIdx.x; k < dm.N; k += blockDim.x) {
    const size_t idx = (size_t)i * dm.N + k;
    const double2 old = sigma[idx];
    const double2 nw = cscale(s[fft_out<R8>(dm, k)], pref);
    const double2 sg = mk(mix * nw.x + (1.0 - mix) * old.x, mix * nw.y + (1.0 - mix) * old.y);
    const double2 d = sg - old;
    dmax = fmax(dmax, cabs2(d));
    smax = fmax(smax, cabs2(sg));
    sigma[idx] = sg;
    const double2 gnew = dyson<R8>(g0[(size_t)e * dm.N + k], sg);
    gk[(size_t)e * dm.N + k] = gnew;
    s2[fft_in<R8>(dm, k)] = gnew;
  }
  dmax = block_max<kFftThreads>(dmax, red_sm);
  smax = block_max<kFftThreads>(smax, red_sm);
  if (threadIdx.x == 0) {
    red[i] = sqrt(dmax);
    red[dm.n_w + i] = sqrt(smax);
  }
  fft_plane<R8, true>(dm, s2, tw);
  const double invN = 1.0 / (double)dm.N;
  for (int r = threadIdx.x; r < dm.N; r += blockDim.x) gr[(size_t)e * dm.N + r] = cscale(s2[fft_out<R8>(dm, r)], invN);
  __syncthreads();
}

// Eq. sd (stages 2a and 2b) for box frequency i: Sigma~_new = (T/2) FFT[sum_W prod]
template <bool R8>
__device__ __forceinline__ void sigma_dyson_plane(const Dims& dm, int i, double mix, const double2* __restrict__ prod,
                                                  const double2* __restrict__ g0, double2* __restrict__ sigma,
                                                  double2* __restrict__ gk, double2* __restrict__ gr,
                                                  double* __restrict__ red, double2* tw, double2* s, double2* s2,
                                                  double* red_sm, int refl = 0) {
  sigma_sum_plane<R8>(dm, i, prod, tw, s, refl);
  sigma_finish_plane<R8>(dm, i, mix, 0.5 * dm.T, s, g0, sigma, gk, gr, red, tw, s2, red_sm);
}

// max over red[0..n) and red[n..2n) into red[2n], red[2n+1] (one block)
__device__ __forceinline__ void residual_reduce_block(int n, double* red, double* red_sm) {
  double a = 0.0, b = 0.0;
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    a = fmax(a, red[j]);
    b = fmax(b, red[n + j]);
  }
  a = block_max<kFftThreads>(a, red_sm);
  b = block_max<kFftThreads>(b, red_sm);
  if (threadIdx.x == 0) {
    red[2 * n] = a;
    red[2 * n + 1] = b;
  }
}

// shared memory of one FFT plane kernel: twiddles + `planes` lattice planes
__host__ __device__ inline size_t fft_smem_bytes(int nk, int N, int planes) {
  return sizeof(double2) * ((size_t)nk / 2 + (size_t)planes * N);
}

}  // namespace df
