// Mixed-precision ladder solve (DF_FP32_IR) of order n <= 32, the method of
// df_mixed64_dev.cuh (S ~ D^-1 by an in-place FP32 sweep, T = S gamma as an exact digit
// product, diag Gamma = diag T + diag((1 - S D) T)), one ladder per WARP: no block
// barrier anywhere, the warps of a block share gamma's digits of one (channel, W).
//
// NP = 16 or 32 is the padded order.
//   * Sweep: lane (lrow, lcol) = (lane % 8, lane / 8) holds rows lrow + 8 i and columns lcol + 4 r.  Step k
//     takes column k's entries by shuffles, finds the pivot row by one warp maximum, its lanes leave it in
//     shared memory and zero their own, and every row adds f u: f = -m / pivot, and 1 / pivot for the
//     pivot row itself, which is scaled at once: scaled at the end instead, its whole
//     magnitude is rounded once more, and R^2 is up to 1.5 times as large.  The columns rotate by one register
//     every four steps (the update writes one register down), so that the pivot column is
//     always register 0 and the loop stays rolled; only the n real columns are swept.
//   * T: S's rows are cut into three base-512 FP16 digits (as in df_mixed64_dev.cuh) and S is
//     then what its digits say (the rest is <= 2^-27 of the row's largest entry, below the sweep's
//     own rounding, and S only has to be an approximate inverse); mma.sync A fragments straight from
//     shared memory.  gamma's six digits (re, im) are kept in B fragment order; 15 pairs x 4
//     real products per 16 x 8 x 16 tile, pairs of equal weight in one exact accumulator.
//   * T's rows pass through a 16-row buffer, diag(R T) summed as they come, which lets
//     twelve ladders (NP = 32) share an SM's shared memory with gamma's digits and words.
// At n <= 32 one ladder fills neither a tcgen05 tile (64 rows) nor a block.  Bound by the FP32
// pipe and issue (three warps per scheduler; the sweep's 950 cycles a step are 3 x 235
// instructions) and, in the product, by the mma.sync rate (960 x 8 cycles per scheduler).
// Measured, 11,264 ladders of order 30: 0.34 ms (1.35 ms with one ladder per 64-thread block,
// [D | gamma] swept and BF16 digits of X0; 0.47 with whole rows per lane, whose pivot row
// costs each lane 16 16-byte loads, and six digits of S; 0.38 with ten warps; 0.33 with rows scaled at the
// end); of order 16: 58 us.  Error against FP64 on the paper's inputs, orders 8 / 16 / 24 / 32, geometric mean of
// a (channel, W) plane's over 24 inputs: 1.1 / 1.5 / 1.6 / 2.0e-14 (the block kernel's: 1.1 / 1.5 / 1.9 / 2.1e-14; with
// rows scaled at the end 1.5 / 2.2 / 2.3 / 2.9e-14).
#pragma once
#include "df_mixed64_dev.cuh"

namespace df {

constexpr int kSDig = 3;                                  // digits of S

template <int NP>
struct M32 {
  static constexpr int RP = NP / 8, CP = NP / 4;          // rows, columns of the sweep's register tile
  static constexpr int NT = NP / 8, KS = NP / 16;         // column tiles, K steps of the product
  static constexpr int kFrag = kDig * 2 * NT * 32 * KS * 8;   // gamma's fragments (bytes)
  static constexpr int kWords = kFrag + NP * 4;           // then its columns' weights, then its words [column][row] (hi, lo)
  static constexpr int kBytes = kWords + NP * NP * 16;    // one matrix, in global and in shared memory
  static constexpr int SLD = NP + 2, TLD = NP + 1;        // row strides of S / R and T (float2)
  // per warp: S / R, 16 rows of T, chi~ hi, lo, the pivot row (two slots), row scales and weights, diag T,
  // pivots, the rows' steps
  static constexpr int oT = NP * SLD * 8, oX = (oT + 16 * TLD * 8 + 15) / 16 * 16, oP = oX + 2 * NP * 8,
                       oS = oP + 2 * NP * 8, oD = oS + 2 * NP * 4, oV = oD + NP * 16,
                       kWarp = oV + 2 * NP * 4;
  static constexpr int kWarps = NP == 32 ? 12 : 16;
  static constexpr int kThreads = 32 * kWarps;
  static constexpr int kItem = kBytes + kWarps * kWarp;   // the batch's queue item (beside it no static shared memory fits)
  static constexpr int kSmem = kItem + 16;
  static_assert(kSmem <= 232448, "a block's shared memory");
};

// gamma's digits of one matrix in global memory, by padded order (orders > 64: df_mixed128_dev.cuh)
__host__ __device__ constexpr size_t mixed_digit_bytes(int np) {
  return np == 16 ? M32<16>::kBytes : np == 32 ? M32<32>::kBytes : np == 64 ? kM64DigBytes : 0;
}

// gamma's digits, weights and words (see M32), `count` n x n matrices (FP64); one warp per column
template <int NP>
__device__ __forceinline__ void gamma_digits_frag(int n, int count, const double2* __restrict__ gam,
                                                  unsigned char* __restrict__ out, int warp_id, int nwarps, int lane) {
  using M = M32<NP>;
  for (int w = warp_id; w < count * NP; w += nwarps) {
    const int mtx = w / NP, j = w - mtx * NP, l = lane;
    const double2* G = gam + (size_t)mtx * n * n;
    unsigned char* O = out + (size_t)mtx * M::kBytes;
    const double2 v = (l < n && j < n) ? G[(size_t)l * n + j] : mk(0.0, 0.0);
    double m = fmax(fabs(v.x), fabs(v.y));
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    int e = -1000;
    if (m > 0.0) frexp(m, &e);                            // m < 2^e
    if (lane == 0)
      reinterpret_cast<float*>(O + M::kFrag)[j] = e > -1000 ? (e - 8 > 127 ? __int_as_float(0x7f800000) : pow2f(e - 8)) : 0.f;
    if (l >= NP) continue;
    const float hx = (float)v.x, hy = (float)v.y;
    reinterpret_cast<float4*>(O + M::kWords)[j * NP + l] =
        make_float4(hx, hy, (float)(v.x - (double)hx), (float)(v.y - (double)hy));
    double re = e > -1000 ? ldexp(v.x, 8 - e) : 0.0, im = e > -1000 ? ldexp(v.y, 8 - e) : 0.0;
    const int ks = l >> 4, reg = (l >> 3) & 1, t4 = (l & 7) >> 1;
#pragma unroll
    for (int s = 0; s < kDig; ++s) {
      const double dr = rint(re), di = rint(im);
      re = (re - dr) * 512.0;
      im = (im - di) * 512.0;
      const double d[2] = {dr, di};
#pragma unroll
      for (int part = 0; part < 2; ++part)
        *reinterpret_cast<__half*>(O + ((((s * 2 + part) * M::NT + (j >> 3)) * 32 + (j & 7) * 4 + t4) * M::KS + ks) * 8 +
                                   reg * 4 + (l & 1) * 2) = __double2half(d[part]);
    }
  }
}

__device__ __forceinline__ void mma_f16(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 "
      "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// c0 + a b for (hi, lo) operands, FP32 result: the leading products exactly, summed by TwoSum
// (one rounding of the result, ~2^-46 relative to the largest term before it)
__device__ __forceinline__ float2 cdf_prod(float2 c0, float2 ah, float2 al, float2 bh, float2 bl) {
  float p, e, s, t, l;
  p = ah.x * bh.x;
  e = fmaf(ah.x, bh.x, -p);
  two_sum(c0.x, p, s, t);
  l = e + t;
  p = -ah.y * bh.y;
  e = fmaf(-ah.y, bh.y, -p);
  two_sum(s, p, s, t);
  l += e + t;
  const float re = s + (l + fmaf(ah.x, bl.x, fmaf(al.x, bh.x, fmaf(-ah.y, bl.y, -al.y * bh.y))));
  p = ah.x * bh.y;
  e = fmaf(ah.x, bh.y, -p);
  two_sum(c0.y, p, s, t);
  l = e + t;
  p = ah.y * bh.x;
  e = fmaf(ah.y, bh.x, -p);
  two_sum(s, p, s, t);
  l += e + t;
  return make_float2(re, s + (l + fmaf(ah.x, bl.y, fmaf(al.x, bh.y, fmaf(ah.y, bl.x, al.y * bh.x)))));
}

// N complex values to shared memory where q is set
__device__ __forceinline__ void st_row_if(bool q, unsigned addr, const float2 (&a)[4]) {
  asm volatile("{\n.reg .pred q;\nsetp.ne.s32 q, %0, 0;\n@q st.shared.v4.f32 [%1], {%2, %3, %4, %5};\n"
               "@q st.shared.v4.f32 [%1 + 16], {%6, %7, %8, %9};\n}\n" ::"r"((int)q), "r"(addr), "f"(a[0].x),
               "f"(a[0].y), "f"(a[1].x), "f"(a[1].y), "f"(a[2].x), "f"(a[2].y), "f"(a[3].x), "f"(a[3].y)
               : "memory");
}
__device__ __forceinline__ void st_row_if(bool q, unsigned addr, const float2 (&a)[8]) {
  asm volatile("{\n.reg .pred q;\nsetp.ne.s32 q, %0, 0;\n@q st.shared.v4.f32 [%1], {%2, %3, %4, %5};\n"
               "@q st.shared.v4.f32 [%1 + 16], {%6, %7, %8, %9};\n@q st.shared.v4.f32 [%1 + 32], {%10, %11, %12, %13};\n"
               "@q st.shared.v4.f32 [%1 + 48], {%14, %15, %16, %17};\n}\n" ::"r"((int)q), "r"(addr), "f"(a[0].x),
               "f"(a[0].y), "f"(a[1].x), "f"(a[1].y), "f"(a[2].x), "f"(a[2].y), "f"(a[3].x), "f"(a[3].y), "f"(a[4].x),
               "f"(a[4].y), "f"(a[5].x), "f"(a[5].y), "f"(a[6].x), "f"(a[6].y), "f"(a[7].x), "f"(a[7].y)
               : "memory");
}

// Where `here` (the same in the whole warp: a branch, not predicated instructions), N complex values
// to shared memory and zeroed in the lanes that set `mine`
__device__ __forceinline__ void take_row(bool here, bool mine, unsigned addr, float2 (&a)[4]) {
  asm volatile(
      "{\n.reg .pred h, q;\nsetp.eq.s32 h, %8, 0;\n@h bra.uni DONE;\nsetp.ne.s32 q, %9, 0;\n"
      "@q st.shared.v4.f32 [%10 + 0], {%0, %1, %2, %3};\n"
      "@q st.shared.v4.f32 [%10 + 16], {%4, %5, %6, %7};\n"
      "@q mov.f32 %0, 0f00000000;\n"
      "@q mov.f32 %1, 0f00000000;\n"
      "@q mov.f32 %2, 0f00000000;\n"
      "@q mov.f32 %3, 0f00000000;\n"
      "@q mov.f32 %4, 0f00000000;\n"
      "@q mov.f32 %5, 0f00000000;\n"
      "@q mov.f32 %6, 0f00000000;\n"
      "@q mov.f32 %7, 0f00000000;\n"
      "DONE:\n}\n"
      : "+f"(a[0].x), "+f"(a[0].y), "+f"(a[1].x), "+f"(a[1].y), "+f"(a[2].x), "+f"(a[2].y), "+f"(a[3].x), "+f"(a[3].y)
      : "r"((int)here), "r"((int)mine), "r"(addr)
      : "memory");
}
__device__ __forceinline__ void take_row(bool here, bool mine, unsigned addr, float2 (&a)[8]) {
  asm volatile(
      "{\n.reg .pred h, q;\nsetp.eq.s32 h, %16, 0;\n@h bra.uni DONE;\nsetp.ne.s32 q, %17, 0;\n"
      "@q st.shared.v4.f32 [%18 + 0], {%0, %1, %2, %3};\n"
      "@q st.shared.v4.f32 [%18 + 16], {%4, %5, %6, %7};\n"
      "@q st.shared.v4.f32 [%18 + 32], {%8, %9, %10, %11};\n"
      "@q st.shared.v4.f32 [%18 + 48], {%12, %13, %14, %15};\n"
      "@q mov.f32 %0, 0f00000000;\n"
      "@q mov.f32 %1, 0f00000000;\n"
      "@q mov.f32 %2, 0f00000000;\n"
      "@q mov.f32 %3, 0f00000000;\n"
      "@q mov.f32 %4, 0f00000000;\n"
      "@q mov.f32 %5, 0f00000000;\n"
      "@q mov.f32 %6, 0f00000000;\n"
      "@q mov.f32 %7, 0f00000000;\n"
      "@q mov.f32 %8, 0f00000000;\n"
      "@q mov.f32 %9, 0f00000000;\n"
      "@q mov.f32 %10, 0f00000000;\n"
      "@q mov.f32 %11, 0f00000000;\n"
      "@q mov.f32 %12, 0f00000000;\n"
      "@q mov.f32 %13, 0f00000000;\n"
      "@q mov.f32 %14, 0f00000000;\n"
      "@q mov.f32 %15, 0f00000000;\n"
      "DONE:\n}\n"
      : "+f"(a[0].x), "+f"(a[0].y), "+f"(a[1].x), "+f"(a[1].y), "+f"(a[2].x), "+f"(a[2].y), "+f"(a[3].x), "+f"(a[3].y),
        "+f"(a[4].x), "+f"(a[4].y), "+f"(a[5].x), "+f"(a[5].y), "+f"(a[6].x), "+f"(a[6].y), "+f"(a[7].x), "+f"(a[7].y)
      : "r"((int)here), "r"((int)mine), "r"(addr)
      : "memory");
}

// One ladder by one warp.  gsm: gamma's fragments, weights and words in shared memory (M32), GGh, GGl the
// (hi, lo) words of gamma o gamma^T (symmetric), ws: the warp's shared memory.  Writes kc[c][a][:][q].
template <int NP>
__device__ __forceinline__ void m32_system(const Dims& dm, int c, int a, int q, const unsigned char* gsm,
                                           const float2* __restrict__ GGh, const float2* __restrict__ GGl, const double2* __restrict__ chi,
                                           double2* __restrict__ kc, int* __restrict__ flags, unsigned char* ws,
                                           const MixedCheck& mc) {
  using M = M32<NP>;
  constexpr int RP = M::RP, CP = M::CP, SLD = M::SLD, TLD = M::TLD, KS = M::KS, NT = M::NT;
  const int n = dm.n_w, N = dm.N, nb = dm.nb;
  const int lane = threadIdx.x & 31, lrow = lane & 7, lcol = lane >> 3;   // sweep: rows lrow + 8 i, columns lcol + 4 r
  float2* S = reinterpret_cast<float2*>(ws);
  float2* T = reinterpret_cast<float2*>(ws + M::oT);
  float2* xh = reinterpret_cast<float2*>(ws + M::oX);
  float2* xl = xh + NP;
  float2* prow = reinterpret_cast<float2*>(ws + M::oP);   // [2][4][CP]
  float* rsc = reinterpret_cast<float*>(ws + M::oS);      // per row of S: digit scale 2^(8 - e), weight 2^(e - 8)
  float* rwt = rsc + NP;
  float4* td = reinterpret_cast<float4*>(ws + M::oD);
  int* piv = reinterpret_cast<int*>(ws + M::oV);
  int* rstep = piv + NP;
  const float* gwt = reinterpret_cast<const float*>(gsm + M::kFrag);
  const float4* words = reinterpret_cast<const float4*>(gsm + M::kWords);

  __syncwarp();
  if (lane < NP) {
    const double2 x = (lane < n) ? chi[((size_t)a * n + lane) * N + q] : mk(0.0, 0.0);
    const float hx = (float)x.x, hy = (float)x.y;
    xh[lane] = make_float2(hx, hy);
    xl[lane] = make_float2((float)(x.x - (double)hx), (float)(x.y - (double)hy));
    piv[lane] = lane;
    rstep[lane] = -1;
  }
  __syncwarp();
  // ---- D in double-float, rounded once ----
  float2 A[RP][CP];
#pragma unroll
  for (int r = 0; r < CP; ++r) {
    const int col = lcol + 4 * r;
    const float2 ch = xh[col], cl = xl[col];
#pragma unroll
    for (int i = 0; i < RP; ++i) {
      const int row = lrow + 8 * i;
      const float4 g = words[col * NP + row];
      A[i][r] = cdf_prod(make_float2(row == col ? 1.f : 0.f, 0.f), make_float2(-g.x, -g.y), make_float2(-g.z, -g.w), ch, cl);
    }
  }
  // ---- in-place Gauss-Jordan sweep, unscaled rows, columns rotating ----
  unsigned km[RP], kr[RP], kmin = ~0u;                    // masks of the rows' keys (used rows: 0)
#pragma unroll
  for (int i = 0; i < RP; ++i) {
    const int row = lrow + 8 * i;
    km[i] = row < n ? ~0x1Fu : 0u;
    kr[i] = row < n ? (unsigned)(31 - row) : 0u;
  }
  const unsigned pa0 = smem_u32(prow) + 8 * CP * lcol;
#pragma unroll 1
  for (int kb = 0; kb < n; kb += 4) {
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      if (kb + s >= n) break;
      float2 m[RP];
      unsigned key = 0u;
#pragma unroll
      for (int i = 0; i < RP; ++i) {
        m[i].x = __shfl_sync(0xffffffffu, A[i][0].x, 8 * s + lrow);
        m[i].y = __shfl_sync(0xffffffffu, A[i][0].y, 8 * s + lrow);
        key = max(key, (__float_as_uint(fabsf(m[i].x) + fabsf(m[i].y)) & km[i]) | kr[i]);
      }
      key = __reduce_max_sync(0xffffffffu, key);
      const int p = (int)(~key & 31u);
      kmin = min(kmin, key);
      const unsigned pa = pa0 + 8 * NP * (s & 1);
      bool is[RP];
#pragma unroll
      for (int i = 0; i < RP; ++i) {
        is[i] = p == lrow + 8 * i;
        km[i] = is[i] ? 0u : km[i];
      }
#pragma unroll
      for (int i = 0; i < RP; ++i) take_row(p >> 3 == i, is[i], pa, A[i]);
      __syncwarp();
      const float2* pr = prow + NP * (s & 1);
      const float2 z = pr[CP * s];
      // approximate reciprocal and one Newton step
      const float zz = fmaf(z.x, z.x, z.y * z.y), d0 = rcp_approx(zz), d = fmaf(d0, fmaf(-zz, d0, 1.f), d0);
      const float2 ainv = make_float2(z.x * d, -z.y * d);
      if (lane == 0) {
        piv[kb + s] = p;
        rstep[p] = kb + s;
      }
      float2 f[RP], nc[RP];                               // the rows' factors: the new column's entries
#pragma unroll
      for (int i = 0; i < RP; ++i) {
        f[i] = cmulf(m[i], make_float2(-ainv.x, -ainv.y));
        f[i].x = is[i] ? ainv.x : f[i].x;
        f[i].y = is[i] ? ainv.y : f[i].y;
        nc[i] = f[i];
      }
      constexpr int kLast = 3;                            // rotate with the last update of four
      const float4* u4 = reinterpret_cast<const float4*>(pr + CP * lcol);
#pragma unroll
      for (int r = 0; r < CP; r += 2) {
        const float4 v = u4[r / 2];
#pragma unroll
        for (int i = 0; i < RP; ++i) {
          float2 t0 = cfmaf2(f[i], make_float2(v.x, v.y), A[i][r]);
          const float2 t1 = cfmaf2(f[i], make_float2(v.z, v.w), A[i][r + 1]);
          if (r == 0) {
            t0.x = lcol == s ? nc[i].x : t0.x;
            t0.y = lcol == s ? nc[i].y : t0.y;
          }
          if (s < kLast) {
            A[i][r] = t0;
            A[i][r + 1] = t1;
          } else {
            if (r == 0)
              nc[i] = t0;
            else
              A[i][r - 1] = t0;
            A[i][r] = t1;
          }
        }
      }
      if (s == kLast) {
#pragma unroll
        for (int i = 0; i < RP; ++i) A[i][CP - 1] = nc[i];
      }
    }
  }
  // an exactly zero FP32 pivot (a used row may then have been taken again, so that rows of S collide: not used)
  const bool zero = (kmin & ~0x1Fu) == 0u;
  if (zero && lane == 0) zero_pivot(mc, flags);
  // ---- S to shared memory in logical order: row `step`, column piv[c]; padding zero ----
  __syncwarp();
  bool bad = zero;
  {
    int pc[CP];                                           // register r holds column lcol + 4 ((r + n / 4) mod CP)
    bool cz[CP];
#pragma unroll
    for (int r = 0; r < CP; ++r) {
      const int col = lcol + 4 * ((r + (n >> 2)) & (CP - 1));
      pc[r] = piv[col];
      cz[r] = col >= n;
    }
#pragma unroll
    for (int i = 0; i < RP; ++i) {
      float mx = 0.f;
      const int st = rstep[lrow + 8 * i];
      const bool real = st >= 0;
      const int k = real ? st : lrow + 8 * i;
#pragma unroll
      for (int r = 0; r < CP; ++r) {
        float2 v = A[i][r];
        if (!real || cz[r]) v = make_float2(0.f, 0.f);
        mx = fmaxf(mx, fmaxf(fabsf(v.x), fabsf(v.y)));
        S[k * SLD + pc[r]] = v;
      }
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
      // a row of S outside 2^(+-100), zero or not finite sends the ladder to the FP64 solve
      const int e = exp_bound_f32(mx);
      const bool rb = !(e > -100 && e < 100);
      bad = bad || (rb && real);
      if (lcol == 0) {
        rsc[k] = rb ? 0.f : __int_as_float((127 + 8 - e) << 23);
        rwt[k] = rb ? 0.f : __int_as_float((127 - 8 + e) << 23);
      }
    }
  }
  __syncwarp();
  // ---- T = S gamma, R = 1 - S + T chi~ in S's place ----
  const int g = lane >> 2, t4 = lane & 3;
  const int nks = (n + 15) >> 4, nnt = (n + 7) >> 3;
  const int j16 = lane & 15, hm = lane >> 4;
  float2 er[2] = {};                                      // (R T)_jj, j = j16 and 16 + j16, half of the terms each
  // er += the terms of 16 m: R's rows r0 + j16 at its columns m0 .., T's rows there (their columns start at t0)
  auto diag_rt = [&](int r0, int m0, int t0) {
    float2 e = make_float2(0.f, 0.f);
#pragma unroll
    for (int m = 0; m < 16; m += 2) {
      const float2 w = S[(r0 + j16) * SLD + m0 + m + hm], tv = T[(m + hm) * TLD + t0 + j16];
      e.x = fmaf(w.x, tv.x, fmaf(-w.y, tv.y, e.x));
      e.y = fmaf(w.x, tv.y, fmaf(w.y, tv.x, e.y));
    }
    er[r0 >> 4].x += e.x;
    er[r0 >> 4].y += e.y;
  };
#pragma unroll 1
  for (int mt = 0; mt < nks; ++mt) {
    const int r0 = 16 * mt + g, r1 = r0 + 8;
    unsigned dr[KS][kSDig][4], di[KS][kSDig][4];
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
#pragma unroll
      for (int x = 0; x < 4; ++x) {                       // fragment registers: (g, lo K), (g + 8, lo), (g, hi), (g + 8, hi)
        const int rw = (x & 1) ? r1 : r0, cl = 16 * ks + 2 * t4 + ((x & 2) ? 8 : 0);
        float4* sp = reinterpret_cast<float4*>(S + rw * SLD + cl);
        const float4 v = *sp;
        const float sc = rsc[rw];
        float a_ = v.x, b_ = v.z, c_ = v.y, d_ = v.w;
#pragma unroll
        for (int dd = 0; dd < kSDig; ++dd) {
          const float fs = dd == 0 ? sc : 512.f;
          const unsigned m0 = dig_next(a_, fs), m1 = dig_next(b_, fs), m2 = dig_next(c_, fs), m3 = dig_next(d_, fs);
          dr[ks][dd][x] = dig_pair(m0, m1);
          di[ks][dd][x] = dig_pair(m2, m3);
        }
        // S is what its digits say: the rest (<= 2^-27 of the row's largest entry) is taken off, exactly
        const float w = -3.814697265625e-06f * rwt[rw];   // 2^-18
        *sp = make_float4(fmaf(a_, w, v.x), fmaf(c_, w, v.y), fmaf(b_, w, v.z), fmaf(d_, w, v.w));
      }
    }
    __syncwarp();                                         // the rows are read before R replaces them
#pragma unroll 1
    for (int nt = 0; nt < nnt; ++nt) {
      float acc[kDig][2][4];
#pragma unroll
      for (int d = 0; d < kDig; ++d)
#pragma unroll
        for (int x = 0; x < 4; ++x) acc[d][0][x] = acc[d][1][x] = 0.f;
#pragma unroll
      for (int sb = 0; sb < kDig; ++sb) {
        uint2 b[3][KS];
#pragma unroll
        for (int part = 0; part < 2; ++part) {
          const unsigned char* src = gsm + (((sb * 2 + part) * NT + nt) * 32 + lane) * KS * 8;
          if constexpr (KS == 2) {
            const uint4 v = *reinterpret_cast<const uint4*>(src);
            b[part][0] = make_uint2(v.x, v.y);
            b[part][1] = make_uint2(v.z, v.w);
          } else {
            b[part][0] = *reinterpret_cast<const uint2*>(src);
          }
        }
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) b[2][ks] = make_uint2(b[1][ks].x ^ 0x80008000u, b[1][ks].y ^ 0x80008000u);
#pragma unroll
        for (int ks = 0; ks < KS; ++ks)
#pragma unroll
          for (int sa = 0; sa < kSDig && sa + sb < kDig; ++sa) {
            mma_f16(acc[sa + sb][0], dr[ks][sa], b[0][ks].x, b[0][ks].y);    // re re
            mma_f16(acc[sa + sb][1], dr[ks][sa], b[1][ks].x, b[1][ks].y);    // re im
            mma_f16(acc[sa + sb][0], di[ks][sa], b[2][ks].x, b[2][ks].y);    // - im im
            mma_f16(acc[sa + sb][1], di[ks][sa], b[0][ks].x, b[0][ks].y);    // im re
          }
      }
      // fold the weights 2^-9d (as in df_mixed64_dev.cuh), two columns packed
      const int col = 8 * nt + 2 * t4;
      const float2 wj = *reinterpret_cast<const float2*>(gwt + col);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int rw = h ? r1 : r0;
        const float wr = rwt[rw];
        const float2 w = make_float2(wr * wj.x, wr * wj.y);
        float2 th[2], tl[2];
#pragma unroll
        for (int part = 0; part < 2; ++part) {
          auto pr = [&](int d) { return make_float2(acc[d][part][2 * h], acc[d][part][2 * h + 1]); };
          const float2 c9 = make_float2(0.001953125f, 0.001953125f);
          const float2 x = x2_fma(x2_fma(pr(5), c9, pr(4)), c9, pr(3));
          const float2 low = x2_mul(x, make_float2(7.450580596923828e-09f, 7.450580596923828e-09f));   // 2^-27
          float2 fh, e, l, e2, e3;
          x2_two_sum(pr(0), x2_mul(pr(1), c9), fh, e);
          x2_two_sum(e, x2_mul(pr(2), make_float2(3.814697265625e-06f, 3.814697265625e-06f)), l, e2);   // 2^-18
          x2_two_sum(fh, l, fh, e3);
          th[part] = x2_mul(fh, w);
          tl[part] = x2_mul(x2_add(e3, x2_add(e2, low)), w);
        }
        float4* sp = reinterpret_cast<float4*>(S + rw * SLD + col);
        const float4 sv = *sp;
        const int tc = mt ? col & 15 : col;               // T's rows 16 .. : 16 columns at a time, over the used ones
        float2 rr[2];
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          const int m = col + x;
          const float2 ti = x ? make_float2(th[0].y, th[1].y) : make_float2(th[0].x, th[1].x);
          const float2 tj = x ? make_float2(tl[0].y, tl[1].y) : make_float2(tl[0].x, tl[1].x);
          float2 c0 = x ? make_float2(-sv.z, -sv.w) : make_float2(-sv.x, -sv.y);
          float e0 = 0.f;
          if (rw == m) {
            two_sum(1.f, c0.x, c0.x, e0);
            td[rw] = make_float4(ti.x, tj.x, ti.y, tj.y);
          }
          rr[x] = cdf_prod(c0, ti, tj, xh[m], xl[m]);
          rr[x].x += e0;
          T[(rw & 15) * TLD + tc + x] = ti;
        }
        *sp = make_float4(rr[0].x, rr[0].y, rr[1].x, rr[1].y);
      }
      if (NP == 32 && mt == 1 && nt == 1) {
        __syncwarp();
        diag_rt(0, 16, 0);
        __syncwarp();
      }
    }
    __syncwarp();
    if (mt == 0) {
      diag_rt(0, 0, 0);
    } else {
      diag_rt(16, 0, 16);
      diag_rt(16, 16, 0);
    }
    __syncwarp();
  }
  // ---- Gamma^(2)_jj = sum_x (gamma_jx gamma_xj) chi~_x, lane j (NP = 16: half of the x each) ----
  constexpr int LPR = 32 / NP;
  const int j = lane % NP, part = lane / NP;
  float sr = 0.f, lr = 0.f, si = 0.f, li = 0.f;
  if (j < n) {
#pragma unroll 4
    for (int x = part; x < n; x += LPR)
      cdf_fma(sr, lr, si, li, __ldg(GGh + x * n + j), __ldg(GGl + x * n + j), xh[x], xl[x]);
  }
#pragma unroll
  for (int h = 0; h < NP / 16; ++h) {
    er[h].x += __shfl_xor_sync(0xffffffffu, er[h].x, 16);
    er[h].y += __shfl_xor_sync(0xffffffffu, er[h].y, 16);
  }
  const float ex = (NP == 32 && hm) ? er[1].x : er[0].x, ey = (NP == 32 && hm) ? er[1].y : er[0].y;
  if constexpr (LPR > 1) {
    const float o0 = __shfl_xor_sync(0xffffffffu, sr, 16), o1 = __shfl_xor_sync(0xffffffffu, lr, 16);
    const float o2 = __shfl_xor_sync(0xffffffffu, si, 16), o3 = __shfl_xor_sync(0xffffffffu, li, 16);
    df_add(sr, lr, o0);
    lr += o1;
    df_add(si, li, o2);
    li += o3;
  }
  float emax = 0.f, gmax = 0.f;
  bool fin = !bad;
  const float4 d0 = j < n ? td[j] : make_float4(0.f, 0.f, 0.f, 0.f);
  if (j < n) {
    emax = fabsf(ex) + fabsf(ey);
    gmax = fabsf(d0.x + ex) + fabsf(d0.z + ey);
    fin = fin && isfinite(emax) && isfinite(gmax);
  }
  for (int o = 16; o > 0; o >>= 1) {
    emax = fmaxf(emax, __shfl_xor_sync(0xffffffffu, emax, o));
    gmax = fmaxf(gmax, __shfl_xor_sync(0xffffffffu, gmax, o));
  }
  if (j < n && part == 0) {
    const double gx = ((double)d0.x + (double)d0.y) + (double)ex, gy = ((double)d0.z + (double)d0.w) + (double)ey;
    const double wgt = (c == 0) ? 1.0 : 3.0;
    kc[(((size_t)c * nb + a) * n + j) * N + q] = mk(wgt * (gx - 0.5 * ((double)sr + (double)lr)),
                                                    wgt * (gy - 0.5 * ((double)si + (double)li)));
  }
  fin = __all_sync(0xffffffffu, fin);
  if (lane == 0) mixed_check_ladder(mc, emax, gmax, fin, ((long)c * nb + a) * N + q, flags);
}

// gamma's fragments, weights and words of one (channel, W) into shared memory (all threads; no ladder running)
template <int NP>
__device__ __forceinline__ void m32_load_gamma(unsigned char* sm, const unsigned char* __restrict__ src) {
  __syncthreads();
  for (int i = threadIdx.x; i < M32<NP>::kBytes / 16; i += blockDim.x)
    reinterpret_cast<uint4*>(sm)[i] = __ldg(reinterpret_cast<const uint4*>(src) + i);
  __syncthreads();
}

}  // namespace df
