// Mixed-precision ladder solve (DF_FP32_IR) of order 32 < n <= 64: Eq. lin_alg_inv,
// D Gamma = gamma with D = 1 - gamma diag(chi~), diag Gamma only, two ladders of
// one (channel, W) at a time per block.
//
// Per ladder (one group of 256 threads):
//   1. D in double-float from the (hi, lo) FP32 words of gamma and chi~, rounded
//      once to FP32 (the diagonal cancels), in registers: warp w holds columns
//      8 w .. 8 w + 7, its lane l rows l and l + 32.
//   2. S ~ D^-1 by an in-place Gauss-Jordan sweep with implicit partial
//      pivoting in FP32, panels of 8 pivot columns.  Panel k is warp k's own
//      columns: it runs the 8 steps with its neighbour (half the rows each) and
//      leaves the factor W = P' - unit columns at the pivot rows in panel k's
//      buffer; after the group's barrier every other warp takes the pivot rows
//      out of its own registers and applies the rank-8 update A += W A[piv, :].
//      One barrier per panel; warp k + 1 starts its panel as soon as it has applied
//      W_k, while the others still update.  S then goes through shared
//      memory to logical order: thread (tr, tc) = (t / 16, t % 16) takes rows
//      tr + 16 i, columns 4 tc + j.
//   3. T = S gamma to ~2^-48 of max|S_i| max|gamma_j| as an exact digit product
//      on the tensor cores: S's rows and gamma's columns are cut into kDig = 6
//      signed base-512 digits (FP16, |digit| <= 256) relative to a power of two
//      per row of S / column of gamma; the 21 digit pairs of weight >= 2^-61
//      are formed, pairs of equal weight summed in one FP32 accumulator (up to
//      4 pairs x 64 x 2^16 <= 2^24: exact where it matters).
//   4. R = 1 - S D = 1 - S + T diag(chi~) in double-float, and
//      diag Gamma = diag T + diag(R T): D^-1 = (1 + R + R^2 ..) S, so one
//      correction leaves ~|R|^2 of Gamma (the error control's rho^2).
// Only D is swept (n^3 multiply-adds, 32 registers of matrix per thread) and
// gamma enters through one product whose gamma operand all ladders of a
// (channel, W) share, so two groups fit a block (222 KB of shared memory,
// 128 registers) and one group's barriers, pivot chain and tensor-core waits
// overlap the other's arithmetic.  Bound by latency: the pivot chain (~60k of a
// group's 119k cycles per ladder at n = 64) with four warps per scheduler,
// issue slots 45% busy, 108k warp instructions per ladder.  Measured, 30,720
// ladders of order 64: 6.12 ms (6.45 with rows of gamma read across n-strided lanes, 11.2 ms with one ladder per block, [D | gamma]
// swept and the residual gamma - D X0 formed after it); 1,536 of order 48, whose
// padding is no longer swept: 0.25 ms (0.57).  Tried: packed f32x2 multiply-adds in the
// update (40k cycles against 34k), a panel on one warp (1000 cycles a step
// against 800), the panels' factors handed over by mbarriers (polling takes the
// panel's issue slots).
#pragma once
#include <cuda_fp16.h>

#include "df_mixed_dev.cuh"

namespace df {

constexpr int kDig = 6;                                   // base-512 digits per value
constexpr int kM64Group = 256;                            // threads per ladder
constexpr int kM64Groups = 2;
constexpr int kM64Threads = kM64Group * kM64Groups;
constexpr int kM64Slice = 128 * 128;                      // one gamma digit slice: [gamma_re; gamma_im] columns j, K = l
constexpr int kM64Shared = kDig * kM64Slice + 64 * 4;     // a matrix's digits and column weights: kept in shared memory
constexpr int kM64DigBytes = kM64Shared + 64 * 64 * 16;   // then its words [column][row] (hi, lo), in global memory
constexpr int kM64TsLd = 65;                              // row stride of T (float2)
constexpr int kM64ELd = 66;                               // row stride of the exchange (float2)
constexpr int kM64Acc = 32 * kDig;                        // TMEM columns of one 16-row block's accumulators

// shared memory of a group, byte offsets
constexpr int kM64Work = 0;          // S digits [kDig][32][64] fp16 | exchange | the sweep's rows
constexpr int kM64WorkBytes = kDig * 32 * 128;
constexpr int kM64Ts = kM64Work + kM64WorkBytes;          // T | S [64][kM64TsLd] | the panels' factors [8][8][64]
constexpr int kM64ChiH = kM64Ts + 64 * kM64TsLd * 8;
constexpr int kM64ChiL = kM64ChiH + 512;
constexpr int kM64G2 = kM64ChiL + 512;
constexpr int kM64Td = kM64G2 + 1024;
constexpr int kM64Ediag = kM64Td + 1024;
constexpr int kM64Piv = kM64Ediag + 512;
constexpr int kM64Step = kM64Piv + 256;
constexpr int kM64Rexp = kM64Step + 256;                  // row weights of the block, then the flag word
constexpr int kM64GroupBytes = (kM64Rexp + 64 + 16 + 1023) / 1024 * 1024;
constexpr int kM64Gexp = kDig * kM64Slice;
constexpr int kM64Base = kM64Gexp + 1024;
constexpr int kM64Smem = kM64Base + kM64Groups * kM64GroupBytes;
static_assert(2 * 16 * kM64ELd * 8 <= kM64WorkBytes && 8 * 512 + 2048 + 512 <= kM64WorkBytes, "the work area's uses");
static_assert(8 * 8 * 64 * 8 <= 64 * kM64TsLd * 8, "the factors fit T's place");

// instruction descriptor, kind::f16: fp16 A and B (K-major), FP32 D, M x N
__host__ __device__ constexpr unsigned umma_idesc_f16(int M, int N) {
  return (1u << 4) | ((unsigned)(N >> 3) << 17) | ((unsigned)(M >> 4) << 24);
}

// The digits of v 2^-e (|v| < 2^e): v 2^(8 - e) = d_0 + d_1 / 512 + ..., d_s the
// nearest integers (|d_s| <= 256), by exact FP32 steps for an FP32 v.  kDigMagic's
// low mantissa bits are the FP16 pattern of 1280, so that a rounded sum's low
// half is the pattern of 1280 + d.
constexpr float kDigMagic = 12582912.f + 25856.f;         // 1.5 2^23 + 0x6500
__device__ __forceinline__ unsigned dig_next(float& r, float scale) {
  const float m = fmaf(r, scale, kDigMagic);
  r = fmaf(r, scale, -(m - kDigMagic));
  return __float_as_uint(m);
}
// digits of two values (low halves of m0, m1) as an FP16 pair
__device__ __forceinline__ unsigned dig_pair(unsigned m0, unsigned m1) {
  const unsigned p = __byte_perm(m0, m1, 0x5410);
  const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&p), __floats2half2_rn(1280.f, 1280.f));
  return *reinterpret_cast<const unsigned*>(&h);
}

// v's FP32 (hi, lo) words
__device__ __forceinline__ float4 split_words(double2 v) {
  const float hx = (float)v.x, hy = (float)v.y;
  return make_float4(hx, hy, (float)(v.x - (double)hx), (float)(v.y - (double)hy));
}

// gamma's digits, `count` n x n matrices (FP64, n <= 64) -> out[count][kM64DigBytes]:
// per column j with the exponent bound e_j over both parts (|gamma_lj| < 2^e_j) the
// weight 2^(e_j - 8) (0 for a zero column), digits at [slice][j (re) or 64 + j (im)][l], 128-byte
// swizzled rows; rows and columns >= n zero.  One warp per column.
__device__ __forceinline__ void gamma_digits_cols(int n, int count, const double2* __restrict__ gam,
                                                  unsigned char* __restrict__ out, int warp_id, int nwarps, int lane) {
  for (int w = warp_id; w < count * 64; w += nwarps) {
    const int mtx = w / 64, j = w - mtx * 64;
    const double2* G = gam + (size_t)mtx * n * n;
    __half* dig = reinterpret_cast<__half*>(out + (size_t)mtx * kM64DigBytes);
    float* colw = reinterpret_cast<float*>(out + (size_t)mtx * kM64DigBytes + kDig * kM64Slice);
    double m = 0.0;
    if (j < n)
      for (int l = lane; l < n; l += 32) m = fmax(m, fmax(fabs(G[(size_t)l * n + j].x), fabs(G[(size_t)l * n + j].y)));
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    int e = -1000;
    if (m > 0.0) frexp(m, &e);                            // m < 2^e
    if (lane == 0) colw[j] = e > -1000 ? (e - 8 > 127 ? __int_as_float(0x7f800000) : pow2f(e - 8)) : 0.f;
    float4* words = reinterpret_cast<float4*>(out + (size_t)mtx * kM64DigBytes + kM64Shared) + j * 64;
    for (int l = lane; l < 64; l += 32) {
      words[l] = split_words(l < n && j < n ? G[(size_t)l * n + j] : mk(0.0, 0.0));
      double re = 0.0, im = 0.0;
      if (l < n && j < n && e > -1000) {
        re = ldexp(G[(size_t)l * n + j].x, 8 - e);
        im = ldexp(G[(size_t)l * n + j].y, 8 - e);
      }
#pragma unroll
      for (int s = 0; s < kDig; ++s) {
        const double dr = rint(re), di = rint(im);
        re = (re - dr) * 512.0;
        im = (im - di) * 512.0;
        dig[(size_t)s * (kM64Slice / 2) + swz(j, l)] = __double2half(dr);
        dig[(size_t)s * (kM64Slice / 2) + swz(64 + j, l)] = __double2half(di);
      }
    }
  }
}

// the group's barrier (1 + g; its two panel warps use 3 + g)
__device__ __forceinline__ void m64_sync(int g) {
  asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "n"(kM64Group) : "memory");
}

// three runs of 16 consecutive FP32 columns of this thread's TMEM lane, one wait
__device__ __forceinline__ void tmem_ld16x3(unsigned t0, unsigned t1, unsigned t2, float* a, float* b, float* c) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%48];\n"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%49];\n"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%32,%33,%34,%35,%36,%37,%38,%39,%40,%41,%42,%43,%44,%45,%46,%47}, [%50];\n"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=f"(a[0]), "=f"(a[1]), "=f"(a[2]), "=f"(a[3]), "=f"(a[4]), "=f"(a[5]), "=f"(a[6]), "=f"(a[7]), "=f"(a[8]),
        "=f"(a[9]), "=f"(a[10]), "=f"(a[11]), "=f"(a[12]), "=f"(a[13]), "=f"(a[14]), "=f"(a[15]), "=f"(b[0]),
        "=f"(b[1]), "=f"(b[2]), "=f"(b[3]), "=f"(b[4]), "=f"(b[5]), "=f"(b[6]), "=f"(b[7]), "=f"(b[8]), "=f"(b[9]),
        "=f"(b[10]), "=f"(b[11]), "=f"(b[12]), "=f"(b[13]), "=f"(b[14]), "=f"(b[15]), "=f"(c[0]), "=f"(c[1]),
        "=f"(c[2]), "=f"(c[3]), "=f"(c[4]), "=f"(c[5]), "=f"(c[6]), "=f"(c[7]), "=f"(c[8]), "=f"(c[9]), "=f"(c[10]),
        "=f"(c[11]), "=f"(c[12]), "=f"(c[13]), "=f"(c[14]), "=f"(c[15])
      : "r"(t0), "r"(t1), "r"(t2)
      : "memory");
}

// packed TwoSum: s + e = a + b in each half
__device__ __forceinline__ void x2_two_sum(float2 a, float2 b, float2& s, float2& e) {
  s = x2_add(a, b);
  const float2 bb = x2_sub(s, a);
  e = x2_add(x2_sub(a, x2_sub(s, bb)), x2_sub(b, bb));
}

__device__ __forceinline__ void st_shared_if(bool on, unsigned addr, float2 a, float2 b) {
  asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %0, 0;\n@p st.shared.v4.f32 [%1], {%2, %3, %4, %5};\n}\n" ::"r"((int)on),
               "r"(addr), "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y)
               : "memory");
}
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// The eight in-place Gauss-Jordan steps of a panel of 32 WARPS rows, one row per
// lane (this lane's row r, its panel columns pv; warp `half` of the team).  Per step each warp's
// unused row with the largest key (|re| + |im| bits with 127 - row in the low
// 7: largest to 2^-16, ties to the lowest row) goes to its slot of cand, its
// key to ckey (two sets of slots in turn), the team's barrier, and all its warps
// take the best row (u); then every row adds f u, f = -m / pivot with m its
// entry of the pivot column (the pivot row, taken as zero: 1 / pivot).  The
// next column and its search come before the rest of the update, so that the
// search's latency is covered.  This chain of n steps is the ladder's critical
// path: ~80 instructions a step and no branches.  W = P' - unit columns at the
// pivot rows goes to wk [step][row].
template <int WARPS>
__device__ __forceinline__ void gj_panel_team(float2 (&pv)[kPanel], int r, int half, int lane, int k0, float2* wk,
                                              float4* cand, unsigned* ckey, int* piv_s, int* rowstep,
                                              const MixedCheck& mc, int* flags, int* badw, int bar) {
  constexpr int kRows = 32 * WARPS;
  const bool taken = rowstep[r] >= 0;
  unsigned km = taken ? 0u : ~0x7Fu, kr = taken ? 0u : (unsigned)(127 - r);   // 0 once the row is a pivot
  int step = -1;
  unsigned kmin = ~0u;
  unsigned key = (__float_as_uint(fabsf(pv[0].x) + fabsf(pv[0].y)) & km) | kr;
#pragma unroll
  for (int i = 0; i < kPanel; ++i) {
    const int par = i & 1;
    const unsigned kw = __reduce_max_sync(0xffffffffu, key);
    const unsigned ca = smem_u32(cand + (par * WARPS + half) * (kPanel / 2));
    const bool best = key == kw;
#pragma unroll
    for (int c = 0; c < kPanel; c += 2) st_shared_if(best, ca + 8 * c, pv[c], pv[c + 1]);
    if (lane == 0) ckey[par * WARPS + half] = kw;
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(kRows) : "memory");
    unsigned kb;
    int wb;
    if constexpr (WARPS == 2) {
      const uint2 ks = *reinterpret_cast<const uint2*>(ckey + par * 2);
      kb = max(ks.x, ks.y);
      wb = ks.y > ks.x ? 1 : 0;
    } else {
      const uint4 ks = *reinterpret_cast<const uint4*>(ckey + par * 4);
      const unsigned k01 = max(ks.x, ks.y), k23 = max(ks.z, ks.w);
      kb = max(k01, k23);
      wb = k23 > k01 ? (ks.w > ks.z ? 3 : 2) : (ks.y > ks.x ? 1 : 0);
    }
    const float4* cb = cand + (par * WARPS + wb) * (kPanel / 2);
    const float2 z = reinterpret_cast<const float2*>(cb)[i];
    float2 u[kPanel];
#pragma unroll
    for (int c = 0; c < kPanel; c += 2) {
      const float4 q = cb[c / 2];
      u[c] = make_float2(q.x, q.y);
      u[c + 1] = make_float2(q.z, q.w);
    }
    kmin = min(kmin, kb);
    const bool is = (int)(~kb & 127u) == r;
    const float2 m = make_float2(is ? -1.f : pv[i].x, is ? 0.f : pv[i].y);
    km = is ? 0u : km;
    kr = is ? 0u : kr;
    step = is ? i : step;
#pragma unroll
    for (int c = 0; c < kPanel; ++c)
      if (c != i) pv[c] = make_float2(is ? 0.f : pv[c].x, is ? 0.f : pv[c].y);
    // approximate reciprocal: the FP32 sweep is corrected later
    const float d = rcp_approx(fmaf(z.x, z.x, z.y * z.y));
    const float2 f = cmulf(m, make_float2(-z.x * d, z.y * d));
    pv[i] = f;
    if (i + 1 < kPanel) {
      pv[i + 1] = cfmaf2(f, u[i + 1], pv[i + 1]);
      key = (__float_as_uint(fabsf(pv[i + 1].x) + fabsf(pv[i + 1].y)) & km) | kr;
    }
#pragma unroll
    for (int c = 0; c < kPanel; ++c)
      if (c != i && c != i + 1) pv[c] = cfmaf2(f, u[c], pv[c]);
  }
#pragma unroll
  for (int c = 0; c < kPanel; ++c) wk[c * kRows + r] = make_float2(step == c ? pv[c].x - 1.f : pv[c].x, pv[c].y);
  if (step >= 0) {
    rowstep[r] = k0 + step;
    piv_s[k0 + step] = r;
  }
  if ((kmin & ~0x7Fu) == 0u && lane == 0) {                 // an exactly zero FP32 pivot
    *badw = 1;
    zero_pivot(mc, flags);
  }
}

struct M64Group {
  unsigned char* sm;      // the group's shared memory
  unsigned tmem;          // its accumulators
  uint64_t* mbar;         // completion barrier of its MMAs
  unsigned phase;
  int g;
  unsigned spins;         // polls of a completion wait
  volatile int* fail;     // shared, per group: a completion wait gave up
};

// One ladder by the kM64Group threads of group gr.  gdig: the block's gamma
// digits in shared memory (their address), gwt the columns' weights 2^(e_j - 8).
// Writes kc[c][a][:][q].  False when a completion wait gave up (the same in the whole group, which then must
// not start another ladder: its MMAs may still read its operands until the tear-down).
__device__ __forceinline__ bool m64_system(const Dims& dm, int c, int a, int q, const float4* __restrict__ words,
                                           const float2* __restrict__ GGh, const float2* __restrict__ GGl,
                                           const double2* __restrict__ chi,
                                           double2* __restrict__ kc, int* __restrict__ flags, M64Group& gr,
                                           unsigned gdig, const float* gwt, const MixedCheck& mc) {
  const int n = dm.n_w, N = dm.N, nb = dm.nb;
  const int n8 = (n + kPanel - 1) / kPanel * kPanel;       // pivot columns (identity padding up to the panel)
  const int npan = n8 / kPanel;
  const int t = threadIdx.x & (kM64Group - 1), warp = t >> 5, lane = t & 31;
  unsigned char* sm = gr.sm;
  float2* Ts = reinterpret_cast<float2*>(sm + kM64Ts);
  float2* chih = reinterpret_cast<float2*>(sm + kM64ChiH);
  float2* chil = reinterpret_cast<float2*>(sm + kM64ChiL);
  float4* g2s = reinterpret_cast<float4*>(sm + kM64G2);
  float4* td = reinterpret_cast<float4*>(sm + kM64Td);
  float2* ediag = reinterpret_cast<float2*>(sm + kM64Ediag);
  int* piv_s = reinterpret_cast<int*>(sm + kM64Piv);
  int* rowstep = reinterpret_cast<int*>(sm + kM64Step);
  float* rwt = reinterpret_cast<float*>(sm + kM64Rexp);
  int* badw = reinterpret_cast<int*>(sm + kM64Rexp + 64);

  if (t >= 128 && t < 192) {
    const int i = t - 128;
    const double2 x = (i < n) ? chi[((size_t)a * n + i) * N + q] : mk(0.0, 0.0);
    const float hx = (float)x.x, hy = (float)x.y;
    chih[i] = make_float2(hx, hy);
    chil[i] = make_float2((float)(x.x - (double)hx), (float)(x.y - (double)hy));
    rowstep[i] = -1;
    piv_s[i] = i;
    if (i == 0) *badw = 0;
  }
  {
    // ---- D into registers (gamma's words loaded ahead of chi~, rows across the lanes) ----
    float2 A[2][kPanel];
    {
      const int c0 = kPanel * warp;
      float4 g[2][kPanel];
#pragma unroll
      for (int ii = 0; ii < 2; ++ii)
#pragma unroll
        for (int jj = 0; jj < kPanel; ++jj) g[ii][jj] = __ldg(words + (c0 + jj) * 64 + lane + 32 * ii);
      m64_sync(gr.g);
#pragma unroll
      for (int ii = 0; ii < 2; ++ii)
#pragma unroll
        for (int jj = 0; jj < kPanel; ++jj) {
          const float2 gh = make_float2(g[ii][jj].x, g[ii][jj].y), gl = make_float2(g[ii][jj].z, g[ii][jj].w);
          float sr = (lane + 32 * ii == c0 + jj) ? 1.f : 0.f, lr = 0.f, si = 0.f, li = 0.f;
          cdf_fma(sr, lr, si, li, make_float2(-gh.x, -gh.y), make_float2(-gl.x, -gl.y), chih[c0 + jj], chil[c0 + jj]);
          A[ii][jj] = make_float2(sr + lr, si + li);
        }
    }
    // ---- in-place Gauss-Jordan sweep ----
    float2* wbuf = Ts;                                      // [panel][step][row]
    float4* prs = reinterpret_cast<float4*>(sm + kM64Work) + warp * 32;   // [step][4]: this warp's columns of the pivot rows
    float2* swap = reinterpret_cast<float2*>(sm + kM64Work + 8 * 512);    // [column][32]: half a panel on its way
    float4* cand = reinterpret_cast<float4*>(swap + kPanel * 32);         // [2][2][kPanel / 2]
    unsigned* ckey = reinterpret_cast<unsigned*>(cand + 2 * kPanel);      // [2][2]
#pragma unroll 1
    for (int kp = 0; kp < npan; ++kp) {
      if (warp == kp || warp == (kp ^ 1)) {
        // the panel on its own warp (rows 0-31) and its neighbour (rows 32-63, handed over and back)
        const int half = warp == kp ? 0 : 1, r = lane + 32 * half;
        if (half == 0) {
#pragma unroll
          for (int c = 0; c < kPanel; ++c) swap[c * 32 + lane] = A[1][c];
        }
        asm volatile("bar.sync %0, 64;" ::"r"(3 + gr.g) : "memory");
        float2 pv[kPanel];
#pragma unroll
        for (int c = 0; c < kPanel; ++c) pv[c] = half ? swap[c * 32 + lane] : A[0][c];
        gj_panel_team<2>(pv, r, half, lane, kPanel * kp, wbuf + kp * 512, cand, ckey, piv_s, rowstep, mc, flags, badw,
                         3 + gr.g);
        if (half == 1) {
#pragma unroll
          for (int c = 0; c < kPanel; ++c) swap[c * 32 + lane] = pv[c];
        }
        asm volatile("bar.sync %0, 64;" ::"r"(3 + gr.g) : "memory");
        if (half == 0) {
#pragma unroll
          for (int c = 0; c < kPanel; ++c) {
            A[0][c] = pv[c];
            A[1][c] = swap[c * 32 + lane];
          }
        }
      } else if (kp == (warp < 2 ? 2 : 0)) {
        // Gamma^(2)_jj = sum_x (gamma_jx gamma_xj) chi~_x in double-float, four lanes per j,
        // while another pair of warps factorises its panel
        const int j = t >> 2, part = t & 3;
        float sr = 0.f, lr = 0.f, si = 0.f, li = 0.f;
#pragma unroll 1
        for (int k0 = 0; k0 < 16; k0 += 4) {
          float2 h[4], l[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int x = part + 4 * (k0 + k);
            const bool ok = j < n && x < n;
            h[k] = ok ? __ldg(GGh + j * n + x) : make_float2(0.f, 0.f);
            l[k] = ok ? __ldg(GGl + j * n + x) : make_float2(0.f, 0.f);
          }
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int x = part + 4 * (k0 + k);
            cdf_fma(sr, lr, si, li, h[k], l[k], chih[x], chil[x]);
          }
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
          const float osr = __shfl_xor_sync(0xffffffffu, sr, o), olr = __shfl_xor_sync(0xffffffffu, lr, o);
          const float osi = __shfl_xor_sync(0xffffffffu, si, o), oli = __shfl_xor_sync(0xffffffffu, li, o);
          df_add(sr, lr, osr);
          lr += olr;
          df_add(si, li, osi);
          li += oli;
        }
        if (part == 0) g2s[j] = make_float4(sr, lr, si, li);
      }
      m64_sync(gr.g);                                       // panel kp's factor
      if (warp != kp && warp < npan) {
        const unsigned pa = smem_u32(prs);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int l = rowstep[lane + 32 * h] - kPanel * kp;
          const bool is = l >= 0 && l < kPanel;
#pragma unroll
          for (int c = 0; c < kPanel; c += 2) st_shared_if(is, pa + 64 * l + 8 * c, A[h][c], A[h][c + 1]);
        }
        __syncwarp();
        const float2* wk = wbuf + kp * 512 + lane;
#pragma unroll 4
        for (int l = 0; l < kPanel; ++l) {
          const float2 w0 = wk[l * 64], w1 = wk[l * 64 + 32];
#pragma unroll
          for (int c = 0; c < kPanel; c += 2) {
            const float4 p = prs[4 * l + c / 2];
            A[0][c] = cfmaf2(w0, make_float2(p.x, p.y), A[0][c]);
            A[1][c] = cfmaf2(w1, make_float2(p.x, p.y), A[1][c]);
            A[0][c + 1] = cfmaf2(w0, make_float2(p.z, p.w), A[0][c + 1]);
            A[1][c + 1] = cfmaf2(w1, make_float2(p.z, p.w), A[1][c + 1]);
          }
        }
        __syncwarp();
      }
    }
    m64_sync(gr.g);                                         // the factors are read
    // S[k][m] = A[row of step k][column c], m = piv_s[c], to shared memory in logical order
    if (warp < npan) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int k = rowstep[lane + 32 * h];
        if (k >= 0) {
#pragma unroll
          for (int c = 0; c < kPanel; ++c) Ts[k * kM64TsLd + piv_s[kPanel * warp + c]] = A[h][c];
        }
      }
    }
    m64_sync(gr.g);
  }
  // rows tr + 16 b, columns 4 tc + jj of S, later of R
  const int tr = t >> 4, tc = t & 15;
  const bool clive = 4 * tc < n8;
  float2 A[kTile][kTile];
#pragma unroll
  for (int ii = 0; ii < kTile; ++ii)
#pragma unroll
    for (int jj = 0; jj < kTile; ++jj)
      A[ii][jj] = clive && tr + 16 * ii < n8 ? Ts[(tr + 16 * ii) * kM64TsLd + 4 * tc + jj] : make_float2(0.f, 0.f);

  // ---- T = S gamma by 16-row blocks, R = 1 - S + T chi~ in S's place ----
  __half* xs = reinterpret_cast<__half*>(sm + kM64Work);               // [kDig][32][64]: rows re 0-15, im 16-31
  float2* E = reinterpret_cast<float2*>(sm + kM64Work);                // [2][16][kM64ELd] (hi, lo) of T re, im
  const unsigned xa = smem_u32(xs);
  const int ksteps = (n + 15) >> 4;
#pragma unroll 1
  for (int b = 0; b < ksteps; ++b) {
    float2 s[kTile];
#pragma unroll
    for (int jj = 0; jj < kTile; ++jj) {
      s[jj] = A[0][jj];
#pragma unroll
      for (int ii = 1; ii < kTile; ++ii)
        if (ii == b) s[jj] = A[ii][jj];
    }
    const int k = tr + 16 * b;                              // S's row
    float mx = 0.f;
#pragma unroll
    for (int jj = 0; jj < kTile; ++jj) mx = fmaxf(mx, fmaxf(fabsf(s[jj].x), fabsf(s[jj].y)));
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    int e = exp_bound_f32(mx);
    // a row of S outside 2^(+-100), zero or not finite sends the ladder to the FP64 solve
    const bool rbad = !(e > -100 && e < 100);
    if (rbad) e = 0;
    if (tc == 0) {
      rwt[tr] = __int_as_float((127 - 8 + e) << 23);
      if (rbad && k < n) *badw = 1;
    }
    const float sc = rbad ? 0.f : __int_as_float((127 + 8 - e) << 23);
    {
      float re[kTile], im[kTile];
#pragma unroll
      for (int jj = 0; jj < kTile; ++jj) {
        re[jj] = rbad ? 0.f : s[jj].x;
        im[jj] = rbad ? 0.f : s[jj].y;
      }
      uint2* o = reinterpret_cast<uint2*>(xs + swz(tr, 4 * tc));          // four consecutive digits: 8 bytes
#pragma unroll
      for (int d = 0; d < kDig; ++d) {
        const float f = d == 0 ? sc : 512.f;
        unsigned mr[kTile], mi[kTile];
#pragma unroll
        for (int jj = 0; jj < kTile; ++jj) {
          mr[jj] = dig_next(re[jj], f);
          mi[jj] = dig_next(im[jj], f);
        }
        o[d * 512] = make_uint2(dig_pair(mr[0], mr[1]), dig_pair(mr[2], mr[3]));
        o[d * 512 + 256] = make_uint2(dig_pair(mi[0], mi[1]), dig_pair(mi[2], mi[3]));
      }
    }
    fence_async_smem();
    tc05_fence_before();
    m64_sync(gr.g);
    if (t == 0) {
      tc05_fence_after();
#pragma unroll
      for (int sa = 0; sa < kDig; ++sa) {
        const unsigned idesc = umma_idesc_f16(128, 32 * (kDig - sa));
#pragma unroll
        for (int ks = 0; ks < 4; ++ks)
          if (ks < ksteps) umma_bf16(gr.tmem + 32 * sa, umma_desc_sw128(gdig + sa * kM64Slice + 32 * ks), umma_desc_sw128(xa + 32 * ks),
                    idesc, (sa > 0 || ks > 0) ? 1u : 0u);
      }
      umma_commit(gr.mbar);
    }
    __syncwarp();
    // a warp that saw the completion may overwrite the operands (with the exchange): the MMAs are done; one that gave up
    // leaves them and the accumulators alone, and after the fold's barrier the whole group knows
    if (!__all_sync(0xffffffffu, mbar_wait(gr.mbar, gr.phase, gr.spins))) {
      *gr.fail = 1;
      m64_sync(gr.g);
      return false;
    }
    gr.phase ^= 1u;
    tc05_fence_after();
    // fold: warp w reads lane quadrant w % 4 (lanes 0-63: gamma_re column j, 64-127:
    // gamma_im) and column half w / 4 (S_re or S_im rows) of the kDig groups: weights
    // 2^-9d, d = 3..5 summed in FP32 (rounding < 2^-27 of the d = 0 unit), 0..2 in double-float
    {
      const int qd = warp & 3, h = warp >> 2;
      const int j = ((qd & 1) << 5) + lane;
      const bool zi = qd >= 2;
      const unsigned tl = gr.tmem + ((unsigned)(32 * qd) << 16) + (unsigned)(16 * h);
      float2 fh[8], fl[8];
      {
        float a3[16], a4[16], a5[16];
        tmem_ld16x3(tl + 32 * 3, tl + 32 * 4, tl + 32 * 5, a3, a4, a5);
        const float2 c9 = make_float2(0.001953125f, 0.001953125f);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float2 x = x2_fma(make_float2(a5[2 * i], a5[2 * i + 1]), c9, make_float2(a4[2 * i], a4[2 * i + 1]));
          fl[i] = x2_mul(x2_fma(x, c9, make_float2(a3[2 * i], a3[2 * i + 1])),
                         make_float2(7.450580596923828e-09f, 7.450580596923828e-09f));      // 2^-27
        }
      }
      {
        float a0[16], a1[16], a2[16];
        tmem_ld16x3(tl, tl + 32, tl + 32 * 2, a0, a1, a2);
        const float wj = gwt[j];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          float2 e, l, e2, e3;
          x2_two_sum(make_float2(a0[2 * i], a0[2 * i + 1]),
                     x2_mul(make_float2(a1[2 * i], a1[2 * i + 1]), make_float2(0.001953125f, 0.001953125f)), fh[i], e);
          x2_two_sum(e, x2_mul(make_float2(a2[2 * i], a2[2 * i + 1]),
                               make_float2(3.814697265625e-06f, 3.814697265625e-06f)), l, e2);   // 2^-18
          x2_two_sum(fh[i], l, fh[i], e3);
          const float2 wi = *reinterpret_cast<const float2*>(rwt + 2 * i);
          const float2 w = x2_mul(wi, make_float2(wj, wj));
          fl[i] = x2_mul(x2_add(e3, x2_add(e2, fl[i])), w);
          fh[i] = x2_mul(fh[i], w);
        }
      }
      tc05_fence_before();
      // T_re = re re - im im, T_im = re im + im re (gamma part, S part): the gamma_im lanes' products cross over
      if (zi) {
        const float sg = h ? -1.f : 1.f;
        float2* Eo = E + (1 - h) * 16 * kM64ELd + j;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          Eo[2 * i * kM64ELd] = make_float2(sg * fh[i].x, sg * fl[i].x);
          Eo[(2 * i + 1) * kM64ELd] = make_float2(sg * fh[i].y, sg * fl[i].y);
        }
      }
      m64_sync(gr.g);
      if (*gr.fail) return false;
      if (!zi) {
        float2* Eo = E + h * 16 * kM64ELd + j;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float2 o0 = Eo[2 * i * kM64ELd], o1 = Eo[(2 * i + 1) * kM64ELd];
          float2 sh, se;
          x2_two_sum(fh[i], make_float2(o0.x, o1.x), sh, se);
          se = x2_add(se, x2_add(fl[i], make_float2(o0.y, o1.y)));
          Eo[2 * i * kM64ELd] = make_float2(sh.x, se.x);
          Eo[(2 * i + 1) * kM64ELd] = make_float2(sh.y, se.y);
        }
      }
      m64_sync(gr.g);
    }
    // R_km = delta_km - S_km + T_km chi~_m, and T's leading words for the correction
#pragma unroll
    for (int jp = 0; jp < kTile; jp += 2) {
      const int m0 = 4 * tc + jp;
      const float4 tr2 = *reinterpret_cast<const float4*>(E + tr * kM64ELd + m0);
      const float4 ti2 = *reinterpret_cast<const float4*>(E + (16 + tr) * kM64ELd + m0);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int jj = jp + h, m = m0 + h;
        const float2 tre = h ? make_float2(tr2.z, tr2.w) : make_float2(tr2.x, tr2.y);
        const float2 tim = h ? make_float2(ti2.z, ti2.w) : make_float2(ti2.x, ti2.y);
        float sr = 0.f, lr = 0.f, si = 0.f, li = 0.f;
        cdf_fma(sr, lr, si, li, make_float2(tre.x, tim.x), make_float2(tre.y, tim.y), chih[m], chil[m]);
        df_add(sr, lr, -s[jj].x);
        df_add(si, li, -s[jj].y);
        if (k == m) {
          df_add(sr, lr, 1.f);
          td[k] = make_float4(tre.x, tre.y, tim.x, tim.y);
        }
        const float2 r = make_float2(sr + lr, si + li);
        Ts[k * kM64TsLd + m] = make_float2(tre.x, tim.x);
#pragma unroll
        for (int ii = 0; ii < kTile; ++ii)
          if (ii == b) A[ii][jj] = r;
      }
    }
    m64_sync(gr.g);                                         // the exchange is read, T's rows are written
  }
  // ---- diag(R T): the 16 threads of a row sum over their columns ----
#pragma unroll
  for (int ii = 0; ii < kTile; ++ii) {
    const int k = tr + 16 * ii;
    float ex = 0.f, ey = 0.f;
    if (ii < ksteps && clive) {
#pragma unroll
      for (int jj = 0; jj < kTile; ++jj) {
        const float2 tv = Ts[(4 * tc + jj) * kM64TsLd + k];
        const float2 w = A[ii][jj];
        ex = fmaf(w.x, tv.x, fmaf(-w.y, tv.y, ex));
        ey = fmaf(w.x, tv.y, fmaf(w.y, tv.x, ey));
      }
    }
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) {
      ex += __shfl_xor_sync(0xffffffffu, ex, o);
      ey += __shfl_xor_sync(0xffffffffu, ey, o);
    }
    if (tc == 0) ediag[k] = make_float2(ex, ey);
  }
  bool fin = *badw == 0;                                    // (the next ladder resets it)
  m64_sync(gr.g);
  // ---- the Eq. sd bracket (warps 0 and 1) and the error control (warp 2); the others go on ----
  if (t < n) {
    const int j = t;
    const float4 d0 = td[j], g2 = g2s[j];
    const float2 ec = ediag[j];
    const double gx = ((double)d0.x + (double)d0.y) + (double)ec.x, gy = ((double)d0.z + (double)d0.w) + (double)ec.y;
    const double wgt = (c == 0) ? 1.0 : 3.0;
    kc[(((size_t)c * nb + a) * n + j) * N + q] = mk(wgt * (gx - 0.5 * ((double)g2.x + (double)g2.y)),
                                                    wgt * (gy - 0.5 * ((double)g2.z + (double)g2.w)));
  }
  if (warp == 2) {
    float emax = 0.f, gmax = 0.f;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int j = lane + 32 * h;
      if (j < n) {
        const float4 d0 = td[j];
        const float2 ec = ediag[j];
        const float ea = fabsf(ec.x) + fabsf(ec.y), ga = fabsf(d0.x + ec.x) + fabsf(d0.z + ec.y);
        fin = fin && isfinite(ea) && isfinite(ga);
        emax = fmaxf(emax, ea);
        gmax = fmaxf(gmax, ga);
      }
    }
    for (int o = 16; o > 0; o >>= 1) {
      emax = fmaxf(emax, __shfl_xor_sync(0xffffffffu, emax, o));
      gmax = fmaxf(gmax, __shfl_xor_sync(0xffffffffu, gmax, o));
    }
    fin = __all_sync(0xffffffffu, fin);
    if (lane == 0) mixed_check_ladder(mc, emax, gmax, fin, ((long)c * nb + a) * N + q, flags);
  }
  return true;
}

// Block-level state: set up by all threads (warp 0 allocates the tensor memory).
struct M64Block {
  unsigned char* sm;      // dynamic shared memory, 1024-aligned
  uint64_t* mbar;         // [kM64Groups] the groups' completion barriers, then their tear-down barriers
  unsigned tmem;
  volatile int* fail;     // [kM64Groups]
  M64Group gr;            // this thread's group
};
// some group of the block gave up (read by all threads while no ladder runs)
__device__ __forceinline__ bool m64_failed(const M64Block& b) {
  int f = 0;
  for (int i = 0; i < kM64Groups; ++i) f |= b.fail[i];
  return f != 0;
}
__device__ __forceinline__ void m64_setup(M64Block& b, unsigned char* sm, uint64_t* mbar, unsigned* tslot,
                                          volatile int* fail, unsigned spins = kMbarSpin) {
  if ((threadIdx.x >> 5) == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tslot)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 0) {
    for (int i = 0; i < 2 * kM64Groups; ++i)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(mbar + i)) : "memory");
    for (int i = 0; i < kM64Groups; ++i) fail[i] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc05_fence_before();
  __syncthreads();
  tc05_fence_after();
  const int g = threadIdx.x / kM64Group;
  b.sm = sm;
  b.mbar = mbar;
  b.tmem = *tslot;
  b.fail = fail;
  b.gr = M64Group{sm + kM64Base + g * kM64GroupBytes, b.tmem + 256u * g, mbar + g, 0u, g, spins, fail + g};
}
// each group's issuing thread commits once more, which completes after every
// MMA it queued (also after a wait that gave up); the wait for it is bounded
__device__ __forceinline__ void m64_teardown(const M64Block& b) {
  if (threadIdx.x % kM64Group == 0) {
    tc05_fence_before();
    umma_commit(b.mbar + kM64Groups + b.gr.g);
    mbar_wait(b.mbar + kM64Groups + b.gr.g, 0u);
  }
  tc05_fence_before();
  __syncthreads();
  tc05_fence_after();
  if ((threadIdx.x >> 5) == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(b.tmem) : "memory");
}
// gamma's digits of one (channel, W) into shared memory (all threads; no ladder running).  False, the same in
// the whole block, once a group gave up: its MMAs may still read the old ones.
__device__ __forceinline__ bool m64_load_digits(const M64Block& b, const unsigned char* __restrict__ gdig) {
  __syncthreads();
  const bool go = !m64_failed(b);
  if (go) {
    const uint4* src = reinterpret_cast<const uint4*>(gdig);
    uint4* dst = reinterpret_cast<uint4*>(b.sm);
    for (int i = threadIdx.x; i < kM64Shared / 16; i += kM64Threads) dst[i] = __ldg(src + i);
    fence_async_smem();
  }
  __syncthreads();
  return go;
}

}  // namespace df
