// Mixed-precision ladder solve (DF_FP32_IR) of order 64 < n <= 128, the method of
// df_mixed64_dev.cuh (S ~ D^-1 by an in-place FP32 sweep of D alone, T = S gamma as an
// exact digit product on the tensor cores, diag Gamma = diag T + diag((1 - S D) T)), one
// ladder at a time per block:
//   * 16 warps of 8 columns each hold D in registers (lane l: rows l + 32 i); a
//     panel is factorised by its warp and the other three of its aligned four
//     (32 rows each), the others apply W A[piv, :] one panel behind;
//   * S goes to shared memory in logical order; R replaces it row by row;
//   * gamma's digits (393 KB at n = 128) do not fit beside it: one thread streams
//     them from L2 by bulk asynchronous copies, per 16-row block of S and
//     64-column tile of gamma kDig slices in pieces of 32 K (8 KB), through a
//     ring of pieces; the block's S digits are the B operand (N = 32 rows per
//     slice), the accumulators 192 columns of tensor memory;
//   * T's leading words stay in tensor memory (lane j, 2 x 128 columns) until
//     all rows of R are there: lane j then sums R_jm T_mj.
// The digit sums: a weight 2^-9d of d + 1 pairs reaches (d + 1) x 128 x 2^16, so that d <= 1 is
// exact (2^24).  d = 2 and 3 could pass 2^24 (by at most 1.5 and 2) where a row of S and a column of gamma
// have digits near 256 of equal sign throughout; a K step beyond rounds by a unit or two, so that the bound on T
// is 2^-28 of max|S_i| max|gamma_j| there.  Measured on matrices a (+-1), Sylvester's of order 128, with a
// chosen to pass 2^24 by a fifth: error 1.9e-12 of the bracket, 1.3e-12 with an a that does not: the
// remainder of the sweep, not these roundings.
// Tile t's finishing lanes 64 t .. 64 t + 63 are the columns j themselves: the
// digit rows are [gamma_re; gamma_im] in tile 0 and [gamma_im; gamma_re] in tile 1.
//
// Cycles per ladder (instrumented copy, n = 96 / 128): D 21k / 28k (with n-strided reads of gamma; its
// words by column since: 4.00 -> 3.89 and 30.1 -> 29.1 ms below), sweep 118k / 182k
// (the updates run near the FMA rate), digits 12k / 16k, products with their
// stream 128k / 211k (92k / 150k of it the stream alone: 1.8 / 3.1 MB per ladder, ~6 TB/s from
// L2 over all SMs), fold, exchange and R 33k / 44k.  Measured: 3,630 ladders of order 96 3.9 ms (9.3 with
// the sweep of [D | gamma] on the tensor cores and a base-128 digit residual streamed in
// 8-column blocks), 17,952 of order 128 29 ms (96.8 with the sweep on the tensor cores and a
// double-float residual on the CUDA cores).  The CUDA-core sweep also leaves a
// smaller residual than three-piece BF16 products: worst rho^2 on the 3D workload
// 1.5e-12 (4.6e-10).
#pragma once
#include "df_mixed64_dev.cuh"

namespace df {

constexpr int kM128Threads = 512;
constexpr int kM128Issuer = 0, kM128Streamer = 32;        // the threads that issue the MMAs and stream the digits
constexpr int kM128Piece = 128 * 64;                      // 128 digit rows x 32 K, 64-byte swizzled
constexpr int kM128Words = 2 * kDig * 4 * kM128Piece + 128 * 4;      // a matrix's digits and column weights,
constexpr int kM128DigBytes = kM128Words + 128 * 128 * 16;           // then its words [column][row] (hi, lo)
constexpr int kM128MaxRing = 10;
constexpr int kM128Atom = kDig * 32 * 128;                // S digits of one 64-wide K block: [kDig][32][64] fp16
constexpr int kM128TmemT = 256;                           // TMEM columns: accumulators [0, 192), T re [256, 384), im [384, 512)

struct M128Layout {
  int ld, s, xs, ex, ring, nring, chih, chil, g2, td, piv, step, rwt, total;   // ld in float2, the rest byte offsets
};
__host__ __device__ inline M128Layout m128_layout(int n) {
  M128Layout L;
  L.ld = (n + 31) / 32 * 32;
  const int rows = (n + 15) / 16 * 16;
  int off = 0;
  auto take = [&](int bytes, int align) {
    off = (off + align - 1) / align * align;
    const int o = off;
    off += bytes;
    return o;
  };
  L.xs = take(2 * kM128Atom, 1024);
  const int sbytes = rows * L.ld * 8, wbytes = (n + 7) / 8 * 8 * 128 * 8;   // S, or the panels' factors before it
  L.s = take(sbytes > wbytes ? sbytes : wbytes, 1024);
  L.ex = take(2 * 16 * 64 * 8, 16);
  L.chih = take(1024, 16);
  L.chil = take(1024, 16);
  L.g2 = take(2048, 16);
  L.td = take(2048, 16);
  L.piv = take(512, 16);
  L.step = take(512, 16);
  L.rwt = take(64 + 16, 16);
  off = (off + 1023) / 1024 * 1024;
  L.nring = (226 * 1024 - off) / kM128Piece;               // 227 KB less the static part
  if (L.nring > kM128MaxRing) L.nring = kM128MaxRing;
  L.ring = take(L.nring * kM128Piece, 1024);
  L.total = off;
  return L;
}

__host__ __device__ constexpr bool m128_supported(int n) { return n > 64 && n <= 128; }

// shared-memory matrix descriptor: K-major, 64-byte swizzle, 8-row groups 512 B apart
__device__ __forceinline__ uint64_t umma_desc_sw64(unsigned saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(512 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)4 << 61);
}

// gamma's digits, `count` n x n matrices (FP64) -> out[count][kM128DigBytes]: per column j the
// weight 2^(e_j - 8), |gamma_lj| < 2^e_j (0 for a zero column); digits at piece (tile, slice, l / 32),
// row j % 64 + 64 h, h = 0 for gamma_re in tile 0 and gamma_im in tile 1.  One warp per column.
__device__ __forceinline__ void gamma_digits_cols128(int n, int count, const double2* __restrict__ gam,
                                                     unsigned char* __restrict__ out, int warp_id, int nwarps,
                                                     int lane) {
  for (int w = warp_id; w < count * 128; w += nwarps) {
    const int mtx = w / 128, j = w - mtx * 128;
    const double2* G = gam + (size_t)mtx * n * n;
    unsigned char* O = out + (size_t)mtx * kM128DigBytes;
    float* colw = reinterpret_cast<float*>(O + 2 * kDig * 4 * kM128Piece);
    double m = 0.0;
    if (j < n)
      for (int l = lane; l < n; l += 32) m = fmax(m, fmax(fabs(G[(size_t)l * n + j].x), fabs(G[(size_t)l * n + j].y)));
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    int e = -1000;
    if (m > 0.0) frexp(m, &e);                            // m < 2^e
    if (lane == 0) colw[j] = e > -1000 ? (e - 8 > 127 ? __int_as_float(0x7f800000) : pow2f(e - 8)) : 0.f;
    const int tile = j >> 6;
    float4* words = reinterpret_cast<float4*>(O + kM128Words) + j * 128;
    for (int l = lane; l < 128; l += 32) {
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
        unsigned char* P = O + (size_t)((tile * kDig + s) * 4 + (l >> 5)) * kM128Piece;
        auto put = [&](int row, double d) {
          *reinterpret_cast<__half*>(P + row * 64 + ((((l & 31) >> 3) ^ ((row >> 1) & 3)) << 4) + (l & 7) * 2) =
              __double2half(d);
        };
        put((j & 63) + (tile ? 64 : 0), dr);
        put((j & 63) + (tile ? 0 : 64), di);
      }
    }
  }
}

__device__ __forceinline__ void m128_sync() { asm volatile("bar.sync 1, 512;" ::: "memory"); }

// The block's state: barriers, tensor memory, the ring's position (the streaming and the
// issuing thread's own counts of pieces since the launch).
struct M128State {
  unsigned char* sm;
  unsigned tmem;
  uint64_t* done;         // the accumulators of a (block, tile) are complete
  uint64_t* full;         // [nring] a piece arrived
  uint64_t* empty;        // [nring] the MMAs that read it completed
  unsigned phase;
  int slot;               // ring position of the thread's next piece and the parity of its round
  unsigned round;
  volatile int* fail;     // shared: a bounded wait gave up
};

__device__ __forceinline__ void m128_bulk_g2s(unsigned dst, const void* src, unsigned bytes, uint64_t* mbar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(mbar)), "r"(bytes) : "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(smem_u32(mbar))
               : "memory");
}

// (the streaming thread) the next `count` pieces of the ladder in the order of use (row block,
// tile, slice, K), each into its ring slot once the MMAs of the slot's last piece completed.  at:
// the piece within the matrix.  False when a wait gave up.
__device__ __forceinline__ bool m128_stream(int count, int& at, int nkat, const M128Layout& L,
                                            const unsigned char* __restrict__ gdig, M128State& st) {
  const unsigned ring = smem_u32(st.sm + L.ring);
  for (int i = 0; i < count; ++i) {
    if (!mbar_wait(st.empty + st.slot, st.round ^ 1u)) return false;   // the first round passes at once
    m128_bulk_g2s(ring + st.slot * kM128Piece, gdig + (size_t)at * kM128Piece, kM128Piece, st.full + st.slot);
    ++at;
    if ((at & 3) == nkat) at += 4 - nkat;                   // pieces are kept four per slice
    if (at == 2 * kDig * 4) at = 0;
    if (++st.slot == L.nring) {
      st.slot = 0;
      st.round ^= 1u;
    }
  }
  return true;
}

// One ladder.  Gh, Gl, GGh, GGl: the (hi, lo) words of gamma and gamma o gamma^T of this
// (channel, W), gdig gamma's digits and column weights.  Returns false when a bounded wait gave
// up (the same in every thread).
__device__ __forceinline__ bool m128_system(const Dims& dm, int c, int a, int q, const float2* __restrict__ GGh,
                                            const float2* __restrict__ GGl,
                                            const unsigned char* __restrict__ gdig,
                                            const double2* __restrict__ chi, double2* __restrict__ kc,
                                            int* __restrict__ flags, const M128Layout& L, M128State& st,
                                            const MixedCheck& mc) {
  const int n = dm.n_w, N = dm.N, nb = dm.nb, ld = L.ld;
  const int n8 = (n + kPanel - 1) / kPanel * kPanel, npan = n8 / kPanel;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  unsigned char* sm = st.sm;
  float2* S = reinterpret_cast<float2*>(sm + L.s);
  float2* chih = reinterpret_cast<float2*>(sm + L.chih);
  float2* chil = reinterpret_cast<float2*>(sm + L.chil);
  float4* g2s = reinterpret_cast<float4*>(sm + L.g2);
  float4* td = reinterpret_cast<float4*>(sm + L.td);
  int* piv_s = reinterpret_cast<int*>(sm + L.piv);
  int* rowstep = reinterpret_cast<int*>(sm + L.step);
  float* rwt = reinterpret_cast<float*>(sm + L.rwt);
  int* badw = reinterpret_cast<int*>(sm + L.rwt + 64);
  // element (k, m) of S and R: pairs of columns swapped within groups of 16 by the row, so
  // that a row read by a warp and a column pair read by 32 rows both spread over the banks
  auto sidx = [&](int k, int m) { return k * ld + ((((m >> 1) ^ (k & 15)) << 1) | (m & 1)); };

  if (t < 128) {
    const double2 x = (t < n) ? chi[((size_t)a * n + t) * N + q] : mk(0.0, 0.0);
    const float hx = (float)x.x, hy = (float)x.y;
    chih[t] = make_float2(hx, hy);
    chil[t] = make_float2((float)(x.x - (double)hx), (float)(x.y - (double)hy));
    rowstep[t] = -1;
    piv_s[t] = t;
    if (t == 0) *badw = 0;
  }
  m128_sync();
  {
    // ---- D into registers ----
    const float4* words = reinterpret_cast<const float4*>(gdig + kM128Words);
    float2 A[4][kPanel];
    const int c0 = kPanel * warp;
#pragma unroll
    for (int ii = 0; ii < 4; ++ii) {
      const int r = lane + 32 * ii;
      float4 g[kPanel];
#pragma unroll
      for (int c2 = 0; c2 < kPanel; ++c2) g[c2] = __ldg(words + (c0 + c2) * 128 + r);   // rows across the lanes
#pragma unroll
      for (int c2 = 0; c2 < kPanel; ++c2) {
        const int col = c0 + c2;
        float sr = (r == col) ? 1.f : 0.f, lr = 0.f, si = 0.f, li = 0.f;
        cdf_fma(sr, lr, si, li, make_float2(-g[c2].x, -g[c2].y), make_float2(-g[c2].z, -g[c2].w), chih[col], chil[col]);
        A[ii][c2] = make_float2(sr + lr, si + li);
      }
    }
    // ---- in-place Gauss-Jordan sweep (the factors in S's place, the rows on their way in the digits') ----
    float2* wbuf = S;                                       // [panel][step][128]
    float4* prs = reinterpret_cast<float4*>(sm + L.xs) + warp * 32;       // [step][4]: this warp's columns of the pivot rows
    float2* swap = reinterpret_cast<float2*>(sm + L.xs + 16 * 512);       // [3][column][32]
    float4* cand = reinterpret_cast<float4*>(swap + 3 * kPanel * 32);     // [2][4][kPanel / 2]
    unsigned* ckey = reinterpret_cast<unsigned*>(cand + 4 * kPanel);      // [2][4]
#pragma unroll 1
    for (int kp = 0; kp < npan; ++kp) {
      if ((warp >> 2) == (kp >> 2)) {
        const int part = (warp ^ kp) & 3, r = lane + 32 * part;
        if (part == 0) {
#pragma unroll
          for (int ii = 1; ii < 4; ++ii)
#pragma unroll
            for (int c2 = 0; c2 < kPanel; ++c2) swap[((ii - 1) * kPanel + c2) * 32 + lane] = A[ii][c2];
        }
        asm volatile("bar.sync 2, 128;" ::: "memory");
        float2 pv[kPanel];
#pragma unroll
        for (int c2 = 0; c2 < kPanel; ++c2) pv[c2] = part ? swap[((part - 1) * kPanel + c2) * 32 + lane] : A[0][c2];
        gj_panel_team<4>(pv, r, part, lane, kPanel * kp, wbuf + kp * kPanel * 128, cand, ckey, piv_s, rowstep, mc, flags,
                         badw, 2);
        if (part) {
#pragma unroll
          for (int c2 = 0; c2 < kPanel; ++c2) swap[((part - 1) * kPanel + c2) * 32 + lane] = pv[c2];
        }
        asm volatile("bar.sync 2, 128;" ::: "memory");
        if (part == 0) {
#pragma unroll
          for (int c2 = 0; c2 < kPanel; ++c2) A[0][c2] = pv[c2];
#pragma unroll
          for (int ii = 1; ii < 4; ++ii)
#pragma unroll
            for (int c2 = 0; c2 < kPanel; ++c2) A[ii][c2] = swap[((ii - 1) * kPanel + c2) * 32 + lane];
        }
      } else if (kp == (warp < 4 ? 4 : 0)) {
        // Gamma^(2)_jj = sum_x (gamma_jx gamma_xj) chi~_x in double-float, four lanes per j,
        // while another team factorises its panel
        const int j = t >> 2, part = t & 3;
        float sr = 0.f, lr = 0.f, si = 0.f, li = 0.f;
#pragma unroll 1
        for (int k0 = 0; k0 < 32; k0 += 4) {
          float2 h[4], l[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int x = part + 4 * (k0 + k);
            const bool in = j < n && x < n;
            h[k] = in ? __ldg(GGh + j * n + x) : make_float2(0.f, 0.f);
            l[k] = in ? __ldg(GGl + j * n + x) : make_float2(0.f, 0.f);
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
      m128_sync();                                          // panel kp's factor
      if (warp != kp && warp < npan) {
        const unsigned pa = smem_u32(prs);
#pragma unroll
        for (int ii = 0; ii < 4; ++ii) {
          const int l = rowstep[lane + 32 * ii] - kPanel * kp;
          const bool is = l >= 0 && l < kPanel;
#pragma unroll
          for (int c2 = 0; c2 < kPanel; c2 += 2) st_shared_if(is, pa + 64 * l + 8 * c2, A[ii][c2], A[ii][c2 + 1]);
        }
        __syncwarp();
        const float2* wk = wbuf + kp * kPanel * 128 + lane;
#pragma unroll 2
        for (int l = 0; l < kPanel; ++l) {
          float2 w[4];
#pragma unroll
          for (int ii = 0; ii < 4; ++ii) w[ii] = wk[l * 128 + 32 * ii];
#pragma unroll
          for (int c2 = 0; c2 < kPanel; c2 += 2) {
            const float4 p = prs[4 * l + c2 / 2];
#pragma unroll
            for (int ii = 0; ii < 4; ++ii) {
              A[ii][c2] = cfmaf2(w[ii], make_float2(p.x, p.y), A[ii][c2]);
              A[ii][c2 + 1] = cfmaf2(w[ii], make_float2(p.z, p.w), A[ii][c2 + 1]);
            }
          }
        }
        __syncwarp();
      }
    }
    m128_sync();                                            // the factors are read
    // S[k][m] = A[row of step k][column c], m = piv_s[c]
    if (warp < npan) {
#pragma unroll
      for (int ii = 0; ii < 4; ++ii) {
        const int k = rowstep[lane + 32 * ii];
        if (k >= 0 && k < n8) {
#pragma unroll
          for (int c2 = 0; c2 < kPanel; ++c2) {
            const int m = piv_s[c0 + c2];
            if (m < ld) S[sidx(k, m)] = A[ii][c2];
          }
        }
      }
    }
    m128_sync();
  }

  // ---- T = S gamma by 16-row blocks and 64-column tiles; R = 1 - S + T chi~ in S's place ----
  const int nblk = (n + 15) >> 4, nkat = (n + 31) >> 5, ksteps = nblk;
  const float* gwt = reinterpret_cast<const float*>(gdig + 2 * kDig * 4 * kM128Piece);
  const int per = kDig * nkat, total = 2 * nblk * per;      // pieces of a (block, tile), of the ladder
  int loaded = 0, at = 0;
  const unsigned xa = smem_u32(sm + L.xs), ring = smem_u32(sm + L.ring);
  float2* E = reinterpret_cast<float2*>(sm + L.ex);         // [2][16][64] (hi, lo) of T re, im
  const int qd = warp & 3, h = (warp >> 2) & 1, e8 = warp >> 3;   // fold: lane quadrant, S part, half of the 16 rows
  const unsigned lq = (32u * qd) << 16;
  const int jl = 32 * qd + lane;
  bool ok = true;
#pragma unroll 1
  for (int b = 0; b < nblk; ++b) {
    const int k = 16 * b + warp;                            // S's row of this warp
    {
      const bool live = k < n8 && 4 * lane < n8;
      const float4* row = reinterpret_cast<const float4*>(S + k * ld);
      const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
      const float4 s0 = live ? row[(2 * lane) ^ (k & 15)] : z, s1 = live ? row[(2 * lane + 1) ^ (k & 15)] : z;
      float mx = fmaxf(fmaxf(fmaxf(fabsf(s0.x), fabsf(s0.y)), fmaxf(fabsf(s0.z), fabsf(s0.w))),
                       fmaxf(fmaxf(fabsf(s1.x), fabsf(s1.y)), fmaxf(fabsf(s1.z), fabsf(s1.w))));
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      int e = exp_bound_f32(mx);
      // a row of S outside 2^(+-100), zero or not finite sends the ladder to the FP64 solve
      const bool rbad = !(e > -100 && e < 100);
      if (rbad) e = 0;
      if (lane == 0) {
        rwt[warp] = __int_as_float((127 - 8 + e) << 23);
        if (rbad && k < n) *badw = 1;
      }
      const float sc = rbad ? 0.f : __int_as_float((127 + 8 - e) << 23);
      float re[4] = {s0.x, s0.z, s1.x, s1.z}, im[4] = {s0.y, s0.w, s1.y, s1.w};
#pragma unroll
      for (int jj = 0; jj < 4; ++jj) {
        re[jj] = rbad ? 0.f : re[jj];
        im[jj] = rbad ? 0.f : im[jj];
      }
      if (4 * lane < 16 * ksteps) {
        __half* xs = reinterpret_cast<__half*>(sm + L.xs) + (lane >> 4) * (kM128Atom / 2);
        uint2* o = reinterpret_cast<uint2*>(xs + swz(warp, 4 * (lane & 15)));
#pragma unroll
        for (int d = 0; d < kDig; ++d) {
          const float f = d == 0 ? sc : 512.f;
          unsigned mr[4], mi[4];
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) {
            mr[jj] = dig_next(re[jj], f);
            mi[jj] = dig_next(im[jj], f);
          }
          o[d * 512] = make_uint2(dig_pair(mr[0], mr[1]), dig_pair(mr[2], mr[3]));
          o[d * 512 + 256] = make_uint2(dig_pair(mi[0], mi[1]), dig_pair(mi[2], mi[3]));
        }
      }
    }
    fence_async_smem();
    tc05_fence_before();
    m128_sync();
#pragma unroll 1
    for (int T = 0; T < 2; ++T) {
      if (t == kM128Streamer) {                             // this tile's pieces, and a ring ahead
        const int to = min(total, (2 * b + T + 1) * per + L.nring);
        if (*st.fail || !m128_stream(to - loaded, at, nkat, L, gdig, st)) *st.fail = 1;
        loaded = to;
      }
      if (t == kM128Issuer) {
        tc05_fence_after();
        bool go = *st.fail == 0;
        const uint64_t da0 = umma_desc_sw64(ring), db0 = umma_desc_sw128(xa);
#pragma unroll
        for (int sa = 0; sa < kDig; ++sa) {
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            if (kk < nkat && go) {
              const int slot = st.slot;
              go = mbar_wait(st.full + slot, st.round);
              if (go) {
                if (++st.slot == L.nring) {
                  st.slot = 0;
                  st.round ^= 1u;
                }
                tc05_fence_after();
                const uint64_t da = da0 + (unsigned)(slot * (kM128Piece >> 4));
#pragma unroll
                for (int k2 = 0; k2 < 2; ++k2) {
                  const int ks = 2 * kk + k2;
                  if (ks < ksteps)
                    umma_bf16(st.tmem + 32 * sa, da + 2 * k2, db0 + ((ks >> 2) * (kM128Atom >> 4) + 2 * (ks & 3)),
                              umma_idesc_f16(128, 32 * (kDig - sa)), (sa > 0 || ks > 0) ? 1u : 0u);
                }
                umma_commit(st.empty + slot);
              }
            }
          }
        }
        if (!go) *st.fail = 1;
        umma_commit(st.done);
      }
      __syncwarp();
      ok = mbar_wait(st.done, st.phase) && ok;
      st.phase ^= 1u;
      tc05_fence_after();
      // fold (as in df_mixed64_dev.cuh): this warp's 8 rows of the block
      const bool cross = (qd >> 1) != T;                    // gamma_im lanes
      const int jt = jl & 63;
      float2 fh[4], fl[4];
      {
        const unsigned tl = st.tmem + lq + (unsigned)(16 * h + 8 * e8);
        float v[6][8];
#pragma unroll
        for (int d = 0; d < 6; ++d)
          asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                       : "=f"(v[d][0]), "=f"(v[d][1]), "=f"(v[d][2]), "=f"(v[d][3]), "=f"(v[d][4]), "=f"(v[d][5]),
                         "=f"(v[d][6]), "=f"(v[d][7])
                       : "r"(tl + 32 * d)
                       : "memory");
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int d = 0; d < 6; ++d)                         // the values are complete only after the wait
#pragma unroll
          for (int i = 0; i < 8; ++i) asm volatile("" : "+f"(v[d][i]));
        const float2 c9 = make_float2(0.001953125f, 0.001953125f);
        const float wj = __ldg(gwt + 64 * T + jt);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          auto pr = [&](int d) { return make_float2(v[d][2 * i], v[d][2 * i + 1]); };
          const float2 x = x2_fma(x2_fma(pr(5), c9, pr(4)), c9, pr(3));
          const float2 low = x2_mul(x, make_float2(7.450580596923828e-09f, 7.450580596923828e-09f));   // 2^-27
          float2 e, l, e2, e3;
          x2_two_sum(pr(0), x2_mul(pr(1), c9), fh[i], e);
          x2_two_sum(e, x2_mul(pr(2), make_float2(3.814697265625e-06f, 3.814697265625e-06f)), l, e2);   // 2^-18
          x2_two_sum(fh[i], l, fh[i], e3);
          const float2 wi = *reinterpret_cast<const float2*>(rwt + 8 * e8 + 2 * i);
          const float2 w = x2_mul(wi, make_float2(wj, wj));
          fl[i] = x2_mul(x2_add(e3, x2_add(e2, low)), w);
          fh[i] = x2_mul(fh[i], w);
        }
      }
      tc05_fence_before();
      if (cross) {
        const float sg = h ? -1.f : 1.f;
        float2* Eo = E + ((1 - h) * 16 + 8 * e8) * 64 + jt;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          Eo[2 * i * 64] = make_float2(sg * fh[i].x, sg * fl[i].x);
          Eo[(2 * i + 1) * 64] = make_float2(sg * fh[i].y, sg * fl[i].y);
        }
      }
      m128_sync();
      if (!cross) {
        float2* Eo = E + (h * 16 + 8 * e8) * 64 + jt;
        float tv[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 o0 = Eo[2 * i * 64], o1 = Eo[(2 * i + 1) * 64];
          float2 sh, se;
          x2_two_sum(fh[i], make_float2(o0.x, o1.x), sh, se);
          se = x2_add(se, x2_add(fl[i], make_float2(o0.y, o1.y)));
          Eo[2 * i * 64] = make_float2(sh.x, se.x);
          Eo[(2 * i + 1) * 64] = make_float2(sh.y, se.y);
          tv[2 * i] = sh.x;
          tv[2 * i + 1] = sh.y;
        }
        // T_ij, i = 16 b + 8 e8 .., at lane j
        asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(
                         st.tmem + lq + (unsigned)(kM128TmemT + 128 * h + 16 * b + 8 * e8)),
                     "f"(tv[0]), "f"(tv[1]), "f"(tv[2]), "f"(tv[3]), "f"(tv[4]), "f"(tv[5]), "f"(tv[6]), "f"(tv[7])
                     : "memory");
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        tc05_fence_before();
      }
      m128_sync();
      // R_km = delta_km - S_km + T_km chi~_m, two columns per thread
      const int m0 = 64 * T + 2 * lane;
      if (m0 < ld) {
        float4* sp = reinterpret_cast<float4*>(S + k * ld) + ((m0 >> 1) ^ (k & 15));
        const bool live = k < n8 && m0 < n8;
        const float4 s = live ? *sp : make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 tr2 = *reinterpret_cast<const float4*>(E + warp * 64 + 2 * lane);
        const float4 ti2 = *reinterpret_cast<const float4*>(E + (16 + warp) * 64 + 2 * lane);
        float2 r[2];
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          const int m = m0 + x;
          const float2 tre = x ? make_float2(tr2.z, tr2.w) : make_float2(tr2.x, tr2.y);
          const float2 tim = x ? make_float2(ti2.z, ti2.w) : make_float2(ti2.x, ti2.y);
          float sr = 0.f, lr = 0.f, si = 0.f, li = 0.f;
          cdf_fma(sr, lr, si, li, make_float2(tre.x, tim.x), make_float2(tre.y, tim.y), chih[m], chil[m]);
          df_add(sr, lr, x ? -s.z : -s.x);
          df_add(si, li, x ? -s.w : -s.y);
          if (k == m) {
            df_add(sr, lr, 1.f);
            td[k] = make_float4(tre.x, tre.y, tim.x, tim.y);
          }
          r[x] = make_float2(sr + lr, si + li);
        }
        *sp = make_float4(r[0].x, r[0].y, r[1].x, r[1].y);
      }
      m128_sync();                                          // the exchange is read
    }
  }
  // ---- diag(R T): lane j against its row of R, the four warps of a quadrant a quarter of m each ----
  tc05_fence_after();
  float2* part = E;                                         // [4][128]
  {
    const int g = warp >> 2, m0 = 32 * g;
    float ex = 0.f, ey = 0.f;
    if (m0 < n8) {
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        float a_[16], b_[16];
        tmem_ld16(st.tmem + lq + (unsigned)(kM128TmemT + m0 + 16 * hh), a_);
        tmem_ld16(st.tmem + lq + (unsigned)(kM128TmemT + 128 + m0 + 16 * hh), b_);
        if (jl < n8) {
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const int m = m0 + 16 * hh + i;
            if (m < n8) {
              const float2 w = S[sidx(jl, m)];
              ex = fmaf(w.x, a_[i], fmaf(-w.y, b_[i], ex));
              ey = fmaf(w.x, b_[i], fmaf(w.y, a_[i], ey));
            }
          }
        }
      }
    }
    part[g * 128 + jl] = make_float2(ex, ey);
  }
  bool fin = *badw == 0;                                    // (the next ladder resets it)
  if (!ok) *st.fail = 1;
  tc05_fence_before();
  m128_sync();
  const bool good = *st.fail == 0;
  // ---- the Eq. sd bracket (warps 0-3) and the error control (warp 4); the others go on ----
  auto corr = [&](int j) {
    const float2 p0 = part[j], p1 = part[128 + j], p2 = part[256 + j], p3 = part[384 + j];
    return make_float2((p0.x + p1.x) + (p2.x + p3.x), (p0.y + p1.y) + (p2.y + p3.y));
  };
  if (t < n) {
    const int j = t;
    const float4 d0 = td[j], g2 = g2s[j];
    const float2 ec = corr(j);
    const double gx = ((double)d0.x + (double)d0.y) + (double)ec.x, gy = ((double)d0.z + (double)d0.w) + (double)ec.y;
    const double wgt = (c == 0) ? 1.0 : 3.0;
    kc[(((size_t)c * nb + a) * n + j) * N + q] = mk(wgt * (gx - 0.5 * ((double)g2.x + (double)g2.y)),
                                                    wgt * (gy - 0.5 * ((double)g2.z + (double)g2.w)));
  }
  if (warp == 4) {
    float emax = 0.f, gmax = 0.f;
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const int j = lane + 32 * x;
      if (j < n) {
        const float4 d0 = td[j];
        const float2 ec = corr(j);
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
  return good;
}

// Set-up and tear-down of a block (all threads); bars: 1 + 2 kM128MaxRing barriers
__device__ __forceinline__ void m128_setup(M128State& st, unsigned char* sm, uint64_t* bars, unsigned* tslot, volatile int* fail) {
  if ((threadIdx.x >> 5) == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tslot)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 0) {
    for (int i = 0; i < 1 + 2 * kM128MaxRing; ++i)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bars + i)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    *fail = 0;
  }
  tc05_fence_before();
  __syncthreads();
  tc05_fence_after();
  st = M128State{sm, *tslot, bars, bars + 1, bars + 1 + kM128MaxRing, 0u, 0, 0u, fail};
}
__device__ __forceinline__ void m128_teardown(const M128State& st) {
  tc05_fence_before();
  __syncthreads();
  tc05_fence_after();
  if ((threadIdx.x >> 5) == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(st.tmem) : "memory");
}
// after a wait that gave up (all threads): the copies in flight land and the MMAs queued complete, both
// bounded, before shared and tensor memory are given back
__device__ __forceinline__ void m128_drain(const M128State& st, const M128Layout& L) {
  if (threadIdx.x == kM128Streamer) {
    // a slot's last copy was of this round below the position, of the round before from it on (a slot
    // never used passes at once)
    for (int i = 0; i < L.nring; ++i) mbar_wait(st.full + i, i < st.slot ? st.round : st.round ^ 1u);
  } else if (threadIdx.x == kM128Issuer) {
    umma_commit(st.done);
    mbar_wait(st.done, st.phase);
  }
}

}  // namespace df
