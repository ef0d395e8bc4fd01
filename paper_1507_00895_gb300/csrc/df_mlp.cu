// Learned warm start of the dual self-energy: a dense network (4 layers,
// n_in -> W -> W -> W -> n_out, tanh between, linear output) evaluated and
// trained with this file's kernels.  Operands of every matrix product are
// rounded to BF16 and multiplied on the tensor cores (tcgen05, FP32
// accumulate in tensor memory); master weights, biases, Adam moments and
// activations are FP32.  The network's output is Sigma~ on the irreducible wedge of the
// square lattice's point group at positive Matsubara frequencies;
// df_warmstart_sigma expands it to the whole grid (D4 images and
// Sigma~(k, -w) = conj Sigma~(k, w)) and sets it as the loop's Sigma~.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <random>
#include <vector>

#include <cuda_bf16.h>

#include "df_mixed_dev.cuh"

namespace df {

// ---- BF16 operands as swizzled atoms ---------------------------------------
// A BF16 matrix X[r][c] that a product reads is kept in global memory as
// 1 KB atoms of 8 rows x 64 columns, the 128-byte-swizzled layout of the
// tensor cores' shared-memory operands: 16-byte chunk q of row r at chunk
// q ^ (r & 7).  Atom (r / 8, c / 64) is at index (c / 64) * rg + r / 8, rg the
// number of 8-row groups (rows and columns padded to 128 with zeros).  A
// run of row groups of one 64-column block is one contiguous piece, so
// that a bulk asynchronous copy brings a whole tile, and the same atoms
// serve a product that sums over the columns (K-major operand) and one that
// sums over the rows (MN-major operand): the network's three products per
// layer read activations, dZ and weights in both ways without a transpose.
__host__ __device__ constexpr long pad128(long x) { return (x + 127) / 128 * 128; }
__host__ __device__ constexpr size_t atoms_bytes(long rows, long cols) { return (size_t)pad128(rows) * pad128(cols) * 2; }
// byte offset of the 16-byte chunk holding columns c .. c + 7 (c a multiple of 8) of row r
__device__ __forceinline__ size_t atom_chunk(int r, int c, int rg) {
  return ((size_t)(c >> 6) * rg + (r >> 3)) * 1024 + (size_t)((r & 7) * 128 + ((((c & 63) >> 3) ^ (r & 7)) << 4));
}
__device__ __forceinline__ unsigned pack_bf16(float lo, float hi) {
  const __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const unsigned*>(&p);
}

// ---- the products ------------------------------------------------------------
// One kernel for every product D[m][n] = sum_k A(m, k) B(k, n) of the network,
// an output tile of TM x TN per block, K in stages of KB blocks of 64:
//   warp 8 (one lane) streams the operand tiles into a ring of NS stages by
//   bulk asynchronous copies; warp 9 (one lane) issues the MMAs (M = TM,
//   N = TN, K = 16, FP32 accumulator in tensor memory) and its commits hand
//   the stages back; warps 0-7 run the epilogue, and where B is the FP32
//   weights (WF32: the forward products) they round the weight tile to BF16
//   into the stage, loading one stage ahead in registers, and with wsh leave
//   the rounded tile in global memory for the backward product.
// AMN / BMN: the operand's M / N index is the atoms' column (MN-major), the
// sum runs over the atoms' rows; else K-major.
// The accumulation runs over k in order whatever the tile, so every tile
// shape gives the same bits.
// A 256-row batch at 512 x 71808 (before: FP32 operands rounded and transposed
// by every block with two-byte stores, two stages, 128 x 128 tiles throughout):
//   forward with the loss     0.11 ms   147 MB of weights, 74 MB of targets read
//   weight gradient           0.056 ms  147 MB of gradients written (HBM: 0.03)
//   activation gradient       0.23 ms   K = 71808; one block per 64 x 16 outputs so that
//                                       128 of the 152 SMs work, bound by the L2 -> shared
//                                       memory traffic of its 1.5 GB of tiles (was 8 blocks,
//                                       ~10 ms); a split K would change the summation order
//                                       and with it BF16 roundings downstream
// and the whole training step 13.1 -> 0.70 ms.
enum GemmEpi {
  kEpiStore = 0,     // C = D
  kEpiTanh = 1,      // a = tanh(D + bias): C = a, Cb = bf16(a)
  kEpiLinear = 2,    // C = D + bias
  kEpiLoss = 3,      // y = D + bias, dZ = 2 (y - aux) scale: Cb = bf16(dZ), column and loss partials
  kEpiBack = 4,      // dZ = D (1 - aux^2): Cb = bf16(dZ), column partials
};

struct GemmArgs {
  int M, N, nkb;                 // outputs; K in 64-blocks
  const unsigned char* A;        // atoms, a_rg row groups
  int a_rg;
  const unsigned char* B;        // atoms, b_rg row groups (not WF32)
  int b_rg;
  const float* W;                // WF32: W[k][n], k < kw rows, ldw = N
  int kw, wvec;
  unsigned char* wsh;            // WF32: the rounded weights' atoms (NULL: not kept)
  int wsh_rg;
  int epi;
  float* C;                      // FP32 output, row stride N
  unsigned char* Cb;             // BF16 atoms of the output
  int cb_rg;
  const float* bias;
  const float* aux;              // kEpiLoss: target, kEpiBack: activations; row stride N
  float scale;
  float* part_col;               // [m tiles * 4][N] sums of dZ over a quadrant's rows
  float* part_loss;              // [blocks] sums of (y - target)^2
  int* err;
};

constexpr int kGemmThreads = 320;

__host__ __device__ constexpr int gemm_stage_bytes(int TM, int TN, int KB) { return (TM + TN) * 128 * KB; }
__host__ __device__ constexpr int gemm_smem_bytes(int TM, int TN, int KB, int NS) {
  const int ring = NS * gemm_stage_bytes(TM, TN, KB), epi = 8 * 32 * 33 * 4;
  return (ring > epi ? ring : epi) + 1024;
}

// shared-memory descriptor of an MN-major operand of 128-byte-swizzled atoms:
// atoms along K 1024 B apart, along M / N (64 elements) 8192 B apart
__device__ __forceinline__ uint64_t umma_desc_mn(unsigned saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(8192 >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

__device__ __forceinline__ void bulk_g2s(unsigned dst, const void* src, unsigned bytes, uint64_t* mbar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(smem_u32(mbar))
               : "memory");
}
__device__ __forceinline__ void mbar_init(uint64_t* b, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint64_t* b, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}

// the tile's loads of one operand for stage `it`: T rows of the product
// (m or n) from t0, KB 64-blocks of k
template <int T, int KB, bool MN>
__device__ __forceinline__ void load_operand(const unsigned char* X, int rg, int t0, int it, unsigned dst,
                                             uint64_t* full) {
  if constexpr (MN) {
    static_assert(KB == 1 && T % 64 == 0, "MN-major tiles are 64-column blocks of 8 row groups");
#pragma unroll
    for (int cb = 0; cb < T / 64; ++cb)
      bulk_g2s(dst + cb * 8192, X + ((size_t)(t0 / 64 + cb) * rg + it * 8) * 1024, 8192, full);
  } else {
#pragma unroll
    for (int kb = 0; kb < KB; ++kb)
      bulk_g2s(dst + kb * T * 128, X + ((size_t)(it * KB + kb) * rg + t0 / 8) * 1024, T * 128, full);
  }
}

template <int TM, int TN, int KB, int NS, bool AMN, bool BMN, bool WF32>
__global__ void __launch_bounds__(kGemmThreads, TM == 128 ? 2 : 1)
gemm_tc_kernel(const GemmArgs g) {
  static_assert(!WF32 || (BMN && KB == 1 && !AMN), "FP32 weights are the forward products' B operand");
  extern __shared__ unsigned char gsm_raw[];
  __shared__ uint64_t full_s[NS], empty_s[NS], done_s;
  __shared__ unsigned tslot_s;
  __shared__ int fail_s;
  __shared__ float loss_s[8];
  unsigned char* gsm = reinterpret_cast<unsigned char*>(((uintptr_t)gsm_raw + 1023) & ~(uintptr_t)1023);
  constexpr int kA = TM * 128 * KB, kB = TN * 128 * KB, kStage = kA + kB;
  constexpr int kTmem = TN < 32 ? 32 : TN;
  // (tiles in a one-dimensional grid, those of one column block together: the other dimensions end at 65,535)
  const int mtiles = (g.M + TM - 1) / TM, bm = blockIdx.x % mtiles, bn = blockIdx.x / mtiles;
  const int m0 = bm * TM, n0 = bn * TN;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nit = (g.nkb + KB - 1) / KB;
  if (warp == 0) tmem_alloc_cols<kTmem>(&tslot_s);
  if (tid == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(&full_s[s], WF32 ? 9 : 1);      // the copies' thread, and the eight converting warps
      mbar_init(&empty_s[s], 1);
    }
    mbar_init(&done_s, 1);
    fail_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc05_fence_before();
  __syncthreads();
  tc05_fence_after();
  const unsigned tmem = tslot_s, ring = smem_u32(gsm);

  if (warp == 8) {
    if (lane == 0) {
      int it = 0;
      for (; it < nit; ++it) {
        const int s = it % NS;
        if (it >= NS && !mbar_wait(&empty_s[s], (unsigned)((it / NS - 1) & 1))) break;
        mbar_expect(&full_s[s], WF32 ? kA : kStage);
        load_operand<TM, KB, AMN>(g.A, g.a_rg, m0, it, ring + s * kStage, &full_s[s]);
        if constexpr (!WF32) load_operand<TN, KB, BMN>(g.B, g.b_rg, n0, it, ring + s * kStage + kA, &full_s[s]);
      }
      if (it < nit) {                           // gave up: its copies in flight land first (bounded)
        fail_s = 1;
        for (int k = it - NS < 0 ? 0 : it - NS; k < it; ++k) mbar_wait(&full_s[k % NS], (unsigned)((k / NS) & 1));
      }
    }
  } else if (warp == 9) {
    if (lane == 0) {
      const unsigned idesc = umma_idesc_bf16(TM, TN) | (AMN ? 1u << 15 : 0u) | (BMN ? 1u << 16 : 0u);
      int it = 0;
      for (; it < nit; ++it) {
        const int s = it % NS;
        if (!mbar_wait(&full_s[s], (unsigned)((it / NS) & 1))) break;
        tc05_fence_after();
        const unsigned a = ring + s * kStage, b = a + kA;
#pragma unroll
        for (int kb = 0; kb < KB; ++kb)
#pragma unroll
          for (int ks = 0; ks < 4; ++ks) {
            const uint64_t da = AMN ? umma_desc_mn(a + 2048 * ks) : umma_desc_sw128(a + kb * TM * 128 + 32 * ks);
            const uint64_t db = BMN ? umma_desc_mn(b + 2048 * ks) : umma_desc_sw128(b + kb * TN * 128 + 32 * ks);
            umma_bf16(tmem, da, db, idesc, (it > 0 || kb > 0 || ks > 0) ? 1u : 0u);
          }
        umma_commit(&empty_s[s]);
      }
      if (it < nit) fail_s = 1;
      umma_commit(&done_s);
    }
  } else {
    if constexpr (WF32) {
      // the weight tile: 64 k x TN n, float4 along n
      constexpr int kPer = 64 * TN / 4 / 256;
      float4 w[kPer];
      auto fetch = [&](int it) {
#pragma unroll
        for (int e = 0; e < kPer; ++e) {
          const int f = tid + 256 * e, k = it * 64 + f / (TN / 4), n = n0 + (f % (TN / 4)) * 4;
          w[e] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (k < g.kw) {
            const float* src = g.W + (size_t)k * g.N + n;
            if (g.wvec && n + 3 < g.N) {
              w[e] = __ldcs(reinterpret_cast<const float4*>(src));
            } else {
              if (n < g.N) w[e].x = src[0];
              if (n + 1 < g.N) w[e].y = src[1];
              if (n + 2 < g.N) w[e].z = src[2];
              if (n + 3 < g.N) w[e].w = src[3];
            }
          }
        }
      };
      fetch(0);
      bool ok = true;
      for (int it = 0; it < nit; ++it) {
        const int s = it % NS;
        if (it >= NS && !(ok = mbar_wait(&empty_s[s], (unsigned)((it / NS - 1) & 1)))) break;
        unsigned char* bt = gsm + s * kStage + kA;
#pragma unroll
        for (int e = 0; e < kPer; ++e) {
          const int f = tid + 256 * e, k = f / (TN / 4), c = (f % (TN / 4)) * 4;
          const uint2 v = make_uint2(pack_bf16(w[e].x, w[e].y), pack_bf16(w[e].z, w[e].w));
          const unsigned o = (unsigned)((k & 7) * 128 + ((((c & 63) >> 3) ^ (k & 7)) << 4) + (c & 4) * 2);
          *reinterpret_cast<uint2*>(bt + (c >> 6) * 8192 + (k >> 3) * 1024 + o) = v;
          if (g.wsh && bm == 0)
            *reinterpret_cast<uint2*>(g.wsh + ((size_t)((n0 + c) >> 6) * g.wsh_rg + it * 8 + (k >> 3)) * 1024 + o) = v;
        }
        if (it + 1 < nit) fetch(it + 1);
        fence_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&full_s[s]);
      }
      if (!ok) fail_s = 1;
    }
    // (the whole sum's products: the limit grows with their number)
    if (!mbar_wait(&done_s, 0u, kMbarSpin * (1u + min(nit >> 12, 1000)))) fail_s = 1;
    tc05_fence_after();
  }
  __syncthreads();
  const bool fail = fail_s != 0;
  if (fail) {
    if (tid == 0) atomicOr(g.err, 1);
  } else if (warp < 8) {
    // epilogue: warp w takes lane quadrant w % 4 and every second group of CW columns
    constexpr int CW = TN >= 64 ? 32 : 16;
    const int q = warp & 3;
    const bool live = TM == 128 || lane < 16;             // TM = 64: rows 16 q .. 16 q + 15 in lanes 0-15
    const int r = m0 + (TM == 128 ? 32 * q + lane : 16 * q + lane);
    const bool in = live && r < g.M;
    float* stg = reinterpret_cast<float*>(gsm) + warp * 32 * 33;
    float loss = 0.f;
#pragma unroll 1
    for (int ci = warp >> 2; ci < TN / CW; ci += 2) {
      float v[CW];
      const unsigned ta = tmem + ((32u * q) << 16) + (unsigned)(CW * ci);
      tmem_ld16(ta, v);
      if constexpr (CW == 32) tmem_ld16(ta + 16, v + 16);
      const int nb = n0 + CW * ci;
      if (g.epi == kEpiTanh || g.epi == kEpiLinear || g.epi == kEpiLoss) {
#pragma unroll
        for (int e = 0; e < CW; ++e)
          if (nb + e < g.N) v[e] += __ldg(g.bias + nb + e);
      }
      if (g.epi == kEpiTanh) {
#pragma unroll
        for (int e = 0; e < CW; ++e) v[e] = tanhf(v[e]);
      }
      const bool dz = g.epi == kEpiLoss || g.epi == kEpiBack;
      if (dz || g.C) {                         // through shared memory: a lane per column, rows coalesced
        constexpr int kRows = TM == 128 ? 32 : 16;
        const int n = nb + lane, rq = m0 + kRows * q, rows = max(0, min(kRows, g.M - rq));
        __syncwarp();
#pragma unroll
        for (int e = 0; e < CW; ++e) stg[lane * 33 + e] = v[e];
        __syncwarp();
        if (lane < CW && n < g.N) {
          if (g.C) {
            float* dst = g.C + (size_t)rq * g.N + n;
            for (int k = 0; k < rows; ++k) __stcs(dst + (size_t)k * g.N, stg[k * 33 + lane]);
          }
          if (dz) {
            const float* ax = g.aux + (size_t)rq * g.N + n;
            float s = 0.f;
#pragma unroll
            for (int k0 = 0; k0 < kRows; k0 += 16) {
              float x[16];
#pragma unroll
              for (int k = 0; k < 16; ++k) x[k] = k0 + k < rows ? __ldg(ax + (size_t)(k0 + k) * g.N) : 0.f;
#pragma unroll
              for (int k = 0; k < 16; ++k) {
                float& y = stg[(k0 + k) * 33 + lane];
                float z = 0.f;
                if (k0 + k < rows) {
                  if (g.epi == kEpiLoss) {
                    const float d = y - x[k];
                    z = 2.f * d * g.scale;
                    loss += d * d;
                  } else {
                    z = y * (1.f - x[k] * x[k]);
                  }
                }
                y = z;
                s += z;
              }
            }
            g.part_col[(size_t)(bm * 4 + q) * g.N + n] = s;
          }
        }
        if (dz) {
          __syncwarp();
#pragma unroll
          for (int e = 0; e < CW; ++e) v[e] = stg[lane * 33 + e];
        }
      }
      if (g.Cb) {                              // padding rows and columns as zeros
#pragma unroll
        for (int e = 0; e < CW; ++e)
          if (!in || nb + e >= g.N) v[e] = 0.f;
        if (live) {
#pragma unroll
          for (int e = 0; e < CW; e += 8)
            *reinterpret_cast<uint4*>(g.Cb + atom_chunk(r, nb + e, g.cb_rg)) =
                make_uint4(pack_bf16(v[e], v[e + 1]), pack_bf16(v[e + 2], v[e + 3]), pack_bf16(v[e + 4], v[e + 5]),
                           pack_bf16(v[e + 6], v[e + 7]));
        }
      }
    }
    if (g.epi == kEpiLoss) {
      for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
      if (lane == 0) loss_s[warp] = loss;
    }
  }
  tc05_fence_before();
  __syncthreads();
  tc05_fence_after();
  if (!fail && g.epi == kEpiLoss && tid == 0) {
    float s = 0.f;
    for (int w = 0; w < 8; ++w) s += loss_s[w];
    g.part_loss[blockIdx.x] = s;
  }
  if (warp == 0) tmem_dealloc_cols<kTmem>(tmem);
}

// x [M][N] FP32 -> BF16 atoms, rows up to the next multiple of 128 and padding columns zero
__global__ void to_atoms_kernel(int M, int N, const float* __restrict__ x, unsigned char* __restrict__ out, int rg) {
  const int cols8 = (int)(pad128(N) / 8);
  const long total = pad128(M) * cols8;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < total; i += (long)gridDim.x * blockDim.x) {
    const int r = (int)(i / cols8), c = (int)(i - (long)r * cols8) * 8;
    float v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = (r < M && c + e < N) ? x[(size_t)r * N + c + e] : 0.f;
    *reinterpret_cast<uint4*>(out + atom_chunk(r, c, rg)) =
        make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
  }
}

// db_l[n] = sum of the layer's row-quadrant partials of dZ (blockIdx.y = layer)
struct BiasGrads {
  const float* part[4];
  float* db[4];
  int n[4], parts[4];
};
__global__ void bias_grad_kernel(const BiasGrads b) {
  const int l = blockIdx.y, N = b.n[l];
  for (int n = blockIdx.x * blockDim.x + threadIdx.x; n < N; n += gridDim.x * blockDim.x) {
    float s = 0.f;
    for (int p = 0; p < b.parts[l]; ++p) s += b.part[l][(size_t)p * N + n];
    b.db[l][n] = s;
  }
}

// bound by HBM: 16 B read and 12 B written per parameter, four parameters per thread and step
__device__ __forceinline__ void adam_one(float& p, float gv, float& m1, float& m2, float lr, float b1, float b2,
                                         float eps, float c1, float c2) {
  const float a = b1 * m1 + (1.f - b1) * gv;
  const float b = b2 * m2 + (1.f - b2) * gv * gv;
  m1 = a;
  m2 = b;
  p -= lr * (a / c1) / (sqrtf(b / c2) + eps);
}
__global__ void __launch_bounds__(256)
adam_kernel(long count, float* __restrict__ p, const float* __restrict__ gr, float* __restrict__ m1,
            float* __restrict__ m2, float lr, float b1, float b2, float eps, float c1, float c2) {
  const long i = (blockIdx.x * (long)blockDim.x + threadIdx.x) * 4;
  if (i + 3 < count) {
    float4 pv = *reinterpret_cast<const float4*>(p + i), av = *reinterpret_cast<const float4*>(m1 + i),
           bv = *reinterpret_cast<const float4*>(m2 + i);
    const float4 gv = *reinterpret_cast<const float4*>(gr + i);
    adam_one(pv.x, gv.x, av.x, bv.x, lr, b1, b2, eps, c1, c2);
    adam_one(pv.y, gv.y, av.y, bv.y, lr, b1, b2, eps, c1, c2);
    adam_one(pv.z, gv.z, av.z, bv.z, lr, b1, b2, eps, c1, c2);
    adam_one(pv.w, gv.w, av.w, bv.w, lr, b1, b2, eps, c1, c2);
    *reinterpret_cast<float4*>(p + i) = pv;
    *reinterpret_cast<float4*>(m1 + i) = av;
    *reinterpret_cast<float4*>(m2 + i) = bv;
  } else {
    for (long k = i; k < count; ++k) adam_one(p[k], gr[k], m1[k], m2[k], lr, b1, b2, eps, c1, c2);
  }
}

// Sigma~[i][r] from the wedge output y [n_wedge][n_w/2][2]: w = kmap[r],
// n = i - n_w/2 >= 0 -> y[w][n], n < 0 -> conj y[w][-n-1]; y de-normalised
// with mean / std of the same layout.
__global__ void warmstart_expand_kernel(int n_w, int N, const int* __restrict__ kmap, const float* __restrict__ y,
                                        const float* __restrict__ mean, const float* __restrict__ sd,
                                        double2* __restrict__ sigma) {
  const int total = n_w * N;
  const int half = n_w / 2;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += gridDim.x * blockDim.x) {
    const int i = idx / N, r = idx - i * N;
    const int n = i - half;
    const int f = n >= 0 ? n : -n - 1;
    const long o = ((long)kmap[r] * half + f) * 2;
    const double re = (double)y[o] * sd[o] + mean[o];
    const double im = (double)y[o + 1] * sd[o + 1] + mean[o + 1];
    sigma[idx] = mk(re, n >= 0 ? im : -im);
  }
}

}  // namespace df

using namespace df;

struct df_mlp {
  int dims[5];
  int max_batch = 0;
  cudaStream_t stream = nullptr;
  std::string err;
  float* params = nullptr;   // W1 b1 W2 b2 W3 b3 W4 b4 (W_l row-major [in][out])
  float* grads = nullptr;
  float* m1 = nullptr;
  float* m2 = nullptr;
  long nparam = 0;
  long off_w[4], off_b[4];
  float* act[4] = {};        // act[l] = output of hidden layer l (l = 1, 2, 3)
  unsigned char* actb[4] = {};  // BF16 atoms: the input (0) and the hidden layers' outputs
  unsigned char* dzb[4] = {};   // BF16 atoms of dZ of layer l's output
  unsigned char* wb[4] = {};    // BF16 atoms of W_l (l >= 1), left by the forward products of a gradient
  float* part_col[4] = {};      // dZ's column sums per row quadrant (bias gradients)
  float* part_loss = nullptr;
  long loss_blocks = 0;         // capacity of part_loss
  int* d_timeout = nullptr;  // set by a tensor-core GEMM whose bounded wait gave up
  long step = 0;
};

namespace {

df_status mfail(df_mlp* m, df_status s, const char* what, cudaError_t e = cudaSuccess) {
  if (m) {
    char buf[256];
    snprintf(buf, sizeof buf, "%s%s%s", what, e != cudaSuccess ? ": " : "", e != cudaSuccess ? cudaGetErrorString(e) : "");
    m->err = buf;
  }
  return s;
}

#define M_CUDA(m, call, what)                                                                  \
  do {                                                                                         \
    cudaError_t e__ = (call);                                                                  \
    if (e__ != cudaSuccess)                                                                    \
      return mfail((m), e__ == cudaErrorMemoryAllocation ? DF_ERR_OOM : DF_ERR_CUDA, (what), e__); \
  } while (0)

template <int TM, int TN, int KB, int NS, bool AMN, bool BMN, bool WF32>
cudaError_t launch_gemm(cudaStream_t s, const GemmArgs& g) {
  constexpr int smem = gemm_smem_bytes(TM, TN, KB, NS);
  auto fn = gemm_tc_kernel<TM, TN, KB, NS, AMN, BMN, WF32>;
  cudaError_t e = cudaFuncSetAttribute((const void*)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const long grid = (long)((g.M + TM - 1) / TM) * (((long)g.N + TN - 1) / TN);
  if (grid > 0x7FFFFFFFL) return cudaErrorInvalidConfiguration;
  fn<<<(unsigned)grid, kGemmThreads, smem, s>>>(g);
  return cudaGetLastError();
}

// forward and weight-gradient tiles: 128 columns, or 64 when 128 leave the
// 152 SMs without a block each (the width-512 layers).  The activation gradient takes 64 x 16 at every size: at
// 256 x 512 outputs that is 128 blocks (8 with 128 x 128); larger batches and widths, whose operands
// wider tiles would read less often, are not tuned
bool wide_tiles(int M, int N) { return (long)((M + 127) / 128) * ((N + 127) / 128) >= 152; }

int rg_of(long rows) { return (int)(pad128(rows) / 8); }
bool vec4(const float* p, int ld) { return ((uintptr_t)p & 15) == 0 && ld % 4 == 0; }

// y: the FP32 output [B][n_out], or with target (and y NULL) dZ of the loss
df_status forward(df_mlp* m, const float* x, int B, float* y, const float* target, bool keep_w) {
  const int rb = rg_of(m->max_batch);
  const long chunks = pad128(B) * (pad128(m->dims[0]) / 8);
  to_atoms_kernel<<<(int)std::min<long>(1024, (chunks + 255) / 256), 256, 0, m->stream>>>(B, m->dims[0], x, m->actb[0],
                                                                                         rb);
  M_CUDA(m, cudaGetLastError(), "input to BF16");
  for (int l = 0; l < 4; ++l) {
    const int in = m->dims[l], out = m->dims[l + 1];
    GemmArgs g{};
    g.M = B; g.N = out; g.nkb = (in + 63) / 64;
    g.A = m->actb[l]; g.a_rg = rb;
    g.W = m->params + m->off_w[l]; g.kw = in; g.wvec = vec4(g.W, out);
    if (keep_w && l > 0) { g.wsh = m->wb[l]; g.wsh_rg = rg_of(in); }
    g.bias = m->params + m->off_b[l];
    g.err = m->d_timeout;
    if (l < 3) {
      g.epi = kEpiTanh; g.C = m->act[l + 1]; g.Cb = m->actb[l + 1]; g.cb_rg = rb;
    } else if (target) {
      g.epi = kEpiLoss; g.aux = target; g.scale = 1.f / (float)((long)B * out);
      g.Cb = m->dzb[3]; g.cb_rg = rb; g.part_col = m->part_col[3]; g.part_loss = m->part_loss;
    } else {
      g.epi = kEpiLinear; g.C = y;
    }
    M_CUDA(m, wide_tiles(B, out) ? (launch_gemm<128, 128, 1, 3, false, true, true>(m->stream, g))
                                 : (launch_gemm<128, 64, 1, 4, false, true, true>(m->stream, g)),
           "forward GEMM");
  }
  return DF_OK;
}

df_status backward(df_mlp* m, int B, float* loss_host) {
  const int rb = rg_of(m->max_batch);
  BiasGrads bg{};
  int nmax = 0;
  for (int l = 3; l >= 0; --l) {
    const int in = m->dims[l], out = m->dims[l + 1];
    bg.part[l] = m->part_col[l];
    bg.db[l] = m->grads + m->off_b[l];
    bg.n[l] = out;
    bg.parts[l] = 4 * (l == 3 ? (B + 127) / 128 : (B + 63) / 64);
    nmax = std::max(nmax, out);
    // dW_l[in][out] = A_l^T dZ_l   (M = in, N = out, K = B)
    GemmArgs w{};
    w.M = in; w.N = out; w.nkb = (B + 63) / 64;
    w.A = m->actb[l]; w.a_rg = rb;
    w.B = m->dzb[l]; w.b_rg = rb;
    w.epi = kEpiStore; w.C = m->grads + m->off_w[l]; w.err = m->d_timeout;
    M_CUDA(m, wide_tiles(in, out) ? (launch_gemm<128, 128, 1, 3, true, true, false>(m->stream, w))
                                  : (launch_gemm<128, 64, 1, 4, true, true, false>(m->stream, w)),
           "weight gradient");
    if (l == 0) break;
    // dZ_{l-1} = (dZ_l W_l^T) (1 - A_l^2)   (M = B, N = in, K = out)
    GemmArgs d{};
    d.M = B; d.N = in; d.nkb = (int)(pad128(out) / 64);
    d.A = m->dzb[l]; d.a_rg = rb;
    d.B = m->wb[l]; d.b_rg = rg_of(in);
    d.epi = kEpiBack; d.aux = m->act[l];
    d.Cb = m->dzb[l - 1]; d.cb_rg = rb; d.part_col = m->part_col[l - 1]; d.err = m->d_timeout;
    M_CUDA(m, (launch_gemm<64, 16, 2, 8, false, false, false>(m->stream, d)), "activation gradient");
  }
  bias_grad_kernel<<<dim3((nmax + 255) / 256, 4), 256, 0, m->stream>>>(bg);
  M_CUDA(m, cudaGetLastError(), "bias gradients");
  if (loss_host) {
    const int nout = m->dims[4];
    const int tn = wide_tiles(B, nout) ? 128 : 64;
    const long nb = (long)((B + 127) / 128) * ((nout + tn - 1) / tn);
    std::vector<float> part(nb);
    M_CUDA(m, cudaMemcpyAsync(part.data(), m->part_loss, sizeof(float) * nb, cudaMemcpyDeviceToHost, m->stream),
           "loss copy");
    int timeout = 0;
    M_CUDA(m, cudaMemcpyAsync(&timeout, m->d_timeout, sizeof(int), cudaMemcpyDeviceToHost, m->stream), "flag copy");
    M_CUDA(m, cudaStreamSynchronize(m->stream), "loss");
    if (timeout) return mfail(m, DF_ERR_TIMEOUT, "a tensor-core GEMM's completion wait gave up");
    double s = 0.0;
    for (float v : part) s += v;
    *loss_host = (float)(s / (double)((long)B * nout));
  }
  return DF_OK;
}

}  // namespace

extern "C" {

df_status df_mlp_create(df_mlp** out, int n_in, int width, int n_out, int max_batch, unsigned long long seed,
                        void* stream) {
  if (!out || n_in < 1 || width < 1 || n_out < 1 || max_batch < 1) return DF_ERR_ARG;
  *out = nullptr;
  df_mlp* m = new (std::nothrow) df_mlp();
  if (!m) return DF_ERR_OOM;
  const int d[5] = {n_in, width, width, width, n_out};
  memcpy(m->dims, d, sizeof d);
  m->max_batch = max_batch;
  m->stream = (cudaStream_t)stream;
  long o = 0;
  for (int l = 0; l < 4; ++l) {
    m->off_w[l] = o;
    o += (long)d[l] * d[l + 1];
    m->off_b[l] = o;
    o += d[l + 1];
  }
  m->nparam = o;
  // Glorot-uniform weights, zero biases (host RNG, seeded)
  std::vector<float> h(o, 0.f);
  std::mt19937_64 rng(seed);
  for (int l = 0; l < 4; ++l) {
    const float lim = std::sqrt(6.f / (float)(d[l] + d[l + 1]));
    std::uniform_real_distribution<float> U(-lim, lim);
    for (long i = 0; i < (long)d[l] * d[l + 1]; ++i) h[m->off_w[l] + i] = U(rng);
  }
  cudaError_t e;
  df_status st = DF_OK;
  if ((e = cudaMalloc(&m->params, sizeof(float) * o)) != cudaSuccess ||
      (e = cudaMalloc(&m->grads, sizeof(float) * o)) != cudaSuccess ||
      (e = cudaMalloc(&m->m1, sizeof(float) * o)) != cudaSuccess ||
      (e = cudaMalloc(&m->m2, sizeof(float) * o)) != cudaSuccess ||
      (e = cudaMalloc(&m->d_timeout, sizeof(int))) != cudaSuccess ||
      (e = cudaMemsetAsync(m->d_timeout, 0, sizeof(int), m->stream)) != cudaSuccess) {
    st = mfail(m, DF_ERR_OOM, "cudaMalloc", e);
  }
  const long pb = pad128(max_batch);
  m->loss_blocks = pb / 128 * ((n_out + 63) / 64);
  // the atoms' padding stays zero; every fill and copy on the network's stream, whose kernels nothing else
  // orders after the legacy stream's work
  auto zalloc = [&](void** p, size_t bytes) {
    if (st != DF_OK) return;
    if ((e = cudaMalloc(p, bytes)) != cudaSuccess || (e = cudaMemsetAsync(*p, 0, bytes, m->stream)) != cudaSuccess)
      st = mfail(m, DF_ERR_OOM, "cudaMalloc activations", e);
  };
  for (int l = 0; l < 4; ++l) {
    zalloc((void**)&m->actb[l], atoms_bytes(max_batch, d[l]));
    zalloc((void**)&m->dzb[l], atoms_bytes(max_batch, d[l + 1]));
    zalloc((void**)&m->part_col[l], sizeof(float) * (size_t)(pb / 64 * 4) * d[l + 1]);
    if (l > 0) {
      zalloc((void**)&m->act[l], sizeof(float) * (size_t)max_batch * d[l]);
      zalloc((void**)&m->wb[l], atoms_bytes(d[l], d[l + 1]));
    }
  }
  zalloc((void**)&m->part_loss, sizeof(float) * m->loss_blocks);
  if (st == DF_OK &&
      ((e = cudaMemcpyAsync(m->params, h.data(), sizeof(float) * o, cudaMemcpyHostToDevice, m->stream)) != cudaSuccess ||
       (e = cudaMemsetAsync(m->m1, 0, sizeof(float) * o, m->stream)) != cudaSuccess ||
       (e = cudaMemsetAsync(m->m2, 0, sizeof(float) * o, m->stream)) != cudaSuccess ||
       (e = cudaMemsetAsync(m->grads, 0, sizeof(float) * o, m->stream)) != cudaSuccess ||
       (e = cudaStreamSynchronize(m->stream)) != cudaSuccess))
    st = mfail(m, DF_ERR_CUDA, "initialise parameters", e);
  if (st != DF_OK) {
    fprintf(stderr, "libdf: df_mlp_create: %s\n", m->err.c_str());
    df_mlp_destroy(m);
    return st;
  }
  *out = m;
  return DF_OK;
}

void df_mlp_destroy(df_mlp* m) {
  if (!m) return;
  cudaFree(m->params);
  cudaFree(m->grads);
  cudaFree(m->m1);
  cudaFree(m->m2);
  cudaFree(m->part_loss);
  cudaFree(m->d_timeout);
  for (int l = 0; l < 4; ++l) {
    cudaFree(m->act[l]);
    cudaFree(m->actb[l]);
    cudaFree(m->dzb[l]);
    cudaFree(m->wb[l]);
    cudaFree(m->part_col[l]);
  }
  delete m;
}

df_status df_mlp_param_count(const df_mlp* m, long* count) {
  if (!m || !count) return DF_ERR_ARG;
  *count = m->nparam;
  return DF_OK;
}

df_status df_mlp_forward(df_mlp* m, const float* x, int batch, float* y) {
  if (!m || !x || !y || batch < 1 || batch > m->max_batch) return DF_ERR_ARG;
  return forward(m, x, batch, y, nullptr, false);
}

df_status df_mlp_gradients(df_mlp* m, const float* x, const float* target, int batch, float* loss_host) {
  if (!m || !x || !target || batch < 1 || batch > m->max_batch) return DF_ERR_ARG;
  df_status s = forward(m, x, batch, nullptr, target, true);
  if (s != DF_OK) return s;
  return backward(m, batch, loss_host);
}

df_status df_mlp_adam_step(df_mlp* m, float lr, float beta1, float beta2, float eps) {
  if (!m) return DF_ERR_ARG;
  ++m->step;
  const float c1 = 1.f - std::pow(beta1, (float)m->step), c2 = 1.f - std::pow(beta2, (float)m->step);
  adam_kernel<<<(unsigned)((m->nparam + 1023) / 1024), 256, 0, m->stream>>>(m->nparam, m->params, m->grads, m->m1, m->m2, lr, beta1,
                                                           beta2, eps, c1, c2);
  M_CUDA(m, cudaGetLastError(), "adam");
  return DF_OK;
}

df_status df_mlp_train_step(df_mlp* m, const float* x, const float* target, int batch, float lr, float* loss_host) {
  df_status s = df_mlp_gradients(m, x, target, batch, loss_host);
  if (s != DF_OK) return s;
  return df_mlp_adam_step(m, lr, 0.9f, 0.999f, 1e-8f);
}

df_status df_mlp_params(df_mlp* m, float* buf, int set, int is_device) {
  if (!m || !buf) return DF_ERR_ARG;
  const cudaMemcpyKind k = set ? (is_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice)
                               : (is_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost);
  M_CUDA(m, cudaMemcpyAsync(set ? m->params : buf, set ? buf : m->params, sizeof(float) * m->nparam, k, m->stream),
         "params");
  M_CUDA(m, cudaStreamSynchronize(m->stream), "params");
  return DF_OK;
}

df_status df_mlp_grads(df_mlp* m, float* buf, int is_device) {
  if (!m || !buf) return DF_ERR_ARG;
  M_CUDA(m, cudaMemcpyAsync(buf, m->grads, sizeof(float) * m->nparam,
                            is_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, m->stream),
         "grads");
  M_CUDA(m, cudaStreamSynchronize(m->stream), "grads");
  return DF_OK;
}

const char* df_mlp_last_error(const df_mlp* m) { return m ? m->err.c_str() : "NULL handle"; }

df_status df_warmstart_sigma(df_ctx* c, const float* y, const float* mean, const float* sd, const int* kmap) {
  if (!c || !y || !mean || !sd || !kmap) return DF_ERR_ARG;
  if (c->dm.n_w & 1) return DF_ERR_ARG;
  const int total = c->dm.n_w * c->dm.N;
  warmstart_expand_kernel<<<(total + 255) / 256, 256, 0, c->stream>>>(c->dm.n_w, c->dm.N, kmap, y, mean, sd, c->sigma);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = launch_dyson_ifft(c, c->dm.m_max, c->dm.n_w);
  if (e != cudaSuccess) {
    c->err = std::string("df_warmstart_sigma: ") + cudaGetErrorString(e);
    return DF_ERR_CUDA;
  }
  return DF_OK;
}

}  // extern "C"
