// Mixed-precision ladder solves (DF_FP32_IR) of order 64 < n <= 128: the default kernel around
// df_mixed128_dev.cuh, and with mixed_sweep = 1 the shared-memory Gauss-Jordan kernel
// (df_mixed_large_dev.cuh: one CTA of 2n threads per ladder, FP32 inversion with row
// exchanges in shared memory, double-float residual on the CUDA cores), which the default
// one beats at every order (3D workload, n = 96: 482 ms of ladders per pass against 182) and
// which shares no code with it.
#include "df_mixed128_dev.cuh"
#include "df_mixed_large_dev.cuh"

namespace df {

// gamma^T's (hi, lo) FP32 words: out_hi[c][a][k][i] = hi(gamma[c][a][i][k])
__global__ void split_gamma_t_kernel(int n, size_t mats, const double2* __restrict__ g, float2* __restrict__ th,
                                     float2* __restrict__ tl) {
  const size_t count = mats * n * n;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < count; e += (size_t)gridDim.x * blockDim.x) {
    const size_t m = e / ((size_t)n * n);
    const int r = (int)(e - m * n * n);
    const int k = r / n, i = r - k * n;
    const double2 v = g[m * n * n + (size_t)i * n + k];
    const float hx = (float)v.x, hy = (float)v.y;
    th[e] = make_float2(hx, hy);
    tl[e] = make_float2((float)(v.x - (double)hx), (float)(v.y - (double)hy));
  }
}

__global__ void __launch_bounds__(256, 1)
bse_gj_ir_kernel(Dims dm, int ch0, int nch, const float2* __restrict__ ghi, const float2* __restrict__ glo,
                 const float2* __restrict__ gth, const float2* __restrict__ gtl, const double2* __restrict__ gg,
                 const double2* __restrict__ chi, double2* __restrict__ kc, int* __restrict__ flags,
                 MixedCheck mc) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ GjShared sh;
  const long systems = (long)nch * dm.na * dm.N;
  for (long sys = blockIdx.x; sys < systems; sys += gridDim.x) {
    const int c = ch0 + (int)(sys / ((long)dm.na * dm.N));
    const int rem = (int)(sys - (long)(c - ch0) * dm.na * dm.N);
    const int a = dm.a0 + rem / dm.N, q = rem - (a - dm.a0) * dm.N;
    gj_ir_system(dm, c, a, q, ghi, glo, gth, gtl, gg, chi, kc, flags, smraw, sh, mc);
  }
}

// The default kernel of these orders (df_mixed128_dev.cuh): one contiguous range of ladders per
// block, one block per SM.
__global__ void gamma_digits128_kernel(int n, int count, const double2* __restrict__ gam,
                                       unsigned char* __restrict__ out) {
  gamma_digits_cols128(n, count, gam, out, (blockIdx.x * blockDim.x + threadIdx.x) >> 5, (gridDim.x * blockDim.x) >> 5,
                       threadIdx.x & 31);
}

__global__ void __launch_bounds__(kM128Threads, 1)
bse_mixed128_kernel(Dims dm, int ch0, int nch, const float2* __restrict__ gg_hi, const float2* __restrict__ gg_lo,
                    const double2* __restrict__ chi, double2* __restrict__ kc, const unsigned char* __restrict__ gdig,
                    int* __restrict__ flags, MixedCheck mc) {
  extern __shared__ __align__(1024) unsigned char sm128[];
  __shared__ uint64_t bars_s[1 + 2 * kM128MaxRing];
  __shared__ unsigned tslot_s;
  __shared__ int fail_s;
  if (smem_u32(sm128) & 1023u) {                 // the swizzled operand tiles need 1024-byte alignment
    if (threadIdx.x == 0) atomicOr(flags, kFlagTcLayout);
    return;
  }
  M128State st;
  m128_setup(st, sm128, bars_s, &tslot_s, &fail_s);
  const M128Layout L = m128_layout(dm.n_w);
  const int N = dm.N, nb = dm.nb, na = dm.na, n = dm.n_w;
  const long systems = (long)nch * na * N;
  const long s0 = systems * blockIdx.x / gridDim.x, s1 = systems * (blockIdx.x + 1) / gridDim.x;
  for (long s = s0; s < s1; ++s) {
    const long plane = s / N;
    const int c = ch0 + (int)(plane / na), a = dm.a0 + (int)(plane % na), key = c * nb + a;
    const size_t mat = (size_t)key * n * n;
    if (!m128_system(dm, c, a, (int)(s - plane * N), gg_hi + mat, gg_lo + mat,
                     gdig + (size_t)key * kM128DigBytes, chi, kc, flags, L, st, mc)) {
      m128_drain(st, L);
      if (threadIdx.x == 0) atomicOr(flags, kFlagTcTimeout);
      break;
    }
  }
  m128_teardown(st);
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

size_t gj_smem_bytes(int n_w) { return (size_t)gj_layout(n_w).total; }

// gamma's digits of the default kernel, after the mixed workspace's other parts
size_t digits128_bytes(const Dims& dm) {
  return m128_supported(dm.n_w) ? (size_t)2 * dm.nb * kM128DigBytes : 0;
}
static unsigned char* digits128_ptr(df_ctx* c) { return (unsigned char*)c->mixed_ws + c->dig128_off; }

// orders > 64: gamma's digits for the default kernel; for the shared-memory Gauss-Jordan kernel
// (mixed_sweep = 1) gamma^T's (hi, lo) words over those of gamma o gamma^T (workspace slots 2 and 3)
cudaError_t launch_gamma_large(df_ctx* c) {
  const Dims& dm = c->dm;
  if (c->opts.mixed_sweep == 0) {
    gamma_digits128_kernel<<<2 * dm.nb * 16, 256, 0, c->stream>>>(dm.n_w, 2 * dm.nb, c->gam, digits128_ptr(c));
    return cudaGetLastError();
  }
  const size_t count = (size_t)2 * dm.nb * dm.n_w * dm.n_w;
  float2* ws = (float2*)c->mixed_ws;
  split_gamma_t_kernel<<<256, 256, 0, c->stream>>>(dm.n_w, (size_t)2 * dm.nb, c->gam, ws + 2 * count, ws + 3 * count);
  return cudaGetLastError();
}

static cudaError_t launch_bse_mixed128(df_ctx* c, int channel_mask, int* flags) {
  const Dims& dm = c->dm;
  const size_t smem = (size_t)m128_layout(dm.n_w).total;
  cudaError_t e = cudaFuncSetAttribute((const void*)bse_mixed128_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  int sms = 0;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device)) != cudaSuccess) return e;
  const size_t count = (size_t)2 * dm.nb * dm.n_w * dm.n_w;
  const float2* hi = (const float2*)c->mixed_ws;
  const int nch = (channel_mask & 1) + ((channel_mask >> 1) & 1), ch0 = (channel_mask & 1) ? 0 : 1;
  const long systems = (long)nch * dm.na * dm.N;
  bse_mixed128_kernel<<<(int)(systems < sms ? systems : sms), kM128Threads, smem, c->stream>>>(
      dm, ch0, nch, hi + 2 * count, hi + 3 * count, c->chi, c->kc, digits128_ptr(c), flags,
      mixed_check(c));
  return cudaGetLastError();
}

cudaError_t launch_bse_mixed_large(df_ctx* c, int channel_mask, int* flags) {
  const Dims& dm = c->dm;
  const int n = dm.n_w;
  if (n > kGjMaxN) return cudaErrorInvalidValue;
  if (c->opts.mixed_sweep == 0) return launch_bse_mixed128(c, channel_mask, flags);
  const size_t smem = gj_smem_bytes(n);
  const int threads = gj_threads(n);
  cudaError_t e = cudaFuncSetAttribute((const void*)bse_gj_ir_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute((const void*)bse_gj_ir_kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                           (int)cudaSharedmemCarveoutMaxShared);
  if (e != cudaSuccess) return e;
  int sms = 0, per_sm = 0;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device)) != cudaSuccess) return e;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (const void*)bse_gj_ir_kernel, threads, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) per_sm = 1;
  const size_t count = (size_t)2 * dm.nb * n * n;
  const float2* ws = (const float2*)c->mixed_ws;
  const MixedCheck mc = mixed_check(c);
  for (int ch = 0; ch < 2; ++ch) {
    if (!(channel_mask & (1 << ch))) continue;
    const long systems = (long)dm.na * dm.N;
    const long grid = (long)sms * per_sm;
    bse_gj_ir_kernel<<<(int)(systems < grid ? systems : grid), threads, smem, c->stream>>>(
        dm, ch, 1, ws, ws + count, ws + 2 * count, ws + 3 * count, gamma_gt_ptr(c), c->chi, c->kc, flags, mc);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace df
