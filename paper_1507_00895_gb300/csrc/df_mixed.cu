// Mixed-precision ladder solves (DF_FP32_IR) of one problem: the kernels around
// the per-ladder bodies of df_mixed64_dev.cuh (orders 33-64, two ladders of
// one (channel, W) at a time per block) and df_mixed32_dev.cuh (orders up to 32,
// one ladder per warp), gamma's words and digits, and the launchers.
#include "df_mixed32_dev.cuh"
#include "df_mixed64_dev.cuh"

namespace df {

// gamma and gamma o gamma^T (FP64) -> (hi, lo) FP32 pairs, same layouts
__global__ void split_gamma_kernel(size_t count, const double2* __restrict__ g, const double2* __restrict__ gg,
                                   float2* __restrict__ hi, float2* __restrict__ lo, float2* __restrict__ gg_hi,
                                   float2* __restrict__ gg_lo) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x) {
    const double2 v = g[i];
    float hx = (float)v.x, hy = (float)v.y;
    hi[i] = make_float2(hx, hy);
    lo[i] = make_float2((float)(v.x - (double)hx), (float)(v.y - (double)hy));
    const double2 w = gg[i];
    hx = (float)w.x; hy = (float)w.y;
    gg_hi[i] = make_float2(hx, hy);
    gg_lo[i] = make_float2((float)(w.x - (double)hx), (float)(w.y - (double)hy));
  }
}

// gamma's digits (once per input upload)
template <int NP>
__global__ void gamma_digits32_kernel(int n, int count, const double2* __restrict__ gam,
                                      unsigned char* __restrict__ out) {
  gamma_digits_frag<NP>(n, count, gam, out, (blockIdx.x * blockDim.x + threadIdx.x) >> 5,
                        (gridDim.x * blockDim.x) >> 5, threadIdx.x & 31);
}

__global__ void gamma_digits64_kernel(int n, int count, const double2* __restrict__ gam,
                                      unsigned char* __restrict__ out) {
  gamma_digits_cols(n, count, gam, out, (blockIdx.x * blockDim.x + threadIdx.x) >> 5, (gridDim.x * blockDim.x) >> 5,
                    threadIdx.x & 31);
}

// Orders up to 32: one contiguous range of systems per block, split where
// (channel, W) changes; the warps of a block take its systems in turn.
template <int NP>
__global__ void __launch_bounds__(M32<NP>::kThreads, 1)
bse_mixed32_kernel(Dims dm, int ch0, int nch, const float2* __restrict__ gg_hi, const float2* __restrict__ gg_lo,
                   const double2* __restrict__ chi, double2* __restrict__ kc, const unsigned char* __restrict__ gdig,
                   int* __restrict__ flags, MixedCheck mc) {
  using M = M32<NP>;
  extern __shared__ __align__(16) unsigned char sm32[];
  unsigned char* ws = sm32 + M::kBytes + (threadIdx.x >> 5) * M::kWarp;
  const int N = dm.N, nb = dm.nb, na = dm.na;
  const long systems = (long)nch * na * N;
  const long s1 = systems * (blockIdx.x + 1) / gridDim.x;
  long s = systems * blockIdx.x / gridDim.x;
  while (s < s1) {
    const long plane = s / N, end = min(s1, (plane + 1) * N);
    const int c = ch0 + (int)(plane / na), a = dm.a0 + (int)(plane % na), key = c * nb + a;
    m32_load_gamma<NP>(sm32, gdig + (size_t)key * M::kBytes);
    const size_t mat = (size_t)key * dm.n_w * dm.n_w;
    for (long x = s + (threadIdx.x >> 5); x < end; x += M::kWarps)
      m32_system<NP>(dm, c, a, (int)(x - plane * N), sm32, gg_hi + mat, gg_lo + mat, chi, kc, flags, ws, mc);
    s = end;
  }
}

// Orders 33-64: one contiguous range of systems per block, split where
// (channel, W) changes; the two groups of a block take its systems in turn.
__global__ void __launch_bounds__(kM64Threads, 1)
bse_mixed64_kernel(Dims dm, int ch0, int nch, const float2* __restrict__ gg_hi, const float2* __restrict__ gg_lo,
                   const double2* __restrict__ chi, double2* __restrict__ kc, const unsigned char* __restrict__ gdig,
                   int* __restrict__ flags, MixedCheck mc, unsigned spins) {
  extern __shared__ __align__(1024) unsigned char sm64[];
  __shared__ uint64_t mbar_s[2 * kM64Groups];
  __shared__ unsigned tslot_s;
  __shared__ int fail_s[kM64Groups];
  if (smem_u32(sm64) & 1023u) {                  // the swizzled operand tiles need 1024-byte alignment
    if (threadIdx.x == 0) atomicOr(flags, kFlagTcLayout);
    return;
  }
  M64Block blk;
  m64_setup(blk, sm64, mbar_s, &tslot_s, fail_s, spins);
  const int N = dm.N, nb = dm.nb, na = dm.na;
  const long systems = (long)nch * na * N;
  const long s1 = systems * (blockIdx.x + 1) / gridDim.x;
  long s = systems * blockIdx.x / gridDim.x;
  while (s < s1) {
    const long plane = s / N, end = min(s1, (plane + 1) * N);
    const int c = ch0 + (int)(plane / na), a = dm.a0 + (int)(plane % na), key = c * nb + a;
    const unsigned char* gd = gdig + (size_t)key * kM64DigBytes;
    if (!m64_load_digits(blk, gd)) break;
    const size_t mat = (size_t)key * dm.n_w * dm.n_w;
    bool ok = true;
    for (long x = s + blk.gr.g; x < end && ok; x += kM64Groups)
      ok = m64_system(dm, c, a, (int)(x - plane * N), reinterpret_cast<const float4*>(gd + kM64Shared), gg_hi + mat,
                 gg_lo + mat, chi, kc, flags, blk.gr, smem_u32(sm64), reinterpret_cast<const float*>(sm64 + kM64Gexp), mc);
    if (!ok && threadIdx.x % kM64Group == 0) atomicOr(flags, kFlagTcTimeout);
    s = end;
  }
  m64_teardown(blk);
}

// Self-test of the bounded wait the ladder kernels' tensor-core products use: one warp
// initialises an mbarrier (one arrival expected), arrives on it only when
// `arrive` is set, and waits for its first phase with a limit of `spins`
// polls; a wait that gives up sets kFlagTcTimeout.  Nothing else runs.
__global__ void wait_selftest_kernel(int arrive, unsigned spins, int* __restrict__ flags) {
  __shared__ uint64_t mbar;
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (arrive && threadIdx.x == 0) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&mbar)) : "memory");
  }
  if (!mbar_wait(&mbar, 0, spins) && threadIdx.x == 0) atomicOr(flags, kFlagTcTimeout);
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

cudaError_t launch_wait_selftest(int arrive, unsigned spins, int* flags, cudaStream_t stream) {
  wait_selftest_kernel<<<1, 32, 0, stream>>>(arrive, spins, flags);
  return cudaGetLastError();
}

static int mixed_np(int n) { return mixed_pad(n); }

bool mixed_supported(int n_w) { return mixed_np(n_w) <= 128; }

// gamma hi, lo (df_chi.cu and mixed_sweep = 1); gamma o gamma^T hi, lo (mixed_sweep = 1: gamma^T hi, lo); gamma's
// digits, weights and words (orders <= 64); then the error control's words: the call's
// largest rho^2 and the hand-back list (count + 2 N_W N system indices)
static size_t mixed_check_offset(const Dims& dm) {
  const int np = mixed_np(dm.n_w);
  const size_t digits = (size_t)2 * dm.nb * mixed_digit_bytes(np);
  return ((size_t)4 * 2 * dm.nb * dm.n_w * dm.n_w * sizeof(float2) + digits + 15) & ~(size_t)15;
}
size_t mixed_digits128_offset(const Dims& dm) {
  return (mixed_check_offset(dm) + sizeof(int) * (4 + (size_t)2 * dm.nb * dm.N) + 1023) & ~(size_t)1023;
}
size_t mixed_workspace_bytes(const Dims& dm) { return mixed_digits128_offset(dm) + digits128_bytes(dm); }
// [0] worst rho^2 (float bits), [1] unused, [2] hand-back count, [3 ..] list
unsigned* mixed_check_words(df_ctx* c) { return (unsigned*)((char*)c->mixed_ws + mixed_check_offset(c->dm)); }

MixedCheck mixed_check(df_ctx* c) {
  unsigned* w = mixed_check_words(c);
  MixedCheck mc;
  mc.worst = w;
  mc.redo = c->opts.ladder_fallback ? (int*)(w + 2) : nullptr;
  mc.rho2_max = (float)c->opts.ladder_tol;
  mc.base = 0;
  return mc;
}

static unsigned char* gdig_ptr(df_ctx* c) {
  const int np = mixed_np(c->dm.n_w);
  if (np > 64) return nullptr;
  return (unsigned char*)c->mixed_ws + (size_t)4 * 2 * c->dm.nb * c->dm.n_w * c->dm.n_w * sizeof(float2);
}

cudaError_t launch_split_gamma(df_ctx* c, const double2* gg) {
  const Dims& dm = c->dm;
  const size_t count = (size_t)2 * dm.nb * dm.n_w * dm.n_w;
  float2* hi = (float2*)c->mixed_ws;
  split_gamma_kernel<<<256, 256, 0, c->stream>>>(count, c->gam, gg, hi, hi + count, hi + 2 * count, hi + 3 * count);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (mixed_np(dm.n_w) > 64) return launch_gamma_large(c);
  if (unsigned char* gd = gdig_ptr(c)) {
    const int np = mixed_np(dm.n_w), rows = 2 * dm.nb * np;
    if (np == 64)
      gamma_digits64_kernel<<<(rows + 7) / 8, 256, 0, c->stream>>>(dm.n_w, 2 * dm.nb, c->gam, gd);
    else
      (np == 32 ? gamma_digits32_kernel<32> : gamma_digits32_kernel<16>)<<<(rows + 7) / 8, 256, 0, c->stream>>>(
          dm.n_w, 2 * dm.nb, c->gam, gd);
    e = cudaGetLastError();
  }
  return e;
}

// orders up to 32: one block per SM, one ladder per warp
template <int NP>
static cudaError_t launch_bse_mixed32(df_ctx* c, int channel_mask, int* flags) {
  using M = M32<NP>;
  const Dims& dm = c->dm;
  cudaError_t e = cudaFuncSetAttribute((const void*)bse_mixed32_kernel<NP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       M::kSmem);
  if (e != cudaSuccess) return e;
  int sms = 0;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device)) != cudaSuccess) return e;
  const size_t count = (size_t)2 * dm.nb * dm.n_w * dm.n_w;
  const float2* gg = (const float2*)c->mixed_ws + 2 * count;
  const int nch = (channel_mask & 1) + ((channel_mask >> 1) & 1), ch0 = (channel_mask & 1) ? 0 : 1;
  const long systems = (long)nch * dm.na * dm.N;
  bse_mixed32_kernel<NP><<<(int)(systems < sms ? systems : sms), M::kThreads, M::kSmem, c->stream>>>(
      dm, ch0, nch, gg, gg + count, c->chi, c->kc, gdig_ptr(c), flags, mixed_check(c));
  return cudaGetLastError();
}

// orders 33-64: one block of two ladder groups per SM
static cudaError_t launch_bse_mixed64(df_ctx* c, int channel_mask, int* flags) {
  const Dims& dm = c->dm;
  cudaError_t e = cudaFuncSetAttribute((const void*)bse_mixed64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kM64Smem);
  if (e != cudaSuccess) return e;
  int sms = 0;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device)) != cudaSuccess) return e;
  const size_t count = (size_t)2 * dm.nb * dm.n_w * dm.n_w;
  const float2* hi = (const float2*)c->mixed_ws;
  const MixedCheck mc = mixed_check(c);
  const int nch = (channel_mask & 1) + ((channel_mask >> 1) & 1), ch0 = (channel_mask & 1) ? 0 : 1;
  const long pairs = ((long)nch * dm.na * dm.N + kM64Groups - 1) / kM64Groups;
  bse_mixed64_kernel<<<(int)(pairs < sms ? pairs : sms), kM64Threads, kM64Smem, c->stream>>>(
      dm, ch0, nch, hi + 2 * count, hi + 3 * count, c->chi, c->kc, gdig_ptr(c), flags, mc,
      c->wait_spins);
  return cudaGetLastError();
}

// the mixed-precision ladder solves of one df_bse call, then the FP64 LU over
// the ladders whose predicted error exceeded the bound (none: its blocks exit
// at once).  The caller zeroes the check words before (run_ladders).
cudaError_t launch_bse_mixed(df_ctx* c, int channel_mask, int* flags) {
  cudaError_t e;
  switch (mixed_np(c->dm.n_w)) {
    case 16: e = launch_bse_mixed32<16>(c, channel_mask, flags); break;
    case 32: e = launch_bse_mixed32<32>(c, channel_mask, flags); break;
    case 64: e = launch_bse_mixed64(c, channel_mask, flags); break;
    case 128: e = launch_bse_mixed_large(c, channel_mask, flags); break;   // df_mixed_large.cu
    default: return cudaErrorInvalidValue;
  }
  if (e != cudaSuccess || !c->opts.ladder_fallback) return e;
  return launch_bse_f64_list(c, (const int*)(mixed_check_words(c) + 2));
}

}  // namespace df
