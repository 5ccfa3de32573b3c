// Transforms of the FP32_HILO (FP32 pair) storage precision: the same steps
// as k_fft.cu's kernels (Alg. 2 steps 1-2, the retransform between the
// stages with the D_t stencil of Sec. II-B.2, the split-K reduction with
// the final IFFT + Truncate), but with every spectrum and every sum carried
// as a double-float pair (df.cuh), so that the rounding of the transforms
// sits near 2^-48 of the signal instead of 2^-24.
//
// Why the pairs: an FFT evaluation rounds relative to the whole 2 Nt-sample
// window, spread evenly over all its samples; when most of a waveform's
// energy arrives after the kept Nt samples (a late arrival), the kept head
// is small against the window and its relative error grows by the ratio of
// the two.  Carrying every spectrum, sum and stored operator as hi + lo
// pairs takes that error down by 2^24.
//
// The transforms are FFTs on pairs (dfft.cuh), one warp per signal, eight
// signals per CTA pass through a shared tile so that the stores of a bin
// cover adjacent rows.  As plain DFT sums (one thread per output) the
// retransform of 6,000 points x 256 steps took 1.0 ms and the slip transform
// of 963 rows 0.092 ms; now 0.063 and 0.016.
#include "dfft.cuh"
#include "s2w_internal.cuh"

namespace s2w {

namespace {

constexpr int kDfThreads = 256;

// tw[m] = exp(-2 pi i m / L) as (re hi, re lo, im hi, im lo), evaluated in
// FP64 and split into FP32 pairs.
__global__ void k_twiddles_df(float4* tw, int L) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= L) return;
  double s, c;
  sincospi(2.0 * static_cast<double>(m) / static_cast<double>(L), &s, &c);
  const double im = -s;
  const float ch = static_cast<float>(c), ih = static_cast<float>(im);
  tw[m] = make_float4(ch, static_cast<float>(c - static_cast<double>(ch)), ih,
                      static_cast<float>(im - static_cast<double>(ih)));
}

__device__ __forceinline__ void load_tw(float4* tws, const float4* __restrict__ tw, int L) {
  for (int m = threadIdx.x; m < L; m += blockDim.x) tws[m] = tw[m];
}

constexpr int kWarps = kDfThreads / 32;
constexpr int kCols = 8;  // signals per CTA pass, one per warp

// Shared memory: twiddles, the tile (kCols or one signal), the warps' scratch.
template <int P>
size_t smem_df(int cols, int warps) {
  return sizeof(float4) * (64 * P + cols * (32 * P + 1) + warps * FftShape<P>::SCR);
}

// Bins 0..N of FP32 rows x[row][0..n_in) zero-padded to L = 2N (samples past
// lens[row / rows_a] read as zero), as pairs to X / X_lo[l * ld_l + (row /
// rows_a) * ld_a + row % rows_a].
template <int P>
__global__ void __launch_bounds__(kDfThreads) k_df_rfft_rows(const float* __restrict__ x, long long rows, int n_in,
                                                             const float4* __restrict__ tw, float2* X, float2* X_lo,
                                                             long long ld_l, long long rows_a, long long ld_a,
                                                             const int* __restrict__ lens) {
  grid_dependency();
  constexpr int N = 32 * P, NB = N + 1;
  extern __shared__ __align__(16) unsigned char smraw[];
  float4* tws = reinterpret_cast<float4*>(smraw);
  float4* tile = tws + 2 * N;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float4* scr = tile + kCols * NB + warp * FftShape<P>::SCR;
  load_tw(tws, tw, 2 * N);
  __syncthreads();
  for (long long r0 = static_cast<long long>(blockIdx.x) * kCols; r0 < rows;
       r0 += static_cast<long long>(gridDim.x) * kCols) {
    const long long row = r0 + warp;
    if (row < rows) {
      const int n_act = lens != nullptr ? min(n_in, max(0, __ldg(lens + row / rows_a))) : n_in;
      dfc z[P];
#pragma unroll
      for (int t = 0; t < P; ++t) {
        const int n = 2 * (lane + 32 * t);
        const float a = n < n_act ? __ldg(x + row * n_in + n) : 0.f;
        const float b = n + 1 < n_act ? __ldg(x + row * n_in + n + 1) : 0.f;
        z[t] = {{a, 0.f}, {b, 0.f}};
      }
      warp_drfft<P>(z, [&](int k, const dfc& v) { tile[warp * NB + k] = dc_pack(v); }, tws, lane, scr);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < kCols * NB; e += kDfThreads) {
      const int c = e % kCols, l = e / kCols;
      const long long r = r0 + c;
      if (r >= rows) continue;
      const float4 v = tile[c * NB + l];
      const long long d = l * ld_l + (r / rows_a) * ld_a + r % rows_a;
      X[d] = make_float2(v.x, v.z);
      X_lo[d] = make_float2(v.y, v.w);
    }
    __syncthreads();
  }
}

// Retransform of grid points i, rupture blockIdx.y, pairs in and out:
//   mhat[l][i] -> IFFT, keep n < N -> m -> v = D_t m (backward difference, or
//   v = m) -> zero-pad to 2N, FFT -> vhat[l][i];  m optionally to
// seafloor[i][n] (rounded to FP32).  inv_dt as a pair.
template <int P>
__global__ void __launch_bounds__(kDfThreads) k_df_retransform(const float2* __restrict__ mhat,
                                                               const float2* __restrict__ mhat_lo, long long Ng,
                                                               long long ld_m, const float4* __restrict__ tw,
                                                               float inv_dt_hi, float inv_dt_lo, int dt_mode,
                                                               float2* vhat, float2* vhat_lo, long long ld_v,
                                                               float* seafloor, long long mhat_ld_b,
                                                               long long vhat_ld_b) {
  grid_dependency();
  constexpr int N = 32 * P, NB = N + 1;
  mhat += blockIdx.y * mhat_ld_b;
  mhat_lo += blockIdx.y * mhat_ld_b;
  vhat += blockIdx.y * vhat_ld_b;
  vhat_lo += blockIdx.y * vhat_ld_b;
  if (seafloor != nullptr) seafloor += static_cast<long long>(blockIdx.y) * Ng * N;
  extern __shared__ __align__(16) unsigned char smraw[];
  float4* tws = reinterpret_cast<float4*>(smraw);
  float4* tile = tws + 2 * N;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float4* scr = tile + kCols * NB + warp * FftShape<P>::SCR;
  load_tw(tws, tw, 2 * N);
  const dfl inv_dt{inv_dt_hi, inv_dt_lo};
  for (long long i0 = static_cast<long long>(blockIdx.x) * kCols; i0 < Ng;
       i0 += static_cast<long long>(gridDim.x) * kCols) {
    for (int e = threadIdx.x; e < kCols * NB; e += kDfThreads) {
      const int c = e % kCols, l = e / kCols;
      const long long i = i0 + c;
      if (i >= Ng) continue;
      const float2 h = __ldg(mhat + l * ld_m + i), o = __ldg(mhat_lo + l * ld_m + i);
      tile[c * NB + l] = make_float4(h.x, o.x, h.y, o.y);
    }
    __syncthreads();
    const long long i = i0 + warp;
    if (i < Ng) {
      float4* Xs = tile + warp * NB;
      dfc z[P];
      warp_dirfft_head<P>([&](int k) { return dc_load(Xs[k]); }, z, tws, lane, scr);
      // (m[2n], m[2n + 1]), n = lane + 32 t < N / 2; the rest is padding
      constexpr int HT = (P + 1) / 2;
      const dfc zero = {{0.f, 0.f}, {0.f, 0.f}};
#pragma unroll
      for (int t = 0; t < P; ++t)
        if (t >= HT || (P == 1 && lane >= 16)) z[t] = zero;
      if (seafloor != nullptr) {
#pragma unroll
        for (int t = 0; t < HT; ++t) {
          const int n = 2 * (lane + 32 * t);
          if (n >= N) continue;
          seafloor[i * N + n] = z[t].re.hi + z[t].re.lo;
          seafloor[i * N + n + 1] = z[t].im.hi + z[t].im.lo;
        }
      }
      if (dt_mode != S2W_DT_NONE) {  // v[n] = (m[n] - m[n-1]) / dt, m[-1] = 0
        dfl prv[HT];
#pragma unroll
        for (int t = 0; t < HT; ++t)
          prv[t] = {__shfl_sync(0xffffffffu, z[t].im.hi, (lane + 31) & 31),
                    __shfl_sync(0xffffffffu, z[t].im.lo, (lane + 31) & 31)};
#pragma unroll
        for (int t = HT - 1; t >= 0; --t) {
          const dfl w = lane > 0 ? prv[t] : (t > 0 ? prv[t > 0 ? t - 1 : 0] : dfl{0.f, 0.f});
          z[t] = {df_mul(df_add(z[t].re, df_neg(w)), inv_dt), df_mul(df_add(z[t].im, df_neg(z[t].re)), inv_dt)};
        }
        if (P == 1 && lane >= 16) z[0] = zero;  // (the padding again: v[N] is not kept)
      }
      warp_drfft<P>(z, [&](int k, const dfc& v) { Xs[k] = dc_pack(v); }, tws, lane, scr);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < kCols * NB; e += kDfThreads) {
      const int c = e % kCols, l = e / kCols;
      if (i0 + c >= Ng) continue;
      const float4 v = tile[c * NB + l];
      vhat[l * ld_v + i0 + c] = make_float2(v.x, v.z);
      vhat_lo[l * ld_v + i0 + c] = make_float2(v.y, v.w);
    }
    __syncthreads();
  }
}

// One CTA per (rupture b, observation o): Qhat[l] = sum over the nseg
// segment partials in fixed order (pairs), then one warp forms q[b][o][n], n <
// n_keep, by the inverse FFT (rounded to FP32), rows n_keep apart.
template <int P>
__global__ void __launch_bounds__(kDfThreads) k_df_reduce_irfft(const float2* __restrict__ part,
                                                                const float2* __restrict__ part_lo, int No, int nseg,
                                                                long long s_b, long long s_l, long long s_s,
                                                                const float4* __restrict__ tw, float* q, int n_keep) {
  grid_dependency();
  constexpr int N = 32 * P;
  extern __shared__ __align__(16) unsigned char smraw[];
  float4* tws = reinterpret_cast<float4*>(smraw);
  float4* Xs = tws + 2 * N;
  float4* scr = Xs + N + 1;
  load_tw(tws, tw, 2 * N);
  const int b = blockIdx.x / No, o = blockIdx.x % No;
  const long long pb = b * s_b + o;
  for (int k = threadIdx.x; k <= N; k += blockDim.x) {
    dacc re{0.f, 0.f}, im{0.f, 0.f};
#pragma unroll 8
    for (int s = 0; s < nseg; ++s) {
      const long long e = pb + k * s_l + s * s_s;
      const float2 h = __ldg(part + e), lo = __ldg(part_lo + e);
      acc_add(re, dfl{h.x, lo.x});
      acc_add(im, dfl{h.y, lo.y});
    }
    Xs[k] = dc_pack({acc_get(re), acc_get(im)});
  }
  __syncthreads();
  if (threadIdx.x >= 32) return;
  float* out = q + static_cast<long long>(blockIdx.x) * n_keep;
  const int lane = threadIdx.x;
  dfc z[P];
  warp_dirfft_head<P>([&](int k) { return dc_load(Xs[k]); }, z, tws, lane, scr);
#pragma unroll
  for (int t = 0; t < (P + 1) / 2; ++t) {
    const int n = 2 * (lane + 32 * t);
    if (n >= N) continue;
    if (n < n_keep) out[n] = z[t].re.hi + z[t].re.lo;
    if (n + 1 < n_keep) out[n + 1] = z[t].im.hi + z[t].im.lo;
  }
}

unsigned df_grid(long long passes) {
  const long long most = 152LL * 3;
  return static_cast<unsigned>(passes < most ? passes : most);
}

template <class K>
cudaError_t allow_smem(K* kernel, size_t bytes) {
  if (bytes <= 48 * 1024) return cudaSuccess;  // allowed without asking
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
}

}  // namespace

cudaError_t launch_twiddles_df(float4* tw, int L, cudaStream_t st) {
  k_twiddles_df<<<(L + 255) / 256, 256, 0, st>>>(tw, L);
  return cudaGetLastError();
}

#define S2W_DISPATCH_P(Nt, ...)                               \
  switch (Nt) {                                               \
    case 32: { constexpr int P = 1; __VA_ARGS__; } break;     \
    case 64: { constexpr int P = 2; __VA_ARGS__; } break;     \
    case 128: { constexpr int P = 4; __VA_ARGS__; } break;    \
    case 256: { constexpr int P = 8; __VA_ARGS__; } break;    \
    case 512: { constexpr int P = 16; __VA_ARGS__; } break;   \
    default: return cudaErrorInvalidValue;                    \
  }

cudaError_t launch_df_rfft_rows(const float* x, long long rows, int n_in, int Nt, const float4* tw, float2* X,
                                float2* X_lo, long long ld_l, long long rows_a, long long ld_a, cudaStream_t st,
                                const int* lens) {
  if (rows <= 0) return cudaSuccess;
  if (n_in < 1 || n_in > Nt) return cudaErrorInvalidValue;
  S2W_DISPATCH_P(Nt, {
    const size_t sm = smem_df<P>(kCols, kWarps);
    const cudaError_t e = allow_smem(k_df_rfft_rows<P>, sm);
    if (e != cudaSuccess) return e;
    launch_next(k_df_rfft_rows<P>, df_grid((rows + kCols - 1) / kCols), kDfThreads, sm, st, x, rows, n_in, tw, X,
                X_lo, ld_l, rows_a, ld_a, lens);
  });
  return cudaGetLastError();
}

cudaError_t launch_df_retransform(const float2* mhat, const float2* mhat_lo, long long Ng, long long ld_m, int Nt,
                                  const float4* tw, double inv_dt, int dt_mode, float2* vhat, float2* vhat_lo,
                                  long long ld_v, float* seafloor, cudaStream_t st, int nb, long long mhat_ld_b,
                                  long long vhat_ld_b) {
  if (Ng <= 0 || nb <= 0) return cudaSuccess;
  if (dt_mode != S2W_DT_BACKWARD && dt_mode != S2W_DT_NONE) return cudaErrorInvalidValue;
  const float ih = static_cast<float>(inv_dt);
  const float il = static_cast<float>(inv_dt - static_cast<double>(ih));
  const dim3 grid(df_grid((Ng + kCols - 1) / kCols), static_cast<unsigned>(nb));
  S2W_DISPATCH_P(Nt, {
    const size_t sm = smem_df<P>(kCols, kWarps);
    const cudaError_t e = allow_smem(k_df_retransform<P>, sm);
    if (e != cudaSuccess) return e;
    launch_next(k_df_retransform<P>, grid, kDfThreads, sm, st, mhat, mhat_lo, Ng, ld_m, tw, ih, il, dt_mode, vhat,
                vhat_lo, ld_v, seafloor, mhat_ld_b, vhat_ld_b);
  });
  return cudaGetLastError();
}

cudaError_t launch_df_reduce_irfft(const float2* part, const float2* part_lo, int B, int No, int nseg, int Nt,
                                   long long s_b, long long s_l, long long s_s, const float4* tw, float* q,
                                   cudaStream_t st, int n_keep) {
  if (n_keep <= 0 || n_keep > Nt) n_keep = Nt;
  const long long n = static_cast<long long>(B) * No;
  if (n <= 0) return cudaSuccess;
  S2W_DISPATCH_P(Nt, {
    const size_t sm = smem_df<P>(1, 1);
    const cudaError_t e = allow_smem(k_df_reduce_irfft<P>, sm);
    if (e != cudaSuccess) return e;
    launch_next(k_df_reduce_irfft<P>, static_cast<unsigned>(n), kDfThreads, sm, st, part, part_lo, No, nseg, s_b,
                s_l, s_s, tw, q, n_keep);
  });
  return cudaGetLastError();
}

}  // namespace s2w
