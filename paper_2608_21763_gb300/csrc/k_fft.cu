// Transform kernels of the pipeline (everything except the per-bin
// contractions): twiddle table, batched zero-padded real FFT (Alg. 2, steps
// 1-2), the stage-1 -> stage-2 retransform (Alg. 2 steps 4-5 for F_G, the
// D_t stencil of Sec. II-B.2, then steps 1-2 for F_q), the split-K reduction
// of stage-2 partials fused with the final IFFT + Truncate, and the load-time
// conversion of FP32 spectra into the resident storage types.
#include "fft.cuh"

namespace s2w {

namespace {

constexpr int kWarps = 8;
constexpr int kThreads = 32 * kWarps;
// CTAs per SM of the transform kernels (registers: 80 a thread, 128 at 512
// points, where they spill: k_rfft_rows 48 bytes, k_irfft_rows 264,
// k_retransform 148, k_rfft_tile up to 32; at 256 points k_retransform 8)
__host__ __device__ constexpr int fft_ctas(int P) { return P >= 16 ? 2 : 3; }
__host__ __device__ constexpr int tile_ctas(int P) { return P >= 8 ? 2 : 3; }  // (shared memory)
__host__ __device__ constexpr int irfft_ctas(int P) { return P >= 8 ? 2 : 3; }  // (a row of bins in flight)
constexpr int kSms = 152;

// tw[m] = exp(-2 pi i m / L), m < L, evaluated in FP64 and stored as FP32.
__global__ void k_twiddles(float2* tw, int L) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= L) return;
  double s, c;
  sincospi(2.0 * static_cast<double>(m) / static_cast<double>(L), &s, &c);
  tw[m] = make_float2(static_cast<float>(c), static_cast<float>(-s));
}

template <int P>
__device__ __forceinline__ void load_twiddles(float2* tw, const float2* __restrict__ twg) {
  for (int m = threadIdx.x; m < 64 * P; m += blockDim.x) tw[m] = twg[m];
}

// Samples 2n, 2n + 1 (n = lane + 32 t) of a real row of n_in, n_act of them
// live; `pair`: the row is 8-byte aligned.
template <int P>
__device__ __forceinline__ void load_pairs(const float* __restrict__ xr, int n_act, bool pair, int lane,
                                           float2 (&z)[P]) {
#pragma unroll
  for (int t = 0; t < P; ++t) {
    const int n = 2 * (lane + 32 * t);
    z[t] = make_float2(0.f, 0.f);
    if (t < (P + 1) / 2) {  // the upper half is zero padding (n_act <= 32 P)
      if (pair && n + 1 < n_act)
        z[t] = __ldg(reinterpret_cast<const float2*>(xr + n));
      else {
        if (n < n_act) z[t].x = __ldg(xr + n);
        if (n + 1 < n_act) z[t].y = __ldg(xr + n + 1);
      }
    }
  }
}

// One warp per row at a time: x[row][0..n_in) zero-padded to L = 2N, bins
// 0..N to X[row * (N + 1) + l].  Persistent warps: the twiddles are read once
// per CTA, and a row's samples are loaded while the row before is
// transformed.  With k_irfft_rows, 246,528 rows of 256 each way (1.5 GB, 0.22
// ms at the copy rate): 0.31 ms; 0.55 with a CTA and a twiddle table per eight
// rows and no row in flight.
template <int P>
__global__ void __launch_bounds__(kThreads, fft_ctas(P)) k_rfft_rows(const float* __restrict__ x, long long rows,
                                                                  int n_in, const float2* __restrict__ twg,
                                                                  float2* __restrict__ X) {
  grid_dependency();
  constexpr int N = 32 * P;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* tw = reinterpret_cast<float2*>(smraw);
  float2* scr = tw + 2 * N + (threadIdx.x >> 5) * FftShape<P>::SCR;
  load_twiddles<P>(tw, twg);
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const FftLane<P> fl = fft_lane<P>(tw, lane);
  const bool pair = (reinterpret_cast<uintptr_t>(x) & 7) == 0 && n_in % 2 == 0;
  const long long step = static_cast<long long>(gridDim.x) * kWarps;
  long long row = static_cast<long long>(blockIdx.x) * kWarps + (threadIdx.x >> 5);
  float2 z[P];
  if (row < rows) load_pairs<P>(x + row * n_in, n_in, pair, lane, z);
  for (; row < rows; row += step) {
    float2 next[P];  // (512 points: the registers are full, the row is loaded after)
    if (P < 16 && row + step < rows) load_pairs<P>(x + (row + step) * n_in, n_in, pair, lane, next);
    float2* out = X + row * (N + 1);
    warp_rfft<P>(z, [&](int k, float2 v) { out[k] = v; }, tw, fl, lane, scr);
    if (P == 16 && row + step < rows) load_pairs<P>(x + (row + step) * n_in, n_in, pair, lane, next);
#pragma unroll
    for (int t = 0; t < P; ++t) z[t] = next[t];
  }
}

// The same with the bins transposed, for the contractions: tile_rows rows per
// CTA pass through a shared tile, so that each bin's stores cover adjacent
// rows (with a warp per row storing one 8-byte entry per bin, 963 x 256 rows
// of 256 samples took 0.58 ms, 0.24 now; with the packing 0.87 -> 0.25).  Bin
// l of row `row`, with a = row / rows_a and c = row % rows_a, goes to X[l *
// ld_l + a * ld_a + c]; or, PACK, into the B operand of the real embedding
// (k_tc.cu: k_pack_b; conj: the conjugate one), rows 2a, 2a + 1 of hi / lo[l *
// ld_l + 2 a * ld_a + c], BF16 pairs.
// Many rows: 32 per tile (128-byte stores of BF16 pairs; 96,300 rows of hi/lo
// pairs 0.24 -> 0.16 ms against 16), 16 at 512 points (shared memory).  Up to
// kFewRows rows: 8 per tile, one per warp, to spread over the SMs.
__host__ __device__ constexpr int tile_rows(int P) { return P >= 16 ? 16 : 32; }
constexpr int kFewRows = 32 * kSms;
template <int P, bool PACK, int kTileRows>
__global__ void __launch_bounds__(kThreads, tile_ctas(P))
    k_rfft_tile(const float* __restrict__ x, long long rows, int n_in, const float2* __restrict__ twg,
                float2* __restrict__ X, long long ld_l, long long rows_a, long long ld_a,
                const int* __restrict__ lens, int conj, __nv_bfloat162* __restrict__ hi,
                __nv_bfloat162* __restrict__ lo) {
  grid_dependency();
  constexpr int N = 32 * P;
  constexpr int NB = N + 1;  // odd: a bin's column of the tile lies on distinct banks
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* tw = reinterpret_cast<float2*>(smraw);
  float2* tile = tw + 2 * N;  // [kTileRows][NB]
  float2* scr = tile + kTileRows * NB + (threadIdx.x >> 5) * FftShape<P>::SCR;
  load_twiddles<P>(tw, twg);
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const FftLane<P> fl = fft_lane<P>(tw, lane);
  const bool pair = (reinterpret_cast<uintptr_t>(x) & 7) == 0 && n_in % 2 == 0;
  const long long step = static_cast<long long>(gridDim.x) * kTileRows;
  float2 next[P];  // the warp's next row, loaded while one is transformed or stored
  auto load = [&](long long row) {
    if (row >= rows) return;
    // lens: active samples per group of rows_a rows (later samples read as 0)
    const int n_act = lens != nullptr ? min(n_in, max(0, __ldg(lens + row / rows_a))) : n_in;
    load_pairs<P>(x + row * n_in, n_act, pair, lane, next);
  };
  load(static_cast<long long>(blockIdx.x) * kTileRows + warp);
  for (long long r0 = static_cast<long long>(blockIdx.x) * kTileRows; r0 < rows; r0 += step) {
    const int nr = static_cast<int>(min(static_cast<long long>(kTileRows), rows - r0));
#pragma unroll 1
    for (int c = warp; c < kTileRows; c += kWarps) {
      float2 z[P];
#pragma unroll
      for (int t = 0; t < P; ++t) z[t] = next[t];
      load(c + kWarps < kTileRows ? r0 + c + kWarps : r0 + step + warp);
      if (c >= nr) continue;
      float2* out = tile + c * NB;
      warp_rfft<P>(z, [&](int k, float2 v) { out[k] = v; }, tw, fl, lane, scr);
    }
    __syncthreads();
    const int c = threadIdx.x % kTileRows;
    if (c < nr) {
      const long long row = r0 + c, a = row / rows_a;
      const float2* col = tile + c * NB;
      if constexpr (PACK) {
        const long long o = 2 * a * ld_a + row % rows_a;
        for (int l = threadIdx.x / kTileRows; l < NB; l += kThreads / kTileRows) {
          const float2 v = col[l];
          const float2 e0 = conj ? make_float2(v.x, v.y) : make_float2(v.x, -v.y);
          const float2 e1 = conj ? make_float2(v.y, -v.x) : make_float2(v.y, v.x);
          const __nv_bfloat162 h0 = __floats2bfloat162_rn(e0.x, e0.y), h1 = __floats2bfloat162_rn(e1.x, e1.y);
          const long long d = l * ld_l + o;
          hi[d] = h0;
          hi[d + ld_a] = h1;
          if (lo != nullptr) {
            lo[d] = __floats2bfloat162_rn(e0.x - __low2float(h0), e0.y - __high2float(h0));
            lo[d + ld_a] = __floats2bfloat162_rn(e1.x - __low2float(h1), e1.y - __high2float(h1));
          }
        }
      } else {
        float2* o = X + a * ld_a + row % rows_a;
        for (int l = threadIdx.x / kTileRows; l < NB; l += kThreads / kTileRows) o[l * ld_l] = col[l];
      }
    }
    __syncthreads();
  }
}

// One warp per row at a time (persistent): bins X[row][0..N] -> first N
// samples x[row][0..N).  Each bin is read once (the mirrored ones through
// the warp's scratch) and the samples leave in pairs, in order.
template <int P>
__global__ void __launch_bounds__(kThreads, irfft_ctas(P)) k_irfft_rows(const float2* __restrict__ X, long long rows,
                                                                   const float2* __restrict__ twg,
                                                                   float* __restrict__ x) {
  grid_dependency();
  constexpr int N = 32 * P;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* tw = reinterpret_cast<float2*>(smraw);
  float2* scr = tw + 2 * N + (threadIdx.x >> 5) * FftShape<P>::SCR;
  load_twiddles<P>(tw, twg);
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const FftLane<P> fl = fft_lane<P>(tw, lane);
  const bool pair = (reinterpret_cast<uintptr_t>(x) & 7) == 0;
  const long long step = static_cast<long long>(gridDim.x) * kWarps;
  long long row = static_cast<long long>(blockIdx.x) * kWarps + (threadIdx.x >> 5);
  float2 in[P], in_n;
  auto load = [&](long long r) {
    const float2* xr = X + r * (N + 1);
#pragma unroll
    for (int t = 0; t < P; ++t) in[t] = __ldg(xr + lane + 32 * t);
    in_n = __ldg(xr + N);
  };
  if (row < rows) load(row);
  for (; row < rows; row += step) {
#pragma unroll
    for (int t = 0; t < P; ++t) scr[lane + 32 * t] = in[t];
    if (lane == 0) scr[N] = in_n;
    __syncwarp();
    float2 z[P];
    // (every bin leaves the scratch before the transform writes to it)
    if (P < 16 && row + step < rows) load(row + step);
    warp_irfft_head<P>([&](int k) { return scr[k]; }, z, tw, fl, lane, scr);
    if (P == 16 && row + step < rows) load(row + step);
    __syncwarp();
    float* out = x + row * N;
#pragma unroll
    for (int t = 0; t < (P + 1) / 2; ++t) {
      const int n = 2 * (lane + 32 * t);
      if (n >= N) continue;
      if (pair)
        *reinterpret_cast<float2*>(out + n) = z[t];
      else
        out[n] = z[t].x, out[n + 1] = z[t].y;
    }
  }
}

// Retransform of kRtCols consecutive grid points per CTA pass, rupture
// blockIdx.y:
//   mhat[l][i] (bins 0..N)  -> IFFT, keep n < N (Truncate)  -> m
//   v = D_t m  (backward difference; or v = m when dt_mode is NONE)
//   v zero-padded to 2N -> FFT -> vhat[l][i]  (FP32, or BF16 pairs when BF16OUT).
// Optionally writes m to seafloor[i][0..N).  The samples stay in registers
// between the two transforms; a neighbour's sample comes by shuffle.  Bound by
// latency between its load, transform and store phases (three CTAs per SM
// overlap them); 37,758 points x 8 ruptures x 256 steps: 0.60 -> 0.47 ms, 0.18
// at the copy rate.
constexpr int kRtCols = 16;
template <int P, bool BF16OUT>
__global__ void __launch_bounds__(kThreads, fft_ctas(P))
    k_retransform(const float2* __restrict__ mhat, long long Ng, long long ld_m, const float2* __restrict__ twg,
                  float inv_dt, int dt_mode, void* __restrict__ vout, long long ld_v, float* __restrict__ seafloor,
                  long long mhat_ld_b, long long vhat_ld_b, __nv_bfloat162* __restrict__ vout_lo, int n_alloc) {
  grid_dependency();
  constexpr int N = 32 * P;
  constexpr int NB = N + 1;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* tw = reinterpret_cast<float2*>(smraw);
  float2* tile = tw + 2 * N;  // [kRtCols][NB]
  float2* scr = tile + kRtCols * NB + (threadIdx.x >> 5) * FftShape<P>::SCR;
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  mhat += blockIdx.y * mhat_ld_b;
  if (seafloor != nullptr) seafloor += static_cast<long long>(blockIdx.y) * Ng * N;
  const bool pair = (reinterpret_cast<uintptr_t>(seafloor) & 7) == 0;
  load_twiddles<P>(tw, twg);
  __syncthreads();
  const FftLane<P> fl = fft_lane<P>(tw, lane);
  for (long long i0 = static_cast<long long>(blockIdx.x) * kRtCols; i0 < Ng;
       i0 += static_cast<long long>(gridDim.x) * kRtCols) {
    // 16 independent loads in flight per thread (a half-warp reads 128
    // contiguous bytes of one bin per load)
    constexpr int kU = 16;
    for (int e0 = threadIdx.x; e0 < NB * kRtCols; e0 += kThreads * kU) {
      float2 v[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int e = e0 + u * kThreads;
        const int l = e / kRtCols, c = e % kRtCols;
        const long long i = i0 + c;
        v[u] = (e < NB * kRtCols && i < Ng) ? __ldg(mhat + l * ld_m + i) : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int e = e0 + u * kThreads;
        if (e < NB * kRtCols) tile[(e % kRtCols) * NB + e / kRtCols] = v[u];
      }
    }
    __syncthreads();
    for (int c = warp; c < kRtCols; c += kWarps) {
      const long long i = i0 + c;
      if (i >= Ng) break;
      float2* X = tile + c * NB;
      float2 z[P];
      warp_irfft_head<P>([&](int k) { return X[k]; }, z, tw, fl, lane, scr);
      // z[t] = (m[2n], m[2n + 1]), n = lane + 32 t < N / 2; the rest is padding
      constexpr int HT = (P + 1) / 2;
#pragma unroll
      for (int t = 0; t < P; ++t)
        if (t >= HT || (P == 1 && lane >= 16)) z[t] = make_float2(0.f, 0.f);
      if (seafloor != nullptr) {
#pragma unroll
        for (int t = 0; t < HT; ++t) {
          const int n = 2 * (lane + 32 * t);
          float* out = seafloor + i * N + n;
          if (n >= N) continue;
          if (pair)
            *reinterpret_cast<float2*>(out) = z[t];
          else
            out[0] = z[t].x, out[1] = z[t].y;
        }
      }
      if (dt_mode == kDtTranspose) {  // D_t^T: u[n] = (w[n] - w[n+1]) / dt, w[N] = 0
        float nxt[HT];
#pragma unroll
        for (int t = 0; t < HT; ++t) nxt[t] = __shfl_sync(0xffffffffu, z[t].x, (lane + 1) & 31);
#pragma unroll
        for (int t = 0; t < HT; ++t) {
          const float w = lane < 31 ? nxt[t] : (t + 1 < HT ? nxt[t + 1 < HT ? t + 1 : t] : 0.f);
          z[t] = make_float2((z[t].x - z[t].y) * inv_dt, (z[t].y - w) * inv_dt);
        }
      } else if (dt_mode != S2W_DT_NONE) {  // backward difference, m[-1] = 0
        float prv[HT];
#pragma unroll
        for (int t = 0; t < HT; ++t) prv[t] = __shfl_sync(0xffffffffu, z[t].y, (lane + 31) & 31);
#pragma unroll
        for (int t = HT - 1; t >= 0; --t) {
          const float w = lane > 0 ? prv[t] : (t > 0 ? prv[t > 0 ? t - 1 : 0] : 0.f);
          z[t] = make_float2((z[t].x - w) * inv_dt, (z[t].y - z[t].x) * inv_dt);
        }
      }
      if (P == 1 && lane >= 16) z[0] = make_float2(0.f, 0.f);  // (the padding again: v[N] is not kept)
      warp_rfft<P>(z, [&](int k, float2 v) { X[k] = v; }, tw, fl, lane, scr);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < NB * kRtCols; e += kThreads) {
      const int l = e / kRtCols, c = e % kRtCols;
      const long long i = i0 + c;
      if (i >= Ng) continue;
      const float2 v = tile[c * NB + l];
      if (BF16OUT && n_alloc > 0) {
        // B operand of the conjugate embedding (tensor-engine adjoint): rows
        // 2b = (Re v, Im v) and 2b+1 = (Im v, -Re v) of [l][n_alloc][ld_v]
        const long long o0 = (static_cast<long long>(l) * n_alloc + 2 * blockIdx.y) * ld_v + i;
        const float2 r[2] = {make_float2(v.x, v.y), make_float2(v.y, -v.x)};
#pragma unroll
        for (int h2 = 0; h2 < 2; ++h2) {
          const __nv_bfloat162 h = __floats2bfloat162_rn(r[h2].x, r[h2].y);
          static_cast<__nv_bfloat162*>(vout)[o0 + h2 * ld_v] = h;
          if (vout_lo != nullptr)
            vout_lo[o0 + h2 * ld_v] = __floats2bfloat162_rn(r[h2].x - __low2float(h), r[h2].y - __high2float(h));
        }
      } else if (BF16OUT) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(v.x, v.y);
        (static_cast<__nv_bfloat162*>(vout) + blockIdx.y * vhat_ld_b)[l * ld_v + i] = h;
        if (vout_lo != nullptr)  // low-order part: v - hi, rounded again
          (vout_lo + blockIdx.y * vhat_ld_b)[l * ld_v + i] =
              __floats2bfloat162_rn(v.x - __low2float(h), v.y - __high2float(h));
      } else
        (static_cast<float2*>(vout) + blockIdx.y * vhat_ld_b)[l * ld_v + i] = v;
    }
    __syncthreads();
  }
}

// Split-K reduction + output transform of OT adjacent observations (or
// subfaults) per CTA:
//   Qhat[l] = sum_{s < nseg} part[b*s_b + l*s_l + s*s_s + o]   (fixed order:
// deterministic), all bins in parallel over the CTA's threads, then a warp per
// output forms q[b][o][n] = IFFT(Qhat)[n], n < N.  OT = 8 reads 64 bytes per
// bin and segment and keeps every warp busy in the transform; OT = 1 spreads
// few outputs over the GPU (launch_reduce_irfft).
template <int P, int OT>
__global__ void __launch_bounds__(kThreads) k_reduce_irfft(const float2* __restrict__ part, int No, int nseg,
                                                           long long s_b, long long s_l, long long s_s,
                                                           const float2* __restrict__ twg, float* __restrict__ q,
                                                           int n_keep) {
  grid_dependency();
  constexpr int N = 32 * P;
  constexpr int NB = N + 1;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* tw = reinterpret_cast<float2*>(smraw);
  float2* xs = tw + 2 * N;      // [OT][NB]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float2* scr = xs + OT * NB + (OT > 1 ? warp * FftShape<P>::SCR : 0);
  load_twiddles<P>(tw, twg);
  const int groups = (No + OT - 1) / OT;
  const int b = blockIdx.x / groups, o0 = blockIdx.x % groups * OT;
  const float2* pb = part + b * s_b + o0;
  for (int e = threadIdx.x; e < OT * NB; e += kThreads) {
    const int k = e / OT, c = e % OT;
    if (OT > 1 && o0 + c >= No) continue;
    const float2* pk = pb + static_cast<long long>(k) * s_l + c;
    float2 acc = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int s = 0; s < nseg; ++s) acc = cadd(acc, pk[static_cast<long long>(s) * s_s]);
    xs[c * NB + k] = acc;
  }
  __syncthreads();
  if (warp >= OT || o0 + warp >= No) return;
  const float2* xw = xs + warp * NB;
  float* out = q + (static_cast<long long>(b) * No + o0 + warp) * n_keep;
  const FftLane<P> fl = fft_lane<P>(tw, lane);
  float2 z[P];
  warp_irfft_head<P>([&](int k) { return xw[k]; }, z, tw, fl, lane, scr);
#pragma unroll
  for (int t = 0; t < (P + 1) / 2; ++t) {
    const int n = 2 * (lane + 32 * t);
    if (n >= N) continue;
    if (n < n_keep) out[n] = z[t].x;
    if (n + 1 < n_keep) out[n + 1] = z[t].y;
  }
}

// part[l][s][e] (l < Nb, s < nseg, e < per): part[l][0][e] becomes the sum
// over s in increasing order (the order k_reduce_irfft adds them in), read
// coalesced along e, so that the reduction reads one segment.
__global__ void k_sum_chunks(float2* __restrict__ part, int Nb, int nseg, long long per) {
  grid_dependency();
  const long long total = static_cast<long long>(Nb) * per;
  for (long long e = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; e < total;
       e += static_cast<long long>(gridDim.x) * blockDim.x) {
    float2* p = part + (e / per) * nseg * per + e % per;
    float2 acc = make_float2(0.f, 0.f);
    for (int s = 0; s < nseg; ++s) acc = cadd(acc, p[static_cast<long long>(s) * per]);
    p[0] = acc;
  }
}

// X[l][r] *= (1 - W_L^l) / dt for l <= L/2, r < per_bin: the spectrum of the
// backward difference, folded into the stage-2 spectra of the single-pass
// variant (no retransform between the stages; L = 4 Nt leaves no wrap).
__global__ void k_scale_dt(float2* __restrict__ X, int Nb, long long per_bin, const float2* __restrict__ twg,
                           float inv_dt) {
  const long long total = static_cast<long long>(Nb) * per_bin;
  for (long long e = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; e < total;
       e += static_cast<long long>(gridDim.x) * blockDim.x) {
    const int l = static_cast<int>(e / per_bin);
    const float2 w = twg[l];
    const float2 d = make_float2((1.f - w.x) * inv_dt, -w.y * inv_dt);
    X[e] = cmul(X[e], d);
  }
}

// FP32 spectra -> resident storage (FP32 / BF16 / BF16 hi+lo), block copy:
// dst[l * ld_dst_l + dst_off + r] = convert(src[l * n_per_l + r]).
__global__ void k_store_blocks(const float2* __restrict__ src, int Nb, long long n_per_l, int el, void* dst,
                               void* dst_lo, long long ld_dst_l, long long dst_off) {
  const long long total = static_cast<long long>(Nb) * n_per_l;
  for (long long e = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; e < total;
       e += static_cast<long long>(gridDim.x) * blockDim.x) {
    const long long l = e / n_per_l, r = e % n_per_l;
    const float2 v = src[e];
    const long long d = l * ld_dst_l + dst_off + r;
    if (el == EL_FP32) {
      static_cast<float2*>(dst)[d] = v;
    } else {
      const __nv_bfloat162 hi = __floats2bfloat162_rn(v.x, v.y);
      static_cast<__nv_bfloat162*>(dst)[d] = hi;
      if (el == EL_BF16_HILO) {
        const float2 h = __bfloat1622float2(hi);
        static_cast<__nv_bfloat162*>(dst_lo)[d] = __floats2bfloat162_rn(v.x - h.x, v.y - h.y);
      }
    }
  }
}

// Stage-2 spectra, staging [l][o][nc] -> resident [l][seg][o][RL] at grid
// column i = c0 + c (seg = i / RL).
__global__ void k_store_adjoint(const float2* __restrict__ src, int Nb, int No, long long nc, long long c0, int RL,
                                int nseg, int el, void* dst) {
  const long long total = static_cast<long long>(Nb) * No * nc;
  for (long long e = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; e < total;
       e += static_cast<long long>(gridDim.x) * blockDim.x) {
    const long long l = e / (No * nc);
    const long long rem = e % (No * nc);
    const long long o = rem / nc, c = rem % nc;
    const long long i = c0 + c;
    const long long d = ((l * nseg + i / RL) * No + o) * RL + (i % RL);
    const float2 v = src[e];
    if (el == EL_FP32)
      static_cast<float2*>(dst)[d] = v;
    else
      static_cast<__nv_bfloat162*>(dst)[d] = __floats2bfloat162_rn(v.x, v.y);
  }
}

// FP8 scales: one CTA per (bin l, 256-row block) of the staging chunk
// [l][rows][Ns_pad]; amax over |Re|, |Im| of the block, then, in FP64,
// scale = amax / 448 (448 = largest finite e4m3).
__global__ void k_fp8_scales(const float2* __restrict__ spec, long long rows, int Ns_pad, long long row0, float* scale,
                             int nblk) {
  const int l = blockIdx.y;
  const long long rb = static_cast<long long>(blockIdx.x) * 256;
  const long long re = min(rows, rb + 256);
  const float2* base = spec + (static_cast<long long>(l) * rows + rb) * Ns_pad;
  const long long n = (re - rb) * Ns_pad;
  float m = 0.f;
  for (long long e = threadIdx.x; e < n; e += blockDim.x) {
    const float2 v = base[e];
    m = fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y)));
  }
  __shared__ float red[32];
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    float mm = 0.f;
    for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) mm = fmaxf(mm, red[w]);
    const double s = static_cast<double>(mm) / 448.0;
    scale[static_cast<long long>(l) * nblk + (row0 + rb) / 256] = static_cast<float>(s);
  }
}

// FP8 quantisation with round-to-nearest-even and saturation:
// dst[l][row0 + r][j] = e4m3(spec[l][r][j] / scale[l][(row0 + r) / 256]).
__global__ void k_fp8_quantize(const float2* __restrict__ spec, int Nb, long long rows, int Ns_pad, long long row0,
                               long long Ng, const float* __restrict__ scale, int nblk,
                               __nv_fp8x2_storage_t* __restrict__ dst) {
  const long long per_l = rows * Ns_pad;
  const long long total = static_cast<long long>(Nb) * per_l;
  for (long long e = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; e < total;
       e += static_cast<long long>(gridDim.x) * blockDim.x) {
    const long long l = e / per_l, rem = e % per_l;
    const long long r = rem / Ns_pad;
    const float sc = scale[l * nblk + (row0 + r) / 256];
    const float inv = sc > 0.f ? static_cast<float>(1.0 / static_cast<double>(sc)) : 0.f;
    const float2 v = spec[e];
    dst[l * Ng * Ns_pad + row0 * Ns_pad + rem] =
        __nv_cvt_float2_to_fp8x2(make_float2(v.x * inv, v.y * inv), __NV_SATFINITE, __NV_E4M3);
  }
}

// Residual and misfit: r = q - d in place of q, loss[b] = 0.5 sum r^2 over the
// rupture's No x Nt samples (one CTA per rupture, fixed summation order).
__global__ void __launch_bounds__(kThreads) k_residual(float* __restrict__ q, const float* __restrict__ d,
                                                       long long n_per_b, float* __restrict__ loss) {
  grid_dependency();
  const long long base = static_cast<long long>(blockIdx.x) * n_per_b;
  float acc = 0.f;
  for (long long e = threadIdx.x; e < n_per_b; e += kThreads) {
    const float r = q[base + e] - d[base + e];
    q[base + e] = r;
    acc = fmaf(r, r, acc);
  }
  __shared__ float red[kWarps];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0 && loss != nullptr) {
    float t = 0.f;
    for (int w = 0; w < kWarps; ++w) t += red[w];
    loss[blockIdx.x] = 0.5f * t;
  }
}

int grid_for(long long n, int threads) {
  long long g = (n + threads - 1) / threads;
  if (g > 152LL * 32) g = 152LL * 32;
  if (g < 1) g = 1;
  return static_cast<int>(g);
}

// Shared memory of the transform kernels: twiddles, a tile of `cols` signals'
// bins, the warps' scratch.
template <int P>
size_t smem_fft(int cols, int warps = kWarps) {
  return sizeof(float2) * (64 * P + cols * (32 * P + 1) + warps * FftShape<P>::SCR);
}

// CTAs for n passes of persistent transform kernels.
template <int P>
unsigned fft_grid(long long n, int ctas = fft_ctas(P)) {
  const long long most = static_cast<long long>(kSms) * ctas;
  return static_cast<unsigned>(n < most ? n : most);
}

template <class K>
cudaError_t allow_smem(K* kernel, size_t bytes) {
  if (bytes <= 48 * 1024) return cudaSuccess;  // allowed without asking
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
}

template <int P, bool PACK, int TR>
cudaError_t run_rfft_tile(const float* x, long long rows, int n_in, const float2* tw, float2* X, long long ld_l,
                          long long rows_a, long long ld_a, const int* lens, int conj, __nv_bfloat162* hi,
                          __nv_bfloat162* lo, cudaStream_t st) {
  const size_t sm = smem_fft<P>(TR);
  const cudaError_t e = allow_smem(k_rfft_tile<P, PACK, TR>, sm);
  if (e != cudaSuccess) return e;
  launch_next(k_rfft_tile<P, PACK, TR>, fft_grid<P>((rows + TR - 1) / TR, tile_ctas(P)), kThreads, sm, st, x, rows,
              n_in, tw, X, ld_l, rows_a, ld_a, lens, conj, hi, lo);
  return cudaGetLastError();
}

}  // namespace

#define S2W_DISPATCH_P(Nt, ...)                               \
  switch (Nt) {                                               \
    case 32: { constexpr int P = 1; __VA_ARGS__; } break;     \
    case 64: { constexpr int P = 2; __VA_ARGS__; } break;     \
    case 128: { constexpr int P = 4; __VA_ARGS__; } break;    \
    case 256: { constexpr int P = 8; __VA_ARGS__; } break;    \
    case 512: { constexpr int P = 16; __VA_ARGS__; } break;   \
    default: return cudaErrorInvalidValue;                    \
  }

cudaError_t launch_residual(float* q, const float* d, int B, long long n_per_b, float* loss, cudaStream_t st) {
  if (B <= 0) return cudaSuccess;
  launch_next(k_residual, B, kThreads, 0, st, q, d, n_per_b, loss);
  return cudaGetLastError();
}

cudaError_t launch_twiddles(float2* tw, int L, cudaStream_t st) {
  k_twiddles<<<(L + 255) / 256, 256, 0, st>>>(tw, L);
  return cudaGetLastError();
}

cudaError_t launch_rfft_rows(const float* x, long long rows, int n_in, int Nt, const float2* tw, float2* X,
                             long long ld_l, long long rows_a, long long ld_a, cudaStream_t st, const int* lens) {
  if (rows <= 0) return cudaSuccess;
  S2W_DISPATCH_P(Nt, {
    cudaError_t e;
    if (ld_l == 1 && rows_a == 1 && ld_a == Nt + 1 && lens == nullptr) {
      const size_t sm = smem_fft<P>(0);
      if ((e = allow_smem(k_rfft_rows<P>, sm)) != cudaSuccess) return e;
      launch_next(k_rfft_rows<P>, fft_grid<P>((rows + kWarps - 1) / kWarps), kThreads, sm, st, x, rows, n_in, tw,
                  X);
    } else if (rows <= kFewRows) {
      e = run_rfft_tile<P, false, 8>(x, rows, n_in, tw, X, ld_l, rows_a, ld_a, lens, 0, nullptr, nullptr, st);
    } else {
      e = run_rfft_tile<P, false, tile_rows(P)>(x, rows, n_in, tw, X, ld_l, rows_a, ld_a, lens, 0, nullptr, nullptr,
                                                st);
    }
    if (e != cudaSuccess) return e;
  });
  return cudaGetLastError();
}

cudaError_t launch_rfft_pack(const float* x, long long rows, int Nt, const float2* tw, long long rows_a,
                             long long Kc, int N_alloc, int conj, void* hi, void* lo, cudaStream_t st,
                             const int* lens) {
  if (rows <= 0) return cudaSuccess;
  __nv_bfloat162* h = static_cast<__nv_bfloat162*>(hi);
  __nv_bfloat162* o = static_cast<__nv_bfloat162*>(lo);
  S2W_DISPATCH_P(Nt, {
    const cudaError_t e =
        rows <= kFewRows
            ? run_rfft_tile<P, true, 8>(x, rows, Nt, tw, nullptr, N_alloc * Kc, rows_a, Kc, lens, conj, h, o, st)
            : run_rfft_tile<P, true, tile_rows(P)>(x, rows, Nt, tw, nullptr, N_alloc * Kc, rows_a, Kc, lens, conj, h,
                                                   o, st);
    if (e != cudaSuccess) return e;
  });
  return cudaGetLastError();
}

cudaError_t launch_irfft_rows(const float2* X, long long rows, int Nt, const float2* tw, float* x, cudaStream_t st) {
  if (rows <= 0) return cudaSuccess;
  S2W_DISPATCH_P(Nt, {
    const size_t sm = smem_fft<P>(0);
    const cudaError_t e = allow_smem(k_irfft_rows<P>, sm);
    if (e != cudaSuccess) return e;
    launch_next(k_irfft_rows<P>, fft_grid<P>((rows + kWarps - 1) / kWarps, irfft_ctas(P)), kThreads, sm, st, X,
                rows, tw, x);
  });
  return cudaGetLastError();
}

cudaError_t launch_retransform(const float2* mhat, long long Ng, long long ld_m, int Nt, const float2* tw,
                               float inv_dt, int dt_mode, float2* vhat, long long ld_v, float* seafloor,
                               cudaStream_t st, int nb, long long mhat_ld_b, long long vhat_ld_b,
                               __nv_bfloat162* vhat_bf, __nv_bfloat162* vhat_bf_lo, int n_alloc) {
  if (Ng <= 0 || nb <= 0) return cudaSuccess;
  S2W_DISPATCH_P(Nt, {
    const dim3 grid(fft_grid<P>((Ng + kRtCols - 1) / kRtCols), static_cast<unsigned>(nb));
    const size_t sm = smem_fft<P>(kRtCols);
    cudaError_t e;
    if (vhat_bf != nullptr) {
      if ((e = allow_smem(k_retransform<P, true>, sm)) != cudaSuccess) return e;
      launch_next(k_retransform<P, true>, grid, kThreads, sm, st, mhat, Ng, ld_m, tw, inv_dt, dt_mode, vhat_bf,
                  ld_v, seafloor, mhat_ld_b, vhat_ld_b, vhat_bf_lo, n_alloc);
    } else {
      if ((e = allow_smem(k_retransform<P, false>, sm)) != cudaSuccess) return e;
      launch_next(k_retransform<P, false>, grid, kThreads, sm, st, mhat, Ng, ld_m, tw, inv_dt, dt_mode, vhat, ld_v,
                  seafloor, mhat_ld_b, vhat_ld_b, nullptr, 0);
    }
  });
  return cudaGetLastError();
}

cudaError_t launch_reduce_irfft(const float2* part, int B, int No, int nseg, int Nt, long long s_b, long long s_l,
                                long long s_s, const float2* tw, float* q, cudaStream_t st, int n_keep) {
  if (n_keep <= 0 || n_keep > Nt) n_keep = Nt;
  const long long n = static_cast<long long>(B) * No;
  if (n <= 0) return cudaSuccess;
  // eight outputs per CTA once that leaves four CTAs per SM
  const bool many = n >= 8LL * 4 * kSms && No >= 8;
  S2W_DISPATCH_P(Nt, {
    cudaError_t e;
    if (many) {
      const size_t sm = smem_fft<P>(8);
      if ((e = allow_smem(k_reduce_irfft<P, 8>, sm)) != cudaSuccess) return e;
      const long long grid = static_cast<long long>(B) * ((No + 7) / 8);
      launch_next(k_reduce_irfft<P, 8>, static_cast<unsigned>(grid), kThreads, sm, st, part, No, nseg, s_b, s_l,
                  s_s, tw, q, n_keep);
    } else {
      const size_t sm = smem_fft<P>(1, 1);
      launch_next(k_reduce_irfft<P, 1>, static_cast<unsigned>(n), kThreads, sm, st, part, No, nseg, s_b, s_l, s_s,
                  tw, q, n_keep);
    }
  });
  return cudaGetLastError();
}

cudaError_t launch_sum_chunks(float2* part, int Nb, int nseg, long long per, cudaStream_t st) {
  launch_next(k_sum_chunks, grid_for(Nb * per, 256), 256, 0, st, part, Nb, nseg, per);
  return cudaGetLastError();
}

cudaError_t launch_scale_dt(float2* X, int Nb, long long per_bin, const float2* tw, float inv_dt, cudaStream_t st) {
  k_scale_dt<<<grid_for(Nb * per_bin, 256), 256, 0, st>>>(X, Nb, per_bin, tw, inv_dt);
  return cudaGetLastError();
}

cudaError_t launch_store_blocks(const float2* src, int Nb, long long n_per_l, int el, void* dst, void* dst_lo,
                                long long ld_dst_l, long long dst_off, cudaStream_t st) {
  k_store_blocks<<<grid_for(Nb * n_per_l, 256), 256, 0, st>>>(src, Nb, n_per_l, el, dst, dst_lo, ld_dst_l, dst_off);
  return cudaGetLastError();
}

cudaError_t launch_store_adjoint(const float2* src, int Nb, int No, long long nc, long long c0, int RL, int nseg,
                                 int el, void* dst, cudaStream_t st) {
  k_store_adjoint<<<grid_for(static_cast<long long>(Nb) * No * nc, 256), 256, 0, st>>>(src, Nb, No, nc, c0, RL, nseg,
                                                                                        el, dst);
  return cudaGetLastError();
}

cudaError_t launch_fp8_store(const float2* spec, int Nb, long long rows, int Ns_pad, long long row0, long long Ng,
                             float* scale, int nblk, void* dst, cudaStream_t st) {
  dim3 g(static_cast<unsigned>((rows + 255) / 256), static_cast<unsigned>(Nb));
  k_fp8_scales<<<g, 256, 0, st>>>(spec, rows, Ns_pad, row0, scale, nblk);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_fp8_quantize<<<grid_for(Nb * rows * Ns_pad, 256), 256, 0, st>>>(spec, Nb, rows, Ns_pad, row0, Ng, scale, nblk,
                                                                     static_cast<__nv_fp8x2_storage_t*>(dst));
  return cudaGetLastError();
}

}  // namespace s2w
