// Warp-level FFTs on double-float pairs, for the FP32-pair precision: the
// algorithm of fft.cuh (one warp per signal, N = 32 P points as P x 32, two
// transposes through the warp's scratch, natural order in and out) with every
// value a complex pair (df.cuh: dfc) and the twiddles of a pair table
// tw[m] = exp(-2 pi i m / L) as (re hi, re lo, im hi, im lo), read from shared
// memory where they are used.  About 2,600 FP32 instructions per lane-warp for
// 256 points, against 50,000 for the plain DFT sums that it replaced.
#pragma once

#include "df.cuh"
#include "fft.cuh"

namespace s2w {

__device__ __forceinline__ dfc dc_load(const float4& w) { return {{w.x, w.y}, {w.z, w.w}}; }
__device__ __forceinline__ float4 dc_pack(const dfc& a) { return make_float4(a.re.hi, a.re.lo, a.im.hi, a.im.lo); }

__device__ __forceinline__ dfc dc_shfl_xor(const dfc& a, int o) {
  return {{__shfl_xor_sync(0xffffffffu, a.re.hi, o), __shfl_xor_sync(0xffffffffu, a.re.lo, o)},
          {__shfl_xor_sync(0xffffffffu, a.im.hi, o), __shfl_xor_sync(0xffffffffu, a.im.lo, o)}};
}
__device__ __forceinline__ dfc dc_shfl(const dfc& a, int l) {
  return {{__shfl_sync(0xffffffffu, a.re.hi, l), __shfl_sync(0xffffffffu, a.re.lo, l)},
          {__shfl_sync(0xffffffffu, a.im.hi, l), __shfl_sync(0xffffffffu, a.im.lo, l)}};
}

// P-point DFT over registers (fft.cuh: reg_dft), table of length 64 PT.
template <int P, int PT = P>
__device__ __forceinline__ void reg_ddft(dfc (&v)[P], const float4* __restrict__ tw) {
  constexpr int L = 64 * PT;
#pragma unroll
  for (int h = P / 2; h >= 1; h >>= 1) {
#pragma unroll
    for (int b = 0; b < P; b += 2 * h) {
#pragma unroll
      for (int j = 0; j < h; ++j) {
        const dfc a = v[b + j], c = v[b + j + h];
        v[b + j] = dc_add(a, c);
        const dfc d = dc_sub(a, c);
        if (j == 0)
          v[b + j + h] = d;
        else if (2 * j == h)  // W = -i
          v[b + j + h] = {d.im, df_neg(d.re)};
        else
          v[b + j + h] = dc_mul(d, dc_load(tw[j * (L / (2 * h))]));
      }
    }
  }
  dfc y[P];
#pragma unroll
  for (int k = 0; k < P; ++k) y[k] = v[bitrev_p<P>(k)];
#pragma unroll
  for (int k = 0; k < P; ++k) v[k] = y[k];
}

// Forward complex DFT of N = 32 P pairs, natural order; scr: the warp's
// scratch of FftShape<P>::SCR entries.
template <int P>
__device__ __forceinline__ void warp_dfft(dfc (&v)[P], const float4* __restrict__ tw, int lane, float4* scr) {
  using SH = FftShape<P>;
  constexpr int N = SH::N, L = 2 * N, Q = SH::Q, RQ = SH::RQ;
  reg_ddft<P>(v, tw);
#pragma unroll
  for (int k = 1; k < P; ++k) v[k] = dc_mul(v[k], dc_load(tw[2 * ((lane * k) & (N - 1))]));
  constexpr int NSH = P == 1 ? 5 : ilog2c(Q / RQ);  // stages across lanes
  const int g = lane / Q, q = lane % Q;             // (P = 1: one group of 32)
  if (P > 1) {
    __syncwarp();
#pragma unroll
    for (int k = 0; k < P; ++k) scr[k * 32 + (lane ^ ((Q * k) & 31))] = dc_pack(v[k]);
    __syncwarp();
#pragma unroll
    for (int j = 0; j < P; ++j) v[j] = dc_load(scr[g * 32 + ((q + Q * j) ^ ((Q * g) & 31))]);
    reg_ddft<P>(v, tw);
#pragma unroll
    for (int a = 1; a < P; ++a) v[a] = dc_mul(v[a], dc_load(tw[((q * a) & 31) * (L / 32)]));
  }
#pragma unroll
  for (int st = 0; st < NSH; ++st) {
    const int h = (Q / 2) >> st;
    const bool upper = (q & h) != 0;
    const dfc w = dc_load(tw[(q & (h - 1)) * (L / (2 * h))]);
#pragma unroll
    for (int a = 0; a < P; ++a) {
      const dfc p = dc_shfl_xor(v[a], h);
      const dfc up = dc_mul(dc_sub(p, v[a]), w), low = dc_add(v[a], p);
      v[a] = upper ? up : low;
    }
  }
  if (P == 1) {
    v[0] = dc_shfl(v[0], rev5(lane));
    return;
  }
  const int ql = q % RQ;
  const int rq =
      (P > 1 && NSH > 0) ? static_cast<int>(__brev(static_cast<unsigned>(q / RQ)) >> (32 - (NSH > 0 ? NSH : 1))) : 0;
  __syncwarp();
#pragma unroll
  for (int a = 0; a < P; ++a) scr[ql * (SH::BLK + SH::SKEW) + g + P * a + P * P * rq] = dc_pack(v[a]);
  __syncwarp();
  constexpr int H = SH::BLK / 32;
#pragma unroll
  for (int h = 0; h < H; ++h) {
    dfc u[RQ];
#pragma unroll
    for (int j = 0; j < RQ; ++j) u[j] = dc_load(scr[j * (SH::BLK + SH::SKEW) + lane + 32 * h]);
    reg_ddft<RQ, P>(u, tw);
#pragma unroll
    for (int j = 0; j < RQ; ++j) v[h + H * j] = u[j];
  }
  __syncwarp();
}

// fft.cuh's warp_rfft and warp_irfft_head on pairs.
template <int P, class Put>
__device__ __forceinline__ void warp_drfft(dfc (&z)[P], Put put, const float4* __restrict__ tw, int lane,
                                           float4* scr) {
  constexpr int N = 32 * P;
  auto bin = [&](int k, const dfc& zk, const dfc& zc) {
    const dfc e = dc_scale(dc_add(zk, zc), 0.5f), d = dc_scale(dc_sub(zk, zc), 0.5f);
    const dfc o = {d.im, df_neg(d.re)};
    put(k, dc_add(e, dc_mul(dc_load(tw[k]), o)));
  };
  warp_dfft<P>(z, tw, lane, scr);
#pragma unroll
  for (int t = 0; t < P; ++t) scr[lane + 32 * t] = dc_pack(z[t]);
  __syncwarp();
#pragma unroll
  for (int t = 0; t < P; ++t) {
    const int k = lane + 32 * t;
    bin(k, z[t], dc_conj(dc_load(scr[(N - k) & (N - 1)])));
  }
  if (lane == 0) bin(N, z[0], dc_conj(z[0]));
  __syncwarp();
}

template <int P, class GetX>
__device__ __forceinline__ void warp_dirfft_head(GetX getx, dfc (&z)[P], const float4* __restrict__ tw, int lane,
                                                 float4* scr) {
  constexpr int N = 32 * P;
#pragma unroll
  for (int t = 0; t < P; ++t) {
    const int k = lane + 32 * t;
    const dfc xk = getx(k), xc = dc_conj(getx(N - k));
    const dfc e = dc_scale(dc_add(xk, xc), 0.5f);
    const dfc o = dc_mul(dc_scale(dc_sub(xk, xc), 0.5f), dc_conj(dc_load(tw[k])));
    // Z = E + i O, conjugated: (E.re - O.im, -(E.im + O.re))
    z[t] = {df_add_fast(e.re, df_neg(o.im)), df_neg(df_add_fast(e.im, o.re))};
  }
  warp_dfft<P>(z, tw, lane, scr);
  const float s = 1.0f / static_cast<float>(N);  // a power of two: exact
#pragma unroll
  for (int t = 0; t < P; ++t) z[t] = dc_scale(dc_conj(z[t]), s);
}

}  // namespace s2w
