// Storage of the streamed operator rows: how a 16-byte chunk of a row unpacks
// into complex FP32 entries, for every storage type.
#pragma once

#include "s2w_internal.cuh"

namespace s2w {

template <int EL>
struct Chunk;  // complex entries per 16-byte chunk and how to unpack them

template <>
struct Chunk<EL_FP32> {
  static constexpr int C = 2;
  __device__ __forceinline__ static void unpack(const uint4& u, float2 (&g)[C]) {
    g[0] = make_float2(__uint_as_float(u.x), __uint_as_float(u.y));
    g[1] = make_float2(__uint_as_float(u.z), __uint_as_float(u.w));
  }
};

__device__ __forceinline__ float2 bf2_to_f2(unsigned w) {
  // bf16 -> f32 is exact: the 16 bits move to the top of the word
  return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}

template <>
struct Chunk<EL_BF16> {
  static constexpr int C = 4;
  __device__ __forceinline__ static void unpack(const uint4& u, float2 (&g)[C]) {
    g[0] = bf2_to_f2(u.x);
    g[1] = bf2_to_f2(u.y);
    g[2] = bf2_to_f2(u.z);
    g[3] = bf2_to_f2(u.w);
  }
};

// Two e4m3 values (bytes 0, 1 of a 16-bit word) widened exactly to an FP16
// pair, and a 32-bit word's two such pairs.
__device__ __forceinline__ __half2 e4m3x2_to_h2(unsigned short v) {
  unsigned r;
  asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(r) : "h"(v));
  return *reinterpret_cast<const __half2*>(&r);
}
__device__ __forceinline__ void e4m3x4_to_h2(unsigned w, __half2& lo, __half2& hi) {
  unsigned short l16, h16;
  asm("mov.b32 {%0, %1}, %2;" : "=h"(l16), "=h"(h16) : "r"(w));
  lo = e4m3x2_to_h2(l16);
  hi = e4m3x2_to_h2(h16);
}

__device__ __forceinline__ float2 fp8x2_to_f2(unsigned short s) {
  const __half2_raw h = __nv_cvt_fp8x2_to_halfraw2(static_cast<__nv_fp8x2_storage_t>(s), __NV_E4M3);
  return __half22float2(*reinterpret_cast<const __half2*>(&h));
}

template <>
struct Chunk<EL_FP8> {
  static constexpr int C = 8;
  __device__ __forceinline__ static void unpack(const uint4& u, float2 (&g)[C]) {
    const unsigned w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      g[2 * k] = fp8x2_to_f2(static_cast<unsigned short>(w[k] & 0xffffu));
      g[2 * k + 1] = fp8x2_to_f2(static_cast<unsigned short>(w[k] >> 16));
    }
  }
};

// Complex products on packed FP32 pairs: a stream of scalar FFMAs with three
// register operands reaches 25.3 TFMA/s on this GPU (register reads), packed
// ones 35.0 of 37.  y + g x in two instructions, from x prepared as (re, im)
// and (-im, re): g.re times the one, then g.im times the other (conj(g) x: the
// second (im, -re)).  The FMAs of g x in scalar form: cmac.
__device__ __forceinline__ float2 cmac2_re(float2 g, float4 x, float2 y) {
  return __ffma2_rn(make_float2(g.x, g.x), make_float2(x.x, x.y), y);
}
__device__ __forceinline__ float2 cmac2_im(float2 g, float4 x, float2 y) {
  return __ffma2_rn(make_float2(g.y, g.y), make_float2(x.z, x.w), y);
}
__device__ __forceinline__ void cmac(float2 g, float2 x, float& re, float& im) {
  re = fmaf(g.x, x.x, re);
  im = fmaf(g.x, x.y, im);
  re = fmaf(-g.y, x.y, re);
  im = fmaf(g.y, x.x, im);
}

}  // namespace s2w
