// Per-bin complex contractions of the FP32-pair precision (FP32_HILO): rows and
// vectors as hi + lo FP32 arrays, y[f] = sum_c rows[f][c] x_vec(f)[c] in
// double-float sums (df.cuh), written as pairs (y, y_lo).
//
// The layout is k_stream_multi's (k_multi.cu): units of (vector group, tile of
// rows), K slabs of 512 bytes per row (hi and lo) and of the vector's hi and
// lo parts by TMA into a shared-memory ring, warp w on kRowsWarp rows of the
// tile, lane l on chunk l of each slab, the accumulators in registers over the
// whole row, one reduce-scatter of pairs over the lanes at the end.  Two
// ruptures at most share a pass.
//
// What bounds it: twelve FP32 operations per real product (TwoProduct with an
// FMA, the two cross terms, TwoSum, two additions into the error sum), 48 per
// 16-byte entry, 0.55 of the FMA pipe when the bytes arrive at the copy rate,
// so HBM, if the pipe is kept fed: real and imaginary part go through packed
// FP32 instructions together (26 per entry and lane pair of products), and
// sixteen warps cover their latency.  With the vector in registers (128 of
// them), eight warps and scalar operations the rows streamed at 0.40 of the
// copy rate: 963 x 6,000 x 64 x 256, stage 1 (24 GB) 8.9 ms, 3.45 here (1.01
// of the copy rate), the whole call 10.5 -> 3.8 ms.  16 x 1,024 x 4 x 32, two
// ruptures, whole call 57 -> 23 us (with the transforms of k_df.cu and
// chained launches).
#include <cuda.h>

#include <type_traits>

#include "chunk.cuh"
#include "df.cuh"

namespace s2w {

namespace {

constexpr int kWarps = 16;
constexpr int kThreads = 32 * (kWarps + 1);
constexpr int kSlabBytes = 512;  // most of each row (and part) per stage
constexpr int kMaxStages = 16;
constexpr int kBudget = 216 * 1024;
__host__ __device__ constexpr int rows_warp(int R) { return 4 / R; }

struct DfArgs {
  int n_vec, rows_per_vec, tiles, mrows;
  int slabs, stages, slab_bytes, nb;
  int x_vec_first;
  long long y_ldb;
  float2 *y, *y_lo;
  int* status;
  unsigned long long wait_ns;
  int fault_skip;
};

__device__ __forceinline__ void tma_words(void* sdst, const CUtensorMap* tm, int c0, int c1, int c2, uint64_t* bar,
                                          uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, "
      "%4}], [%5], %6;" ::"r"(smem_u32(sdst)),
      "l"(reinterpret_cast<uint64_t>(tm)), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar)), "l"(policy)
      : "memory");
}

// (s, c) += (g + gl) (x + xl) for two real products at once (x: two values):
// TwoProduct, the two cross terms and TwoSum of df.cuh on packed pairs; a - b
// is fma(b, -1, a).
__device__ __forceinline__ void pmac(float2& s, float2& c, float g, float gl, float2 x, float2 xl) {
  const float2 m1 = make_float2(-1.f, -1.f), g2 = make_float2(g, g);
  const float2 p = __fmul2_rn(g2, x);
  const float2 e = __ffma2_rn(g2, x, __fmul2_rn(make_float2(-g, -g), x));  // g x - p, exactly
  const float2 cross = __ffma2_rn(g2, xl, __ffma2_rn(make_float2(gl, gl), x, e));
  const float2 t = __fadd2_rn(s, p);
  const float2 bb = __ffma2_rn(s, m1, t);
  const float2 lo = __fadd2_rn(__ffma2_rn(__ffma2_rn(bb, m1, t), m1, s), __ffma2_rn(bb, m1, p));
  s = t;
  c = __fadd2_rn(c, __fadd2_rn(lo, cross));
}

// LPR lanes per row: 32, or 8 / 16 for rows of at most that many chunks (a
// warp then takes 32 / LPR times the rows); SHORT: rows shorter than a slab.
template <int R, bool SHORT, int LPR>
__global__ void __launch_bounds__(kThreads, 1)
    k_stream_df(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmAlo,
                const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmXlo, const DfArgs a) {
  grid_dependency();
  constexpr int RW = rows_warp(R);
  constexpr int G = 32 / LPR;  // row groups per warp
  const int slab_bytes = SHORT ? a.slab_bytes : kSlabBytes;
  const int pitch = slab_bytes / 16;
  extern __shared__ __align__(128) unsigned char sm[];
  const int S = a.stages;
  uint64_t* full = reinterpret_cast<uint64_t*>(sm);
  uint64_t* empty = full + kMaxStages;
  const int a_bytes = a.mrows * slab_bytes;
  const int x_bytes = (R * slab_bytes + 127) & ~127;
  const int stage_bytes = 2 * (a_bytes + x_bytes);
  unsigned char* ring = sm + 2 * 8 * kMaxStages;
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int sub = lane % LPR, grp = lane / LPR;
  const long long units = static_cast<long long>(a.n_vec) * a.tiles;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, kWarps);
    }
    fence_mbar_init();
  }
  __syncthreads();

  if (warp == kWarps) {
    if (lane != 0) return;
    const uint64_t first = l2_policy_evict_first();
    uint64_t last;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(last));
    int it = 0, s = 0;
    uint32_t ph = 1;
    bool ok = true;
    for (long long u = blockIdx.x; u < units && ok; u += gridDim.x) {
      const int vec = static_cast<int>(u / a.tiles), tile = static_cast<int>(u % a.tiles);
      const int xa = a.x_vec_first ? vec : 0, xb = a.x_vec_first ? 0 : vec;
      for (int k = 0; k < a.slabs; ++k, ++it) {
        if (it >= S && !mbar_wait_bounded(empty + s, ph, a.status, DEV_ERR_TIMEOUT_EMPTY, a.wait_ns)) {
          ok = false;
          break;
        }
        if (!(a.fault_skip && it == 0)) {  // (test hook: stage 0 never fills)
          unsigned char* st = ring + s * stage_bytes;
          const int c0 = k * (slab_bytes / 4);
          mbar_arrive_expect_tx(full + s, 2 * (a_bytes + R * slab_bytes));
          tma_words(st, &tmA, c0, tile * a.mrows, vec, full + s, first);
          tma_words(st + a_bytes, &tmAlo, c0, tile * a.mrows, vec, full + s, first);
          tma_words(st + 2 * a_bytes, &tmX, c0, xa, xb, full + s, last);
          tma_words(st + 2 * a_bytes + x_bytes, &tmXlo, c0, xa, xb, full + s, last);
        }
        if (++s == S) s = 0, ph ^= 1;
      }
    }
    // never leave the CTA with copies in flight
    for (int kk = (it > S ? it - S : 0); kk < it; ++kk)
      mbar_wait_bounded(full + kk % S, (kk / S) & 1, a.status, DEV_ERR_TIMEOUT_FULL, a.wait_ns);
    return;
  }

  int s = 0;
  uint32_t ph = 0;
  for (long long u = blockIdx.x; u < units; u += gridDim.x) {
    const int vec = static_cast<int>(u / a.tiles), tile = static_cast<int>(u % a.tiles);
    const int nr = min(a.mrows, a.rows_per_vec - tile * a.mrows);
    // a full tile gives each warp adjacent rows, a partial one deals its rows
    // out over the warps
    const bool whole = nr == kWarps * RW * G;
    const int r_i = whole ? 1 : kWarps * G, row0 = (warp * G + grp) * (whole ? RW : 1);
    float2 sum[RW * R], err[RW * R];  // (re, im) and their errors
#pragma unroll
    for (int k = 0; k < RW * R; ++k) sum[k] = err[k] = make_float2(0.f, 0.f);
    for (int k = 0; k < a.slabs; ++k) {
      if (!mbar_wait_bounded(full + s, ph, a.status, DEV_ERR_TIMEOUT_FULL, a.wait_ns)) return;
      const unsigned char* st = ring + s * stage_bytes;
      const float4* rows = reinterpret_cast<const float4*>(st) + sub;
      const float4* rows_lo = reinterpret_cast<const float4*>(st + a_bytes) + sub;
      const float4* xs = reinterpret_cast<const float4*>(st + 2 * a_bytes) + sub;
      const float4* xs_lo = reinterpret_cast<const float4*>(st + 2 * a_bytes + x_bytes) + sub;
      if (!SHORT || sub < pitch) {
        float4 x[R], xl[R];
#pragma unroll
        for (int b = 0; b < R; ++b) {
          x[b] = xs[b * pitch];
          xl[b] = xs_lo[b * pitch];
        }
#pragma unroll
        for (int i = 0; i < RW; ++i) {
          const int row = row0 + i * r_i;
          if (row >= nr) continue;
          const float4 g = rows[row * pitch], gl = rows_lo[row * pitch];
#pragma unroll
          for (int b = 0; b < R; ++b) {
            float2& sv = sum[i * R + b];
            float2& ev = err[i * R + b];
            pmac(sv, ev, g.x, gl.x, make_float2(x[b].x, x[b].y), make_float2(xl[b].x, xl[b].y));
            pmac(sv, ev, g.y, gl.y, make_float2(-x[b].y, x[b].x), make_float2(-xl[b].y, xl[b].x));
            pmac(sv, ev, g.z, gl.z, make_float2(x[b].z, x[b].w), make_float2(xl[b].z, xl[b].w));
            pmac(sv, ev, g.w, gl.w, make_float2(-x[b].w, x[b].z), make_float2(-xl[b].w, xl[b].z));
          }
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(empty + s);
      if (++s == S) s = 0, ph ^= 1;
    }
    // eight pairs ((row, rupture), component) over the row's lanes: three
    // steps that halve them, then plain ones; every LPR / 8 lanes hold one
    dacc v[8];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[2 * k] = {sum[k].x, err[k].x};
      v[2 * k + 1] = {sum[k].y, err[k].y};
    }
#pragma unroll
    for (int o = LPR / 2, n = 4; o > 0; o >>= 1, n >>= 1) {
      const bool up = n > 0 && (lane & o) != 0;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (k >= (n > 0 ? n : 1)) continue;
        const dacc keep = up ? v[k + n] : v[k];
        const dacc send = up || n == 0 ? v[k] : v[k + n];
        v[k] = acc_merge(keep, {__shfl_xor_sync(0xffffffffu, send.s, o), __shfl_xor_sync(0xffffffffu, send.c, o)});
      }
    }
    const int idx = sub / (LPR / 8), b = (idx >> 1) % R;
    const int row = row0 + (idx >> 1) / R * r_i;
    if (sub % (LPR / 8) == 0 && row < nr && b < a.nb) {
      const dfl r = acc_get(v[0]);
      const long long f = static_cast<long long>(vec) * a.rows_per_vec + tile * a.mrows + row + b * a.y_ldb;
      reinterpret_cast<float*>(a.y + f)[idx & 1] = r.hi;
      reinterpret_cast<float*>(a.y_lo + f)[idx & 1] = r.lo;
    }
  }
}

template <int R, bool SHORT, int LPR>
cudaError_t launch_r(const StreamArgs& a, int num_sms, cudaStream_t st) {
  const long long row_bytes = 8LL * a.row_len, vec_bytes = row_bytes * a.rows_per_vec;
  DfArgs m{};
  m.slab_bytes = SHORT ? static_cast<int>(row_bytes) : kSlabBytes;
  m.rows_per_vec = static_cast<int>(a.rows_per_vec);
  m.n_vec = static_cast<int>(a.F / a.rows_per_vec);
  constexpr int tile_rows = kWarps * rows_warp(R) * (32 / LPR);
  m.mrows = a.rows_per_vec >= tile_rows ? tile_rows : static_cast<int>((a.rows_per_vec + 7) / 8 * 8);
  m.tiles = (m.rows_per_vec + m.mrows - 1) / m.mrows;
  m.slabs = static_cast<int>((row_bytes + m.slab_bytes - 1) / m.slab_bytes);
  const int stage = 2 * (m.mrows * m.slab_bytes + ((R * m.slab_bytes + 127) & ~127));
  m.stages = kBudget / stage < kMaxStages ? kBudget / stage : kMaxStages;
  m.nb = a.nb;
  m.y = a.y;
  m.y_lo = a.y_lo;
  m.y_ldb = a.y_ldb;
  m.status = a.status;
  m.wait_ns = a.wait_ns ? a.wait_ns : kWaitLimitNs;
  m.fault_skip = a.fault_skip;
  // the vector map's dimensions go up in pitch; ruptures past nb read as
  // zeros (TMA fill), their sums are never stored
  m.x_vec_first = a.nb == 1 || a.x_stride < a.x_ldb ? 1 : 0;
  const long long b_pitch = a.nb == 1 ? 8 * a.x_stride * m.n_vec : 8 * a.x_ldb;
  auto rows_map = [&](CUtensorMap* tm, const void* base) {
    return tc_encode_words(tm, base, row_bytes / 4, a.rows_per_vec, row_bytes, m.n_vec, vec_bytes, m.slab_bytes / 4,
                           m.mrows);
  };
  auto vec_map = [&](CUtensorMap* tm, const float2* base) {
    return m.x_vec_first ? tc_encode_words(tm, base, row_bytes / 4, m.n_vec, 8 * a.x_stride, a.nb, b_pitch,
                                           m.slab_bytes / 4, 1, R)
                         : tc_encode_words(tm, base, row_bytes / 4, a.nb, 8 * a.x_ldb, m.n_vec, 8 * a.x_stride,
                                           m.slab_bytes / 4, R);
  };
  CUtensorMap ta, tl, tx, txl;
  cudaError_t e;
  if ((e = rows_map(&ta, a.rows)) != cudaSuccess || (e = rows_map(&tl, a.rows_lo)) != cudaSuccess ||
      (e = vec_map(&tx, a.x)) != cudaSuccess || (e = vec_map(&txl, a.x_lo)) != cudaSuccess)
    return e;
  const size_t smem = 2 * 8 * kMaxStages + static_cast<size_t>(m.stages) * stage;
  if ((e = cudaFuncSetAttribute(k_stream_df<R, SHORT, LPR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                static_cast<int>(smem))) != cudaSuccess)
    return e;
  long long grid = static_cast<long long>(m.n_vec) * m.tiles;
  if (grid > num_sms) grid = num_sms;
  launch_next(k_stream_df<R, SHORT, LPR>, static_cast<unsigned>(grid), kThreads, smem, st, ta, tl, tx, txl, m);
  return cudaGetLastError();
}

}  // namespace

namespace {
template <int R>
cudaError_t launch_nb(const StreamArgs& a, int num_sms, cudaStream_t st) {
  const int chunks = a.row_len / 2;
  if (chunks <= 8) return launch_r<R, true, 8>(a, num_sms, st);
  if (chunks <= 16) return launch_r<R, true, 16>(a, num_sms, st);
  if (chunks < 32) return launch_r<R, true, 32>(a, num_sms, st);
  return launch_r<R, false, 32>(a, num_sms, st);
}
}  // namespace

cudaError_t launch_stream_df(const StreamArgs& a, int num_sms, cudaStream_t st) {
  if (a.rows_lo == nullptr || a.x_lo == nullptr || a.y_lo == nullptr || a.rows_per_vec < 1 ||
      a.rows_per_vec > 0x7fffff00 || a.F % a.rows_per_vec != 0)
    return cudaErrorInvalidValue;
  for (int b = 0; b < a.nb; b += 2) {
    StreamArgs h = a;
    h.nb = a.nb - b < 2 ? 1 : 2;
    h.x = a.x + b * a.x_ldb;
    h.x_lo = a.x_lo + b * a.x_ldb;
    h.y = a.y + b * a.y_ldb;
    h.y_lo = a.y_lo + b * a.y_ldb;
    const cudaError_t e = h.nb == 1 ? launch_nb<1>(h, num_sms, st) : launch_nb<2>(h, num_sms, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace s2w
