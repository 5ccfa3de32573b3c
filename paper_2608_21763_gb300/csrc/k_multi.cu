// Per-bin complex contractions for a handful of ruptures (2 .. 8) on
// CUDA cores: y_b[f] = sum_c rows[f][c] x_b[c] for all of them while the row
// is in shared memory, so that the batch reads the operator from HBM once
// (k_stream.cu reads it once per rupture).
//
// A unit is (vector group, tile of up to 64 rows); persistent CTAs take units
// round robin.  One elected lane streams K slabs through a shared-memory ring
// by TMA: the tile's rows (512 bytes of each, 32 chunks of 16) and the same
// columns of the R vectors, which come from L2 after their first use.  Warp w
// owns eight of the rows, lane l chunk l of each slab, and the FP32
// accumulators of all 8 x R products stay in registers over the whole row, or
// half of a long one; then one butterfly reduce-scatter over the lanes sums
// them.
//
// What bounds it: 4 FMAs per stored entry and rupture.  At eight ruptures an
// FP32 entry costs 32 FMAs for 8 bytes; scalar FFMAs with three register
// operands run at 25 TFMA/s here, so the FMAs take as long as the bytes at
// the copy rate at about six ruptures.  Rows are cut into K slabs (not whole
// rows per warp) because eight warps with eight whole rows each would need
// 0.5 MB of shared memory, and eight rows per warp because each vector entry
// read from shared memory must serve several rows.  Packed FP32 products (35
// TFMA/s) on (re, im) pairs were slower here: they want the vectors twice
// (rotated), in registers or in shared-memory reads, at two warps per
// scheduler (also twelve warps with four or six rows each).
//
// Each lane sums its chunks l, l + 32, ... in column order into one
// accumulator per component, then the lanes are added over xor 16, 8, 4, 2, 1;
// a row of more than two slabs goes in two blocks (chain_slabs), each reduced
// by itself, then added: k_stream_dot's order, so a rupture's result is the
// same bits alone or in a batch.  The two blocks round like two accumulators
// per component, for which there are no registers (128 hold one each).  They
// cost eight ruptures a second reduction, about 500 instructions per 64 rows
// and lane; dealing each lane its rows in an order that the reduction wants
// takes the selections out of it.  Stage 1 of 963 x 8,000 x 64 x 256: one
// rupture 2.25 ms, two 2.28, four 2.39, six 2.34, eight 2.78 (2.61 in one
// block; 18.0 eight times over).  Whole calls, operators read once per
// rupture, then one block, then as it is: 480 x 37,758 x 32 x 256, eight
// ruptures, 46.0 -> 7.94 -> 8.65 ms; 333 x 4,999 x 17 x 512 with seafloor
// output, five, 6.66 -> 1.37 -> 1.52 ms.  Other ways to the same rounding, at
// the first of these: two accumulators with four rows per warp 10.4 ms, the
// first block's sums kept in tensor memory 8.7 - 9.4.
#include <cuda.h>

#include <type_traits>

#include "chunk.cuh"

namespace s2w {

namespace {

constexpr int kWarps = 8;
// Two warpgroups of consumers and one whose first lane produces.  The launch
// gives every thread 168 registers; the producer group hands most of its
// share to the consumers, whose accumulators and operands need ~200
// (2 x 128 x 232 + 128 x 40 = 384 x 168).
constexpr int kThreads = 32 * (kWarps + 4);
constexpr int kRegsConsumer = 232, kRegsProducer = 40;
constexpr int RW = 8;                 // rows per warp, of a full tile
constexpr int kSlabBytes = 512;       // most of each row per stage: one 16-byte chunk per lane
constexpr int kMaxStages = 16;
constexpr int kBudget = 208 * 1024;   // ring bytes

struct MultiArgs {
  int n_vec, rows_per_vec, tiles, mrows;  // tiles of mrows rows per vector group
  int slabs, stages;
  int block;        // slabs of the first block (chain_slabs), all of them in rows that are not cut
  int slab_bytes;   // of each row per stage: kSlabBytes, or the whole of a shorter row
  int nb;
  int x_vec_first;  // the vector map's dimensions are (entry, vector, rupture), else (entry, rupture, vector)
  long long y_ldb;
  float2* y;
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

__device__ __forceinline__ uint64_t l2_policy_evict_last() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}

// SHORT: rows shorter than a slab (the stage holds whole rows).
template <int EL, bool HILO, int R, bool SHORT>
__global__ void __launch_bounds__(kThreads, 1)
    k_stream_multi(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmAlo,
                   const __grid_constant__ CUtensorMap tmX, const MultiArgs a) {
  grid_dependency();
  using CH = Chunk<EL>;
  constexpr int C = CH::C;
  const int slab_bytes = SHORT ? a.slab_bytes : kSlabBytes;
  const int pitch = slab_bytes / 16;                  // 16-byte chunks of a row in a stage
  const int x_bytes = slab_bytes * (C / 2);           // of a vector in a stage
  extern __shared__ __align__(128) unsigned char sm[];
  const int S = a.stages;
  uint64_t* full = reinterpret_cast<uint64_t*>(sm);
  uint64_t* empty = full + kMaxStages;
  const int a_bytes = a.mrows * slab_bytes;
  const int fill_bytes = a_bytes * (HILO ? 2 : 1) + R * x_bytes;  // what TMA brings per stage
  const int stage_bytes = (fill_bytes + 127) & ~127;
  unsigned char* ring = sm + 2 * 8 * kMaxStages;
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const long long units = static_cast<long long>(a.n_vec) * a.tiles;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, kWarps);
    }
    fence_mbar_init();
  }
  __syncthreads();

  if (warp >= kWarps) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsProducer));
    if (warp == kWarps && lane == 0) {
      const uint64_t first = l2_policy_evict_first(), last = l2_policy_evict_last();
      int it = 0, s = 0;
      uint32_t ph = 1;  // parity of the empty barrier's phase (first lap passes)
      bool ok = true;
      for (long long u = blockIdx.x; u < units && ok; u += gridDim.x) {
        const int vec = static_cast<int>(u / a.tiles), tile = static_cast<int>(u % a.tiles);
        for (int k = 0; k < a.slabs; ++k, ++it) {
          if (it >= S && !mbar_wait_bounded(empty + s, ph, a.status, DEV_ERR_TIMEOUT_EMPTY, a.wait_ns)) {
            ok = false;
            break;
          }
          if (!(a.fault_skip && it == 0)) {  // (test hook: stage 0 never fills)
            unsigned char* st = ring + s * stage_bytes;
            mbar_arrive_expect_tx(full + s, fill_bytes);
            tma_words(st, &tmA, k * (slab_bytes / 4), tile * a.mrows, vec, full + s, first);
            if (HILO)
              tma_words(st + a_bytes, &tmAlo, k * (slab_bytes / 4), tile * a.mrows, vec, full + s, first);
            tma_words(st + a_bytes * (HILO ? 2 : 1), &tmX, k * (x_bytes / 4), a.x_vec_first ? vec : 0,
                      a.x_vec_first ? 0 : vec, full + s, last);
          }
          if (++s == S) s = 0, ph ^= 1;
        }
      }
      // never leave the CTA with copies in flight
      for (int kk = (it > S ? it - S : 0); kk < it; ++kk)
        mbar_wait_bounded(full + kk % S, (kk / S) & 1, a.status, DEV_ERR_TIMEOUT_FULL, a.wait_ns);
    }
    return;
  }

  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsConsumer));
  int s = 0;
  uint32_t ph = 0;
  for (long long u = blockIdx.x; u < units; u += gridDim.x) {
    const int vec = static_cast<int>(u / a.tiles), tile = static_cast<int>(u % a.tiles);
    const int nr = min(a.mrows, a.rows_per_vec - tile * a.mrows);
    // a full tile gives each warp eight adjacent rows (64-byte stores), a
    // partial one deals its rows out over the warps.  The lanes of a full
    // tile's warp take their eight rows in an order of their own, so that
    // the reduction's first three steps need no selection
    const bool whole = nr == kWarps * RW;
    const int r_w = whole ? RW : 1, r_i = whole ? 1 : kWarps;
    const int row0 = warp * r_w;
    const int deal = !SHORT && whole ? lane >> 2 : 0;  // slot i of the lane is row i ^ deal of the warp's
    constexpr int PL = RW * R / 16;  // sums of a lane
    float sum[PL];
    for (int k0 = 0, k1 = a.block; k0 < a.slabs; k0 = k1, k1 = a.slabs) {
      float acc[RW * R * 2];
#pragma unroll
      for (int k = 0; k < RW * R * 2; ++k) acc[k] = 0.f;
      for (int k = k0; k < k1; ++k) {
        if (!mbar_wait_bounded(full + s, ph, a.status, DEV_ERR_TIMEOUT_FULL, a.wait_ns)) return;
        const unsigned char* st = ring + s * stage_bytes;
        const uint4* rows = reinterpret_cast<const uint4*>(st) + lane;
        const uint4* rows_lo = reinterpret_cast<const uint4*>(st + a_bytes) + lane;
        const float4* xs = reinterpret_cast<const float4*>(st + a_bytes * (HILO ? 2 : 1)) + lane * (C / 2);
        auto slab = [&](auto whole_tag) {
          constexpr bool WHOLE = decltype(whole_tag)::value;
#pragma unroll
          for (int h = 0; h < C / 2; ++h) {  // two entries of the lane's chunk at a time
            float4 x[R];
#pragma unroll
            for (int b = 0; b < R; ++b) x[b] = xs[b * pitch * (C / 2) + h];
#pragma unroll
            for (int i = 0; i < RW; ++i) {
              const int row = WHOLE ? row0 + (i ^ deal) : row0 + kWarps * i;
              if (!WHOLE && row >= nr) continue;
              float2 g[C];
              CH::unpack(rows[row * pitch], g);
              if (HILO) {
                float2 gl[C];
                CH::unpack(rows_lo[row * pitch], gl);
#pragma unroll
                for (int q = 0; q < C; ++q) g[q] = cadd(g[q], gl[q]);
              }
              const float2 g0 = g[2 * h], g1 = g[2 * h + 1];
#pragma unroll
              for (int b = 0; b < R; ++b) {
                cmac(g0, make_float2(x[b].x, x[b].y), acc[(i * R + b) * 2], acc[(i * R + b) * 2 + 1]);
                cmac(g1, make_float2(x[b].z, x[b].w), acc[(i * R + b) * 2], acc[(i * R + b) * 2 + 1]);
              }
            }
          }
        };
        if (!SHORT || lane < pitch) {  // (a row shorter than a slab leaves lanes without a chunk)
          if (whole)
            slab(std::true_type{});
          else
            slab(std::false_type{});
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(empty + s);
        if (++s == S) s = 0, ph ^= 1;
      }
      // reduce-scatter over the lanes: after the step with lane bit o a lane
      // keeps the half of its values that the bit selects, summed with its
      // partner's; value index ((row * R) + b) * 2 + component
#pragma unroll
      for (int o = 16, n = RW * R; o > 0; o >>= 1, n >>= 1) {
        const bool up = (lane & o) != 0;
        if (!SHORT && o > 2 && whole) {  // the rows are dealt so that the first half is the lane's own
#pragma unroll
          for (int k = 0; k < n; ++k) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k + n], o);
        } else {
#pragma unroll
          for (int k = 0; k < n; ++k) {
            const float keep = up ? acc[k + n] : acc[k];
            const float send = up ? acc[k] : acc[k + n];
            acc[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
          }
        }
      }
#pragma unroll
      for (int j = 0; j < PL; ++j) sum[j] = k0 == 0 ? acc[j] : sum[j] + acc[j];
    }
    float2* y = a.y + static_cast<long long>(vec) * a.rows_per_vec + tile * a.mrows;
#pragma unroll
    for (int j = 0; j < PL; ++j) {
      const int v = lane * PL + j;  // (each step's bit selects a half: lane major)
      const int row = row0 + v / (2 * R) * r_i, b = v / 2 % R;
      if (row < nr && b < a.nb) reinterpret_cast<float*>(y + b * a.y_ldb + row)[v & 1] = sum[j];
    }
  }
}

template <int EL, bool HILO, int R, bool SHORT = false>
cudaError_t launch_r(const StreamArgs& a, int num_sms, cudaStream_t st) {
  using CH = Chunk<EL>;
  const long long row_bytes = static_cast<long long>(a.row_len) * (16 / CH::C);
  MultiArgs m{};
  m.slab_bytes = row_bytes < kSlabBytes ? static_cast<int>(row_bytes) : kSlabBytes;
  const int x_bytes = m.slab_bytes * (CH::C / 2);
  m.rows_per_vec = static_cast<int>(a.rows_per_vec);
  m.n_vec = static_cast<int>(a.F / a.rows_per_vec);
  constexpr int tile_rows = kWarps * RW;
  m.mrows = a.rows_per_vec >= tile_rows ? tile_rows : static_cast<int>((a.rows_per_vec + 7) / 8 * 8);
  m.tiles = (m.rows_per_vec + m.mrows - 1) / m.mrows;
  m.slabs = static_cast<int>((row_bytes + kSlabBytes - 1) / kSlabBytes);
  m.block = chain_slabs(m.slabs) > 0 ? chain_slabs(m.slabs) : m.slabs;
  const int stage = (m.mrows * m.slab_bytes * (HILO ? 2 : 1) + R * x_bytes + 127) & ~127;
  m.stages = kBudget / stage < kMaxStages ? kBudget / stage : kMaxStages;
  m.nb = a.nb;
  m.y = a.y;
  m.y_ldb = a.y_ldb;
  m.status = a.status;
  m.wait_ns = a.wait_ns ? a.wait_ns : kWaitLimitNs;
  m.fault_skip = a.fault_skip;
  CUtensorMap ta, tl, tx;
  cudaError_t e;
  const long long vec_bytes = row_bytes * a.rows_per_vec;
  if ((e = tc_encode_words(&ta, a.rows, row_bytes / 4, a.rows_per_vec, row_bytes, m.n_vec, vec_bytes, m.slab_bytes / 4,
                           m.mrows)) != cudaSuccess)
    return e;
  tl = ta;
  if (HILO && (e = tc_encode_words(&tl, a.rows_lo, row_bytes / 4, a.rows_per_vec, row_bytes, m.n_vec, vec_bytes,
                                   m.slab_bytes / 4, m.mrows)) != cudaSuccess)
    return e;
  // ruptures past nb read as zeros (TMA fill); their sums are never stored.
  // The map's dimensions go up in pitch
  m.x_vec_first = a.x_stride < a.x_ldb ? 1 : 0;
  e = m.x_vec_first
          ? tc_encode_words(&tx, a.x, 2LL * a.row_len, m.n_vec, 8 * a.x_stride, a.nb, 8 * a.x_ldb, x_bytes / 4, 1, R)
          : tc_encode_words(&tx, a.x, 2LL * a.row_len, a.nb, 8 * a.x_ldb, m.n_vec, 8 * a.x_stride, x_bytes / 4, R);
  if (e != cudaSuccess) return e;
  const size_t smem = 2 * 8 * kMaxStages + static_cast<size_t>(m.stages) * stage;
  if ((e = cudaFuncSetAttribute(k_stream_multi<EL, HILO, R, SHORT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                static_cast<int>(smem))) != cudaSuccess)
    return e;
  long long grid = static_cast<long long>(m.n_vec) * m.tiles;
  if (grid > num_sms) grid = num_sms;
  launch_next(k_stream_multi<EL, HILO, R, SHORT>, static_cast<unsigned>(grid), kThreads, smem, st, ta, tl, tx, m);
  return cudaGetLastError();
}

template <int EL, bool HILO>
cudaError_t launch_el(const StreamArgs& a, int num_sms, cudaStream_t st) {
  if (a.row_len * (16 / Chunk<EL>::C) < kSlabBytes)
    return a.nb <= 4 ? launch_r<EL, HILO, 4, true>(a, num_sms, st) : launch_r<EL, HILO, 8, true>(a, num_sms, st);
  if (a.nb <= 2) return launch_r<EL, HILO, 2>(a, num_sms, st);
  if (a.nb <= 4) return launch_r<EL, HILO, 4>(a, num_sms, st);
  if (a.nb <= 6) return launch_r<EL, HILO, 6>(a, num_sms, st);
  return launch_r<EL, HILO, 8>(a, num_sms, st);
}

}  // namespace

cudaError_t launch_stream_multi(const StreamArgs& a, int num_sms, cudaStream_t st) {
  if (a.nb < 2 || a.nb > kStreamMulti || a.rows_per_vec < 1 || a.rows_per_vec > 0x7fffff00 ||
      a.F % a.rows_per_vec != 0)
    return cudaErrorInvalidValue;
  switch (a.el) {
    case EL_FP32: return launch_el<EL_FP32, false>(a, num_sms, st);
    case EL_BF16: return launch_el<EL_BF16, false>(a, num_sms, st);
    case EL_BF16_HILO: return launch_el<EL_BF16, true>(a, num_sms, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace s2w
