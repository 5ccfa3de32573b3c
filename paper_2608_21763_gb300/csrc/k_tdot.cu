// Transposed contraction on the HBM-streaming path (the adjoint, a
// correlation with the conjugate spectra), for 1 .. 8 ruptures per pass:
//   y_b[u][c] = sum_{f in unit u} conj(rows[f][c]) w_b[f].
// A unit is `Rc` consecutive rows of one group of G1 rows (chunk u % nchunk
// of group u / nchunk); rupture b's weight of row f is w[w_base + b w_ldb +
// (g / wa) wb + (f - g G1)] with g = f / G1, times the FP8 row scale.
//
// Persistent CTAs take units round robin; one lane streams the unit's rows
// (contiguous) through a ring by cp.async.bulk, its warp brings the rows'
// weights into the stage beside them.  The consumer warps split the
// columns: a thread owns one 16-byte chunk of every row and keeps the
// sums of its columns for all R ruptures in registers, so nothing is reduced
// across threads over long rows.  Each time a multiple of 64 rows is passed
// (whole stages, so after 64 to 127 rows) they are added to sums in shared
// memory (1.5 % of the instructions), since one accumulation over a whole unit
// showed in the result (3.2e-7 against 2.6e-7 of FP32 rounding at 501 x 10,007
// x 33 x 128).  With fewer chunks than threads, groups of
// threads take the rows in turn and are added up at the end of the unit, in
// fixed order.  A row's weights are one shared-memory broadcast per two
// ruptures.
//
// What bounds it: HBM up to about four FP32 ruptures, then the FMAs (4 per
// stored entry and rupture) and their issue: packed FP32 products (chunk.cuh)
// with the weights prepared by the producer warp, sixteen FP32 warps (four
// per scheduler; at six and eight ruptures their 96 registers spill 12 and 28
// bytes).  Measured, adjoint of 963 x 8,000 x 64 x 256: one rupture
// 2.57 ms (2.61 before, rows split over eight warps), two 2.61, four 2.90,
// eight 4.2 (20.8 one by one; eight warps with scalar FMAs 4.8, sixteen 4.5);
// BF16, one 1.31 ms (1.87), eight 3.3 (14.8); 60 x 60,000 x 4 x 256, one 1.5 ms
// (10.7: the old kernel gave a short row to a whole warp).  FP32 gradient
// through autograd, 501 x 10,007 x 33 x 128, six ruptures, forward and
// backward: 11.5 -> 2.17 ms.  The sums do not depend on R: a rupture's result
// is the same bits alone or in a batch.
#include "chunk.cuh"

namespace s2w {

namespace {

// Consumer warps: the chunks of the longest row (512 FP32, 256 BF16, 128 FP8)
// on one thread each, at least eight warps.
__host__ __device__ constexpr int tdot_warps(int el) { return el == EL_FP32 ? 16 : 8; }
constexpr int kMaxRowLen = 1024;
constexpr int kMaxStages = 8;
constexpr int kStageRows = 64;         // most rows per stage (their weights share the stage)
constexpr int kMaxGroups = 32;
constexpr int kStageBytes = 32 * 1024;
constexpr int kFlushRows = 64;         // rows per FP32 accumulation; the blocks' sums are added up apart
constexpr int kBudget = 208 * 1024;    // ring and sums (up to 64 KB)

template <int EL, bool HILO, int R>
__global__ void __launch_bounds__(32 * (tdot_warps(EL) + 1), 1)
    k_stream_tdot(const StreamTArgs a, int stage_rows, int stages, int cols, int groups) {
  grid_dependency();
  using CH = Chunk<EL>;
  constexpr int C = CH::C;
  constexpr int kWarps = tdot_warps(EL);
  constexpr int kCons = 32 * kWarps;
  extern __shared__ __align__(128) unsigned char sm[];
  uint64_t* full = reinterpret_cast<uint64_t*>(sm);
  uint64_t* empty = full + kMaxStages;
  const int row_bytes = a.row_len * (16 / C);
  const int rows_bytes = stage_rows * row_bytes;
  const int stage_bytes = rows_bytes * (HILO ? 2 : 1) + stage_rows * R * 16;
  unsigned char* ring = sm + 2 * 8 * kMaxStages;
  // sums over whole kFlushRows blocks, one 16-byte slot per thread and step
  float4* part = reinterpret_cast<float4*>(ring + stages * ((stage_bytes + 15) & ~15)) + threadIdx.x;
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(full + s, 2);  // the copies' lane, and the weights' warp
      mbar_init(empty + s, kWarps);
    }
    fence_mbar_init();
  }
  __syncthreads();

  auto unit_rows = [&](long long u, long long& g, long long& f0, int& w0, int& n) {
    g = u / a.nchunk;
    w0 = static_cast<int>(u % a.nchunk) * a.Rc;  // first row within the group
    n = static_cast<int>(min(static_cast<long long>(a.Rc), a.G1 - w0));
    f0 = g * a.G1 + w0;
  };

  if (warp == kWarps) {
    const uint64_t pol = l2_policy_evict_first();
    // the stage being filled: unit u, rows r0 .. r0 + nr of it
    long long u = blockIdx.x, g = 0, f0 = 0;
    int w0 = 0, n = 0, r0 = 0;
    const float2* wu = nullptr;  // the unit's weights
    auto seek = [&]() {
      if (u >= a.n_units) return;
      unit_rows(u, g, f0, w0, n);
      wu = a.w + a.w_base + (g / a.wa) * a.wb + w0;
    };
    auto next = [&]() {
      r0 += stage_rows;
      if (r0 >= n) u += gridDim.x, r0 = 0, seek();
    };
    auto weight = [&](int e) {  // entry e = row R + b of the stage's weights
      const int b = e % R, row = e / R;
      float2 w = make_float2(0.f, 0.f);
      if (row < min(stage_rows, n - r0) && b < a.nb) {
        w = __ldg(wu + b * a.w_ldb + r0 + row);
        if (EL == EL_FP8) {
          const float sc = a.scale[g * a.nblk + (w0 + r0 + row) / 256];
          w.x *= sc;
          w.y *= sc;
        }
      }
      return w;
    };
    seek();
    float2 pre[4];  // the stage's first 128 weights, loaded one stage ahead
    if (u < a.n_units)
#pragma unroll
      for (int j = 0; j < 4; ++j) pre[j] = weight(lane + 32 * j);
    int it = 0, s = 0;
    uint32_t ph = 1;
    for (; u < a.n_units; ++it) {
      const int nr = min(stage_rows, n - r0);
      // (a vote: the lanes leave together)
      if (it >= stages &&
          !__all_sync(0xffffffffu, mbar_wait_bounded(empty + s, ph, a.status, DEV_ERR_TIMEOUT_EMPTY)))
        break;
      unsigned char* st = ring + s * ((stage_bytes + 15) & ~15);
      if (lane == 0) {
        const uint32_t bytes = static_cast<uint32_t>(nr) * row_bytes;
        mbar_arrive_expect_tx(full + s, HILO ? 2 * bytes : bytes);
        bulk_g2s(st, static_cast<const unsigned char*>(a.rows) + (f0 + r0) * row_bytes, bytes, full + s, pol);
        if (HILO)
          bulk_g2s(st + rows_bytes, static_cast<const unsigned char*>(a.rows_lo) + (f0 + r0) * row_bytes, bytes,
                   full + s, pol);
      }
      float4* ws = reinterpret_cast<float4*>(st + rows_bytes * (HILO ? 2 : 1));
      auto put = [&](int e, float2 w) {  // prepared for conj(g) w on packed pairs (chunk.cuh)
        if (e < nr * R) ws[e] = make_float4(w.x, w.y, w.y, -w.x);
      };
#pragma unroll
      for (int j = 0; j < 4; ++j) put(lane + 32 * j, pre[j]);
      for (int e = lane + 128; e < nr * R; e += 32) put(e, weight(e));
      __syncwarp();
      if (lane == 0) mbar_arrive(full + s);
      if (++s == stages) s = 0, ph ^= 1;
      next();
      if (u < a.n_units)
#pragma unroll
        for (int j = 0; j < 4; ++j) pre[j] = weight(lane + 32 * j);
    }
    // never leave the CTA with copies in flight
    if (lane == 0)
      for (int kk = (it > stages ? it - stages : 0); kk < it; ++kk)
        mbar_wait_bounded(full + kk % stages, (kk / stages) & 1, a.status, DEV_ERR_TIMEOUT_FULL);
    return;
  }

  const int c0 = threadIdx.x % cols, grp = threadIdx.x / cols;
  const bool mine = grp < groups;
  int s = 0;
  uint32_t ph = 0;
  for (long long u = blockIdx.x; u < a.n_units; u += gridDim.x) {
    long long g, f0;
    int w0, n;
    unit_rows(u, g, f0, w0, n);
    float2 acc[R][C];
#pragma unroll
    for (int b = 0; b < R; ++b)
#pragma unroll
      for (int q = 0; q < C; ++q) acc[b][q] = make_float2(0.f, 0.f);
    bool ok = true, flushed = false;
    auto flush = [&](bool clear) {  // acc += the earlier blocks' sums, to `part` when `clear`
#pragma unroll
      for (int k = 0; k < R * C / 2; ++k) {
        float2& lo = acc[k / (C / 2)][k % (C / 2) * 2];
        float2& hi = acc[k / (C / 2)][k % (C / 2) * 2 + 1];
        if (flushed) {
          const float4 v = part[k * kCons];
          lo = make_float2(v.x + lo.x, v.y + lo.y);
          hi = make_float2(v.z + hi.x, v.w + hi.y);
        }
        if (clear) {
          part[k * kCons] = make_float4(lo.x, lo.y, hi.x, hi.y);
          lo = hi = make_float2(0.f, 0.f);
        }
      }
      flushed = true;
    };
    for (int r0 = 0; r0 < n; r0 += stage_rows) {
      if (r0 / kFlushRows != (r0 - stage_rows) / kFlushRows && r0 > 0) flush(true);
      if (!mbar_wait_bounded(full + s, ph, a.status, DEV_ERR_TIMEOUT_FULL)) {
        ok = false;
        break;
      }
      const int nr = min(stage_rows, n - r0);
      const unsigned char* st = ring + s * ((stage_bytes + 15) & ~15);
      const float4* ws = reinterpret_cast<const float4*>(st + rows_bytes * (HILO ? 2 : 1));
      if (mine) {
#pragma unroll 2
        for (int row = grp; row < nr; row += groups) {
          float4 w[R];
#pragma unroll
          for (int b = 0; b < R; ++b) w[b] = ws[row * R + b];
          float2 gv[C];
          CH::unpack(*reinterpret_cast<const uint4*>(st + row * row_bytes + c0 * 16), gv);
          if (HILO) {
            float2 gl[C];
            CH::unpack(*reinterpret_cast<const uint4*>(st + rows_bytes + row * row_bytes + c0 * 16), gl);
#pragma unroll
            for (int q = 0; q < C; ++q) gv[q] = cadd(gv[q], gl[q]);
          }
#pragma unroll
          for (int q = 0; q < C; ++q) {  // conj(g) w
#pragma unroll
            for (int b = 0; b < R; ++b) acc[b][q] = cmac2_re(gv[q], w[b], acc[b][q]);
#pragma unroll
            for (int b = 0; b < R; ++b) acc[b][q] = cmac2_im(gv[q], w[b], acc[b][q]);
          }
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(empty + s);
      if (++s == stages) s = 0, ph ^= 1;
    }
    float2* y = a.y + u * a.row_len;
    const int nc = static_cast<int>(  // columns that are not padding
        max(0LL, min(static_cast<long long>(a.row_len), a.cols - (g % a.wa) * a.row_len)));
    flush(groups > 1);
    if (groups == 1) {
      if (!ok) return;
      if (mine) {
#pragma unroll
        for (int b = 0; b < R; ++b)
          if (b < a.nb)
#pragma unroll
            for (int q = 0; q < C; q += 2) {
              float2* yc = y + b * a.y_ldb + c0 * C + q;
              if (c0 * C + q + 1 < nc)
                *reinterpret_cast<float4*>(yc) =
                    make_float4(acc[b][q].x, acc[b][q].y, acc[b][q + 1].x, acc[b][q + 1].y);
              else if (c0 * C + q < nc)
                *yc = acc[b][q];
            }
      }
      continue;
    }
    // the row groups' sums, added in group order
    asm volatile("bar.sync 1, %0;" ::"r"(kCons) : "memory");
    const int live = a.nb * a.row_len;
    const float2* all = reinterpret_cast<const float2*>(part - threadIdx.x);
    for (int e = threadIdx.x; e < live; e += kCons) {
      const int b = e / a.row_len, col = e - b * a.row_len;
      if (col >= nc) continue;
      const int at = 2 * ((b * (C / 2) + col % C / 2) * kCons + col / C) + (col & 1);
      float2 p[4];  // four partial sums: shorter chains, less rounding
#pragma unroll
      for (int k = 0; k < 4; ++k) p[k] = k < groups ? all[at + 2 * k * cols] : make_float2(0.f, 0.f);
      for (int k0 = 4; k0 < groups; k0 += 4)
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (k0 + k < groups) p[k] = cadd(p[k], all[at + 2 * (k0 + k) * cols]);
      const float2 sum = cadd(cadd(p[0], p[1]), cadd(p[2], p[3]));
      y[b * a.y_ldb + col] = sum;
    }
    // second barrier doubles as a vote: if any consumer warp gave up on a
    // wait, all of them leave together (none is left behind on this barrier)
    int any_failed;
    asm volatile(
        "{\n\t.reg .pred pin, pout;\n\t"
        "setp.eq.u32 pin, %1, 0;\n\t"
        "bar.red.or.pred pout, 1, %2, pin;\n\t"
        "selp.u32 %0, 1, 0, pout;\n\t}"
        : "=r"(any_failed)
        : "r"(ok ? 1u : 0u), "r"(kCons)
        : "memory");
    if (any_failed) return;
  }
}

template <int EL, bool HILO, int R>
cudaError_t launch_r(const StreamTArgs& a, int num_sms, cudaStream_t st) {
  constexpr int C = Chunk<EL>::C;
  constexpr int kCons = 32 * tdot_warps(EL);
  const int row_bytes = a.row_len * (16 / C), cols = row_bytes / 16;
  int groups = kCons / cols;
  if (groups > kMaxGroups) groups = kMaxGroups;
  // whole rounds of the row groups per stage, so that a row's group does not
  // depend on the stage it falls into
  int stage_rows = kStageBytes / (row_bytes * (HILO ? 2 : 1));
  if (stage_rows > kStageRows) stage_rows = kStageRows;
  stage_rows = stage_rows / groups * groups;
  if (stage_rows < groups) stage_rows = groups;
  const int stage_bytes = (stage_rows * (row_bytes * (HILO ? 2 : 1) + R * 16) + 15) & ~15;
  constexpr int part_bytes = sizeof(float2) * kCons * R * C;
  int stages = (kBudget - part_bytes) / stage_bytes;
  if (stages > kMaxStages) stages = kMaxStages;
  const size_t smem = 2 * 8 * kMaxStages + static_cast<size_t>(stages) * stage_bytes + part_bytes;
  cudaError_t e = cudaFuncSetAttribute(k_stream_tdot<EL, HILO, R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  const long long grid = a.n_units < num_sms ? a.n_units : num_sms;
  launch_next(k_stream_tdot<EL, HILO, R>, static_cast<unsigned>(grid), kCons + 32, smem, st, a, stage_rows, stages,
              cols, groups);
  return cudaGetLastError();
}

template <int EL, bool HILO>
cudaError_t launch_el(const StreamTArgs& a, int num_sms, cudaStream_t st) {
  // FP8 chunks hold eight entries: sums for four ruptures fill the registers
  constexpr int most = EL == EL_FP8 ? 4 : kStreamMulti;
  if (a.nb > most) {
    StreamTArgs h = a;
    h.nb = most;
    const cudaError_t e = launch_el<EL, HILO>(h, num_sms, st);
    if (e != cudaSuccess) return e;
    h.nb = a.nb - most;
    h.w = a.w + most * a.w_ldb;
    h.y = a.y + most * a.y_ldb;
    return launch_el<EL, HILO>(h, num_sms, st);
  }
  if (a.nb == 1) return launch_r<EL, HILO, 1>(a, num_sms, st);
  if (a.nb == 2) return launch_r<EL, HILO, 2>(a, num_sms, st);
  if (a.nb <= 4) return launch_r<EL, HILO, 4>(a, num_sms, st);
  if constexpr (most > 4) {
    if (a.nb <= 6) return launch_r<EL, HILO, 6>(a, num_sms, st);
    return launch_r<EL, HILO, 8>(a, num_sms, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_stream_tdot(const StreamTArgs& a, int num_sms, cudaStream_t st) {
  if (a.n_units <= 0 || a.nb <= 0) return cudaSuccess;
  if (a.row_len <= 0 || a.row_len > kMaxRowLen || (a.row_len % 8) != 0 || a.Rc < 1 || a.nchunk < 1 ||
      a.nb > kStreamMulti)
    return cudaErrorInvalidValue;
  switch (a.el) {
    case EL_FP32: return launch_el<EL_FP32, false>(a, num_sms, st);
    case EL_BF16: return launch_el<EL_BF16, false>(a, num_sms, st);
    case EL_BF16_HILO: return launch_el<EL_BF16, true>(a, num_sms, st);
    case EL_FP8: return launch_el<EL_FP8, false>(a, num_sms, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace s2w
