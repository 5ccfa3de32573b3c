// Per-bin complex contractions on the HBM-streaming path (Alg. 2 step 3,
// yhat_l = Fhat_l xhat_l, for a small rupture batch).
//
// Both stages are one kernel (batches of FP32 / BF16 rows: k_multi.cu, and
// the R > 1 variants here for short rows).  The resident spectrum is a sequence of F
// contiguous rows of `row_len` complex entries; row f is dotted with the
// vector x_vec(f) = x + (f / rows_per_vec) * x_stride:
//   stage 1: rows (l, i) of Ghat [l][i][Ns_pad], x_vec = shat_l     -> mhat[l][i]
//   stage 2: rows (l, seg, o) of Phat [l][seg][o][RL],
//            x_vec = vhat_l[seg * RL ..]                           -> partial[l][seg][o]
//
// Each CTA owns one contiguous range of rows (balanced to the row) and streams
// it through a 3-stage shared-memory ring filled by cp.async.bulk (one bulk
// copy per stage, L2 evict-first: every operator byte is read exactly once).
// Eight consumer warps take rows in passes: a long row gets a whole warp (lane
// l handles the 16-byte chunks l, l + 32, ..., so a warp reads 512 contiguous
// bytes per step); a short row (a few subfaults) gets a power-of-two group of
// lanes with about four chunks each, several rows per warp pass.  Each lane
// keeps its slice of x_vec in registers across rows that share it.  Products
// accumulate in FP32; FP8 rows are widened exactly to FP16 pairs (one
// conversion per complex entry) and multiplied by the vector held as FP16
// pairs scaled by a power of two (its largest magnitude into [2, 4)), with
// packed FP16 multiply-adds (independent accumulators per lane, each summing
// at most 8 products) flushed into FP32 at the end of the row, so that a
// streamed byte costs about two instructions; long FP8 rows go four per warp
// pass with one butterfly reduction over the lanes for the four;
// the per-(bin, 256-row block) scale and the power of two are undone after
// the dot product.  FP32_HILO (FP32 pairs): k_dfdot.cu.
#include <type_traits>

#include "chunk.cuh"

namespace s2w {

namespace {

constexpr int kStages = 3;
constexpr int kMaxRowLen = 1024;

// EL selects the unpacker (EL_BF16 also serves the hi/lo pair when HILO);
// SHORT: rows of at most 64 chunks, shared by lane groups.
// Consumer warps of k_stream_dot.  FP8 rows carry half the bytes of BF16
// ones, so per-row work (the lane reduction, the scale) weighs more: long FP8
// rows are taken four per warp pass (one reduction for the four), short ones
// by twelve warps (more rows in flight; ~120 registers each, no spills).
// One rupture's short FP32 / BF16 rows take twelve warps too.
__host__ __device__ constexpr int stream_warps(bool short_rows, int r) {
  return (short_rows && r == 1) ? 12 : 8;
}

// R > 1 (short FP32 / BF16 rows): the row meets the vectors of R ruptures,
// each lane's slices of all R held in registers, so a batch reads the
// operator once per R ruptures.  Otherwise a batch takes one grid slice (y)
// per rupture.
// BLK: slabs in the first block of a long FP32 / BF16 row (chain_slabs), so
// the row has 2 BLK or 2 BLK + 1 of them.  A kernel for each count keeps the
// blocks' border and the empty slabs of shorter rows out of the row loop,
// which is bound by its instructions below about 500 entries: stage 1, one
// rupture, 190 x 20,000 x 256 FP32 2.01 ms in one kernel for all lengths, 1.12
// here; 300 x 12,000 1.44 -> 1.08; 300 x 8,000 BF16 0.71 -> 0.53; 963 x 8,000 FP32
// 2.30 -> 2.25 (its bytes), BF16 1.16 -> 1.15.
template <int EL, bool HILO, bool SHORT, int R = 1, int BLK = 0>
__global__ void __launch_bounds__(32 * (stream_warps(SHORT, R) + 1), 1)
    k_stream_dot(const StreamArgs a, int stage_rows) {
  grid_dependency();
  constexpr int kConsumerWarps = stream_warps(SHORT, R);
  static_assert(R == 1 || (SHORT && EL != EL_FP8), "several vectors: short FP32 or BF16 rows");
  using CH = Chunk<EL>;
  constexpr int C = CH::C;
  // chunk slots per lane: a short row gives each lane at most four chunks
  constexpr int kMostSlabs = kMaxRowLen / (32 * C);
  constexpr int T = SHORT ? 4 : (BLK > 0 && 2 * BLK + 1 < kMostSlabs ? 2 * BLK + 1 : kMostSlabs);
  extern __shared__ __align__(128) unsigned char sm[];
  uint64_t* full = reinterpret_cast<uint64_t*>(sm);
  uint64_t* empty = full + kStages;
  unsigned char* buf = sm + 128;
  const int row_bytes = a.row_len * (16 / C);
  const int stage_bytes = stage_rows * row_bytes;
  unsigned char* buf_lo = buf + kStages * stage_bytes;
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const long long r0 = a.F * blockIdx.x / gridDim.x;
  const long long r1 = a.F * (blockIdx.x + 1) / gridDim.x;
  const int nst = static_cast<int>((r1 - r0 + stage_rows - 1) / stage_rows);
  const unsigned long long wlim = a.wait_ns ? a.wait_ns : kWaitLimitNs;
  const float2* const ax = a.x + blockIdx.y * a.x_ldb;
  float2* const ay = a.y + blockIdx.y * a.y_ldb;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, kConsumerWarps);
    }
    fence_mbar_init();
  }
  __syncthreads();

  if (warp == kConsumerWarps) {  // producer warp: one elected lane issues the copies
    if (lane == 0) {
      const uint64_t pol = l2_policy_evict_first();
      int k = 0;
      for (; k < nst; ++k) {
        const int s = k % kStages;
        if (k >= kStages &&
            !mbar_wait_bounded(empty + s, ((k / kStages) - 1) & 1, a.status, DEV_ERR_TIMEOUT_EMPTY, wlim))
          break;
        if (a.fault_skip && k == 0) continue;  // test hook: stage 0 never fills (no copy, no expected bytes)
        const long long rs = r0 + static_cast<long long>(k) * stage_rows;
        const int nr = static_cast<int>(min(static_cast<long long>(stage_rows), r1 - rs));
        const uint32_t bytes = static_cast<uint32_t>(nr) * row_bytes;
        mbar_arrive_expect_tx(full + s, HILO ? 2 * bytes : bytes);
        bulk_g2s(buf + s * stage_bytes, static_cast<const unsigned char*>(a.rows) + rs * row_bytes, bytes, full + s,
                 pol);
        if (HILO)
          bulk_g2s(buf_lo + s * stage_bytes, static_cast<const unsigned char*>(a.rows_lo) + rs * row_bytes, bytes,
                   full + s, pol);
      }
      // Never leave the CTA with copies in flight: wait for the last stages issued.
      for (int kk = (k > kStages ? k - kStages : 0); kk < k; ++kk)
        mbar_wait_bounded(full + kk % kStages, (kk / kStages) & 1, a.status, DEV_ERR_TIMEOUT_FULL, wlim);
    }
    return;
  }

  // consumer warps: a row is shared by `lpr` lanes (a power of two, chosen so
  // a lane takes about four chunks of a short row), so a warp takes 32 / lpr
  // rows per pass and the row sums need log2(lpr) shuffle steps
  const int nchunk = row_bytes / 16;
  int lpr = 32;
  if (SHORT)
    while (lpr > 1 && 4 * (lpr / 2) >= nchunk) lpr >>= 1;
  const int rpp = 32 / lpr;     // rows per warp pass
  const int sub = lane % lpr;   // lane within its row group
  const int grp = lane / lpr;   // row group within the warp
  constexpr bool F8 = EL == EL_FP8;
  float2 xr[R][F8 ? 1 : T][F8 ? 1 : C];
  // FP8: x_vec times a power of two sx (max |component| into [2, 4)) as FP16
  // pairs (Re, Re) and (Im, Im) for the packed products, and 1 / sx
  __half2 xrr[F8 ? T : 1][F8 ? C : 1], xii[F8 ? T : 1][F8 ? C : 1];
  float x_unscale = 1.f;
  long long vec = -1, vec_end = 0;  // x_vec of rows [vec_end - rows_per_vec, vec_end); rows rise per lane
  if constexpr (F8 && !SHORT) {
    // Long FP8 rows, four per warp pass, all 32 lanes on each: the lane's
    // products of the four rows accumulate side by side (sixteen FP16 pair
    // chains per kind), then one butterfly reduce-scatter over the lanes sums
    // the 8 values (Re and Im of four rows) with 9 shuffles instead of 40;
    // lanes 4v hold value v.  Rows of a pass that fall into the next bin are
    // taken in a second round after the vector reload.
    for (int k = 0; k < nst; ++k) {
      const int s = k % kStages;
      if (!mbar_wait_bounded(full + s, (k / kStages) & 1, a.status, DEV_ERR_TIMEOUT_FULL, wlim)) return;
      const long long rs = r0 + static_cast<long long>(k) * stage_rows;
      const int nr = static_cast<int>(min(static_cast<long long>(stage_rows), r1 - rs));
      for (int base = warp * 4; base < nr; base += kConsumerWarps * 4) {
        int j = 0;
        while (j < 4 && base + j < nr) {
          if (rs + base + j >= vec_end) {  // warp-uniform: every lane works on the same rows
            vec = (rs + base + j) / a.rows_per_vec;
            vec_end = (vec + 1) * a.rows_per_vec;
            const float4* xv = reinterpret_cast<const float4*>(ax + vec * a.x_stride);
            float amax = 0.f;
#pragma unroll
            for (int t = 0; t < T; ++t) {
              const int c = lane + 32 * t;
#pragma unroll
              for (int q = 0; q < C / 2; ++q) {
                const float4 v = (c < nchunk) ? __ldg(xv + c * (C / 2) + q) : make_float4(0.f, 0.f, 0.f, 0.f);
                amax = fmaxf(amax, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
              }
            }
            for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
            int e = 0;
            frexpf(amax, &e);  // amax = m 2^e, m in [0.5, 1)
            const float sx = amax > 0.f ? ldexpf(1.f, 2 - e) : 1.f;
            x_unscale = amax > 0.f ? ldexpf(1.f, e - 2) : 1.f;
#pragma unroll
            for (int t = 0; t < T; ++t) {
              const int c = lane + 32 * t;
#pragma unroll
              for (int q = 0; q < C / 2; ++q) {
                const float4 v = (c < nchunk) ? __ldg(xv + c * (C / 2) + q) : make_float4(0.f, 0.f, 0.f, 0.f);
                xrr[t][2 * q] = __float2half2_rn(v.x * sx);
                xii[t][2 * q] = __float2half2_rn(v.y * sx);
                xrr[t][2 * q + 1] = __float2half2_rn(v.z * sx);
                xii[t][2 * q + 1] = __float2half2_rn(v.w * sx);
              }
            }
          }
          int je = j + 1;  // rows j .. je-1 of the pass share this bin's vector
          while (je < 4 && base + je < nr && rs + base + je < vec_end) ++je;
          __half2 ha[4][4], hb[4][4];
#pragma unroll
          for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int q = 0; q < 4; ++q) ha[r][q] = hb[r][q] = __float2half2_rn(0.f);
          // ALL: the four rows share the bin (the usual case): no per-row tests
          auto accumulate = [&](auto all_tag) {
            constexpr bool ALL = decltype(all_tag)::value;
#pragma unroll
            for (int t = 0; t < T; ++t) {
              const int c = lane + 32 * t;
              if (c < nchunk) {
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                  if (ALL || (r >= j && r < je)) {
                    const uint4 u =
                        reinterpret_cast<const uint4*>(buf + s * stage_bytes + (base + r) * row_bytes)[c];
                    const unsigned w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                      __half2 g[2];
                      e4m3x4_to_h2(w[q], g[0], g[1]);
#pragma unroll
                      for (int h = 0; h < 2; ++h) {
                        ha[r][q] = __hfma2(g[h], xrr[t][2 * q + h], ha[r][q]);  // (gr xr, gi xr)
                        hb[r][q] = __hfma2(g[h], xii[t][2 * q + h], hb[r][q]);  // (gr xi, gi xi)
                      }
                    }
                  }
                }
              }
            }
          };
          if (j == 0 && je == 4)
            accumulate(std::true_type{});
          else
            accumulate(std::false_type{});
          float v[8];
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            float ar = 0.f, ai = 0.f;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const float2 fa = __half22float2(ha[r][q]), fb = __half22float2(hb[r][q]);
              ar += fa.x - fb.y;
              ai += fb.x + fa.y;
            }
            v[2 * r] = ar;
            v[2 * r + 1] = ai;
          }
          // reduce-scatter: after the step with lane bit b, the lane keeps the
          // half of its values selected by that bit, summed with its partner's
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const bool up = lane & 16;
            const float keep = up ? v[i + 4] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, up ? v[i] : v[i + 4], 16);
          }
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const bool up = lane & 8;
            const float keep = up ? v[i + 2] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, up ? v[i] : v[i + 2], 8);
          }
          {
            const bool up = lane & 4;
            const float keep = up ? v[1] : v[0];
            v[0] = keep + __shfl_xor_sync(0xffffffffu, up ? v[0] : v[1], 4);
          }
          v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
          v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
          const int idx = ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
          const int r = idx >> 1;
          if ((lane & 3) == 0 && r >= j && r < je) {
            const long long f = rs + base + r;
            const float sc = a.scale[vec * a.nblk + (f - (vec_end - a.rows_per_vec)) / 256] * x_unscale;
            reinterpret_cast<float*>(ay + f)[idx & 1] = v[0] * sc;
          }
          j = je;
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(empty + s);
    }
    return;
  }
  for (int k = 0; k < nst; ++k) {
    const int s = k % kStages;
    if (!mbar_wait_bounded(full + s, (k / kStages) & 1, a.status, DEV_ERR_TIMEOUT_FULL, wlim)) return;
    const long long rs = r0 + static_cast<long long>(k) * stage_rows;
    const int nr = static_cast<int>(min(static_cast<long long>(stage_rows), r1 - rs));
    for (int base = warp * rpp; base < nr; base += kConsumerWarps * rpp) {
      const int lr = base + grp;
      const bool valid = lr < nr;
      const long long f = rs + (valid ? lr : base);
      if (f >= vec_end) {
        vec = f / a.rows_per_vec;
        vec_end = (vec + 1) * a.rows_per_vec;
        const float4* xv = reinterpret_cast<const float4*>(ax + vec * a.x_stride);
        if constexpr (F8) {
          // two passes over the lane's slice (cached loads): the largest
          // magnitude over the row group's whole vector, then the scaled
          // FP16 pairs; the lanes of one row group take this branch together
          float amax = 0.f;
#pragma unroll
          for (int t = 0; t < T; ++t) {
            const int c = sub + lpr * t;
#pragma unroll
            for (int q = 0; q < C / 2; ++q) {
              const float4 v = (c < nchunk) ? __ldg(xv + c * (C / 2) + q) : make_float4(0.f, 0.f, 0.f, 0.f);
              amax = fmaxf(amax, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
            }
          }
          const unsigned gmask = lpr == 32 ? 0xffffffffu : ((1u << lpr) - 1u) << (grp * lpr);  // this row group
          for (int o = lpr / 2; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(gmask, amax, o));
          int e = 0;
          frexpf(amax, &e);  // amax = m 2^e, m in [0.5, 1)
          const float sx = amax > 0.f ? ldexpf(1.f, 2 - e) : 1.f;
          x_unscale = amax > 0.f ? ldexpf(1.f, e - 2) : 1.f;
#pragma unroll
          for (int t = 0; t < T; ++t) {
            const int c = sub + lpr * t;
#pragma unroll
            for (int q = 0; q < C / 2; ++q) {
              const float4 v = (c < nchunk) ? __ldg(xv + c * (C / 2) + q) : make_float4(0.f, 0.f, 0.f, 0.f);
              xrr[t][2 * q] = __float2half2_rn(v.x * sx);
              xii[t][2 * q] = __float2half2_rn(v.y * sx);
              xrr[t][2 * q + 1] = __float2half2_rn(v.z * sx);
              xii[t][2 * q + 1] = __float2half2_rn(v.w * sx);
            }
          }
        } else {
#pragma unroll
          for (int t = 0; t < T; ++t) {
            const int c = sub + lpr * t;
#pragma unroll
            for (int q = 0; q < C / 2; ++q) {
#pragma unroll
              for (int b = 0; b < R; ++b) {  // (slots past the last rupture repeat it; never stored)
                const float4* xb = b == 0 ? xv : xv + min(b, a.nb - 1) * (a.x_ldb / 2);
                const float4 v = (c < nchunk) ? __ldg(xb + c * (C / 2) + q) : make_float4(0.f, 0.f, 0.f, 0.f);
                xr[b][t][2 * q] = make_float2(v.x, v.y);
                xr[b][t][2 * q + 1] = make_float2(v.z, v.w);
              }
            }
          }
        }
      }
      const int rrow = valid ? lr : base;
      const uint4* row = reinterpret_cast<const uint4*>(buf + s * stage_bytes + rrow * row_bytes);
      const uint4* row_lo = reinterpret_cast<const uint4*>(buf_lo + s * stage_bytes + rrow * row_bytes);
      if constexpr (F8) {
        // e4m3 pairs (Re, Im) widen exactly to FP16 pairs (one cvt per
        // complex entry); g * (xr, xr) and g * (xi, xi) accumulate as FP16
        // pairs over the lane's T = 4 chunks of the row (eight independent
        // accumulator chains of 8 products each: |g| <= 448, |x sx| < 4, so
        // |sum| < 2^14, inside the FP16 range), then into FP32
        static_assert(!F8 || T <= 4, "FP16 accumulation bound: at most 8 products per accumulator");
        float ar = 0.f, ai = 0.f;
        __half2 ha[4], hb[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) ha[k] = hb[k] = __float2half2_rn(0.f);
#pragma unroll
        for (int t = 0; t < T; ++t) {
          const int c = sub + lpr * t;
          if (valid && c < nchunk) {
            const uint4 u = row[c];
            const unsigned w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              __half2 g[2];
              e4m3x4_to_h2(w[k], g[0], g[1]);
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                ha[k] = __hfma2(g[h], xrr[t][2 * k + h], ha[k]);  // (gr xr, gi xr)
                hb[k] = __hfma2(g[h], xii[t][2 * k + h], hb[k]);  // (gr xi, gi xi)
              }
            }
          }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float2 fa = __half22float2(ha[k]), fb = __half22float2(hb[k]);
          ar += fa.x - fb.y;
          ai += fb.x + fa.y;
        }
        for (int o = lpr / 2; o > 0; o >>= 1) {
          ar += __shfl_xor_sync(0xffffffffu, ar, o);
          ai += __shfl_xor_sync(0xffffffffu, ai, o);
        }
        if (valid && sub == 0) {
          const float sc = a.scale[vec * a.nblk + (f - (vec_end - a.rows_per_vec)) / 256] * x_unscale;
          ay[f] = make_float2(ar * sc, ai * sc);
        }
      } else {
        // The order of k_stream_multi (chunk c on lane c mod 32, one chain per
        // component and lane, then the lanes added over xor 16, 8, .. 1; a long
        // row's blocks of slabs each by itself, then one after the other), so
        // that a rupture's result does not depend on the batch.  A short row's
        // lane holds four of those lanes' chunks: with 16 lanes per row the
        // chunks t and t + 2 are one chain, with fewer all four are apart.
        constexpr int H = SHORT ? 2 : 1;  // chains per lane and component
        float first_a = 0.f, first_i = 0.f;  // a long row's first block (R = 1)
        float xa[H][R], xi[H][R], sa[H][R], si[H][R];
#pragma unroll
        for (int h = 0; h < H; ++h)
#pragma unroll
          for (int b = 0; b < R; ++b) xa[h][b] = xi[h][b] = sa[h][b] = si[h][b] = 0.f;
#pragma unroll
        for (int t = 0; t < T; ++t) {
          const int c = sub + lpr * t;
          if (!SHORT && t == BLK) {
            first_a = xa[0][0], first_i = xi[0][0];
            xa[0][0] = xi[0][0] = 0.f;
          }
          if (SHORT && t == 2 && lpr < 16) {
#pragma unroll
            for (int h = 0; h < H; ++h)
#pragma unroll
              for (int b = 0; b < R; ++b) {
                sa[h][b] = xa[h][b];
                si[h][b] = xi[h][b];
                xa[h][b] = xi[h][b] = 0.f;
              }
          }
          if ((!SHORT || valid) && (t < 2 * BLK - 1 || c < nchunk)) {
            float2 g[C];
            CH::unpack(row[c], g);
            if (HILO) {
              float2 gl[C];
              CH::unpack(row_lo[c], gl);
#pragma unroll
              for (int q = 0; q < C; ++q) g[q] = cadd(g[q], gl[q]);
            }
#pragma unroll
            for (int q = 0; q < C; ++q) {
#pragma unroll
              for (int b = 0; b < R; ++b) {
                cmac(g[q], xr[b][t][q], xa[t % H][b], xi[t % H][b]);
              }
            }
          }
        }
        float ar[R], ai[R];
#pragma unroll
        for (int b = 0; b < R; ++b) {
          ar[b] = SHORT ? (sa[0][b] + xa[0][b]) + (sa[H - 1][b] + xa[H - 1][b]) : xa[0][b];
          ai[b] = SHORT ? (si[0][b] + xi[0][b]) + (si[H - 1][b] + xi[H - 1][b]) : xi[0][b];
        }
        if constexpr (SHORT) {
          for (int o = lpr / 2; o > 0; o >>= 1) {
#pragma unroll
            for (int b = 0; b < R; ++b) {
              ar[b] += __shfl_xor_sync(0xffffffffu, ar[b], o);
              ai[b] += __shfl_xor_sync(0xffffffffu, ai[b], o);
            }
          }
          if (valid && sub == 0) {
#pragma unroll
            for (int b = 0; b < R; ++b)
              if (R == 1 || b < a.nb) ay[b * a.y_ldb + f] = make_float2(ar[b], ai[b]);
          }
        } else {
          // reduce-scatter: lane bit 16 selects the block, bit 8 the component
          const bool last = (lane & 16) != 0, im = (lane & 8) != 0;
          float re = (last ? ar[0] : first_a) + __shfl_xor_sync(0xffffffffu, last ? first_a : ar[0], 16);
          float iv = (last ? ai[0] : first_i) + __shfl_xor_sync(0xffffffffu, last ? first_i : ai[0], 16);
          float v = (im ? iv : re) + __shfl_xor_sync(0xffffffffu, im ? re : iv, 8);
#pragma unroll
          for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
          v += __shfl_xor_sync(0xffffffffu, v, 16);  // the two blocks
          if ((lane & ~8) == 0) reinterpret_cast<float*>(ay + f)[lane >> 3] = v;
        }
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(empty + s);
  }
}

template <int EL, bool HILO, bool SHORT, int R = 1, int BLK = 0>
cudaError_t launch_t(const StreamArgs& a, int num_sms, cudaStream_t st) {
  constexpr int C = Chunk<EL>::C;
  const int row_bytes = a.row_len * (16 / C);
  const int budget = HILO ? 32 * 1024 : 64 * 1024;
  int stage_rows = budget / row_bytes;
  if (stage_rows >= 8) stage_rows -= stage_rows % 8;
  if (stage_rows < 1) stage_rows = 1;
  const size_t smem = 128 + static_cast<size_t>(kStages) * stage_rows * row_bytes * (HILO ? 2 : 1);
  cudaError_t e = cudaFuncSetAttribute(k_stream_dot<EL, HILO, SHORT, R, BLK>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  long long grid = num_sms;
  if (grid > a.F) grid = a.F;
  if (grid < 1) grid = 1;
  const dim3 g(static_cast<unsigned>(grid), R == 1 ? static_cast<unsigned>(a.nb) : 1u);
  launch_next(k_stream_dot<EL, HILO, SHORT, R, BLK>, g, 32 * (stream_warps(SHORT, R) + 1), smem, st, a, stage_rows);
  return cudaGetLastError();
}

// Rows of at most 64 16-byte chunks (C complex entries each) take the
// lane-group variant.
bool short_rows(const StreamArgs& a, int C) { return a.row_len / C <= 64; }

}  // namespace

namespace {
// Rows of at most this many chunks stay on the lane groups in a batch.
constexpr int kShortestChunks = 16;
// Long rows of one rupture, by the slabs of their first block.
template <int EL, bool HILO, int BLK = 1>
cudaError_t launch_long(const StreamArgs& a, int num_sms, cudaStream_t st) {
  constexpr int C = Chunk<EL>::C, most = chain_slabs(kMaxRowLen / (32 * C));
  if constexpr (BLK < most)
    if (chain_slabs((a.row_len / C + 31) / 32) > BLK) return launch_long<EL, HILO, BLK + 1>(a, num_sms, st);
  return launch_t<EL, HILO, false, 1, BLK>(a, num_sms, st);
}
// One launch for a.nb ruptures of FP32 / BF16 storage (nb <= kStreamMulti).
template <int EL, bool HILO>
cudaError_t launch_plain(const StreamArgs& a, int num_sms, cudaStream_t st) {
  if (a.nb == 1)
    return short_rows(a, Chunk<EL>::C) ? launch_t<EL, HILO, true>(a, num_sms, st) : launch_long<EL, HILO>(a, num_sms, st);
  // A batch: k_stream_multi, whose warps take eight rows at about the same
  // cost however short they are; the shortest rows in lane groups here, at
  // most kMostVectors at a time (a lane holds its slices of every vector)
  if (a.row_len / Chunk<EL>::C > kShortestChunks) return launch_stream_multi(a, num_sms, st);
  constexpr int kMostVectors = EL == EL_FP32 ? 4 : 2;
  for (int b = 0; b < a.nb; b += kMostVectors) {
    StreamArgs h = a;
    h.nb = a.nb - b < kMostVectors ? a.nb - b : kMostVectors;
    h.x = a.x + b * a.x_ldb;
    h.y = a.y + b * a.y_ldb;
    const cudaError_t e = launch_t<EL, HILO, true, kMostVectors>(h, num_sms, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}
}  // namespace

cudaError_t launch_stream_dot(const StreamArgs& a, int num_sms, cudaStream_t st) {
  if (a.F <= 0 || a.nb <= 0) return cudaSuccess;
  if (a.row_len <= 0 || a.row_len > kMaxRowLen || (a.row_len % 8) != 0 || a.nb > kStreamMulti)
    return cudaErrorInvalidValue;
  switch (a.el) {
    case EL_FP32: return launch_plain<EL_FP32, false>(a, num_sms, st);
    case EL_BF16: return launch_plain<EL_BF16, false>(a, num_sms, st);
    case EL_BF16_HILO: return launch_plain<EL_BF16, true>(a, num_sms, st);
    case EL_FP8:
      return short_rows(a, 8) ? launch_t<EL_FP8, false, true>(a, num_sms, st)
                              : launch_t<EL_FP8, false, false>(a, num_sms, st);
    case EL_FP32_HILO: return launch_stream_df(a, num_sms, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace s2w
