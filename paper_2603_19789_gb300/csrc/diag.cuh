// diag.cuh -- device side of the FP32 diagnostics reduction (totals of the five compartments in
// FP64, peak of I), shared by the single-grid (io_kernels.cu) and the ensemble (ensemble.cu) launches.
#pragma once
#include <float.h>
#include <stdint.h>

#include "bounds.cuh"
#include "sslbm_internal.cuh"

namespace sslbm {
namespace {

// Block-wide reduction of kDiagSlots values (sums of slots 0..4, max of slot 5) in a fixed
// order, result valid in thread 0.
__device__ void block_reduce6(double (&v)[kDiagSlots]) {
  __shared__ double sh[32][kDiagSlots];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
    for (int j = 0; j < 5; ++j) v[j] += __shfl_down_sync(0xffffffffu, v[j], off);
    v[5] = fmax(v[5], __shfl_down_sync(0xffffffffu, v[5], off));
  }
  if (lane == 0) {
#pragma unroll
    for (int j = 0; j < kDiagSlots; ++j) sh[warp][j] = v[j];
  }
  __syncthreads();
  if (warp == 0) {
    const int nw = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int j = 0; j < 5; ++j) v[j] = lane < nw ? sh[lane][j] : 0.0;
    v[5] = lane < nw ? sh[lane][5] : -DBL_MAX;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
      for (int j = 0; j < 5; ++j) v[j] += __shfl_down_sync(0xffffffffu, v[j], off);
      v[5] = fmax(v[5], __shfl_down_sync(0xffffffffu, v[5], off));
    }
  }
}

// Knuth's TwoSum: hi + lo <- hi + x with the rounding error of the addition carried into lo,
// so that FP32 arithmetic keeps the running sum to about twice FP32's precision.
__device__ __forceinline__ void two_sum_add(float& hi, float& lo, float x) {
  const float s = __fadd_rn(hi, x);
  const float bp = __fsub_rn(s, hi);
  const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(x, bp));
  hi = s;
  lo = __fadd_rn(lo, e);
}

// The FP32 partials of diag_partial_kernel without per-cell FP64 arithmetic (few FP64 units
// on this GPU): each thread reads 4 cells per plane at a time (16-byte loads; the pitch and
// the plane stride are multiples of 4) and keeps its share of the rows as a TwoSum pair per
// compartment, renormalised (Fast2Sum) after every 4 cells and added to the FP64 partial every
// kFlushRows rows and at the end.  After a renormalisation the pair's low part is at most half
// an ulp of its high part, so the pair's own rounding stays near FP32's unit roundoff squared
// per group of 4 cells.  (Adding the pair to FP64 after every row, the earlier form, took
// 265 us per 8192^2 call against 255 us now: GB300 has few FP64 units.)
// NCOMP: the first NCOMP compartments carry a compensation plane (0; 1 for the split S; 5 for
// Kahan), subtracted from the values.  The peak of I is taken in FP32 (the same value as in
// FP64), or in FP64 as value minus compensation when I has one.
// One of `nb` blocks of 256 threads: its rows' partial (6 doubles) goes to out.
template <int LAYOUT, int NCOMP>
__device__ __forceinline__ void diag_rows_f32x4(const GridView& g, const float* __restrict__ st,
                                                const float* __restrict__ comp, int block, int nb,
                                                double* __restrict__ out) {
  constexpr int kFlushRows = 16;
  double v[kDiagSlots] = {0.0, 0.0, 0.0, 0.0, 0.0, -DBL_MAX};
  float hi[5] = {0.f, 0.f, 0.f, 0.f, 0.f}, lo[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
  float pk = -FLT_MAX;
  int rows = 0;
  auto flush = [&]() {
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      v[c] += (double)hi[c] + (double)lo[c];
      hi[c] = lo[c] = 0.f;
    }
  };
  for (int64_t y = block; y < g.ny; y += nb) {
    for (int64_t x = 4 * (int64_t)threadIdx.x; x < g.nx; x += 4 * (int64_t)blockDim.x) {
      if (!SSLBM_IN(x, 4, g.pitch, 30)) continue;
      const int64_t idx = y * g.pitch + x;
      const int nv = g.nx - x < 4 ? (int)(g.nx - x) : 4;
      float r[5][4];
      if (LAYOUT == 0) {
#pragma unroll
        for (int c = 0; c < 5; ++c) {
          const float4 a = *reinterpret_cast<const float4*>(st + c * g.plane + idx);
          r[c][0] = a.x, r[c][1] = a.y, r[c][2] = a.z, r[c][3] = a.w;
        }
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          float4 a = *reinterpret_cast<const float4*>(st + (c * 5) * g.plane + idx);
#pragma unroll
          for (int i = 1; i < 5; ++i) {
            const float4 b = *reinterpret_cast<const float4*>(st + (c * 5 + i) * g.plane + idx);
            a.x = __fadd_rn(a.x, b.x), a.y = __fadd_rn(a.y, b.y), a.z = __fadd_rn(a.z, b.z), a.w = __fadd_rn(a.w, b.w);
          }
          r[c][0] = a.x, r[c][1] = a.y, r[c][2] = a.z, r[c][3] = a.w;
        }
        const float4 d = *reinterpret_cast<const float4*>(st + 20 * g.plane + idx);
        r[4][0] = d.x, r[4][1] = d.y, r[4][2] = d.z, r[4][3] = d.w;
      }
      float q[5][4];
      if (NCOMP > 0) {
#pragma unroll
        for (int c = 0; c < NCOMP; ++c) {
          const float4 b = *reinterpret_cast<const float4*>(comp + c * g.plane + idx);
          q[c][0] = b.x, q[c][1] = b.y, q[c][2] = b.z, q[c][3] = b.w;
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (j >= nv) break;
#pragma unroll
        for (int c = 0; c < 5; ++c) {
          two_sum_add(hi[c], lo[c], r[c][j]);
          if (c < NCOMP) two_sum_add(hi[c], lo[c], -q[c][j]);
        }
        if (NCOMP > 2)
          v[5] = fmax(v[5], (double)r[2][j] - (double)q[2][j]);
        else
          pk = fmaxf(pk, r[2][j]);
      }
#pragma unroll
      for (int c = 0; c < 5; ++c) {  // Fast2Sum: |lo| <= ulp(hi) / 2 again
        const float t = __fadd_rn(hi[c], lo[c]);
        lo[c] = __fsub_rn(lo[c], __fsub_rn(t, hi[c]));
        hi[c] = t;
      }
    }
    if (++rows == kFlushRows) {
      flush();
      rows = 0;
    }
  }
  flush();
  if (NCOMP <= 2) v[5] = fmax(v[5], (double)pk);
  block_reduce6(v);
  if (threadIdx.x == 0 && SSLBM_IN(block, 1, kDiagBlocks, 31)) {
#pragma unroll
    for (int j = 0; j < kDiagSlots; ++j) out[j] = v[j];
  }
}

// The fixed-order total of nblocks partials, by one block of 256 threads.
__device__ __forceinline__ void diag_total(const double* __restrict__ partials, int nblocks,
                                           double* __restrict__ result) {
  double v[kDiagSlots] = {0.0, 0.0, 0.0, 0.0, 0.0, -DBL_MAX};
  for (int b = threadIdx.x; b < nblocks; b += blockDim.x) {
#pragma unroll
    for (int j = 0; j < 5; ++j) v[j] += partials[b * kDiagSlots + j];
    v[5] = fmax(v[5], partials[b * kDiagSlots + 5]);
  }
  block_reduce6(v);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int j = 0; j < kDiagSlots; ++j) result[j] = v[j];
  }
}

// Blocks of the reduction of a grid that an ensemble may hold (FP32, deviation and split storages): a
// block's FP64 reduction costs as much as the sums of about 4096 cells, so a block takes up to four
// rows, but no more than that many cells (a block per row: 533 us for an ensemble of 32 scenarios, now
// 186; four rows each on 12000 x 300: 64 us, with a row each 42).  The same for a grid alone and in an
// ensemble, so that both add in the same order.  FP64 and the compensated storages, whose cells
// cost more, take a block per row.
__host__ __device__ inline int64_t diag_blocks(int64_t nx, int64_t ny) {
  const int64_t rows = nx >= 4096 ? 1 : nx >= 2048 ? 2 : 4, b = (ny + rows - 1) / rows;
  return b < 1 ? 1 : b < kDiagBlocks ? b : kDiagBlocks;
}
__host__ __device__ inline int64_t diag_blocks_by_row(int64_t ny) { return ny < kDiagBlocks ? ny : kDiagBlocks; }

}  // namespace
}  // namespace sslbm
