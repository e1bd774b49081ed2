// io_kernels.cu -- conversion between the caller's contiguous ny x nx planes and the
// solver's pitched storage, and the diagnostics reduction of Sec. II.C 'Mass conservation'
// (per-compartment totals in double precision, peak infected density).
#include <float.h>
#include <stdint.h>

#include "bounds.cuh"
#include "diag.cuh"
#include "pdl.cuh"
#include "sslbm_internal.cuh"

SSLBM_OOB_ACCESSOR(io)

namespace sslbm {

namespace {

// The caller's contiguous ny x nx planes (type U) to or from the pitched planes (type T), planes c0
// .. c0 + gridDim.z - 1 of a state in one launch.  A stored value is v - comp[c] for the first n_comp
// planes (comps != NULL: on write the rounding residue of the value, so that value - compensation
// reproduces the input), and s_ref - v for plane 0 under dev_S; both are evaluated in double.  Planes
// stored as given are copied.
// Bound by HBM on large grids and by the launch on small ones: a launch per plane (or a strided
// copy per plane) cost an ensemble of 32 scenarios 957 us to write and 1232 to read, now 186 and 524;
// the strided device copies of an 8192^2 state took 1.33 ms each way, this 0.39.  Conversions are bound
// by the FP64 pipe; 3786 x 4055, us, the earlier launch per plane and this: double to Kahan 718 and 554,
// FP64 to float 339 and 162, one plane of deviations to double 70 and 60; 64 x 20000, Kahan to double 72
// and 38.
// vec: nx is a multiple of 4 and the caller's planes are 16-byte aligned, so a thread moves four
// cells at a time; else single cells.  A CTA is bx columns (cells or groups of four) by blockDim.x / bx
// rows, so that narrow grids keep its lanes busy; on large grids a thread has the loads of four such
// rows in flight before it stores the first, on small ones the FP64 arithmetic of the compensated
// storages is spread over more and smaller CTAs.
template <int N, typename T>
__device__ __forceinline__ void ld_cells(T (&r)[N], const T* p) {
  if constexpr (N == 1) {
    r[0] = *p;
  } else if constexpr (sizeof(T) == 4) {
    *reinterpret_cast<float4*>(r) = *reinterpret_cast<const float4*>(p);
  } else {
    *reinterpret_cast<double2*>(r) = *reinterpret_cast<const double2*>(p);
    *reinterpret_cast<double2*>(r + 2) = *reinterpret_cast<const double2*>(p + 2);
  }
}
template <int N, typename T>
__device__ __forceinline__ void st_cells(T* p, const T (&r)[N]) {
  if constexpr (N == 1) {
    *p = r[0];
  } else if constexpr (sizeof(T) == 4) {
    *reinterpret_cast<float4*>(p) = *reinterpret_cast<const float4*>(r);
  } else {
    *reinterpret_cast<double2*>(p) = *reinterpret_cast<const double2*>(r);
    *reinterpret_cast<double2*>(p + 2) = *reinterpret_cast<const double2*>(r + 2);
  }
}

constexpr int kIoThreads = 256;

// What a stored value is: the value, value - compensation, or s_ref - the value.  Each kind is a loop of
// its own, so that values stored as given see no FP64 arithmetic, of which this GPU has little.
enum { IO_PLAIN, IO_COMP, IO_DEV };

template <typename T, typename U, int N>
struct IoCells {
  alignas(16) T hi[N], lo[N];
  alignas(16) U v[N];
};

template <typename T, typename U, bool WRITE, int KIND, int N, int ROWS>
__device__ __forceinline__ void io_rows(const GridView& g, U* up, T* pp, T* cp, const double s_ref, const int bx) {
  const int64_t x = (int64_t)N * ((int64_t)blockIdx.x * bx + ((int)threadIdx.x & (bx - 1)));
  if (x >= g.nx) return;
  const int by = (int)blockDim.x / bx;
  for (int64_t y0 = (int64_t)blockIdx.y * ROWS * by + (int)threadIdx.x / bx; y0 < g.ny;
       y0 += (int64_t)gridDim.y * ROWS * by) {
    IoCells<T, U, N> q[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      const int64_t y = y0 + r * by;
      if (y >= g.ny) continue;
      if (WRITE) {
        ld_cells<N>(q[r].v, up + y * g.nx + x);
      } else {
        ld_cells<N>(q[r].hi, pp + y * g.pitch + x);
        if (KIND == IO_COMP) ld_cells<N>(q[r].lo, cp + y * g.pitch + x);
      }
    }
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      const int64_t y = y0 + r * by;
      if (y >= g.ny) continue;
#pragma unroll
      for (int e = 0; e < N; ++e) {
        if (WRITE) {
          if (KIND == IO_PLAIN) {
            q[r].hi[e] = (T)q[r].v[e];
          } else {
            const double v = KIND == IO_DEV ? s_ref - (double)q[r].v[e] : (double)q[r].v[e];
            q[r].hi[e] = (T)v;
            if (KIND == IO_COMP) q[r].lo[e] = (T)((double)q[r].hi[e] - v);
          }
        } else if (KIND == IO_PLAIN) {
          q[r].v[e] = (U)q[r].hi[e];
        } else {
          q[r].v[e] = (U)(KIND == IO_DEV ? s_ref - (double)q[r].hi[e] : (double)q[r].hi[e] - (double)q[r].lo[e]);
        }
      }
      if (WRITE) {
        st_cells<N>(pp + y * g.pitch + x, q[r].hi);
        if (KIND == IO_COMP) st_cells<N>(cp + y * g.pitch + x, q[r].lo);
      } else {
        st_cells<N>(up + y * g.nx + x, q[r].v);
      }
    }
  }
}

template <typename T, typename U, bool WRITE, int N, int ROWS>
__global__ void __launch_bounds__(kIoThreads) planes_io_kernel(const GridView g, U* user, T* planes, T* comps,
                                                               const int n_comp, const int c0, const int dev_S,
                                                               const double s_ref, const int bx) {
  pdl_enter();
  const int c = c0 + (int)blockIdx.z;
  U* up = user + (int64_t)blockIdx.z * g.nx * g.ny;
  T* pp = planes + (int64_t)blockIdx.z * g.plane;
  if (comps != nullptr && c < n_comp)
    io_rows<T, U, WRITE, IO_COMP, N, ROWS>(g, up, pp, comps + (int64_t)blockIdx.z * g.plane, s_ref, bx);
  else if (dev_S && c == 0)
    io_rows<T, U, WRITE, IO_DEV, N, ROWS>(g, up, pp, nullptr, s_ref, bx);
  else
    io_rows<T, U, WRITE, IO_PLAIN, N, ROWS>(g, up, pp, nullptr, s_ref, bx);
}

template <typename T, typename U, bool WRITE>
cudaError_t planes_io_t(const GridView& g, void* user, void* planes, void* comps, int n_comp, int c0, int nplanes,
                        int dev_S, double s_ref, cudaStream_t s) {
  const bool vec = g.nx % 4 == 0 && reinterpret_cast<uintptr_t>(user) % 16 == 0;
  const int64_t cols = vec ? g.nx / 4 : g.nx;
  // threads per CTA, columns (a power of two) and rows per thread: the largest CTAs of which there are
  // enough for the GPU
  int threads = 0, rows = 0, bx = 0;
  int64_t gx = 0, gy = 0;
  for (int t = 0; t < 3; ++t) {
    threads = t < 2 ? kIoThreads : 64, rows = t == 0 ? 4 : 1;
    for (bx = 8; bx < threads && bx < cols;) bx *= 2;
    gx = (cols + bx - 1) / bx;
    gy = (g.ny + (int64_t)rows * (threads / bx) - 1) / ((int64_t)rows * (threads / bx));
    if (gx * gy * nplanes >= 1024) break;
  }
  const dim3 grid((unsigned)gx, (unsigned)(gy < 65535 ? gy : 65535), (unsigned)nplanes);
  auto kern = vec ? (rows == 4 ? planes_io_kernel<T, U, WRITE, 4, 4> : planes_io_kernel<T, U, WRITE, 4, 1>)
                  : (rows == 4 ? planes_io_kernel<T, U, WRITE, 1, 4> : planes_io_kernel<T, U, WRITE, 1, 1>);
  return launch_pdl(kern, grid, dim3(threads), 0, s, g, static_cast<U*>(user), static_cast<T*>(planes),
                    static_cast<T*>(comps), n_comp, c0, dev_S, s_ref, bx);
}

template <bool WRITE>
cudaError_t planes_io(int precision, const GridView& g, void* user, int dtype, void* planes, void* comps, int n_comp,
                      int c0, int nplanes, int dev_S, double s_ref, cudaStream_t s) {
  const bool t64 = precision == SSLBM_FP64, u64 = dtype == SSLBM_DT_F64;
  if (t64)
    return u64 ? planes_io_t<double, double, WRITE>(g, user, planes, comps, n_comp, c0, nplanes, dev_S, s_ref, s)
               : planes_io_t<double, float, WRITE>(g, user, planes, comps, n_comp, c0, nplanes, dev_S, s_ref, s);
  return u64 ? planes_io_t<float, double, WRITE>(g, user, planes, comps, n_comp, c0, nplanes, dev_S, s_ref, s)
             : planes_io_t<float, float, WRITE>(g, user, planes, comps, n_comp, c0, nplanes, dev_S, s_ref, s);
}

// Per-block partial totals of the five compartments and the maximum of I.
// LAYOUT 0: SSLBM planes (value minus Kahan compensation when comp != nullptr);
// LAYOUT 1: BGK populations, rho^C = sum_i f_i^C, and D in plane 20.
template <typename T, int LAYOUT>
__global__ void __launch_bounds__(256) diag_partial_kernel(const GridView g,
                                                           const T* __restrict__ st,
                                                           const T* __restrict__ comp,
                                                           double* __restrict__ partials, int n_comp) {
  double v[kDiagSlots] = {0.0, 0.0, 0.0, 0.0, 0.0, -DBL_MAX};
  for (int64_t y = blockIdx.x; y < g.ny; y += gridDim.x) {
    for (int64_t x = threadIdx.x; x < g.nx; x += blockDim.x) {
      const int64_t idx = y * g.pitch + x;
      double r[5];
      if (LAYOUT == 0) {
#pragma unroll
        for (int c = 0; c < 5; ++c) {
          r[c] = (double)st[c * g.plane + idx];
          if (comp && c < n_comp) r[c] -= (double)comp[c * g.plane + idx];
        }
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          T a = st[(c * 5) * g.plane + idx];
#pragma unroll
          for (int i = 1; i < 5; ++i) a = add_rn(a, st[(c * 5 + i) * g.plane + idx]);
          r[c] = (double)a;
        }
        r[4] = (double)st[20 * g.plane + idx];
      }
#pragma unroll
      for (int c = 0; c < 5; ++c) v[c] += r[c];
      v[5] = fmax(v[5], r[2]);
    }
  }
  block_reduce6(v);
  if (threadIdx.x == 0 && SSLBM_IN(blockIdx.x, 1, kDiagBlocks, 31)) {
#pragma unroll
    for (int j = 0; j < kDiagSlots; ++j) partials[blockIdx.x * kDiagSlots + j] = v[j];
  }
}

template <int LAYOUT, int NCOMP>
__global__ void __launch_bounds__(256) diag_partial_f32x4_kernel(const GridView g, const float* __restrict__ st,
                                                                 const float* __restrict__ comp,
                                                                 double* __restrict__ partials) {
  diag_rows_f32x4<LAYOUT, NCOMP>(g, st, comp, (int)blockIdx.x, (int)gridDim.x, partials + blockIdx.x * kDiagSlots);
}

// Sum of the per-block partials in a fixed order (deterministic).
__global__ void __launch_bounds__(256) diag_final_kernel(const double* __restrict__ partials,
                                                         int nblocks, double* __restrict__ result) {
  diag_total(partials, nblocks, result);
}

}  // namespace

cudaError_t launch_planes_write(int precision, const GridView& g, const void* src, int src_dtype, void* planes,
                                void* comps, int n_comp, int c0, int nplanes, int dev_S, double s_ref, cudaStream_t s) {
  return planes_io<true>(precision, g, const_cast<void*>(src), src_dtype, planes, comps, n_comp, c0, nplanes, dev_S,
                         s_ref, s);
}

cudaError_t launch_planes_read(int precision, const GridView& g, const void* planes, const void* comps, int n_comp,
                               int c0, int nplanes, int dev_S, double s_ref, void* dst, int dst_dtype, cudaStream_t s) {
  return planes_io<false>(precision, g, dst, dst_dtype, const_cast<void*>(planes), const_cast<void*>(comps), n_comp,
                          c0, nplanes, dev_S, s_ref, s);
}

cudaError_t launch_diagnostics(int precision, int layout, const GridView& g, const void* planes,
                               const void* comp_planes, double* partials, double* result,
                               cudaStream_t s, int n_comp) {
  if (!comp_planes) n_comp = 0;
  if (n_comp != 0 && n_comp != 1 && n_comp != 5) return cudaErrorInvalidValue;
  const int64_t blocks =
      precision == SSLBM_FP64 || layout == 1 || n_comp == 5 ? diag_blocks_by_row(g.ny) : diag_blocks(g.nx, g.ny);
  if (precision == SSLBM_FP64) {
    if (layout == 0)
      diag_partial_kernel<double, 0><<<(unsigned)blocks, 256, 0, s>>>(
          g, (const double*)planes, (const double*)comp_planes, partials, n_comp);
    else
      diag_partial_kernel<double, 1><<<(unsigned)blocks, 256, 0, s>>>(g, (const double*)planes,
                                                                      nullptr, partials, 0);
  } else if (g.pitch % 4 == 0 && g.plane % 4 == 0 && reinterpret_cast<uintptr_t>(planes) % 16 == 0 &&
             reinterpret_cast<uintptr_t>(comp_planes) % 16 == 0) {
    const float* st = (const float*)planes;
    const float* cp = (const float*)comp_planes;
    if (layout == 1)
      diag_partial_f32x4_kernel<1, 0><<<(unsigned)blocks, 256, 0, s>>>(g, st, nullptr, partials);
    else if (n_comp == 5)
      diag_partial_f32x4_kernel<0, 5><<<(unsigned)blocks, 256, 0, s>>>(g, st, cp, partials);
    else if (n_comp == 1)
      diag_partial_f32x4_kernel<0, 1><<<(unsigned)blocks, 256, 0, s>>>(g, st, cp, partials);
    else
      diag_partial_f32x4_kernel<0, 0><<<(unsigned)blocks, 256, 0, s>>>(g, st, nullptr, partials);
  } else {
    if (layout == 0)
      diag_partial_kernel<float, 0><<<(unsigned)blocks, 256, 0, s>>>(
          g, (const float*)planes, (const float*)comp_planes, partials, n_comp);
    else
      diag_partial_kernel<float, 1><<<(unsigned)blocks, 256, 0, s>>>(g, (const float*)planes,
                                                                     nullptr, partials, 0);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  diag_final_kernel<<<1, 256, 0, s>>>(partials, (int)blocks, result);
  return cudaGetLastError();
}

cudaError_t launch_diag_final(const double* partials, int nblocks, double* result, cudaStream_t s) {
  if (nblocks < 1 || nblocks > kDiagBlocks) return cudaErrorInvalidValue;
  diag_final_kernel<<<1, 256, 0, s>>>(partials, nblocks, result);
  return cudaGetLastError();
}

namespace {
// One index check with no memory access behind it (site 999).
__global__ void oob_probe_kernel(long long v, long long limit) { (void)SSLBM_IN(v, 1, limit, 999); }
}  // namespace

cudaError_t launch_oob_probe(long long v, long long limit, cudaStream_t s) {
  oob_probe_kernel<<<1, 1, 0, s>>>(v, limit);
  return cudaGetLastError();
}

}  // namespace sslbm
