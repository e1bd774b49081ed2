// sslbm_kernels.cu -- SSLBM time-step kernels (Sec. II.C, Eq. sslbm_final_clean with the
// sources of Eq. sources and the deceased update of Eq. rhoD).
//
//   step1_kernel    one FP64 step per launch, a cell per thread; neighbours come from L1/L2.  The FP32
//                   storages advance one step per launch in the streaming kernel (stream.cu).
//   pipe_kernel     (pipe_launch.cuh) K steps per launch (temporal blocking, K = 2..8) for
//                   FP32, FP32 deviation-S and FP32 split-S (a sixth plane); pipe_d2q9*.cu and
//                   pipe_vard.cu instantiate it for FP32 on the D2Q9 lattice (periodic, or no-flux with the
//                   bounce-back substituted into the row update) and on the varying-diffusion
//                   lattice (the scale rows in a static shared-memory ring), as a pipeline of
//                   K warps per
//                   CTA: warp s computes level s+1 of the time-step wavefront.  A CTA owns a
//                   128-column strip (4 columns per lane, 16-byte accesses) with a K-column halo
//                   on each side and streams down a segment of rows, two rows per step of the
//                   pipeline.  Warp 0 brings level-0 rows in with cp.async into a shared-memory
//                   ring three row pairs ahead; every level's output pair goes through a
//                   double-buffered shared-memory slot (dynamic shared memory) to the next
//                   warp, one CTA barrier per pair; the last warp writes level K to global
//                   memory.  Each warp keeps only its own level's rows in four register
//                   buffers (about 110 registers per thread), so two or more CTAs share an SM.
//                   x neighbours come from warp shuffles.  Rows and columns outside the domain
//                   are loaded as ghost images (periodic wrap or the even mirror extension),
//                   which the uniform stencil keeps consistent, so no boundary logic is needed
//                   inside the pipeline.  DRAM traffic is one read and one write of the five
//                   planes per K steps.
// The pipeline and the streaming kernel evaluate the same packed per-cell expressions
// (sslbm_internal.cuh), so a blocked launch gives the same bits as K one-step launches.
#include <atomic>

#include "bounds.cuh"
#include "pdl.cuh"
#include "sslbm_internal.cuh"
#include "pipe_launch.cuh"

SSLBM_OOB_ACCESSOR(kernels)

namespace sslbm {

namespace {

constexpr int kStep1Threads = 1024;

// One FP64 step, a cell per thread: the cells are numbered along the rows (x fastest), CTA b takes
// the `per` cells from b * per on.  Bound by the FP64 pipe (two lanes per SM): 38 operations per cell,
// 15.2 GLUPS at 2 GHz; wider accesses would not help, the pipe takes 16 times longer over a cell
// than its 21 loads do.  8192^2 13.95 GLUPS; two cells per thread with the earlier force_quot 11.8.
__global__ void __launch_bounds__(kStep1Threads) step1_kernel(const GridView g, const Coeffs<double> k,
                                                              const double* in, double* out, const int per) {
  pdl_enter();
  if ((int)threadIdx.x >= per) return;
  int64_t x, y;
  const int64_t i = (int64_t)blockIdx.x * per + threadIdx.x;
  if (g.nx <= 0x7fffffff && i <= 0x7fffffff) {
    const unsigned yy = (unsigned)i / (unsigned)g.nx;
    y = yy;
    x = (unsigned)i - yy * (unsigned)g.nx;
  } else {
    y = i / g.nx;
    x = i - y * g.nx;
  }
  if (y >= g.ny) return;
  const int64_t yu = link_index(y - 1, g.ny, g.bc), yd = link_index(y + 1, g.ny, g.bc);
  const int64_t xl = link_index(x - 1, g.nx, g.bc), xr = link_index(x + 1, g.nx, g.bc);
  if (!(SSLBM_IN(yu, 1, g.ny, 10) && SSLBM_IN(yd, 1, g.ny, 11) && SSLBM_IN(x, 1, g.nx, 12) &&
        SSLBM_IN(xl, 1, g.nx, 13) && SSLBM_IN(xr, 1, g.nx, 14)))
    return;
  const int64_t rc = y * g.pitch, o = rc + x;
  double c[5], l[4], r[4], u[4], d[4];
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    const double* P = in + f * g.plane;
    c[f] = P[o], l[f] = P[rc + xl], r[f] = P[rc + xr];
    u[f] = P[yu * g.pitch + x], d[f] = P[yd * g.pitch + x];
  }
  c[4] = in[4 * g.plane + o];
  double lap[4], n[5];
#pragma unroll
  for (int f = 0; f < 4; ++f) lap[f] = lap5(c[f], l[f], r[f], u[f], d[f]);
  seird_cell(k, c[0], c[1], c[2], c[3], c[4], lap[0], lap[1], lap[2], lap[3], n[0], n[1], n[2], n[3], n[4]);
#pragma unroll
  for (int f = 0; f < 5; ++f) out[f * g.plane + o] = n[f];
}

// Small grids (at most kStep1Threads cells per SM): one CTA per SM with an equal share of the cells,
// and enough shared memory reserved that an SM holds no more than two, one of this launch and one of
// the next: with small CTAs the dependent launch's go where there is room and some SMs get twice the
// work (200^2, us per step: 10.3 with 64 x 8 blocks of two cells, 8.2 with 64-thread CTAs, 10.6 with
// those and dependent launches, 5.2 with even shares).  Above 576 cells per SM (about 296^2) the
// registers, 56 per thread, leave room for one CTA, and the next launch starts when it ends; even
// shares stay ahead of 64-thread CTAs to the limit: 350^2 11.1 and 14.4, 394^2 13.3 and 14.5.  Only a step after a step is a dependent
// launch: after another kernel, two CTAs may go to one SM, and stay together from step to step (8.0).
// Larger grids: 64-thread CTAs.
cudaError_t launch_step1_fp64(const GridView& g, const void* coeffs, const void* in, void* out, bool chained,
                              cudaStream_t s) {
  constexpr size_t kReserve = 100 * 1024;
  static std::atomic<int> sms_of[64];  // multiprocessors; set after the kernel's shared-memory limit
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  int sms = sms_of[dev & 63].load(std::memory_order_acquire);
  if (!sms) {
    if ((e = cudaFuncSetAttribute(step1_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kReserve)) != cudaSuccess)
      return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    sms_of[dev & 63].store(sms, std::memory_order_release);
  }
  const int64_t cells = g.nx * g.ny;
  const bool even = cells <= (int64_t)kStep1Threads * sms;
  const int per = even ? (int)((cells + sms - 1) / sms) : 64;
  const int64_t ctas = (cells + per - 1) / per;  // up to 2^31 - 1: 1.4e11 cells, 5.5 TB per state
  if (ctas > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  return launch_pdl_if(chained, step1_kernel, dim3((unsigned)ctas), dim3((per + 31) / 32 * 32), even ? kReserve : 0, s,
                       g, *static_cast<const Coeffs<double>*>(coeffs), static_cast<const double*>(in),
                       static_cast<double*>(out), per);
}

}  // namespace

int blocked_default_seg_rows(int precision, const GridView& g, int depth) {
  if (precision == SSLBM_FP32) return default_seg_rows_mode<MODE_PLAIN>(g, depth);
  if (precision == SSLBM_FP32_DEV) return default_seg_rows_mode<MODE_DEV>(g, depth);
  if (precision == SSLBM_FP32_SPLIT) return default_seg_rows_mode<MODE_SPLIT>(g, depth);
  if (precision == SSLBM_FP32_KAHAN) return blocked_kahan_default_seg_rows(g, depth);
  return 0;
}

bool blocked_supported(int precision, const GridView&) {
  return precision == SSLBM_FP32 || precision == SSLBM_FP32_DEV || precision == SSLBM_FP32_SPLIT ||
         precision == SSLBM_FP32_KAHAN;
}

cudaError_t launch_sslbm_step1(int precision, const GridView& g, const void* coeffs, const void* in,
                               void* out, bool chained, cudaStream_t s) {
  switch (precision) {
    case SSLBM_FP64: return launch_step1_fp64(g, coeffs, in, out, chained, s);
    case SSLBM_FP32:
    case SSLBM_FP32_DEV:
    case SSLBM_FP32_SPLIT:
    case SSLBM_FP32_KAHAN: return launch_stream_d2q5(precision, g, coeffs, in, out, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_sslbm_blocked(int precision, const GridView& g, const void* coeffs,
                                 const void* in, void* out, int depth, int seg_rows, bool chained,
                                 cudaStream_t s) {
  if (precision == SSLBM_FP32)
    return launch_blocked_mode<MODE_PLAIN>(g, coeffs, in, out, depth, seg_rows, chained, s);
  if (precision == SSLBM_FP32_DEV)
    return launch_blocked_mode<MODE_DEV>(g, coeffs, in, out, depth, seg_rows, chained, s);
  if (precision == SSLBM_FP32_SPLIT)
    return launch_blocked_mode<MODE_SPLIT>(g, coeffs, in, out, depth, seg_rows, chained, s);
  if (precision == SSLBM_FP32_KAHAN) return launch_kahan_blocked(g, coeffs, in, out, depth, seg_rows, chained, s);
  return cudaErrorInvalidValue;
}

}  // namespace sslbm
