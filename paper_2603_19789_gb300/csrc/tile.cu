// tile.cu -- K steps per pass on grids too small to fill the GPU with the row pipeline: a CTA keeps
// a region of the grid in registers and advances it K steps (overlapped tiling in time).
//
// A region is 64 columns (two per lane: one warp spans a row) times 16 NR rows (NR per warp).  Its
// outer K rows and columns are a halo that is recomputed: after K steps the inner part is exact.
// x neighbours come from warp shuffles, rows within a warp from its registers, and each step the
// warps exchange only their first and last rows through shared memory, one barrier per step.
// Cells outside the domain are loaded as ghost images (periodic wrap or mirror), which the uniform
// stencil keeps consistent; the D2Q9 no-flux walls are substituted into the row update, as in the
// row pipeline.  The cell updates are the packed forms of the other kernels in the same order, so a
// pass gives the bits of K one-step launches.
//
// What bounds it: on small grids the launch and the load of the region (2 to 4.5 us per pass), and
// per step the FP32 arithmetic of the region's rows, halo included (0.38 us for 16 rows, 0.44 for
// 32, 0.77 for 64; 0.35 at 100% of the FP32 pipes for 64).  The row pipeline needs one barrier per
// two rows and 12 rows of fill whatever the grid, so a 128^2 pass of 4 steps takes 16.5 us there;
// here 14 steps take 9.7.  us per step of 40, pipeline (depth 4, without dependent launches) and tiles:
// 128^2 4.1 and 0.64, 512^2 4.6 and 1.2, 1000^2 5.9 and 3.7; 2048^2, where the pipeline stays ahead, 12.8 and
// 16.7; D2Q9 with walls 1500 x 1100 19.8 and 10.7; varying diffusion 1000^2 9.2 and 6.6.  Passes use programmatic dependent launch: the next one
// is resident and has its indices ready when the current one ends.
#include <cuda_runtime.h>

#include <atomic>

#include "bounds.cuh"
#include "pdl.cuh"
#include "sslbm_internal.cuh"
#include "tile.cuh"

SSLBM_OOB_ACCESSOR(tile)

namespace sslbm {
namespace {

constexpr int kTW = kTileWarps;     // warps per CTA
constexpr int kTCols = kTileCols;  // region columns

// planes with neighbours: the exchanged ones
constexpr int kTX = 4;

struct TileSmem {
  float2 ex[2][kTW][2][kTX][32];  // [step parity][warp][first, last row][plane][lane]
};

// ghost_index (sslbm_internal.cuh) in 32-bit arithmetic, one fold without a division: a region
// reaches past the domain by less than its own size, so only tiny grids need the general form.
__device__ __forceinline__ int ghost32(int i, int n, int bc) {
  if (i >= 0 && i < n) return i;
  const int j = bc == 0 ? (i < 0 ? i + n : i - n) : (i < 0 ? -1 - i : 2 * n - 1 - i);
  if (j >= 0 && j < n) return j;
  if (bc == 0) {
    const int r = i % n;
    return r < 0 ? r + n : r;
  }
  int r = (int)((unsigned)i % (2u * (unsigned)n));
  if (i < 0) {
    r = (int)((unsigned)(-(i + 1)) % (2u * (unsigned)n));
    r = 2 * n - 1 - r;
  }
  return r < n ? r : 2 * n - 1 - r;
}

// Neighbour values of a row: what lies left of the lane's first and right of its second column.
struct Side {
  float l[kTX], r[kTX];
};
__device__ __forceinline__ void sides(const float2* v, Side& s) {
#pragma unroll
  for (int f = 0; f < kTX; ++f) {
    s.l[f] = __shfl_up_sync(0xffffffffu, v[f].y, 1);
    s.r[f] = __shfl_down_sync(0xffffffffu, v[f].x, 1);
  }
}

// The link coefficients of a cell pair on the varying-diffusion lattice.
struct Links {
  float2 xp, xm, yp, ym;
};

// One row of the update: C (with D in C[4]) and its neighbour rows P, N (S, E, I, R) -> M.
template <int MODE>
__device__ __forceinline__ void tile_row(const Coeffs<float>& k, const float2* P, const float2* C, const float2* N,
                                         const Side& sP, const Side& sC, const Side& sN, const Links& q, bool wl,
                                         bool wr0, bool wr1, bool wd, bool wu, float2 (&M)[5]) {
  float2 lp[kTX];
#pragma unroll
  for (int f = 0; f < kTX; ++f) {
    const float2 c = C[f];
    if constexpr (MODE == MODE_D2Q9 || MODE == MODE_D2Q9_NOFLUX) {
      constexpr bool W = MODE == MODE_D2Q9_NOFLUX;
      // pair sums row[x-1] + row[x+1]; a link through a wall sees the cell itself
      auto pair = [&](const float2& v, float l, float r) {
        const float a0 = W && wl ? c.x : l, b0 = W && wr0 ? c.x : v.y, b1 = W && wr1 ? c.y : r;
        return make_float2(__fadd_rn(a0, b0), __fadd_rn(v.x, b1));
      };
      float2 Pv = P[f], Nv = N[f];
      float2 hP = pair(P[f], sP.l[f], sP.r[f]), hN = pair(N[f], sN.l[f], sN.r[f]);
      const float2 hC = pair(c, sC.l[f], sC.r[f]);
      if (W && wd) Pv = c, hP = add2(c, c);
      if (W && wu) Nv = c, hN = add2(c, c);
      lp[f] = mul2(fma2(splat2(-20.f), c, fma2(splat2(4.f), add2(hC, add2(Nv, Pv)), add2(hN, hP))), splat2(1.f / 6.f));
    } else if constexpr (MODE == MODE_VARD) {
      const float2 nc = neg2(c);
      const float2 t1 = mul2(q.xp, add2(make_float2(c.y, sC.r[f]), nc));
      const float2 t2 = mul2(q.yp, add2(N[f], nc));
      const float2 t3 = mul2(q.xm, add2(make_float2(sC.l[f], c.x), nc));
      const float2 t4 = mul2(q.ym, add2(P[f], nc));
      lp[f] = make_float2(__fadd_rn(__fadd_rn(t1.x, t3.x), __fadd_rn(t2.x, t4.x)),
                          __fadd_rn(__fadd_rn(t1.y, t3.y), __fadd_rn(t2.y, t4.y)));
    } else {
      const float2 lr = make_float2(__fadd_rn(sC.l[f], c.y), __fadd_rn(c.x, sC.r[f]));
      lp[f] = lap5x2(c, lr, P[f], N[f]);
    }
  }
  seird_cell2<MODE == MODE_DEV>(k, C[0], C[1], C[2], C[3], C[4], lp[0], lp[1], lp[2], lp[3], M[0], M[1], M[2], M[3],
                                M[4]);
}

template <int MODE, int NR>
__global__ void __launch_bounds__(32 * kTW, 1) tile_kernel(const GridView g, const Coeffs<float> k,
                                                           const float* in, float* out, const float* kx,
                                                           const float* ky, const int K, const int ntx) {
  constexpr int R = kTW * NR;
  constexpr bool Q9 = MODE == MODE_D2Q9 || MODE == MODE_D2Q9_NOFLUX;
  extern __shared__ __align__(16) unsigned char tile_smem[];
  TileSmem& sm = *reinterpret_cast<TileSmem*>(tile_smem);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int ke = (K + 1) & ~1;  // halo columns: even, so that a lane's pair is one aligned load
  const int nx = (int)g.nx, ny = (int)g.ny, bc = g.bc;
  const int x = (int)(blockIdx.x % ntx) * (kTCols - 2 * ke) - ke + 2 * lane;
  const int yr = (int)(blockIdx.x / ntx) * (R - 2 * K) - K + w * NR;  // the warp's first row
  const bool pair = x >= 0 && x + 1 < nx;
  const bool c0 = x >= -K && x < nx + K, c1 = x + 1 >= -K && x + 1 < nx + K;  // cells that can matter
  const int x0 = ghost32(x, nx, bc), x1 = ghost32(x + 1, nx, bc);

  pdl_enter();

  auto load = [&](const float* p, int64_t row) {
    float2 v = make_float2(0.f, 0.f);
    if (pair) {
      if (SSLBM_IN(x, 2, nx, 1)) v = *reinterpret_cast<const float2*>(p + row + x);
    } else {
      if (c0 && SSLBM_IN(x0, 1, nx, 2)) v.x = p[row + x0];
      if (c1 && SSLBM_IN(x1, 1, nx, 3)) v.y = p[row + x1];
    }
    return v;
  };
  float2 X[NR][5];
  Links q[MODE == MODE_VARD ? NR : 1];
#pragma unroll
  for (int j = 0; j < NR; ++j) {
    const int y = yr + j;
    const int yq = ghost32(y, ny, bc);
    const bool in_range = y >= -K && y < ny + K && SSLBM_IN(yq, 1, ny, 4);
#pragma unroll
    for (int f = 0; f < 5; ++f) X[j][f] = in_range ? load(in + f * g.plane, yq * g.pitch) : make_float2(0.f, 0.f);
  }
  if constexpr (MODE == MODE_VARD) {
    const float2 half = splat2(0.5f);
    float2 b[3];
    auto ky_row = [&](int y) {
      const int yq = ghost32(y, ny, bc);
      return y >= -K && y < ny + K && SSLBM_IN(yq, 1, ny, 5) ? load(ky, yq * g.pitch) : make_float2(0.f, 0.f);
    };
    b[0] = ky_row(yr - 1);
    b[1] = ky_row(yr);
#pragma unroll
    for (int j = 0; j < NR; ++j) {
      const int y = yr + j;
      const int yq = ghost32(y, ny, bc);
      const float2 a = y >= -K && y < ny + K && SSLBM_IN(yq, 1, ny, 6) ? load(kx, yq * g.pitch)
                                                                          : make_float2(0.f, 0.f);
      const float aL = __shfl_up_sync(0xffffffffu, a.y, 1), aR = __shfl_down_sync(0xffffffffu, a.x, 1);
      b[2] = ky_row(y + 1);
      q[j].xp = mul2(half, add2(a, make_float2(a.y, aR)));
      q[j].xm = mul2(half, add2(a, make_float2(aL, a.x)));
      q[j].yp = mul2(half, add2(b[1], b[2]));
      q[j].ym = mul2(half, add2(b[1], b[0]));
      b[0] = b[1];
      b[1] = b[2];
    }
  }
  const bool wl = MODE == MODE_D2Q9_NOFLUX && x == 0;
  const bool wr0 = MODE == MODE_D2Q9_NOFLUX && x == nx - 1, wr1 = MODE == MODE_D2Q9_NOFLUX && x + 1 == nx - 1;
  const bool beyond = yr >= ny + K;  // no row of this warp can matter

  for (int s = 0; s < K; ++s) {
    float2(&ex)[kTW][2][kTX][32] = sm.ex[s & 1];
#pragma unroll
    for (int f = 0; f < kTX; ++f) {
      ex[w][0][f][lane] = X[0][f];
      if (NR > 1) ex[w][1][f][lane] = X[NR - 1][f];
    }
    __syncthreads();
    // rows that the halo's shrinking validity still reaches: region rows [s + 1, R - s - 1)
    if (beyond || (w + 1) * NR <= s + 1 || w * NR >= R - s - 1) continue;
    float2 P[5], U[kTX], D[kTX];
#pragma unroll
    for (int f = 0; f < kTX; ++f) {
      U[f] = ex[w > 0 ? w - 1 : 0][NR > 1 ? 1 : 0][f][lane];
      D[f] = ex[w < kTW - 1 ? w + 1 : w][0][f][lane];
    }
#pragma unroll
    for (int f = 0; f < kTX; ++f) P[f] = U[f];
    Side sP, sC, sN;
    if (Q9) sides(P, sP);
    sides(X[0], sC);
#pragma unroll
    for (int j = 0; j < NR; ++j) {
      const float2* N = j + 1 < NR ? X[j + 1 < NR ? j + 1 : j] : D;
      if (Q9 || j + 1 < NR) sides(N, sN);
      float2 M[5];
      tile_row<MODE>(k, P, X[j], N, sP, sC, sN, q[MODE == MODE_VARD ? j : 0], wl, wr0, wr1,
                     MODE == MODE_D2Q9_NOFLUX && yr + j == 0, MODE == MODE_D2Q9_NOFLUX && yr + j == ny - 1, M);
#pragma unroll
      for (int f = 0; f < kTX; ++f) P[f] = X[j][f];
#pragma unroll
      for (int f = 0; f < 5; ++f) X[j][f] = M[f];
      sP = sC;
      sC = sN;
    }
  }

  // the exact part: columns [ke, 64 - ke), rows [K, R - K) of the region
  if (2 * lane < ke || 2 * lane >= kTCols - ke || x >= nx) return;
#pragma unroll
  for (int j = 0; j < NR; ++j) {
    const int rr = w * NR + j;
    const int y = yr + j;
    if (rr < K || rr >= R - K || y >= ny || !SSLBM_IN(y, 1, ny, 7) || !SSLBM_IN(x, 1, nx, 8)) continue;
    float* o = out + y * g.pitch + x;
#pragma unroll
    for (int f = 0; f < 5; ++f) {
      if (pair)
        *reinterpret_cast<float2*>(o + f * g.plane) = X[j][f];
      else
        o[f * g.plane] = X[j][f].x;
    }
  }
}

template <int MODE, int NR>
cudaError_t launch_t(const GridView& g, const void* coeffs, const void* in, void* out, const void* kx, const void* ky,
                     int K, cudaStream_t s) {
  // the dynamic shared-memory limit, set once per device (a bit per device in an atomic mask: host
  // threads may launch concurrently; setting it twice is harmless)
  static std::atomic<unsigned long long> done{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (!(done.load(std::memory_order_acquire) & (1ull << (dev & 63)))) {
    if ((e = cudaFuncSetAttribute(tile_kernel<MODE, NR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)sizeof(TileSmem))) != cudaSuccess)
      return e;
    done.fetch_or(1ull << (dev & 63), std::memory_order_release);
  }
  const int ke = (K + 1) & ~1;
  if (K < 1 || 2 * ke >= kTCols || 2 * K >= kTW * NR) return cudaErrorInvalidValue;
  const int64_t ntx = (g.nx + kTCols - 2 * ke - 1) / (kTCols - 2 * ke);
  const int64_t nty = (g.ny + kTW * NR - 2 * K - 1) / (kTW * NR - 2 * K);
  if (ntx * nty > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  return launch_pdl(tile_kernel<MODE, NR>, dim3((unsigned)(ntx * nty)), dim3(32 * kTW), sizeof(TileSmem), s, g,
                    *static_cast<const Coeffs<float>*>(coeffs), static_cast<const float*>(in), static_cast<float*>(out),
                    static_cast<const float*>(kx), static_cast<const float*>(ky), K, (int)ntx);
}

template <int MODE>
cudaError_t launch_nr(const GridView& g, const void* coeffs, const void* in, void* out, const void* kx, const void* ky,
                      int nr, int K, cudaStream_t s) {
  switch (nr) {
    case 1: return launch_t<MODE, 1>(g, coeffs, in, out, kx, ky, K, s);
    case 2: return launch_t<MODE, 2>(g, coeffs, in, out, kx, ky, K, s);
    case 4: return launch_t<MODE, 4>(g, coeffs, in, out, kx, ky, K, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

int sm_count() {
  static std::atomic<int> cache[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 1;
  int v = cache[dev & 63].load(std::memory_order_relaxed);
  if (!v && cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess)
    cache[dev & 63].store(v, std::memory_order_relaxed);
  return v > 0 ? v : 1;
}

cudaError_t launch_tile(int lattice, int precision, const GridView& g, const void* coeffs, const void* in, void* out,
                        const void* kx, const void* ky, int nr, int K, cudaStream_t s) {
  if (lattice == SSLBM_LATTICE_D2Q5 && precision == SSLBM_FP32)
    return launch_nr<MODE_PLAIN>(g, coeffs, in, out, nullptr, nullptr, nr, K, s);
  if (lattice == SSLBM_LATTICE_D2Q5 && precision == SSLBM_FP32_DEV)
    return launch_nr<MODE_DEV>(g, coeffs, in, out, nullptr, nullptr, nr, K, s);
  if (lattice == SSLBM_LATTICE_D2Q9 && precision == SSLBM_FP32)
    return g.bc == 0 ? launch_nr<MODE_D2Q9>(g, coeffs, in, out, nullptr, nullptr, nr, K, s)
                     : launch_nr<MODE_D2Q9_NOFLUX>(g, coeffs, in, out, nullptr, nullptr, nr, K, s);
  if (lattice == SSLBM_LATTICE_D2Q5_VARD && precision == SSLBM_FP32)
    return launch_nr<MODE_VARD>(g, coeffs, in, out, kx, ky, nr, K, s);
  return cudaErrorInvalidValue;
}

}  // namespace sslbm
