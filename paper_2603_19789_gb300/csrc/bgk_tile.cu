// bgk_tile.cu -- K BGK steps per pass in FP32 (Sec. II.B, Eq. pdf): a CTA keeps a region of the grid's
// populations in registers and collides and streams it K times (overlapped tiling in time).
//
// A region is 64 columns (two per lane: a warp spans a row) times 2 NW rows (two per warp), its outer K
// rows and columns a halo that is recomputed.  A step collides every cell in place, then streams:
// along x by warp shuffles, along y within a warp by renaming, and between warps by exchanging the
// populations that cross (f_2 of the last row up, f_4 of the first row down) through shared memory,
// one barrier per step.  Periodic halos are loaded wrapped; at a no-flux wall a population that
// would leave returns in the opposite direction (halfway bounce-back), so cells outside the domain
// are never read.  The operations and their order are those of bgk_step_kernel, so a pass gives
// the bits of K of its launches.
//
// What bounds it: one step per launch moves 168 bytes per cell and step (39.5 GLUPS is 99% of HBM); a
// pass moves the same once for K steps, 42 bytes per cell and step at four, which is 46% of HBM at
// 2048^2.  The rest is instruction issue (170 operations per cell and step, half of them on packed
// pairs, on a third more cells than are written) and the exchange of each step, so deeper passes gain
// nothing.  Per step, one step per launch and four per pass: 2048^2 107.6 and 57.1 us, 4096^2 419 and 221 (76
// GLUPS), 200^2 4.3 and 2.3; two steps 72.9 at 2048^2, three 58.3, six 57.1.
#include <cuda_runtime.h>

#include "bounds.cuh"
#include "pdl.cuh"
#include "sslbm_internal.cuh"

SSLBM_OOB_ACCESSOR(bgk_tile)

namespace sslbm {
namespace {

constexpr int kBCols = 64;

// Collision of a cell pair: f[c][i] <- f + (w rho - f)/tau + w Psi dt; D <- D + phi gamma I dt.
__device__ __forceinline__ void collide2(const Coeffs<float>& k, float2 (&f)[4][5], float2& D) {
  float2 rho[4], psi[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) rho[c] = add2(add2(add2(add2(f[c][0], f[c][1]), f[c][2]), f[c][3]), f[c][4]);
  const float2 F = force_dt2(k, rho[0], rho[1], rho[2], rho[3]);
  psi[0] = neg2(F);
  psi[1] = fma2(splat2(-k.adt), rho[1], F);
  psi[2] = fma2(splat2(k.adt), rho[1], neg2(mul2(splat2(k.gdt), rho[2])));
  psi[3] = mul2(splat2(k.rdt), rho[2]);
  D = fma2(splat2(k.ddt), rho[2], D);
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      const float2 w = splat2(i == 0 ? 1.f / 3.f : 1.f / 6.f);
      const float2 relax = mul2(fma2(w, rho[c], neg2(f[c][i])), splat2(k.itau[c]));
      // scalar adds: a packed add of a packed product may be fused into one operation
      const float2 a = make_float2(__fadd_rn(f[c][i].x, relax.x), __fadd_rn(f[c][i].y, relax.y));
      f[c][i] = fma2(w, psi[c], a);
    }
}

template <int NW>
__global__ void __launch_bounds__(32 * NW, NW > 8 ? 1 : 2) bgk_tile_kernel(const GridView g, const Coeffs<float> k,
                                                                          const float* fin, float* fout, const int K,
                                                                          const int ntx) {
  constexpr int R = 2 * NW;
  // [step parity][warp][f_2 of the last row, f_4 of the first][compartment][lane]
  __shared__ float2 ex[2][NW][2][4][32];
  const int nx = (int)g.nx, ny = (int)g.ny;
  const bool walls = g.bc != 0;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int ke = (K + 1) & ~1;  // halo columns: even, so that a lane's pair is one aligned access
  const int x = (int)(blockIdx.x % ntx) * (kBCols - 2 * ke) - ke + 2 * lane;
  const int yr = (int)(blockIdx.x / ntx) * (R - 2 * K) - K + 2 * w;
  const bool pair = x >= 0 && x + 1 < nx;
  // position of a (halo) column or row, -1 where nothing is read: beyond a wall, or further out
  // than K steps reach
  auto pos = [&](int i, int n) {
    if (i >= 0 && i < n) return i;
    if (walls || i < -K || i >= n + K) return -1;
    const int r = i % n;
    return r < 0 ? r + n : r;
  };
  const int x0 = pos(x, nx), x1 = pos(x + 1, nx);
  pdl_enter();

  float2 f[2][4][5], D[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int yq = pos(yr + j, ny);
    const bool row_ok = yq >= 0 && SSLBM_IN(yq, 1, ny, 1);
    const float* row = fin + (int64_t)(yq < 0 ? 0 : yq) * g.pitch;
    auto load = [&](int plane) {
      float2 v = make_float2(0.f, 0.f);
      const float* p = row + plane * g.plane;
      if (row_ok && pair) {
        if (SSLBM_IN(x, 2, nx, 2)) v = *reinterpret_cast<const float2*>(p + x);
      } else if (row_ok) {
        if (x0 >= 0 && SSLBM_IN(x0, 1, nx, 3)) v.x = p[x0];
        if (x1 >= 0 && SSLBM_IN(x1, 1, nx, 4)) v.y = p[x1];
      }
      return v;
    };
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int i = 0; i < 5; ++i) f[j][c][i] = load(c * 5 + i);
    D[j] = load(20);
  }
  const bool wl = walls && x == 0;                                         // column 0 is x = 0
  const bool wr0 = walls && x == nx - 1, wr1 = walls && x + 1 == nx - 1;   // column 0 / 1 is x = nx - 1

  for (int s = 0; s < K; ++s) {
    collide2(k, f[0], D[0]);
    collide2(k, f[1], D[1]);
    float2(&e)[NW][2][4][32] = ex[s & 1];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      e[w][0][c][lane] = f[1][c][2];
      e[w][1][c][lane] = f[0][c][4];
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      // the rows beyond the warp's two; the region's outermost receive a leftover that no written
      // cell depends on
      const float2 below = e[w > 0 ? w - 1 : 0][0][c][lane], above = e[w < NW - 1 ? w + 1 : w][1][c][lane];
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const float2 f1 = f[j][c][1], f3 = f[j][c][3];
        const float l = __shfl_up_sync(0xffffffffu, f1.y, 1), r = __shfl_down_sync(0xffffffffu, f3.x, 1);
        f[j][c][1] = make_float2(wl ? f3.x : l, f1.x);
        f[j][c][3] = make_float2(wr0 ? f1.x : f3.y, wr1 ? f1.y : r);
      }
      const float2 a2 = f[0][c][2], b2 = f[1][c][2], a4 = f[0][c][4], b4 = f[1][c][4];
      f[0][c][2] = walls && yr == 0 ? a4 : below;
      f[1][c][2] = walls && yr + 1 == 0 ? b4 : a2;
      f[0][c][4] = walls && yr == ny - 1 ? a2 : b4;
      f[1][c][4] = walls && yr + 1 == ny - 1 ? b2 : above;
    }
  }

  // the exact part: columns [ke, 64 - ke), rows [K, R - K) of the region
  if (2 * lane < ke || 2 * lane >= kBCols - ke || x >= nx) return;
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int rr = 2 * w + j, y = yr + j;
    if (rr < K || rr >= R - K || y >= ny || !SSLBM_IN(y, 1, ny, 5) || !SSLBM_IN(x, 1, nx, 6)) continue;
    float* o = fout + (int64_t)y * g.pitch + x;
    auto store = [&](int plane, float2 v) {
      if (pair)
        *reinterpret_cast<float2*>(o + plane * g.plane) = v;
      else
        o[plane * g.plane] = v.x;
    };
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int i = 0; i < 5; ++i) store(c * 5 + i, f[j][c][i]);
    store(20, D[j]);
  }
}

template <int NW>
cudaError_t launch_t(const GridView& g, const void* coeffs, const void* f_in, void* f_out, int K, cudaStream_t s) {
  const int ke = (K + 1) & ~1;
  const int64_t ntx = (g.nx + kBCols - 2 * ke - 1) / (kBCols - 2 * ke);
  const int64_t nty = (g.ny + 2 * NW - 2 * K - 1) / (2 * NW - 2 * K);
  if (K < 1 || K >= NW || ntx * nty > 0x7fffffffLL || g.nx > (1 << 30) || g.ny > (1 << 30))
    return cudaErrorInvalidConfiguration;
  return launch_pdl(bgk_tile_kernel<NW>, dim3((unsigned)(ntx * nty)), dim3(32 * NW), 0, s, g,
                    *static_cast<const Coeffs<float>*>(coeffs), static_cast<const float*>(f_in),
                    static_cast<float*>(f_out), K, (int)ntx);
}

}  // namespace

namespace {

// regions of 2 NW rows that cover the grid with K steps per pass
int64_t regions(const GridView& g, int K, int nw) {
  const int ke = (K + 1) & ~1;
  return (g.nx + kBCols - 2 * ke - 1) / (kBCols - 2 * ke) * ((g.ny + 2 * nw - 2 * K - 1) / (2 * nw - 2 * K));
}

}  // namespace

cudaError_t launch_bgk_tile(const GridView& g, const void* coeffs, const void* f_in, void* f_out, int K, cudaStream_t s) {
  // regions of 16 rows (two CTAs per SM) while they make at most one wave, else of 32, whose halo is
  // relatively smaller: four steps per pass, us per step with 16 and 32 rows: 200^2 2.3 and 3.0,
  // 501 x 377 4.3 and 3.2, 2048^2 58.8 and 57.1, 4096^2 229 and 221
  return regions(g, K, 8) <= 2 * (int64_t)sm_count() ? launch_t<8>(g, coeffs, f_in, f_out, K, s)
                                                     : launch_t<16>(g, coeffs, f_in, f_out, K, s);
}

bool bgk_pair_pays(const GridView& g) {
  const int64_t sms = sm_count(), waves = (regions(g, 2, 16) + sms - 1) / sms;
  return regions(g, 2, 8) <= 2 * sms || 8.6 * (double)waves < 2 * 168 / 5.6e6 * (double)g.nx * (double)g.ny;
}

}  // namespace sslbm
