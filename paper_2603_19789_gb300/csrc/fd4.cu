// fd4.cu -- the fourth-order finite-difference reference of Sec. III on the GPU (and, for the
// cost comparison of Sec. IV, its second-order counterpart, sslbm_fd4_set_order): classical
// RK4 in time and the fourth-order centred Laplacian in space,
//   L4 u = sum over axes of (-u[-2] + 16 u[-1] - 30 u[0] + 16 u[+1] - u[+2]) / (12 dx^2),
//   d/dt C = Psi^C + d^C L4 C (C = S, E, I, R),  d/dt D = phi gamma I   (Eqs. EqSEIRD_S..D),
// with the reactions of Eq. (sources) evaluated at every stage.  Ghost cells: periodic wrap,
// or (no-flux) the even reflection about the boundary face, u[-1] = u[0], u[-2] = u[1].
//
// One step is four stage launches in FP64; in FP32 two launches of two stages each, or the four on grids
// where those are faster (plan_step).  Stage s reads the previous stage's state with the stencil and
// writes the next stage's state and the running sum of the slopes:
//   s = 1: acc = k1,         t = u + (dt/2) k1
//   s = 2: acc = acc + 2 k2, t = u + (dt/2) k2
//   s = 3: acc = acc + 2 k3, t = u + dt k3
//   s = 4: u = u + (dt/6) (acc + k4)
// Every operation is rounded on its own (no contraction) in the order of the formulas
// above, so the FP64 path reproduces a plain evaluation of them operation by operation.
// Stage launches: one cell per thread on 32 x 8 tiles.  Pairs: four cells per thread on tiles of 128 x 8
// or 16; both evaluate the same expressions.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <new>
#include <utility>

#include "pdl.cuh"
#include "sslbm.h"

namespace sslbm {
int record_error(int status, const char* msg);
}

namespace {

int err(int status, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  return sslbm::record_error(status, buf);
}

int cuda_err(cudaError_t e, const char* what) {
  return err(SSLBM_ERR_CUDA, "%s: %s (%s)", what, cudaGetErrorName(e), cudaGetErrorString(e));
}

#define CK(call, what)                                  \
  do {                                                  \
    cudaError_t e_ = (call);                            \
    if (e_ != cudaSuccess) return cuda_err(e_, what);   \
  } while (0)

__device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float dvd(float a, float b) { return __fdiv_rn(a, b); }
__device__ __forceinline__ double dvd(double a, double b) { return __ddiv_rn(a, b); }

template <typename T>
struct Fd4Coeffs {
  T beta, alpha, gamma, rg, dg;  // rg = (1 - phi) gamma, dg = phi gamma
  T d[4];                        // diffusivities of S, E, I, R
  T inv, inv2;                   // 1 / (12 dx^2), 1 / dx^2
  T half_dt, dt, dt6;            // dt/2, dt, dt/6
};

// index of a (possibly ghost) cell along an axis of n cells
__device__ __forceinline__ int64_t ghost2(int64_t i, int64_t n, int bc) {
  if (i >= 0 && i < n) return i;
  if (bc == SSLBM_BC_PERIODIC) {
    int64_t r = i % n;
    return r < 0 ? r + n : r;
  }
  if (i < 0) i = -1 - i;
  if (i >= n) i = 2 * n - 1 - i;
  if (i < 0) i = 0;  // grids narrower than the stencil
  if (i >= n) i = n - 1;
  return i;
}

constexpr int kTX = 32, kTY = 8, kH = 2;  // tile of cells per CTA and the stencil's halo

// One RK4 stage on a kTX x kTY tile of cells: the four mobile planes of the stage input are
// staged in shared memory with a halo of two cells (ghost cells resolved once, at load),
// then every cell evaluates its right-hand side from the tile.
template <typename T, int STAGE, int ORDER>
__global__ void __launch_bounds__(kTX * kTY) fd4_stage_kernel(int64_t nx, int64_t ny, int bc, const Fd4Coeffs<T> k,
                                                              const T* __restrict__ src, const T* u, T* acc,
                                                              T* dst) {
  constexpr int SX = kTX + 2 * kH, SY = kTY + 2 * kH;
  __shared__ T tile[4][SY][SX];
  const int64_t M = nx * ny;
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * kTX + tx;
  const int64_t bx0 = (int64_t)blockIdx.x * kTX;
  for (int64_t by0 = (int64_t)blockIdx.y * kTY; by0 < ny; by0 += (int64_t)gridDim.y * kTY) {
    __syncthreads();  // the previous tile's readers are done
    for (int i = tid; i < SX * SY; i += kTX * kTY) {
      const int sy = i / SX, sx = i - sy * SX;
      const int64_t gx = ghost2(bx0 + sx - kH, nx, bc), gy = ghost2(by0 + sy - kH, ny, bc);
      const int64_t off = gy * nx + gx;
#pragma unroll
      for (int c = 0; c < 4; ++c) tile[c][sy][sx] = src[c * M + off];
    }
    __syncthreads();
    const int64_t x = bx0 + tx, y = by0 + ty;
    if (x >= nx || y >= ny) continue;
    const int64_t c0 = y * nx + x;
    const int cx = tx + kH, cy = ty + kH;
    const T S = tile[0][cy][cx], E = tile[1][cy][cx], I = tile[2][cy][cx], R = tile[3][cy][cx];
    // reactions, Eq. (sources)
    const T Nc = add(add(add(S, E), I), R);
    const T F = Nc != T(0) ? dvd(mul(mul(k.beta, S), I), Nc) : T(0);
    const T aE = mul(k.alpha, E);
    T rhs[5];
    rhs[0] = -F;
    rhs[1] = sub(F, aE);
    rhs[2] = sub(aE, mul(k.gamma, I));
    rhs[3] = mul(k.rg, I);
    rhs[4] = mul(k.dg, I);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const T u0 = tile[c][cy][cx];
      T lx, ly;
      if (ORDER == 4) {
        lx = sub(add(sub(add(-tile[c][cy][cx - 2], mul(T(16), tile[c][cy][cx - 1])), mul(T(30), u0)),
                     mul(T(16), tile[c][cy][cx + 1])),
                 tile[c][cy][cx + 2]);
        ly = sub(add(sub(add(-tile[c][cy - 2][cx], mul(T(16), tile[c][cy - 1][cx])), mul(T(30), u0)),
                     mul(T(16), tile[c][cy + 1][cx])),
                 tile[c][cy + 2][cx]);
      } else {  // second order: u[-1] - 2 u[0] + u[+1]
        lx = add(sub(tile[c][cy][cx - 1], mul(T(2), u0)), tile[c][cy][cx + 1]);
        ly = add(sub(tile[c][cy - 1][cx], mul(T(2), u0)), tile[c][cy + 1][cx]);
      }
      rhs[c] = add(rhs[c], mul(mul(k.d[c], add(lx, ly)), ORDER == 4 ? k.inv : k.inv2));
    }
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      const int64_t i = c * M + c0;
      const T r = rhs[c];
      if (STAGE == 1) {
        acc[i] = r;
        dst[i] = add(u[i], mul(k.half_dt, r));
      } else if (STAGE == 2) {
        acc[i] = add(acc[i], mul(T(2), r));
        dst[i] = add(u[i], mul(k.half_dt, r));
      } else if (STAGE == 3) {
        acc[i] = add(acc[i], mul(T(2), r));
        dst[i] = add(u[i], mul(k.dt, r));
      } else {
        dst[i] = add(u[i], mul(k.dt6, add(acc[i], r)));
      }
    }
  }
}

// Two RK4 stages in one launch, FP32: stages 1 and 2 (PAIR 0) or 3 and 4 (PAIR 1) on tiles of
// 128 x TY cells.  A CTA stages its tile of the input with a halo of four cells, evaluates the first
// stage on the tile and two cells around it (into shared memory), then the second stage on the
// tile; the first stage's slopes of the tile stay in registers.
//   PAIR 0: k1 = f(u), t = u + (dt/2) k1 (on chip), k2 = f(t); writes u + (dt/2) k2 and k1 + 2 k2
//   PAIR 1: k3 = f(src), v = u + dt k3 (on chip), k4 = f(v); writes u + (dt/6) (acc + 2 k3 + k4)
// The second stage's ghost cells: with periodic wrap the cells beyond an edge evaluate the first
// stage on wrapped values, which are the wrapped results; under no-flux the results are copied from
// the cells they mirror (evaluating the reflected neighbourhood would add its terms in the
// reverse order).  Every cell performs the operations of fd4_stage_kernel in its order.
//
// What bounds it: the operations, 90 per cell and stage of which none may contract, at 1.15 stage
// evaluations per cell (TY = 16), and latency; the separate stages moved 85 planes a step through
// HBM or L2 (340 bytes per cell), this moves 32.
// Four separate stages and these, us per step: 200^2 25.7 and 19.0, 1000^2 79.7 and 58.5, 2048^2 314
// and 176, 8192^2 4476 and 2462 (27.3 GLUPS; issue 59% busy, 200 instructions per cell and stage); widths
// that are no multiple of four, moved cell by cell: 1023 x 1025 78 and 73, 2047 x 2049 375 and 244.
// The loads of u and acc wait for HBM if issued where they are used (8192^2 3117); they are
// requested before the right-hand sides.
// ghost2 in 32-bit arithmetic, the wrap by one fold without a division on all but tiny grids (with
// 64-bit modulos the tiles at an edge took 18 us)
__device__ __forceinline__ int ghost2i(int i, int n, int bc) {
  if (i >= 0 && i < n) return i;
  if (bc == SSLBM_BC_PERIODIC) {
    const int j = i < 0 ? i + n : i - n;
    if (j >= 0 && j < n) return j;
    const int r = i % n;
    return r < 0 ? r + n : r;
  }
  if (i < 0) i = -1 - i;
  if (i >= n) i = 2 * n - 1 - i;
  return i < 0 ? 0 : i >= n ? n - 1 : i;  // grids narrower than the stencil
}

constexpr int kPX = 128;          // tile columns
constexpr int kPS = kPX + 8;      // floats per shared row: columns -4 .. 131

// o[0..1] = a v[0..1], each rounded as mul
__device__ __forceinline__ void mul2(float a, const float* v, float* o) {
  const float2 r = __fmul2_rn(make_float2(a, a), make_float2(v[0], v[1]));
  o[0] = r.x, o[1] = r.y;
}

// Right-hand sides of S, E, I, R (rhs[0..3]) and D (rhs[4]) for NE consecutive cells: rows are
// pointers to the cells' first column in rows y-2 .. y+2 of field 0, fields fs floats apart.
template <int ORDER, int NE>
__device__ __forceinline__ void fd4_rhs(const float* m2, const float* m1, const float* c0, const float* p1,
                                        const float* p2, const int fs, const Fd4Coeffs<float>& k, float (&rhs)[5][NE]) {
#pragma unroll
  for (int e = 0; e < NE; ++e) {  // reactions, Eq. (sources)
    const float S = c0[e], E = c0[fs + e], I = c0[2 * fs + e], R = c0[3 * fs + e];
    const float Nc = add(add(add(S, E), I), R);
    const float F = Nc != 0.f ? dvd(mul(mul(k.beta, S), I), Nc) : 0.f;
    const float aE = mul(k.alpha, E);
    rhs[0][e] = -F;
    rhs[1][e] = sub(F, aE);
    rhs[2][e] = sub(aE, mul(k.gamma, I));
    rhs[3][e] = mul(k.rg, I);
    rhs[4][e] = mul(k.dg, I);
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    float h[NE + 4], u2[NE], u1[NE], d1[NE], d2[NE];
    if (NE == 4) {
      const float2 hl = *reinterpret_cast<const float2*>(c0 + c * fs - 2);
      const float4 hc = *reinterpret_cast<const float4*>(c0 + c * fs);
      const float2 hr = *reinterpret_cast<const float2*>(c0 + c * fs + 4);
      const float hv[8] = {hl.x, hl.y, hc.x, hc.y, hc.z, hc.w, hr.x, hr.y};
      const float4 a1 = *reinterpret_cast<const float4*>(m1 + c * fs), b1 = *reinterpret_cast<const float4*>(p1 + c * fs);
      float4 a2 = make_float4(0.f, 0.f, 0.f, 0.f), b2 = a2;
      if (ORDER == 4) {
        a2 = *reinterpret_cast<const float4*>(m2 + c * fs);
        b2 = *reinterpret_cast<const float4*>(p2 + c * fs);
      }
      const float av[4] = {a1.x, a1.y, a1.z, a1.w}, bv[4] = {b1.x, b1.y, b1.z, b1.w};
      const float aw[4] = {a2.x, a2.y, a2.z, a2.w}, bw[4] = {b2.x, b2.y, b2.z, b2.w};
#pragma unroll
      for (int e = 0; e < NE + 4; ++e) h[e] = hv[e < 8 ? e : 0];
#pragma unroll
      for (int e = 0; e < NE; ++e) u1[e] = av[e & 3], d1[e] = bv[e & 3], u2[e] = aw[e & 3], d2[e] = bw[e & 3];
    } else {
#pragma unroll
      for (int e = 0; e < NE + 4; ++e) h[e] = c0[c * fs + e - 2];
#pragma unroll
      for (int e = 0; e < NE; ++e)
        u2[e] = m2[c * fs + e], u1[e] = m1[c * fs + e], d1[e] = p1[c * fs + e], d2[e] = p2[c * fs + e];
    }
    if constexpr (NE == 4 && ORDER == 4) {
      // the products two at a time; the sums that take a product stay scalar (packed, the compiler
      // may fuse the product into them)
      float m[8], mu[4], md[4], m30[4], l[4];
      mul2(16.f, h, m), mul2(16.f, h + 2, m + 2), mul2(16.f, h + 4, m + 4), mul2(16.f, h + 6, m + 6);
      mul2(16.f, u1, mu), mul2(16.f, u1 + 2, mu + 2), mul2(16.f, d1, md), mul2(16.f, d1 + 2, md + 2);
      mul2(30.f, h + 2, m30), mul2(30.f, h + 4, m30 + 2);
#pragma unroll
      for (int e = 0; e < 4; ++e)
        l[e] = add(sub(add(sub(add(-h[e], m[1 + e]), m30[e]), m[3 + e]), h[4 + e]),
                   sub(add(sub(add(-u2[e], mu[e]), m30[e]), md[e]), d2[e]));
      mul2(k.d[c], l, l), mul2(k.d[c], l + 2, l + 2);
      mul2(k.inv, l, l), mul2(k.inv, l + 2, l + 2);
#pragma unroll
      for (int e = 0; e < 4; ++e) rhs[c][e] = add(rhs[c][e], l[e]);
    } else {
#pragma unroll
    for (int e = 0; e < NE; ++e) {
      const float u0 = h[2 + e];
      float lx, ly;
      if (ORDER == 4) {
        lx = sub(add(sub(add(-h[e], mul(16.f, h[1 + e])), mul(30.f, u0)), mul(16.f, h[3 + e])), h[4 + e]);
        ly = sub(add(sub(add(-u2[e], mul(16.f, u1[e])), mul(30.f, u0)), mul(16.f, d1[e])), d2[e]);
      } else {
        lx = add(sub(h[1 + e], mul(2.f, u0)), h[3 + e]);
        ly = add(sub(u1[e], mul(2.f, u0)), d1[e]);
      }
      rhs[c][e] = add(rhs[c][e], mul(mul(k.d[c], add(lx, ly)), ORDER == 4 ? k.inv : k.inv2));
    }
    }
  }
}

template <int TY>
constexpr size_t fd4_pair_smem() {
  return sizeof(float) * 4 * (2 * TY + 12) * kPS;
}

// u: the step's state; src: the input of the pair (PAIR 0: u); acc: running sum of the slopes
// (PAIR 0: written); dst: PAIR 0 the next stage's state (S, E, I, R), PAIR 1 the next state, not
// u or src.  VEC: nx is a multiple of 4, so that every row starts on a 16-byte boundary and four
// cells move at a time; else one by one.
template <int PAIR, int ORDER, int TY, bool VEC>
__global__ void __launch_bounds__(256, TY > 8 ? 2 : 3)
    fd4_pair_kernel(const int nx, const int ny, const int bc, const Fd4Coeffs<float> k,
                    const float* src, const float* u, float* acc, float* dst) {
  constexpr int RA = TY + 8, RB = TY + 4, FA = RA * kPS, FB = RB * kPS, NR = TY / 8;
  static_assert(TY % 8 == 0, "whole rows per warp");
  extern __shared__ __align__(16) float fd4_smem[];
  float* A = fd4_smem;          // [4][RA][kPS]: the input, rows by0 - 4 ..
  float* B = fd4_smem + 4 * FA;  // [4][RB][kPS]: the first stage's result, rows by0 - 2 ..
  const int64_t M = (int64_t)nx * ny;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int ntx = (nx + kPX - 1) / kPX;
  const int bx0 = (int)(blockIdx.x % ntx) * kPX, by0 = (int)(blockIdx.x / ntx) * TY;
  const float cA = PAIR == 0 ? k.half_dt : k.dt;
  static_assert(4 * RB <= 128, "a thread per cell of the side columns");

  sslbm::pdl_enter();

  // the input tile: rows of 34 groups of four columns, one warp per row; rows past the domain's
  // last needed one are skipped (no cell that is written reads them)
  for (int j = w; j < 4 * RA; j += 8) {
    const int c = j / RA, r = j - c * RA;
    if (by0 + r - 4 >= ny + 4) continue;
    const float* row = src + c * M + (int64_t)ghost2i(by0 + r - 4, ny, bc) * nx;
    float* d = A + c * FA + r * kPS;
    if constexpr (VEC) {
      for (int q = lane; q < kPS / 4; q += 32) {
        const int x = bx0 - 4 + 4 * q;
        if (x >= nx + 4) continue;
        if (x >= 0 && x + 3 < nx) {
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(
                           (unsigned)__cvta_generic_to_shared(d + 4 * q)),
                       "l"(row + x)
                       : "memory");
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(
                             (unsigned)__cvta_generic_to_shared(d + 4 * q + e)),
                         "l"(row + ghost2i(x + e, nx, bc))
                         : "memory");
        }
      }
    } else {  // a lane per column
      for (int q = lane; q < kPS; q += 32) {
        const int x = bx0 - 4 + q;
        if (x < nx + 4)
          asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"((unsigned)__cvta_generic_to_shared(d + q)),
                       "l"(row + ghost2i(x, nx, bc))
                       : "memory");
      }
    }
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  __syncthreads();

  const int x = bx0 + 4 * lane;
  // four cells of a row of a global plane, those that lie in the grid
  auto load4 = [&](const float* p, float (&v)[4]) {
    if (VEC) {
      const float4 t = x < nx ? *reinterpret_cast<const float4*>(p) : make_float4(0.f, 0.f, 0.f, 0.f);
      v[0] = t.x, v[1] = t.y, v[2] = t.z, v[3] = t.w;
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = x + e < nx ? p[e] : 0.f;
    }
  };
  auto store4 = [&](float* p, const float (&v)[4]) {
    if (VEC) {
      if (x < nx) *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (x + e < nx) p[e] = v[e];
    }
  };
  // first stage of tile row r (-2 .. TY + 1), the lane's four columns; u is requested before the
  // right-hand sides are evaluated
  auto stage1 = [&](int r, float (&rhs)[5][4]) {
    const float* c0 = A + (r + 4) * kPS + 4 + 4 * lane;
    float uv[4][4];
    const float* ur = u + (int64_t)ghost2i(by0 + r, ny, bc) * nx;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      if (PAIR == 0) {
        const float4 t = *reinterpret_cast<const float4*>(c0 + c * FA);
        uv[c][0] = t.x, uv[c][1] = t.y, uv[c][2] = t.z, uv[c][3] = t.w;
      } else if (x + 3 < nx) {
        load4(ur + c * M + x, uv[c]);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) uv[c][e] = x + e < nx + 2 ? ur[c * M + ghost2i(x + e, nx, bc)] : 0.f;
      }
    }
    fd4_rhs<ORDER, 4>(c0 - 2 * kPS, c0 - kPS, c0, c0 + kPS, c0 + 2 * kPS, FA, k, rhs);
    float* o = B + (r + 2) * kPS + 4 + 4 * lane;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      float v[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = add(uv[c][e], mul(cA, rhs[c][e]));
      *reinterpret_cast<float4*>(o + c * FB) = make_float4(v[0], v[1], v[2], v[3]);
    }
  };
  float ka[NR][5][4];  // the first stage's slopes of the warp's tile rows
#pragma unroll
  for (int i = 0; i < NR; ++i) stage1(w + 8 * i, ka[i]);
  if (w < 4) {  // the two rows above and below
    float t[5][4];
    stage1(w < 2 ? w - 2 : TY + w - 2, t);
  }
  if (tid >= 128 && tid < 128 + 4 * RB) {  // the two columns on each side
    const int r = (tid - 128) >> 2, h = tid & 3, col = h < 2 ? h - 2 : kPX + h - 2;
    const float* c0 = A + (r + 2) * kPS + 4 + col;
    float t[5][1];
    fd4_rhs<ORDER, 1>(c0 - 2 * kPS, c0 - kPS, c0, c0 + kPS, c0 + 2 * kPS, FA, k, t);
    const int64_t row = (int64_t)ghost2i(by0 + r - 2, ny, bc) * nx;
    const int64_t gx = ghost2i(bx0 + col, nx, bc);
#pragma unroll
    for (int c = 0; c < 4; ++c)
      B[c * FB + r * kPS + 4 + col] = add(PAIR == 0 ? c0[c * FA] : u[c * M + row + gx], mul(cA, t[c][0]));
  }
  __syncthreads();

  if (bc != SSLBM_BC_PERIODIC && (bx0 == 0 || by0 == 0 || bx0 + kPX + 2 > nx || by0 + TY + 2 > ny)) {
    // mirror images of the first stage's results: columns beyond the walls, then rows
    for (int i = tid; i < 4 * RB * 4; i += 256) {
      const int h = i & 3, r = (i >> 2) % RB, c = (i >> 2) / RB;
      const int gx = h < 2 ? h - 2 : nx + h - 2;  // -2, -1, nx, nx + 1
      if (gx >= bx0 - 2 && gx < bx0 + kPX + 2)
        B[c * FB + r * kPS + 4 + gx - bx0] = B[c * FB + r * kPS + 4 + ghost2i(gx, nx, bc) - bx0];
    }
    __syncthreads();
    for (int i = tid; i < 4 * 4 * (kPX + 4); i += 256) {
      const int col = i % (kPX + 4) - 2, h = i / (kPX + 4) & 3, c = i / (kPX + 4) / 4;
      const int gy = h < 2 ? h - 2 : ny + h - 2;
      if (gy >= by0 - 2 && gy < by0 + TY + 2)
        B[c * FB + (gy - by0 + 2) * kPS + 4 + col] = B[c * FB + (ghost2i(gy, ny, bc) - by0 + 2) * kPS + 4 + col];
    }
    __syncthreads();
  }

#pragma unroll
  for (int i = 0; i < NR; ++i) {
    const int r = w + 8 * i, y = by0 + r;
    if (y >= ny) continue;
    const float* c0 = B + (r + 2) * kPS + 4 + 4 * lane;
    float rhs[5][4];
    const int64_t o = (int64_t)y * nx + x;
    float ag[5][4], ug[5][4];
    if (PAIR == 1) {  // requested before the right-hand sides
#pragma unroll
      for (int c = 0; c < 5; ++c) {
        load4(acc + c * M + o, ag[c]);
        load4(u + c * M + o, ug[c]);
      }
    }
    fd4_rhs<ORDER, 4>(c0 - 2 * kPS, c0 - kPS, c0, c0 + kPS, c0 + 2 * kPS, FB, k, rhs);
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      float out[4];
      if (PAIR == 0) {
        float av[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) av[e] = add(ka[i][c][e], mul(2.f, rhs[c][e]));
        store4(acc + c * M + o, av);
        if (c < 4) {  // D enters no right-hand side
          const float* uc = A + c * FA + (r + 4) * kPS + 4 + 4 * lane;
#pragma unroll
          for (int e = 0; e < 4; ++e) out[e] = add(uc[e], mul(k.half_dt, rhs[c][e]));
          store4(dst + c * M + o, out);
        }
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
          out[e] = add(ug[c][e], mul(k.dt6, add(add(ag[c][e], mul(2.f, ka[i][c][e])), rhs[c][e])));
        store4(dst + c * M + o, out);
      }
    }
  }
}

template <typename A, typename B>
__global__ void convert_kernel(const A* __restrict__ a, B* __restrict__ b, int64_t n) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
    b[t] = (B)a[t];
}

unsigned blocks1(int64_t n) { return (unsigned)std::min<int64_t>(65536, (n + 255) / 256); }

size_t rup(size_t v) { return (v + 255) / 256 * 256; }

int check_grid(const sslbm_grid* g) {
  if (!g) return err(SSLBM_ERR_BAD_ARG, "grid is NULL");
  if (g->nx < 1 || g->ny < 1 || g->nx > (1 << 20) || g->ny > (1 << 20))
    return err(SSLBM_ERR_BAD_ARG, "grid %lld x %lld out of range", (long long)g->nx, (long long)g->ny);
  if (!(g->dx > 0) || !(g->dt > 0) || !std::isfinite(g->dx) || !std::isfinite(g->dt))
    return err(SSLBM_ERR_BAD_ARG, "dx and dt must be finite and > 0");
  if (g->bc != SSLBM_BC_PERIODIC && g->bc != SSLBM_BC_NOFLUX) return err(SSLBM_ERR_BAD_ARG, "bc %d", g->bc);
  if (g->precision != SSLBM_FP64 && g->precision != SSLBM_FP32)
    return err(SSLBM_ERR_UNSUPPORTED, "the FD4 reference runs in FP64 or FP32");
  return SSLBM_OK;
}

size_t state_bytes(const sslbm_grid* g) {
  return rup((size_t)5 * g->nx * g->ny * (g->precision == SSLBM_FP64 ? 8 : 4));
}

}  // namespace

struct sslbm_fd4 {
  sslbm_grid g;
  cudaStream_t stream = nullptr;
  int device = 0;
  char* ws = nullptr;
  size_t sb = 0;  // bytes of one 5-plane state
  Fd4Coeffs<double> k64;
  Fd4Coeffs<float> k32;
  int64_t steps = 0;
  int order = 4;  // order of the Laplacian: 4 (the reference) or 2
  int sms = 1;    // multiprocessors of the device
  // 0 u, the state; scratch of a step: FP64 1 t1, 2 t2, 3 acc, FP32 1 t, 2 acc, 3 the next state
  void* buf(int i) const { return ws + (size_t)i * sb; }
};

namespace {

struct DevGuard {
  int prev = -1;
  explicit DevGuard(int dev) {
    if (cudaGetDevice(&prev) == cudaSuccess && prev != dev) cudaSetDevice(dev);
    else prev = -1;
  }
  ~DevGuard() {
    if (prev >= 0) cudaSetDevice(prev);
  }
};

template <int PAIR, int ORDER, int TY, bool VEC>
cudaError_t launch_pair(const sslbm_fd4* f, const float* src, const float* u, float* acc, float* dst) {
  // the dynamic shared-memory limit, once per device (a bit per device; setting it twice is harmless)
  static std::atomic<unsigned long long> done{0};
  auto kern = fd4_pair_kernel<PAIR, ORDER, TY, VEC>;
  if (!(done.load(std::memory_order_acquire) & (1ull << (f->device & 63)))) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fd4_pair_smem<TY>());
    if (e != cudaSuccess) return e;
    done.fetch_or(1ull << (f->device & 63), std::memory_order_release);
  }
  const int64_t nx = f->g.nx, ny = f->g.ny;
  const int64_t ctas = (nx + kPX - 1) / kPX * ((ny + TY - 1) / TY);
  if (ctas > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  // Ordinary launches where the next one's CTAs would fit beside this one's on more than half of the SMs:
  // launched early they settle two to an SM beside empty ones, and stay so from launch to launch
  // (333 x 257 no-flux, 20 steps, 32 us per step dependent, 29 ordinary).
  const bool beside = 2 * ctas > f->sms && 2 * ctas <= (TY > 8 ? 2 : 3) * (int64_t)f->sms;
  return sslbm::launch_pdl_if(!beside, kern, dim3((unsigned)ctas), dim3(256), fd4_pair_smem<TY>(), f->stream, (int)nx,
                              (int)ny, (int)f->g.bc, f->k32, src, u, acc, dst);
}

// One FP32 step from u to next: two launches.
template <int ORDER, int TY, bool VEC>
cudaError_t run_step_pairs(const sslbm_fd4* f, const float* u, float* next) {
  float* t = static_cast<float*>(f->buf(1));
  float* acc = static_cast<float*>(f->buf(2));
  cudaError_t e = launch_pair<0, ORDER, TY, VEC>(f, u, u, acc, t);
  return e == cudaSuccess ? launch_pair<1, ORDER, TY, VEC>(f, t, u, acc, next) : e;
}

// One step of four stage launches, in place.
template <typename T, int ORDER>
cudaError_t run_step(const sslbm_fd4* f, const Fd4Coeffs<T>& k) {
  const int64_t nx = f->g.nx, ny = f->g.ny;
  dim3 block(kTX, kTY);
  dim3 grid((unsigned)((nx + kTX - 1) / kTX), (unsigned)std::min<int64_t>(65535, (ny + kTY - 1) / kTY));
  T* u = static_cast<T*>(f->buf(0));
  T* t1 = static_cast<T*>(f->buf(1));
  T* t2 = static_cast<T*>(f->buf(2));
  T* acc = static_cast<T*>(f->buf(3));
  const int bc = f->g.bc;
  fd4_stage_kernel<T, 1, ORDER><<<grid, block, 0, f->stream>>>(nx, ny, bc, k, u, u, acc, t1);
  fd4_stage_kernel<T, 2, ORDER><<<grid, block, 0, f->stream>>>(nx, ny, bc, k, t1, u, acc, t2);
  fd4_stage_kernel<T, 3, ORDER><<<grid, block, 0, f->stream>>>(nx, ny, bc, k, t2, u, acc, t1);
  fd4_stage_kernel<T, 4, ORDER><<<grid, block, 0, f->stream>>>(nx, ny, bc, k, t1, u, acc, u);
  return cudaGetLastError();
}

// How FP32 steps are launched: the two-stage kernel with 8 or 16 rows per tile, or the four one-cell
// stage launches; and whether the last of an odd number of steps takes the stage launches, which work
// in place, rather than a pair and the copy into buffer 0.
struct StepPlan {
  int rows;  // 0: stage launches
  bool odd_in_place;
};

// By the costs measured (us per step, 40 grids from 32^2 to 2048^2 and 3 x 100000 to 20000 x 3, both
// boundaries).  A pair step takes whole waves of its tiles, 3 CTAs per SM with 8 rows and 2 with 16:
// 1000^2 59 and 58, 800 x 600 40 and 34 (two waves and one), 20000 x 64 65 and 76, 2048^2 187 and 177.
// Grids narrower than a tile waste most of it, where the 32 x 8 stage tiles do not: 64 x 20000 no-flux
// 152 as pairs and 103 as stages, 3 x 100000 570 and 180, but 96 x 20000 155 and 181.  On small no-flux
// grids the pairs' mirror passes cost what the launches save, most where a tile spans the domain
// (64 x 1000 26.8 and 22.9, 20000 x 8 26.2 and 25.0).  The copy after an odd step is worth it only on
// larger grids: one step at 128^2 31 with it and 22 in place, at 2048^2 206 and 363.
StepPlan plan_step(const sslbm_grid& g, int sms) {
  const double cells = (double)g.nx * g.ny, m = 1e-6;
  const int64_t cols = (g.nx + kPX - 1) / kPX;
  const bool walls = g.bc != SSLBM_BC_PERIODIC, vec = g.nx % 4 == 0;
  const int64_t t8 = cols * ((g.ny + 7) / 8), t16 = cols * ((g.ny + 15) / 16);
  const int64_t w8 = (t8 + 3 * sms - 1) / (3 * sms), w16 = (t16 + 2 * sms - 1) / (2 * sms);
  const double edge = walls ? 2.5 + (cols == 1 || g.ny <= 8 ? 6.0 : 0.0) : 0.0;
  double p8, p16;
  if (w8 == 1) {  // one wave of 8-row tiles is never behind
    p8 = 2 * t8 <= sms ? 18.5 + (vec ? 0.0 : 2.0) : t8 <= sms ? (vec ? 24.0 : 27.5) : vec ? 26.5 : 30.5;
    p16 = 1e30;
  } else {
    p8 = (6.0 + 20.2 * w8) * (vec ? 1.0 : 1.3);
    p16 = (6.0 + 25.5 * w16) * (vec ? 1.0 : 1.3);
  }
  const double pair = (p8 <= p16 ? p8 : p16) + edge;
  // the stage launches: cells of whole 32 x 8 tiles, slower beyond what L2 holds
  const double tiles = m * (double)((g.nx + kTX - 1) / kTX * kTX) * (double)((g.ny + kTY - 1) / kTY * kTY);
  const double stage = 20.0 + (tiles > 0.02 ? 2.5 : 1.0) + 55.0 * std::min(tiles, 1.0) +
                       85.0 * std::max(tiles - 1.0, 0.0) + (walls ? 0.0 : 3.5);
  StepPlan plan;
  plan.rows = pair > stage ? 0 : p8 <= p16 ? 8 : 16;
  plan.odd_in_place = pair + 7.0 + 6.9 * m * cells > stage;
  return plan;
}

// n FP32 steps: pairs alternate between buffers 0 and 3 and the state ends in buffer 0, so that every
// call finds it there and a captured call can be replayed for any n.
template <int ORDER, bool VEC>
cudaError_t run_steps_f32(sslbm_fd4* f, int64_t n) {
  const StepPlan plan = plan_step(f->g, f->sms);
  float* a = static_cast<float*>(f->buf(0));
  float* b = static_cast<float*>(f->buf(3));
  cudaError_t e = cudaSuccess;
  for (int64_t i = 0; i < n && e == cudaSuccess; ++i) {
    const bool last_odd = a == f->buf(0) && i + 1 == n;
    if (plan.rows == 0 || (last_odd && plan.odd_in_place)) {
      e = run_step<float, ORDER>(f, f->k32);
    } else {
      e = plan.rows == 8 ? run_step_pairs<ORDER, 8, VEC>(f, a, b) : run_step_pairs<ORDER, 16, VEC>(f, a, b);
      if (e == cudaSuccess) std::swap(a, b);
    }
    if (e == cudaSuccess) ++f->steps;
  }
  if (a != f->buf(0)) {
    const size_t bytes = (size_t)5 * f->g.nx * f->g.ny * sizeof(float);
    const cudaError_t ce = cudaMemcpyAsync(b, a, bytes, cudaMemcpyDeviceToDevice, f->stream);
    if (e == cudaSuccess) e = ce;
  }
  return e;
}

template <typename T>
Fd4Coeffs<T> make_coeffs(const sslbm_grid* g, const sslbm_params* p) {
  Fd4Coeffs<T> k;
  k.beta = (T)p->beta;
  k.alpha = (T)p->alpha;
  k.gamma = (T)p->gamma;
  k.rg = (T)((1.0 - p->phi) * p->gamma);
  k.dg = (T)(p->phi * p->gamma);
  for (int c = 0; c < 4; ++c) k.d[c] = (T)p->d[c];
  k.inv = (T)(1.0 / (12.0 * g->dx * g->dx));
  k.inv2 = (T)(1.0 / (g->dx * g->dx));
  k.half_dt = (T)(0.5 * g->dt);
  k.dt = (T)g->dt;
  k.dt6 = (T)(g->dt / 6.0);
  return k;
}

}  // namespace

extern "C" {

int sslbm_fd4_workspace_bytes(const sslbm_grid* g, size_t* bytes) {
  if (!bytes) return err(SSLBM_ERR_BAD_ARG, "bytes is NULL");
  int st = check_grid(g);
  if (st) return st;
  *bytes = 4 * state_bytes(g);
  return SSLBM_OK;
}

int sslbm_fd4_create(const sslbm_grid* g, const sslbm_params* p, void* dev_ws, size_t ws_bytes, void* stream,
                     sslbm_fd4** out) {
  if (!out) return err(SSLBM_ERR_BAD_ARG, "out is NULL");
  *out = nullptr;
  int st = check_grid(g);
  if (st) return st;
  if (!p) return err(SSLBM_ERR_BAD_ARG, "params is NULL");
  if (p->use_tau) return err(SSLBM_ERR_BAD_ARG, "the FD4 reference takes diffusivities d, not tau");
  const double rates[4] = {p->beta, p->alpha, p->gamma, p->phi};
  for (double r : rates)
    if (!std::isfinite(r) || r < 0) return err(SSLBM_ERR_BAD_ARG, "rates must be finite and >= 0");
  if (p->phi > 1) return err(SSLBM_ERR_BAD_ARG, "phi %g > 1", p->phi);
  for (int c = 0; c < 4; ++c)
    if (!std::isfinite(p->d[c]) || p->d[c] < 0) return err(SSLBM_ERR_BAD_ARG, "d[%d] must be finite and >= 0", c);
  if (p->d[4] != 0) return err(SSLBM_ERR_BAD_ARG, "d[D] must be 0 (D does not move)");
  // RK4 is stable on the negative real axis up to |z| = 2.78; the fourth-order Laplacian's
  // most negative eigenvalue is -(64/12) per axis / dx^2, so d dt / dx^2 <= 0.26 in 2D
  for (int c = 0; c < 4; ++c)
    if (p->d[c] * g->dt / (g->dx * g->dx) > 0.26)
      return err(SSLBM_ERR_UNSTABLE, "d[%d] dt / dx^2 = %g > 0.26 (RK4 with the fourth-order Laplacian)", c,
                 p->d[c] * g->dt / (g->dx * g->dx));
  const size_t need = 4 * state_bytes(g);
  if (!dev_ws || reinterpret_cast<uintptr_t>(dev_ws) % 256)
    return err(SSLBM_ERR_WORKSPACE, "workspace missing or not 256-byte aligned");
  if (ws_bytes < need) return err(SSLBM_ERR_WORKSPACE, "workspace of %zu bytes < %zu", ws_bytes, need);
  cudaPointerAttributes attr;
  CK(cudaPointerGetAttributes(&attr, dev_ws), "cudaPointerGetAttributes");
  if (attr.type != cudaMemoryTypeDevice && attr.type != cudaMemoryTypeManaged)
    return err(SSLBM_ERR_WORKSPACE, "workspace is not device memory");
  sslbm_fd4* f = new (std::nothrow) sslbm_fd4();
  if (!f) return err(SSLBM_ERR_BAD_ARG, "out of host memory");
  f->g = *g;
  f->ws = static_cast<char*>(dev_ws);
  f->sb = state_bytes(g);
  f->stream = static_cast<cudaStream_t>(stream);
  f->device = attr.device;
  f->k64 = make_coeffs<double>(g, p);
  f->k32 = make_coeffs<float>(g, p);
  DevGuard dg(f->device);
  if (cudaDeviceGetAttribute(&f->sms, cudaDevAttrMultiProcessorCount, f->device) != cudaSuccess || f->sms < 1)
    f->sms = 1;
  cudaError_t e = cudaMemsetAsync(f->ws, 0, need, f->stream);
  if (e != cudaSuccess) {
    delete f;
    return cuda_err(e, "zero workspace");
  }
  *out = f;
  return SSLBM_OK;
}

void sslbm_fd4_destroy(sslbm_fd4* f) { delete f; }

int sslbm_fd4_write(sslbm_fd4* f, const void* src, int src_dtype, int src_on_device) {
  if (!f || !src) return err(SSLBM_ERR_BAD_ARG, "NULL argument");
  if (src_dtype != SSLBM_DT_F64 && src_dtype != SSLBM_DT_F32) return err(SSLBM_ERR_BAD_ARG, "dtype %d", src_dtype);
  DevGuard dg(f->device);
  const int64_t n = 5 * f->g.nx * f->g.ny;
  const size_t esz = src_dtype == SSLBM_DT_F64 ? 8 : 4;
  const bool f64 = f->g.precision == SSLBM_FP64;
  if ((src_dtype == SSLBM_DT_F64) == f64) {
    CK(cudaMemcpyAsync(f->buf(0), src, (size_t)n * esz,
                       src_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, f->stream),
       "copy");
  } else {
    const void* s = src;
    if (!src_on_device) {  // stage through the scratch buffers (two when FP32 holds FP64)
      CK(cudaMemcpyAsync(f->buf(1), src, (size_t)n * esz, cudaMemcpyHostToDevice, f->stream), "host -> device");
      s = f->buf(1);
    }
    if (f64)
      convert_kernel<float, double><<<blocks1(n), 256, 0, f->stream>>>(static_cast<const float*>(s),
                                                                       static_cast<double*>(f->buf(0)), n);
    else
      convert_kernel<double, float><<<blocks1(n), 256, 0, f->stream>>>(static_cast<const double*>(s),
                                                                       static_cast<float*>(f->buf(0)), n);
    CK(cudaGetLastError(), "convert");
  }
  if (!src_on_device) CK(cudaStreamSynchronize(f->stream), "sync");
  f->steps = 0;
  return SSLBM_OK;
}

int sslbm_fd4_read(sslbm_fd4* f, void* dst, int dst_dtype, int dst_on_device) {
  if (!f || !dst) return err(SSLBM_ERR_BAD_ARG, "NULL argument");
  if (dst_dtype != SSLBM_DT_F64 && dst_dtype != SSLBM_DT_F32) return err(SSLBM_ERR_BAD_ARG, "dtype %d", dst_dtype);
  DevGuard dg(f->device);
  const int64_t n = 5 * f->g.nx * f->g.ny;
  const size_t esz = dst_dtype == SSLBM_DT_F64 ? 8 : 4;
  const bool f64 = f->g.precision == SSLBM_FP64;
  if ((dst_dtype == SSLBM_DT_F64) == f64) {
    CK(cudaMemcpyAsync(dst, f->buf(0), (size_t)n * esz, dst_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                       f->stream),
       "copy");
  } else {
    void* d = dst_on_device ? dst : f->buf(1);
    if (f64)
      convert_kernel<double, float><<<blocks1(n), 256, 0, f->stream>>>(static_cast<const double*>(f->buf(0)),
                                                                       static_cast<float*>(d), n);
    else
      convert_kernel<float, double><<<blocks1(n), 256, 0, f->stream>>>(static_cast<const float*>(f->buf(0)),
                                                                       static_cast<double*>(d), n);
    CK(cudaGetLastError(), "convert");
    if (!dst_on_device) CK(cudaMemcpyAsync(dst, d, (size_t)n * esz, cudaMemcpyDeviceToHost, f->stream), "device -> host");
  }
  CK(cudaStreamSynchronize(f->stream), "sync");
  return SSLBM_OK;
}

int sslbm_fd4_step(sslbm_fd4* f, int64_t n) {
  if (!f) return err(SSLBM_ERR_BAD_ARG, "NULL handle");
  if (n < 0) return err(SSLBM_ERR_BAD_ARG, "n < 0");
  DevGuard dg(f->device);
  if (f->g.precision == SSLBM_FP32) {
    const bool vec = f->g.nx % 4 == 0;
    const cudaError_t e = f->order == 4 ? (vec ? run_steps_f32<4, true>(f, n) : run_steps_f32<4, false>(f, n))
                                        : (vec ? run_steps_f32<2, true>(f, n) : run_steps_f32<2, false>(f, n));
    return e == cudaSuccess ? SSLBM_OK : cuda_err(e, "FD4 stage launch");
  }
  for (int64_t i = 0; i < n; ++i) {
    cudaError_t e = f->order == 4 ? run_step<double, 4>(f, f->k64) : run_step<double, 2>(f, f->k64);
    if (e != cudaSuccess) return cuda_err(e, "FD4 stage launch");
    ++f->steps;
  }
  return SSLBM_OK;
}

int64_t sslbm_fd4_steps_done(const sslbm_fd4* f) { return f ? f->steps : -1; }

int sslbm_fd4_set_order(sslbm_fd4* f, int order) {
  if (!f) return err(SSLBM_ERR_BAD_ARG, "NULL handle");
  if (order != 2 && order != 4) return err(SSLBM_ERR_BAD_ARG, "order %d is not 2 or 4", order);
  f->order = order;  // the create-time stability check (d dt / dx^2 <= 0.26) covers both orders
  return SSLBM_OK;
}

}  // extern "C"
