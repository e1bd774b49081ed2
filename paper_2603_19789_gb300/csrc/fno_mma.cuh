// fno_mma.cuh -- the warp-level pieces the surrogate's fused row kernels share (fno_fused.cu, the
// forward pass; fno_bwd.cu, the backward pass): cp.async copies, ldmatrix fragment loads, the
// BF16 mma.sync with FP32 accumulation, GELU and its derivative.
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

namespace sslbm {
namespace fno_fused {
namespace {

typedef __nv_bfloat16 bf16;
typedef __nv_bfloat162 bf162;

__device__ __forceinline__ unsigned saddr(const void* p) {
  return static_cast<unsigned>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void cp16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(saddr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void wait_groups() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// ldmatrix: four (or two) 8x8 b16 tiles; lane l supplies the address of row l % 8 of tile l / 8
__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], const bf16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(saddr(p)));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t (&r)[4], const bf16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(saddr(p)));
}
__device__ __forceinline__ void ldsm_x2(uint32_t (&r)[2], const bf16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];\n"
               : "=r"(r[0]), "=r"(r[1])
               : "r"(saddr(p)));
}
__device__ __forceinline__ void ldsm_x2_t(uint32_t (&r)[2], const bf16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n"
               : "=r"(r[0]), "=r"(r[1])
               : "r"(saddr(p)));
}

__device__ __forceinline__ void mma(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The A fragment of a 16 x 16 tile of a row-major [m][k] array with row stride ld (elements)
__device__ __forceinline__ void load_a(uint32_t (&a)[4], const bf16* base, int ld, int m0, int k0, int lane) {
  ldsm_x4(a, base + (m0 + (lane & 15)) * ld + k0 + (lane >> 4) * 8);
}
// The A fragment of a 16 x 16 tile of A^T, from A stored [k][m] (m contiguous) with row stride ld
__device__ __forceinline__ void load_a_t(uint32_t (&a)[4], const bf16* base, int ld, int m0, int k0, int lane) {
  ldsm_x4_t(a, base + (k0 + (lane & 7) + (lane >> 4) * 8) * ld + m0 + ((lane >> 3) & 1) * 8);
}
// B fragments (k16 x n8) of n tiles n0 and n0 + 8 from a [k][n] array (n contiguous)
__device__ __forceinline__ void load_b_kn2(uint32_t (&b)[4], const bf16* base, int ld, int k0, int n0, int lane) {
  ldsm_x4_t(b, base + (k0 + (lane & 15)) * ld + n0 + (lane >> 4) * 8);
}
__device__ __forceinline__ void load_b_kn1(uint32_t (&b)[2], const bf16* base, int ld, int k0, int n0, int lane) {
  ldsm_x2_t(b, base + (k0 + (lane & 15)) * ld + n0);
}
// B fragments from an [n][k] array (k contiguous)
__device__ __forceinline__ void load_b_nk2(uint32_t (&b)[4], const bf16* base, int ld, int k0, int n0, int lane) {
  ldsm_x4(b, base + (n0 + (lane & 7) + (lane >> 4) * 8) * ld + k0 + ((lane >> 3) & 1) * 8);
}
__device__ __forceinline__ void load_b_nk1(uint32_t (&b)[2], const bf16* base, int ld, int k0, int n0, int lane) {
  ldsm_x2(b, base + (n0 + (lane & 7)) * ld + k0 + ((lane >> 3) & 1) * 8);
}

// acc[u] += A B of the T adjacent n tiles from n0 on ([k][n] array): one A fragment for all of them
template <int T>
__device__ __forceinline__ void mma_tiles_kn(float (&acc)[T][4], const uint32_t (&af)[4], const bf16* base, int ld,
                                             int k0, int n0, int lane) {
#pragma unroll
  for (int u = 0; u + 1 < T; u += 2) {
    uint32_t bf[4];
    load_b_kn2(bf, base, ld, k0, n0 + 8 * u, lane);
    mma(acc[u], af, bf[0], bf[1]);
    mma(acc[u + 1], af, bf[2], bf[3]);
  }
  if (T % 2) {
    uint32_t bf[2];
    load_b_kn1(bf, base, ld, k0, n0 + 8 * (T - 1), lane);
    mma(acc[T - 1], af, bf[0], bf[1]);
  }
}

// GELU as on the unfused path -- the tanh form, 0.5 z (1 + tanh(u)), u = sqrt(2/pi) (z + 0.044715 z^3)
// = z (c + 0.044715 c z^2), with the hardware tanh (tanh.approx.f32) -- and its derivative,
// 0.5 (1 + t) + 0.5 z (1 - t^2) du/dz, two values at a time in packed FP32: 4 instructions per value
// instead of 8, where these and the fragment traffic fill the row kernels' issue slots.
constexpr float kGeluC = 0.7978845608028654f, kGeluC3 = 0.044715f * 0.7978845608028654f;
__device__ __forceinline__ float2 splat(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 tanh2(float2 u) {
  float2 t;
  asm("tanh.approx.f32 %0, %1;" : "=f"(t.x) : "f"(u.x));
  asm("tanh.approx.f32 %0, %1;" : "=f"(t.y) : "f"(u.y));
  return t;
}
__device__ __forceinline__ float2 gelu2(float2 z) {
  const float2 p = __ffma2_rn(splat(kGeluC3), __fmul2_rn(z, z), splat(kGeluC));
  const float2 t = tanh2(__fmul2_rn(z, p));
  const float2 h = __fmul2_rn(splat(0.5f), z);
  return __ffma2_rn(h, t, h);
}
__device__ __forceinline__ float2 gelu_grad2(float2 z) {
  const float2 zz = __fmul2_rn(z, z);
  const float2 t = tanh2(__fmul2_rn(z, __ffma2_rn(splat(kGeluC3), zz, splat(kGeluC))));
  const float2 du = __ffma2_rn(splat(3.f * kGeluC3), zz, splat(kGeluC));
  const float2 a = __fmul2_rn(__fmul2_rn(splat(0.5f), z), du);
  const float2 w = __ffma2_rn(make_float2(-t.x, -t.y), t, splat(1.f));
  return __ffma2_rn(a, w, __ffma2_rn(splat(0.5f), t, splat(0.5f)));
}

__device__ __forceinline__ void st_bf2(bf16* p, float a, float b) {
  *reinterpret_cast<bf162*>(p) = __floats2bfloat162_rn(a, b);
}

}  // namespace
}  // namespace fno_fused
}  // namespace sslbm
