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

// the same GELU as the unfused path: the tanh form, 0.5 z (1 + tanh(sqrt(2/pi) (z + 0.044715 z^3))),
// with the hardware tanh (tanh.approx.f32)
__device__ __forceinline__ float gelu(float z) {
  float t;
  asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(0.7978845608028654f * fmaf(0.044715f * z, z * z, z)));
  const float h = 0.5f * z;
  return fmaf(h, t, h);
}

// its derivative, 0.5 (1 + t) + 0.5 z (1 - t^2) du/dz
__device__ __forceinline__ float gelu_grad(float z) {
  float t;
  asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(0.7978845608028654f * fmaf(0.044715f * z, z * z, z)));
  const float du = 0.7978845608028654f * fmaf(3.f * 0.044715f * z, z, 1.f);
  return fmaf(0.5f * z * du, fmaf(-t, t, 1.f), 0.5f * (1.f + t));
}

__device__ __forceinline__ void st_bf2(bf16* p, float a, float b) {
  *reinterpret_cast<bf162*>(p) = __floats2bfloat162_rn(a, b);
}

}  // namespace
}  // namespace fno_fused
}  // namespace sslbm
