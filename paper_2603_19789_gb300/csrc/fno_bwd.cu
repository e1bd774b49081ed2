// fno_bwd.cu -- fused backward kernels of the learned surrogate (the shapes of fno_fused.cuh).
//
// With dz_l = dL/dz_l (FP32 in memory), the backward pass runs as 1 + 5L launches after the seed:
//
//   row kernel, last:  dd = the seed (clamp and rescale), dp = Q2^T dd, dzp = dp gelu'(zp),
//                      dz_L = Q1^T dzp;  the gradients of Q2, q2, Q1, q1
//   per layer l = L .. 1:
//     y kernel:         dU = Fyi^T dG1 (per channel), its adjoint expansion dG
//     mix kernel:       dR_l (over the batch) and dhat = dG conj(R_l), per mode
//     inverse y kernel: dH1 = Fy^T dT(dhat)
//     row kernel, mid:  dz_{l-1} = gelu'(z_{l-1}) (B_l^T dz_l + dH1 Fx^T)      (l > 1)
//     row kernel, first: dh_0 = B_1^T dz_1 + dH1 Fx^T, the gradients of A0, a0  (l = 1)
//   and every row kernel, while a row of its dz is on chip, adds the row to the gradients of
//   its bias and channel map (dB = dz h^T) and (last, mid) transforms it along x, dG1 = dz Fx / n^2.
//
// What bounds it: the row kernels move dz (FP32), z and h (BF16) once each -- per cell and layer
// 4W read + 4W written + 2W + 2W bytes -- where the separate kernels they replace (a product per
// contraction, a pass for gelu', one for the bias sums) read or wrote dz nine times.  A row is
// taken in chunks of 128 columns (the last kernel, with 6 rows of operands instead of 4, of 64), so that two stages and
// two CTAs fit an SM: cp.async copies the next chunk while the current one is computed (the last
// kernel with one stage of 128 columns: 220 us), and the transform along x accumulates in
// registers across the chunks.  Weight and bias gradients accumulate in registers over all rows of a CTA and are added
// to memory once.  Products: mma.sync, BF16 operands rounded where the separate kernels rounded
// them, FP32 accumulation.
// One training step (B = 16, 256 x 256, W = 32, m = 12, L = 4, H = 64) took 5317 us with the separate
// kernels and takes 1403 us: its backward pass 3.7 ms then, under 0.8 ms now (ncu, per launch before
// the packed gelu': last 208, mid 107, first 59, y 14.6, mix 10.9, inverse y 10.3).  Mid moves 402 MB (60 us at 6.7 TB/s), last
// 600 MB (90 us); both issue the rest of the time (fragment loads, gelu').
#include <cuda_bf16.h>

#include <atomic>

#include "fno_bwd.cuh"
#include "fno_mma.cuh"

namespace sslbm {
namespace fno_fused {
namespace {

constexpr int kThreads = 256;  // 8 warps; warp w owns the chunk's columns [w CC/8, (w+1) CC/8)
constexpr int kCin = 8;

template <int W, int KF, int H, int CC, int NCH, int MODE>
struct BwdSmem {
  static constexpr int n = CC * NCH, SF = KF + 8, SC = CC + 8, SB = W + 8, SR = CC + 4;
  static constexpr int SQ1 = H + 8, SQ2 = 24;
  static constexpr bool last = MODE == BWD_LAST, mid = MODE == BWD_MID;
  static constexpr size_t align16(size_t v) { return (v + 15) / 16 * 16; }
  static constexpr size_t oF = 0;                                  // bf16 [n][SF]
  // bf16 [W][SC] the chunk of dz produced; at the end of a row f32 [W][KF] partial sums
  static constexpr size_t oDz = oF + align16((size_t)n * SF * 2);
  static constexpr size_t dz_bytes = (size_t)W * SC * 2 > (size_t)W * KF * 4 ? (size_t)W * SC * 2 : (size_t)W * KF * 4;
  static constexpr size_t oB = oDz + align16(dz_bytes);            // bf16 [W][SB]: B^T (mid, first)
  static constexpr size_t oH1 = oB + (last ? 0 : align16((size_t)W * SB * 2));   // bf16 [W][SF] (mid, first)
  static constexpr size_t oQ2 = oH1 + (last ? 0 : align16((size_t)W * SF * 2));   // bf16 [H][SQ2]: Q2^T
  static constexpr size_t oQ1 = oQ2 + (last ? align16((size_t)H * SQ2 * 2) : 0);  // bf16 [W][SQ1]: Q1^T
  static constexpr size_t oDD = oQ1 + (last ? align16((size_t)W * SQ1 * 2) : 0);  // bf16 [16][SC]: the seed
  static constexpr size_t oStage = oDD + (last ? align16((size_t)16 * SC * 2) : 0);
  // last: {zp [H][SC], p [H][SC], h_L [W][SC], h_{L-1} [W][SC]} bf16
  // mid, first: dz f32 [W][SR]; mid: {z [W][SC], h [W][SC]} bf16; first: x f32 [8][SR]
  static constexpr size_t raw = align16((size_t)W * SR * 4);
  static constexpr size_t stage = last ? (size_t)(2 * H + 2 * W) * SC * 2 : raw + (mid ? (size_t)2 * W * SC * 2 : (size_t)kCin * SR * 4);
  static constexpr size_t bytes = oStage + 2 * stage;
};

// rows of a BF16 field [b][C][y][x] (plane stride P): chunk of CC columns into [C][SC]
template <int CC, int SC>
__device__ __forceinline__ void copy_rows(bf16* dst, const bf16* src, int C, int64_t P, int tid) {
  for (int i = tid; i < C * (CC / 8); i += kThreads) {
    const int c = i / (CC / 8), j = i - c * (CC / 8);
    cp16(dst + c * SC + 8 * j, src + (size_t)c * P + 8 * j);
  }
}

template <int W, int KF, int H, int CC, int NCH, int MODE>
__global__ void __launch_bounds__(kThreads, 2) bwd_row_kernel(const BwdArgs a) {
  using S = BwdSmem<W, KF, H, CC, NCH, MODE>;
  constexpr int n = S::n, SF = S::SF, SC = S::SC, SB = S::SB, SR = S::SR, SQ1 = S::SQ1, SQ2 = S::SQ2;
  constexpr bool last = S::last, mid = S::mid, first = MODE == BWD_FIRST;
  constexpr int MT = W / 16, NT = CC / 64;  // 16-row tiles of W; 8-column tiles per warp
  constexpr int MH = H / 16;
  constexpr int64_t P = (int64_t)n * n;
  extern __shared__ __align__(16) unsigned char smem[];
  bf16* sF = reinterpret_cast<bf16*>(smem + S::oF);
  bf16* sDz = reinterpret_cast<bf16*>(smem + S::oDz);
  float* sRed = reinterpret_cast<float*>(smem + S::oDz);
  bf16* sB = reinterpret_cast<bf16*>(smem + S::oB);
  bf16* sH1 = reinterpret_cast<bf16*>(smem + S::oH1);
  bf16* sQ2 = reinterpret_cast<bf16*>(smem + S::oQ2);
  bf16* sQ1 = reinterpret_cast<bf16*>(smem + S::oQ1);
  bf16* sDD = reinterpret_cast<bf16*>(smem + S::oDD);
  unsigned char* stage0 = smem + S::oStage;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int gr = lane >> 2, tg = lane & 3;
  const int x0 = warp * (CC / 8);
  const int rows = a.B * n;

  // constants, published by the first barrier of the loop
  for (int i = tid; i < n * (KF / 8); i += kThreads) {
    const int r = i / (KF / 8), c = i - r * (KF / 8);
    *reinterpret_cast<uint4*>(sF + r * SF + 8 * c) = *reinterpret_cast<const uint4*>(a.F + (size_t)r * KF + 8 * c);
  }
  if (last) {
    for (int i = tid; i < H * 16; i += kThreads) {
      const int h = i / 16, c = i - h * 16;
      sQ2[h * SQ2 + c] = c < 5 ? a.Q2[c * H + h] : __float2bfloat16_rn(0.f);
    }
    for (int i = tid; i < H * W; i += kThreads) sQ1[(i % W) * SQ1 + i / W] = a.Q1[i];
    for (int i = tid; i < 11 * SC; i += kThreads) sDD[5 * SC + i] = __float2bfloat16_rn(0.f);
  } else {
    for (int i = tid; i < W * W; i += kThreads) sB[(i % W) * SB + i / W] = a.Bl[i];
  }

  // item it: chunk it % NCH of the CTA's row it / NCH
  auto row_of = [&](int it) { return (int64_t)blockIdx.x + (int64_t)(it / NCH) * gridDim.x; };
  auto issue = [&](int it, int s) {
    const int64_t row = row_of(it);
    if (row < rows) {
      const int64_t b = row / n, y = row - b * n;
      const int64_t off = y * n + (it % NCH) * CC;
      unsigned char* st = stage0 + s * S::stage;
      if (last) {
        bf16* d = reinterpret_cast<bf16*>(st);
        copy_rows<CC, SC>(d, a.zp + b * H * P + off, H, P, tid);
        copy_rows<CC, SC>(d + H * SC, a.p + b * H * P + off, H, P, tid);
        copy_rows<CC, SC>(d + 2 * H * SC, a.hL + b * W * P + off, W, P, tid);
        copy_rows<CC, SC>(d + (2 * H + W) * SC, a.hprev + b * W * P + off, W, P, tid);
      } else {
        float* dr = reinterpret_cast<float*>(st);
        const float* src = a.dzin + b * W * P + off;
        for (int i = tid; i < W * (CC / 4); i += kThreads) {
          const int c = i / (CC / 4), j = i - c * (CC / 4);
          cp16(dr + c * SR + 4 * j, src + (size_t)c * P + 4 * j);
        }
        if (mid) {
          bf16* d = reinterpret_cast<bf16*>(st + S::raw);
          copy_rows<CC, SC>(d, a.z + b * W * P + off, W, P, tid);
          copy_rows<CC, SC>(d + W * SC, a.hprev + b * W * P + off, W, P, tid);
        } else {
          float* dx = reinterpret_cast<float*>(st + S::raw);
          for (int i = tid; i < kCin * (CC / 4); i += kThreads) {
            const int c = i / (CC / 4), j = i - c * (CC / 4);
            cp16(dx + c * SR + 4 * j, a.x + (b * kCin + c) * P + off + 4 * j);
          }
        }
      }
    }
    commit();  // possibly empty: every thread keeps the same group count
  };

  // dH1 of the next row, in registers until its first chunk
  constexpr int NH1 = W * KF / 2 / kThreads;
  static_assert(W * KF / 2 % kThreads == 0, "dH1 pairs per thread");
  float2 h1[NH1];
  auto fetch_h1 = [&](int64_t row) {
    if (row < rows)
#pragma unroll
      for (int k = 0; k < NH1; ++k)
        h1[k] = reinterpret_cast<const float2*>(a.dH1 + (size_t)row * W * KF)[tid + k * kThreads];
  };

  // the seed's operands of the next chunk (last): y and dy of up to NSD channels of a column
  constexpr int G = kThreads / CC, NSD = (5 + G - 1) / G;
  float ysd[NSD], dsd[NSD];
  auto fetch_seed = [&](int it) {
    const int64_t row = row_of(it);
    if (row < rows) {
      const int64_t b = row / n, y = row - b * n;
#pragma unroll
      for (int k = 0; k < NSD; ++k) {
        const int c = tid / CC + G * k;
        if (c < 5) {
          const int64_t i = (b * 5 + c) * P + y * n + (it % NCH) * CC + tid % CC;
          ysd[k] = a.y[i];
          dsd[k] = a.dy[i];
        }
      }
    }
  };

  // accumulators over the CTA's rows
  constexpr int TW = MT * (W / 8), UW = first ? 1 : (TW + 7) / 8;   // dB tiles, per warp
  constexpr int KS = 8 / MT < CC / 16 ? 8 / MT : CC / 16;           // first: warps per dA0 tile
  constexpr int TQ = MH * (W / 8), UQ = (TQ + 7) / 8;               // dQ1 tiles
  float accW[UW][4], accQ1[UQ][4], accQ2[4];
  float bs[MT][2], bq1[MH][2], bq2[NSD];
#pragma unroll
  for (int u = 0; u < UW; ++u) accW[u][0] = accW[u][1] = accW[u][2] = accW[u][3] = 0.f;
#pragma unroll
  for (int u = 0; u < UQ; ++u) accQ1[u][0] = accQ1[u][1] = accQ1[u][2] = accQ1[u][3] = 0.f;
  accQ2[0] = accQ2[1] = accQ2[2] = accQ2[3] = 0.f;
#pragma unroll
  for (int i = 0; i < MT; ++i) bs[i][0] = bs[i][1] = 0.f;
#pragma unroll
  for (int i = 0; i < MH; ++i) bq1[i][0] = bq1[i][1] = 0.f;
#pragma unroll
  for (int k = 0; k < NSD; ++k) bq2[k] = 0.f;
  // the transform along x: tile group g, half kh of the chunk's columns
  constexpr int TPG = MT * (KF / 8) / 4;
  static_assert(MT * (KF / 8) % 4 == 0, "tile groups");
  const int g = warp & 3, kh = warp >> 2;
  float acc2[TPG][4];
#pragma unroll
  for (int u = 0; u < TPG; ++u) acc2[u][0] = acc2[u][1] = acc2[u][2] = acc2[u][3] = 0.f;

  if (last) fetch_seed(0);
  else fetch_h1(row_of(0));
  issue(0, 0);
  for (int it = 0; row_of(it) < rows; ++it) {
    const int64_t row = row_of(it), b = row / n, y = row - b * n;
    const int ch = it % NCH;
    const int64_t off = y * n + ch * CC;
    unsigned char* st = stage0 + (it & 1) * S::stage;
    float acc[MT][NT][4];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[mt][nt][r] = 0.f;

    issue(it + 1, (it + 1) & 1);
    if (last) {
      {  // the seed dd = sigma r [y > 0] (dy - lambda), lambda = sum(dy y) / sum y
        const float lam = a.seed[b], sg = a.seed[a.B + b], r = a.ratio[b];
#pragma unroll
        for (int k = 0; k < NSD; ++k) {
          const int c = tid / CC + G * k;
          if (c < 5) {
            const float f = ((c == 1 || c == 2) ? sg : 1.f) * r;
            const float d = ysd[k] > 0.f ? f * (dsd[k] - lam) : 0.f;
            bq2[k] += d;
            sDD[c * SC + tid % CC] = __float2bfloat16_rn(d);
          }
        }
      }
      fetch_seed(it + 1);
      wait_groups<1>();
      __syncthreads();
      bf16* sZ = reinterpret_cast<bf16*>(st);
      const bf16* sP = sZ + H * SC;
      {  // dzp = (Q2^T dd) gelu'(zp), in place of zp; the bias gradient from the FP32 values
        float acc3[MH][NT][4];
#pragma unroll
        for (int mh = 0; mh < MH; ++mh)
#pragma unroll
          for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int r = 0; r < 4; ++r) acc3[mh][nt][r] = 0.f;
        uint32_t bf[NT][2];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) load_b_kn1(bf[nt], sDD, SC, 0, x0 + nt * 8, lane);
#pragma unroll
        for (int mh = 0; mh < MH; ++mh) {
          uint32_t af[4];
          load_a(af, sQ2, SQ2, mh * 16, 0, lane);
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) mma(acc3[mh][nt], af, bf[nt][0], bf[nt][1]);
        }
#pragma unroll
        for (int mh = 0; mh < MH; ++mh)
#pragma unroll
          for (int h2 = 0; h2 < 2; ++h2)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
              bf162* q = reinterpret_cast<bf162*>(sZ + (mh * 16 + gr + 8 * h2) * SC + x0 + nt * 8 + 2 * tg);
              const float2 z = __bfloat1622float2(*q);
              const float2 d = gelu_grad2(z);
              const float v0 = acc3[mh][nt][2 * h2] * d.x, v1 = acc3[mh][nt][2 * h2 + 1] * d.y;
              bq1[mh][h2] += v0 + v1;
              *q = __floats2bfloat162_rn(v0, v1);
            }
      }
      if (warp < H / 8) {  // dQ2 += dd p^T
#pragma unroll
        for (int k0 = 0; k0 < CC; k0 += 16) {
          uint32_t af[4], bf[2];
          load_a(af, sDD, SC, 0, k0, lane);
          load_b_nk1(bf, sP, SC, k0, warp * 8, lane);
          mma(accQ2, af, bf[0], bf[1]);
        }
      }
      __syncwarp();
      // dz_L = Q1^T dzp on the warp's own columns
#pragma unroll
      for (int k0 = 0; k0 < H; k0 += 16) {
        uint32_t bf[NT][2];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) load_b_kn1(bf[nt], sZ, SC, k0, x0 + nt * 8, lane);
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
          uint32_t af[4];
          load_a(af, sQ1, SQ1, mt * 16, k0, lane);
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) mma(acc[mt][nt], af, bf[nt][0], bf[nt][1]);
        }
      }
    } else {
      if (ch == 0) {
#pragma unroll
        for (int k = 0; k < NH1; ++k) {
          const int i = 2 * (tid + k * kThreads);
          st_bf2(sH1 + (i / KF) * SF + i % KF, h1[k].x, h1[k].y);
        }
      }
      wait_groups<1>();
      __syncthreads();
      if (ch == NCH - 1) fetch_h1(row + gridDim.x);
      // dh = B^T dz + dH1 Fx^T; dz is rounded to BF16 as an operand
      const float* dr = reinterpret_cast<const float*>(st);
#pragma unroll
      for (int k0 = 0; k0 < W; k0 += 16) {
        uint32_t bf[NT][2];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
          const float* q = dr + (k0 + 2 * tg) * SR + x0 + nt * 8 + gr;
          const bf162 lo = __floats2bfloat162_rn(q[0], q[SR]), hi = __floats2bfloat162_rn(q[8 * SR], q[9 * SR]);
          bf[nt][0] = *reinterpret_cast<const uint32_t*>(&lo);
          bf[nt][1] = *reinterpret_cast<const uint32_t*>(&hi);
        }
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
          uint32_t af[4];
          load_a(af, sB, SB, mt * 16, k0, lane);
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) mma(acc[mt][nt], af, bf[nt][0], bf[nt][1]);
        }
      }
#pragma unroll
      for (int k0 = 0; k0 < KF; k0 += 16) {
        uint32_t bf[NT][2];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) load_b_nk1(bf[nt], sF + ch * CC * SF, SF, k0, x0 + nt * 8, lane);
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
          uint32_t af[4];
          load_a(af, sH1, SF, mt * 16, k0, lane);
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) mma(acc[mt][nt], af, bf[nt][0], bf[nt][1]);
        }
      }
    }

    // dz of this chunk: times gelu'(z) (mid), to memory in FP32 (last, mid), to sDz in BF16, and
    // into the bias sums
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
      for (int h2 = 0; h2 < 2; ++h2)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
          const int o = mt * 16 + gr + 8 * h2, xx = x0 + nt * 8 + 2 * tg;
          float v0 = acc[mt][nt][2 * h2], v1 = acc[mt][nt][2 * h2 + 1];
          if (mid) {
            const float2 z = __bfloat1622float2(*reinterpret_cast<const bf162*>(
                reinterpret_cast<const bf16*>(st + S::raw) + o * SC + xx));
            const float2 d = gelu_grad2(z);
            v0 *= d.x;
            v1 *= d.y;
          }
          if (!first) *reinterpret_cast<float2*>(a.dz + (b * W + o) * P + off + xx) = make_float2(v0, v1);
          bs[mt][h2] += v0 + v1;
          st_bf2(sDz + o * SC + xx, v0, v1);
        }
    __syncthreads();

    // the channel map's gradient: dB += dz h^T (first: dA0 += dh0 x^T, its few tiles cut along x)
    if (first) {
      const float* xr = reinterpret_cast<const float*>(st + S::raw);
      const int mt = warp % MT, ks = warp / MT;
      if (ks < KS) {
#pragma unroll
        for (int k0 = ks * (CC / KS); k0 < (ks + 1) * (CC / KS); k0 += 16) {
          const float2 v0 = *reinterpret_cast<const float2*>(xr + gr * SR + k0 + 2 * tg);
          const float2 v1 = *reinterpret_cast<const float2*>(xr + gr * SR + k0 + 8 + 2 * tg);
          const bf162 lo = __floats2bfloat162_rn(v0.x, v0.y), hi = __floats2bfloat162_rn(v1.x, v1.y);
          uint32_t af[4];
          load_a(af, sDz, SC, mt * 16, k0, lane);
          mma(accW[0], af, *reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
        }
      }
    } else {
      const bf16* sIn = last ? reinterpret_cast<const bf16*>(st) + (2 * H + W) * SC
                             : reinterpret_cast<const bf16*>(st + S::raw) + W * SC;
#pragma unroll
      for (int u = 0; u < UW; ++u) {
        const int t = warp + 8 * u;
        if (t < TW) {
          const int mt = t / (W / 8), nt = t - mt * (W / 8);
#pragma unroll
          for (int k0 = 0; k0 < CC; k0 += 16) {
            uint32_t af[4], bf[2];
            load_a(af, sDz, SC, mt * 16, k0, lane);
            load_b_nk1(bf, sIn, SC, k0, nt * 8, lane);
            mma(accW[u], af, bf[0], bf[1]);
          }
        }
      }
    }
    if (last) {  // dQ1 += dzp h_L^T
      const bf16* sZ = reinterpret_cast<const bf16*>(st);
      const bf16* sHL = sZ + 2 * H * SC;
#pragma unroll
      for (int u = 0; u < UQ; ++u) {
        const int t = warp + 8 * u;
        if (t < TQ) {
          const int mt = t / (W / 8), nt = t - mt * (W / 8);
#pragma unroll
          for (int k0 = 0; k0 < CC; k0 += 16) {
            uint32_t af[4], bf[2];
            load_a(af, sZ, SC, mt * 16, k0, lane);
            load_b_nk1(bf, sHL, SC, k0, nt * 8, lane);
            mma(accQ1[u], af, bf[0], bf[1]);
          }
        }
      }
    }
    if (!first) {  // dG1 += dz Fx over this chunk's half
      static_assert((KF / 8) % TPG == 0, "a group's tiles share their 16 channels");
      const int gm = g * TPG / (KF / 8) * 16, gn = g * TPG % (KF / 8) * 8;
#pragma unroll
      for (int k0 = kh * (CC / 2); k0 < (kh + 1) * (CC / 2); k0 += 16) {
        uint32_t af[4];
        load_a(af, sDz, SC, gm, k0, lane);
        mma_tiles_kn<TPG>(acc2, af, sF + ch * CC * SF, SF, k0, gn, lane);
      }
    }
    __syncthreads();  // the stage and sDz are free

    if (!first && ch == NCH - 1) {
      // the row's dG1: the upper halves through shared memory, the lower halves add and store
      if (kh == 1) {
#pragma unroll
        for (int u = 0; u < TPG; ++u) {
          const int t = g * TPG + u, mt = t / (KF / 8), nt = t - mt * (KF / 8);
#pragma unroll
          for (int h2 = 0; h2 < 2; ++h2)
            *reinterpret_cast<float2*>(sRed + (mt * 16 + gr + 8 * h2) * KF + nt * 8 + 2 * tg) =
                make_float2(acc2[u][2 * h2], acc2[u][2 * h2 + 1]);
        }
      }
      __syncthreads();
      if (kh == 0) {
        float* dst = a.dG1 + (size_t)row * W * KF;
#pragma unroll
        for (int u = 0; u < TPG; ++u) {
          const int t = g * TPG + u, mt = t / (KF / 8), nt = t - mt * (KF / 8);
#pragma unroll
          for (int h2 = 0; h2 < 2; ++h2) {
            const int i = (mt * 16 + gr + 8 * h2) * KF + nt * 8 + 2 * tg;
            const float2 q = *reinterpret_cast<const float2*>(sRed + i);
            *reinterpret_cast<float2*>(dst + i) =
                make_float2((acc2[u][2 * h2] + q.x) * a.scale, (acc2[u][2 * h2 + 1] + q.y) * a.scale);
          }
        }
      }
#pragma unroll
      for (int u = 0; u < TPG; ++u) acc2[u][0] = acc2[u][1] = acc2[u][2] = acc2[u][3] = 0.f;
    }
  }
  wait_groups<0>();

  // the CTA's sums into the gradients
  auto add_tile = [&](float* dst, const float (&v)[4], int r0, int c0, int rows_, int cols) {
#pragma unroll
    for (int h2 = 0; h2 < 2; ++h2) {
      const int r = r0 + gr + 8 * h2, c = c0 + 2 * tg;
      if (r < rows_) {
        atomicAdd(dst + r * cols + c, v[2 * h2]);
        atomicAdd(dst + r * cols + c + 1, v[2 * h2 + 1]);
      }
    }
  };
  auto add_bias = [&](float* dst, float v) {  // the four lanes of a row hold its columns
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    if (tg == 0) atomicAdd(dst, v);
  };
  if (first) {
    if (warp / MT < KS) add_tile(a.gW, accW[0], warp % MT * 16, 0, W, kCin);
  } else {
#pragma unroll
    for (int u = 0; u < UW; ++u) {
      const int t = warp + 8 * u;
      if (t < TW) add_tile(a.gW, accW[u], t / (W / 8) * 16, t % (W / 8) * 8, W, W);
    }
  }
#pragma unroll
  for (int mt = 0; mt < MT; ++mt)
#pragma unroll
    for (int h2 = 0; h2 < 2; ++h2) add_bias(a.gb + mt * 16 + gr + 8 * h2, bs[mt][h2]);
  if (last) {
#pragma unroll
    for (int u = 0; u < UQ; ++u) {
      const int t = warp + 8 * u;
      if (t < TQ) add_tile(a.gQ1, accQ1[u], t / (W / 8) * 16, t % (W / 8) * 8, H, W);
    }
    if (warp < H / 8) add_tile(a.gQ2, accQ2, 0, warp * 8, 5, H);
#pragma unroll
    for (int mh = 0; mh < MH; ++mh)
#pragma unroll
      for (int h2 = 0; h2 < 2; ++h2) add_bias(a.gq1 + mh * 16 + gr + 8 * h2, bq1[mh][h2]);
#pragma unroll
    for (int k = 0; k < NSD; ++k) {
      float v = bq2[k];  // a warp's lanes share their channel
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      const int c = tid / CC + G * k;
      if (lane == 0 && c < 5) atomicAdd(a.gq2 + c, v);
    }
  }
}

// ---- adjoint of the inverse transform along y ------------------------------------------------

// CTA = (sample b, CG channels): D[c] = Fyi^T (2m x n) dG1[b, :, c, :] (n x 4m), then the adjoint
// of the expansion, dG[b, c, j, q] = c_q (D[2q, 2j] + D[2q+1, 2j+1], D[2q, 2j+1] - D[2q+1, 2j])
template <int KF, int CG>
__global__ void __launch_bounds__(128) bwd_y_kernel(const float* __restrict__ dG1, const bf16* __restrict__ Fyi,
                                                    float2* __restrict__ dG, int W, int n) {
  constexpr int M2 = KF / 2, m = KF / 4, NC = CG * KF, SC = NC + 8, SY = 40, modes = 2 * m * m;
  constexpr int TPW = NC / 8 / 4;
  static_assert(NC / 8 % 4 == 0 && M2 <= 32 && M2 % 8 == 0, "tiling");
  extern __shared__ __align__(16) unsigned char smem[];
  bf16* sFyi = reinterpret_cast<bf16*>(smem);          // [n][SY], columns >= 2m zero
  bf16* sT = sFyi + (size_t)n * SY;                     // [n][SC]
  float* sO = reinterpret_cast<float*>(sT);             // [2m][NC], after the product
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int gr = lane >> 2, tg = lane & 3;
  const int b = blockIdx.y, c0 = blockIdx.x * CG;
  for (int i = tid; i < n * 4; i += 128) {
    const int yy = i >> 2, j = i & 3;
    *reinterpret_cast<uint4*>(sFyi + yy * SY + 8 * j) =
        8 * j < M2 ? *reinterpret_cast<const uint4*>(Fyi + (size_t)yy * M2 + 8 * j) : make_uint4(0, 0, 0, 0);
  }
#pragma unroll 4
  for (int i = tid; i < n * (NC / 4); i += 128) {
    const int yy = i / (NC / 4), j = i - yy * (NC / 4);
    const float4 v = *reinterpret_cast<const float4*>(dG1 + (((size_t)b * n + yy) * W + c0) * KF + 4 * j);
    st_bf2(sT + yy * SC + 4 * j, v.x, v.y);
    st_bf2(sT + yy * SC + 4 * j + 2, v.z, v.w);
  }
  __syncthreads();
  float acc[2][TPW][4];
#pragma unroll
  for (int mt = 0; mt < 2; ++mt)
#pragma unroll
    for (int u = 0; u < TPW; ++u)
#pragma unroll
      for (int r = 0; r < 4; ++r) acc[mt][u][r] = 0.f;
  for (int k0 = 0; k0 < n; k0 += 16) {
    uint32_t af[2][4];
    load_a_t(af[0], sFyi, SY, 0, k0, lane);
    load_a_t(af[1], sFyi, SY, 16, k0, lane);
#pragma unroll
    for (int u = 0; u < TPW; ++u) {
      uint32_t bf[2];
      load_b_kn1(bf, sT, SC, k0, (warp * TPW + u) * 8, lane);
      mma(acc[0][u], af[0], bf[0], bf[1]);
      mma(acc[1][u], af[1], bf[0], bf[1]);
    }
  }
  __syncthreads();
#pragma unroll
  for (int mt = 0; mt < 2; ++mt)
#pragma unroll
    for (int u = 0; u < TPW; ++u)
#pragma unroll
      for (int h2 = 0; h2 < 2; ++h2) {
        const int r = mt * 16 + gr + 8 * h2, col = (warp * TPW + u) * 8 + 2 * tg;
        if (r < M2) *reinterpret_cast<float2*>(sO + r * NC + col) = make_float2(acc[mt][u][2 * h2], acc[mt][u][2 * h2 + 1]);
      }
  __syncthreads();
  for (int i = tid; i < CG * modes; i += 128) {
    const int cc = i / modes, k = i - cc * modes, j = k / m, q = k - j * m;
    const float* D = sO + cc * KF;
    const float c = q == 0 ? 1.f : 2.f;
    dG[((size_t)b * W + c0 + cc) * modes + k] =
        make_float2(c * (D[(2 * q) * NC + 2 * j] + D[(2 * q + 1) * NC + 2 * j + 1]),
                    c * (D[(2 * q) * NC + 2 * j + 1] - D[(2 * q + 1) * NC + 2 * j]));
  }
}

// ---- spectral mix, adjoint ------------------------------------------------------------------

// CTA = MC modes, each mode's weights, modes and gradients read once: for blockIdx.y = 0
// dhat[b, i, k] = sum_o dG[b, o, k] conj(R[i, o, k]), for 1 dR[i, o, k] = sum_b conj(hat[b, i, k])
// dG[b, o, k], all b, i, o.
template <int W, int MC, int BC>
__global__ void __launch_bounds__(16 * W) bwd_mix_kernel(const float2* __restrict__ hat, const float2* __restrict__ dG,
                                                         const float2* __restrict__ R, float2* __restrict__ dR,
                                                         float2* __restrict__ dhat, int B, int modes) {
  extern __shared__ __align__(16) unsigned char smem[];
  float2* sG = reinterpret_cast<float2*>(smem);  // [BC][W][MC]
  float2* sR = sG + (size_t)BC * W * MC;         // dhat: R transposed, [o][i][MC]; dR: hat, [BC][W][MC]
  constexpr int NT = 16 * W, NI = W * W / NT;    // threads; (i, o) pairs per thread
  const int tid = threadIdx.x, k0 = blockIdx.x * MC;
  const int mc = min(MC, modes - k0);
  const float2 zero = make_float2(0.f, 0.f);
  const bool weights = blockIdx.y == 1;
  if (!weights)
    for (int t = tid; t < W * W * MC; t += NT) {
      const int io = t / MC, kk = t - io * MC, i = io / W, o = io - i * W;
      sR[(o * W + i) * MC + kk] = kk < mc ? R[(size_t)io * modes + k0 + kk] : zero;
    }
  const int o = tid % W, i0 = tid / W;
  float2 acc[NI][MC];
#pragma unroll
  for (int u = 0; u < NI; ++u)
#pragma unroll
    for (int kk = 0; kk < MC; ++kk) acc[u][kk] = zero;
  for (int b0 = 0; b0 < B; b0 += BC) {
    const int nb = min(BC, B - b0);
    __syncthreads();
    for (int t = tid; t < nb * W * MC; t += NT) {
      const int bi = t / MC, kk = t - bi * MC;
      const size_t off = ((size_t)b0 * W + bi) * modes + k0 + kk;
      sG[t] = kk < mc ? dG[off] : zero;
      if (weights) sR[t] = kk < mc ? hat[off] : zero;
    }
    __syncthreads();
    if (weights) {
      for (int b = 0; b < nb; ++b) {
#pragma unroll
        for (int kk = 0; kk < MC; ++kk) {
          const float2 d = sG[(b * W + o) * MC + kk];
#pragma unroll
          for (int u = 0; u < NI; ++u) {
            const float2 h = sR[(b * W + i0 + (NT / W) * u) * MC + kk];
            acc[u][kk].x = fmaf(h.x, d.x, fmaf(h.y, d.y, acc[u][kk].x));
            acc[u][kk].y = fmaf(h.x, d.y, fmaf(-h.y, d.x, acc[u][kk].y));
          }
        }
      }
    } else {
      for (int t = tid; t < nb * W; t += NT) {
        const int bl = t / W, i = t - bl * W;
        float2 s[MC];
#pragma unroll
        for (int kk = 0; kk < MC; ++kk) s[kk] = zero;
#pragma unroll 8
        for (int oo = 0; oo < W; ++oo)
#pragma unroll
          for (int kk = 0; kk < MC; ++kk) {
            const float2 d = sG[(bl * W + oo) * MC + kk], r = sR[(oo * W + i) * MC + kk];
            s[kk].x = fmaf(d.x, r.x, fmaf(d.y, r.y, s[kk].x));
            s[kk].y = fmaf(d.y, r.x, fmaf(-d.x, r.y, s[kk].y));
          }
#pragma unroll
        for (int kk = 0; kk < MC; ++kk)
          if (kk < mc) dhat[((size_t)(b0 + bl) * W + i) * modes + k0 + kk] = s[kk];
      }
    }
  }
  if (weights) {
#pragma unroll
    for (int u = 0; u < NI; ++u)
#pragma unroll
      for (int kk = 0; kk < MC; ++kk)
        if (kk < mc) dR[(size_t)((i0 + (NT / W) * u) * W + o) * modes + k0 + kk] = acc[u][kk];
  }
}

// ---- adjoint of the transform along y --------------------------------------------------------

// CTA = (sample b, OG channels): T[c] = the adjoint combination of dhat[b, c] (2m x 4m), then
// dH1[b, y, c, :] = Fy[:, y]^T T[c], FP32
template <int KF, int OG>
__global__ void __launch_bounds__(256) bwd_iy_kernel(const float2* __restrict__ dhat, const bf16* __restrict__ Fy,
                                                     float* __restrict__ dH1, int W, int n) {
  constexpr int M2 = KF / 2, m = KF / 4, modes = 2 * m * m, NC = OG * KF, SU = NC + 8;
  constexpr int NTT = NC / 8;
  static_assert(NTT % 2 == 0 && M2 <= 32, "tiling");
  extern __shared__ __align__(16) unsigned char smem[];
  const int SY = n + 8;
  bf16* sFy = reinterpret_cast<bf16*>(smem);  // [32][SY], rows >= 2m zero
  bf16* sU = sFy + (size_t)32 * SY;            // [32][SU], rows >= 2m zero
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int gr = lane >> 2, tg = lane & 3;
  const int b = blockIdx.y, c0 = blockIdx.x * OG;
  for (int i = tid; i < 32 * (n / 8); i += 256) {
    const int r = i / (n / 8), j = i - r * (n / 8);
    *reinterpret_cast<uint4*>(sFy + r * SY + 8 * j) =
        r < M2 ? *reinterpret_cast<const uint4*>(Fy + (size_t)r * n + 8 * j) : make_uint4(0, 0, 0, 0);
  }
  const bf16 zero = __float2bfloat16_rn(0.f);
  for (int i = tid; i < (32 - M2) * NC; i += 256) sU[(M2 + i / NC) * SU + i % NC] = zero;
  for (int i = tid; i < OG * modes; i += 256) {
    const int cc = i / modes, k = i - cc * modes;
    const float2 v = dhat[((size_t)b * W + c0 + cc) * modes + k];
    const int j = k / m, q = k - j * m;
    bf16* U = sU + cc * KF;
    U[(2 * q) * SU + 2 * j] = __float2bfloat16_rn(v.x);
    U[(2 * q + 1) * SU + 2 * j + 1] = __float2bfloat16_rn(-v.x);
    U[(2 * q) * SU + 2 * j + 1] = __float2bfloat16_rn(v.y);
    U[(2 * q + 1) * SU + 2 * j] = __float2bfloat16_rn(v.y);
  }
  __syncthreads();
  for (int mt = warp; mt < n / 16; mt += 8) {
    float acc[NTT][4];
#pragma unroll
    for (int t = 0; t < NTT; ++t)
#pragma unroll
      for (int r = 0; r < 4; ++r) acc[t][r] = 0.f;
#pragma unroll
    for (int k0 = 0; k0 < 32; k0 += 16) {
      uint32_t af[4];
      load_a_t(af, sFy, SY, mt * 16, k0, lane);
#pragma unroll
      for (int t = 0; t < NTT; t += 2) {
        uint32_t bf[4];
        load_b_kn2(bf, sU, SU, k0, t * 8, lane);
        mma(acc[t], af, bf[0], bf[1]);
        mma(acc[t + 1], af, bf[2], bf[3]);
      }
    }
#pragma unroll
    for (int t = 0; t < NTT; ++t)
#pragma unroll
      for (int h2 = 0; h2 < 2; ++h2) {
        const int yy = mt * 16 + gr + 8 * h2, col = t * 8 + 2 * tg;
        *reinterpret_cast<float2*>(dH1 + (((size_t)b * n + yy) * W + c0) * KF + col) =
            make_float2(acc[t][2 * h2], acc[t][2 * h2 + 1]);
      }
  }
}

// ---- launchers -------------------------------------------------------------------------------

constexpr int kMaxDev = 64;

template <int W, int KF, int H, int CC, int NCH, int MODE>
cudaError_t launch_t(const BwdArgs& a, cudaStream_t s) {
  using S = BwdSmem<W, KF, H, CC, NCH, MODE>;
  static std::atomic<int> resident[kMaxDev];  // CTAs on the device; set after the kernel's attribute
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDev) return cudaErrorInvalidDevice;
  auto kern = bwd_row_kernel<W, KF, H, CC, NCH, MODE>;
  int ctas = resident[dev].load(std::memory_order_acquire);
  if (!ctas) {
    int per = 0, sms = 0;
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::bytes)) != cudaSuccess)
      return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, kThreads, S::bytes)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if (per < 1) return cudaErrorInvalidConfiguration;
    ctas = per * sms;
    resident[dev].store(ctas, std::memory_order_release);
  }
  const int rows = a.B * S::n;
  kern<<<rows < ctas ? rows : ctas, kThreads, S::bytes, s>>>(a);
  return cudaGetLastError();
}

template <int W, int KF, int H, int MODE>
cudaError_t by_n(int n, const BwdArgs& a, cudaStream_t s) {
  constexpr int CC = MODE == BWD_LAST ? 64 : 128;  // columns per chunk (two stages of it in shared memory)
  switch (n) {
    case 64: return launch_t<W, KF, H, 64, 1, MODE>(a, s);
    case 128: return launch_t<W, KF, H, CC, 128 / CC, MODE>(a, s);
    case 256: return launch_t<W, KF, H, CC, 256 / CC, MODE>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

template <int W, int KF, int H>
cudaError_t by_mode(int mode, int n, const BwdArgs& a, cudaStream_t s) {
  switch (mode) {
    case BWD_LAST: return by_n<W, KF, H, BWD_LAST>(n, a, s);
    case BWD_MID: return by_n<W, KF, H, BWD_MID>(n, a, s);
    case BWD_FIRST: return by_n<W, KF, H, BWD_FIRST>(n, a, s);
    default: return cudaErrorInvalidValue;
  }
}

template <int W, int KF>
cudaError_t spectral_t(int B, int n, const BwdSpectral& a, cudaStream_t s) {
  constexpr int CG = 2, MC = 2, BC = 16, m = KF / 4, modes = 2 * m * m, NC = CG * KF;
  const size_t by = (size_t)n * 40 * 2 + (size_t)n * (NC + 8) * 2;
  cudaError_t e = cudaFuncSetAttribute(bwd_y_kernel<KF, CG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)by);
  if (e != cudaSuccess) return e;
  bwd_y_kernel<KF, CG><<<dim3(W / CG, B), 128, by, s>>>(a.dG1, a.Fyi, reinterpret_cast<float2*>(a.dG), W, n);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const size_t bm = ((size_t)(W > BC ? W : BC) * W * MC + (size_t)BC * W * MC) * sizeof(float2);
  e = cudaFuncSetAttribute(bwd_mix_kernel<W, MC, BC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bm);
  if (e != cudaSuccess) return e;
  bwd_mix_kernel<W, MC, BC><<<dim3((modes + MC - 1) / MC, 2), 16 * W, bm, s>>>(
      reinterpret_cast<const float2*>(a.hat), reinterpret_cast<const float2*>(a.dG),
      reinterpret_cast<const float2*>(a.R), reinterpret_cast<float2*>(a.dR), reinterpret_cast<float2*>(a.dhat), B,
      modes);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const size_t bi = (size_t)32 * (n + 8) * 2 + (size_t)32 * (NC + 8) * 2;
  e = cudaFuncSetAttribute(bwd_iy_kernel<KF, CG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bi);
  if (e != cudaSuccess) return e;
  bwd_iy_kernel<KF, CG><<<dim3(W / CG, B), 256, bi, s>>>(reinterpret_cast<const float2*>(a.dhat), a.Fy, a.dH1, W, n);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_bwd_row(int mode, int W, int m, int H, int n, const BwdArgs& a, cudaStream_t s) {
  if (!supported(W, m, H, n) || a.B < 1) return cudaErrorInvalidValue;
  if (W == 32) return by_mode<32, 48, 64>(mode, n, a, s);
  return by_mode<16, 32, 32>(mode, n, a, s);
}

cudaError_t launch_bwd_spectral(int W, int m, int H, int B, int n, const BwdSpectral& a, cudaStream_t s) {
  if (!supported(W, m, H, n) || B < 1) return cudaErrorInvalidValue;
  if (W == 32) return spectral_t<32, 48>(B, n, a, s);
  return spectral_t<16, 32>(B, n, a, s);
}

}  // namespace fno_fused
}  // namespace sslbm
