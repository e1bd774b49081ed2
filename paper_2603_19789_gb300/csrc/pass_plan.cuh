// pass_plan.cuh -- how a call of n steps is cut into passes, by rules and measured costs (host code only).
//
// A pass reads one state buffer and writes the other, so the buffer that holds the state after a call
// depends on the number of passes.  A captured call is replayed from the buffer it was captured on:
// it advances the state again only if the state is back there, which takes an even number of
// passes.  Under the default blocking and in the multi-step BGK passes, where the number is a matter of
// speed alone, it is therefore even in a captured call, and has the parity of the plain cut --
// ceil(n / depth) passes, for BGK n -- in every later call of that handle, so that calls between
// replays leave the state in the buffer where the plain cut would.
#pragma once
#include <stddef.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "sslbm.h"

namespace sslbm {

enum { kAnyParity = -1, kEvenPasses = 0, kOddPasses = 1 };

// Passes of at most `depth` steps that cover n: the fewest, one more where their number has to be
// odd or even (a single step is one pass).
inline int64_t pass_count(int64_t n, int depth, int parity) {
  const int64_t p = (n + depth - 1) / depth;
  return parity != kAnyParity && (p & 1) != parity && p < n ? p + 1 : p;
}

// Required parity of a call's passes: `captured` is whether this call is being captured, `was_captured`
// whether an earlier one of the handle was; depth: that of the plain cut.
inline int pass_parity(int64_t n, int depth, bool captured, bool was_captured) {
  if (captured) return kEvenPasses;
  return was_captured ? (int)(((n + depth - 1) / depth) & 1) : kAnyParity;
}

// Depth of the next of the pipeline passes that cover n steps: passes deeper than depth are taken
// whole, where they leave at least three steps or none; else the n steps are cut into passes whose
// depths differ by at most one (100 steps at depth 7: 10 of 7 and 5 of 6), rather than full passes and
// a shallow remainder, which runs at a lower rate per step.  parity: of the passes that remain.
inline int next_pass_depth(int64_t n, int depth, int deep, int parity) {
  if (deep > depth && ((n == deep && parity != kEvenPasses) || n >= deep + 3)) return deep;
  const int64_t passes = pass_count(n, depth, parity);
  return (int)((n + passes - 1) / passes);
}

// Parity of the passes that remain after one more.
inline int flip_parity(int parity) { return parity == kAnyParity ? parity : 1 - parity; }

// ---- what passes cost ------------------------------------------------------------------------

// Shared memory of a row-pipeline CTA of depth K: eight rows of level 0 and four of each further level
// but the last, `planes` planes of 128 columns each, and on the varying-diffusion lattice 32 rows of
// the two scale planes; and the CTAs that an SM holds (228 KB, 1 KB of it per CTA, 16 warps at the
// kernels' register limit).
constexpr size_t pipe_bytes(int planes, int K, bool scales) {
  return (size_t)512 * planes * (8 + 4 * (K - 1)) + (scales ? (size_t)32 * 2 * 512 : 0);
}
constexpr int pipe_ctas_per_sm(size_t bytes, int K) {
  const int by_smem = (int)(228 * 1024 / (bytes + 1024)), by_regs = 16 / K;
  return by_smem < 1 ? 1 : by_smem < by_regs ? by_smem : by_regs;
}

// Measured on a GB300 (us): a row-pipeline pass of depth K takes pass + waves * iterations * (it +
// it_warp * K * CTAs per SM), and one wave of register-tile passes fix + depth * step, by rows per warp
// (1, 2, 4; no tile pass: 0).
struct PassCost {
  int planes;      // of the pipeline's rows
  bool whole;      // fitted with the CTAs that fit an SM, and those of the fullest SM; else 16 / K and the average
  int segments;    // row segments in units of what fits at once
  int deep;        // a default depth beside 4, or 4
  double pass, it, it_warp;
  double shallow[2];  // factors of passes of two and three steps
  double fix[3], step[3];
};
constexpr PassCost kCostD2q5{5, false, 1, 4, 6.4, 0.43, 0.053, {1.15, 1.0}, {2.1, 3.5, 4.5}, {0.38, 0.44, 0.77}};
constexpr PassCost kCostD2q9{5, false, 1, 4, 5.9, 0.54, 0.068, {1.15, 1.0}, {2.1, 3.5, 4.5}, {0.40, 0.50, 1.05}};
constexpr PassCost kCostD2q9Walls{5, false, 2, 4, 18.9, 0.21, 0.134, {1.1, 1.0}, {2.1, 2.8, 4.0}, {0.47, 0.85, 1.90}};
constexpr PassCost kCostVard{5, true, 1, 6, 4.1, 0.66, 0.070, {1.3, 1.25}, {2.1, 2.8, 6.0}, {0.42, 0.80, 1.55}};
constexpr PassCost kCostSplit{6, true, 1, 8, 4.0, 0.52, 0.061, {1.0, 1.0}, {0, 0, 0}, {0, 0, 0}};
constexpr PassCost kCostKahan{10, true, 1, 8, 4.0, 0.70, 0.117, {1.0, 1.0}, {0, 0, 0}, {0, 0, 0}};

inline const PassCost* pass_cost(int lattice, int precision, int bc) {
  if (lattice == SSLBM_LATTICE_D2Q5 && (precision == SSLBM_FP32 || precision == SSLBM_FP32_DEV)) return &kCostD2q5;
  if (lattice == SSLBM_LATTICE_D2Q5 && precision == SSLBM_FP32_SPLIT) return &kCostSplit;
  if (lattice == SSLBM_LATTICE_D2Q5 && precision == SSLBM_FP32_KAHAN) return &kCostKahan;
  if (precision != SSLBM_FP32) return nullptr;
  if (lattice == SSLBM_LATTICE_D2Q5_VARD) return &kCostVard;
  if (lattice == SSLBM_LATTICE_D2Q9) return bc == SSLBM_BC_PERIODIC ? &kCostD2q9 : &kCostD2q9Walls;
  return nullptr;
}

// A pipeline pass of depth k at its automatic segments.
inline double pipe_pass_us(const PassCost& c, int64_t nx, int64_t ny, int k, int sms) {
  const int per = c.whole ? pipe_ctas_per_sm(pipe_bytes(c.planes, k, &c == &kCostVard), k) : 16 / k;
  const double res = (double)sms * per, strips = std::ceil((double)nx / (128 - 8 * ((k + 3) / 4)));
  const double segs = std::max(1.0, std::floor(c.segments * res / strips));
  const double rows = std::max(4.0 * k, std::ceil((double)ny / segs)), ctas = strips * std::ceil((double)ny / rows);
  const double load = std::min((double)per, c.whole ? std::ceil(ctas / sms) : ctas / sms);
  const double us = c.pass + std::ceil(ctas / res) * (std::floor((rows + 4 * k - 3) / 2) + 1) * (c.it + c.it_warp * k * load);
  return k < 4 ? us * c.shallow[k - 2] : us;
}

// Depth of the pipeline passes that the default blocking takes where n allows: 4, or the update's deeper
// one where the estimate has it ahead per step.  A deeper pass saves passes over memory but fills for
// 4 K - 3 rows per segment and leaves fewer, larger CTAs.  us per step at depth 4 and deeper: varying
// diffusion (6) 2048^2 22.1 and 19.9, 430 x 5304 13.7 and 12.6, 1500 x 1100 10.3 and 10.4, 12000 x 300 17.9
// and 22.5; split (8) 2048^2 15.8 and 15.2, 800 x 600 5.5 and 4.2, 3786 x 4055 51.0 and 51.6, 12000 x 300
// 14.9 and 17.1; Kahan (8) 2048^2 30.1 and 29.4, 800 x 600 7.3 and 6.8, 3000 x 2200 41.3 and 47.9, 350^2 5.6
// and 6.8, 12000 x 300 24.2 and 33.3.  The plain storage and D2Q9 gain and lose a few percent unevenly at
// every depth and stay at 4.
inline int default_pass_depth(const PassCost& c, int64_t nx, int64_t ny, int sms) {
  return pipe_pass_us(c, nx, ny, c.deep, sms) / c.deep < pipe_pass_us(c, nx, ny, 4, sms) / 4 ? c.deep : 4;
}

constexpr int kTileCols = 64, kTileWarps = 16;  // a register tile's columns and warps (tile.cu)

// The tile passes' rows per warp and depth for n steps of a grid, or false where the row pipeline
// (passes of `deep` steps and the rest of up to 4) is expected to be faster or the update has no tile
// pass: tile passes recompute their halo but need no pipeline fill, so they win where a pipeline would
// have only short segments to stream.  parity: of the number of passes.
// Of the choices measured (10 grids from 200^2 to 2048^2, 12000 x 300 and 430 x 5304, 2 to 20 steps) the one it
// picks is 1.3% slower on average than the fastest for D2Q5, 0.8% D2Q9, 0.4% with walls, 0.8% the
// varying diffusion; at most 19% (1500 x 1100 D2Q5, two steps).
// The lines, in us per step of 24 (tile, pipeline): D2Q5 430 x 5304 9.2 and 8.7, 1300 x 1000 5.0 and
// 5.8; D2Q9 walls 2048^2 27.6 and 31.4, 3000 x 2200 43.7 and 37.1.
struct TilePlan {
  int nr, depth;
};
inline bool tile_plan(const PassCost& c, int64_t nx, int64_t ny, int64_t n, int deep, int parity, int sms,
                      TilePlan* plan) {
  // beyond 32 cells per column and SM the pipeline is ahead whatever the estimate's error
  if (c.step[0] <= 0 || n < 2 || nx > (1 << 22) || ny > (1 << 22) || nx * ny > (int64_t)1 << 24) return false;
  double best = 1e300;
  for (int i = 0; i < 3; ++i) {
    const int nr = 1 << i, rows = kTileWarps * nr;
    for (int k = 2; k <= n && 2 * k < rows && k < 29; ++k) {
      const int ke = (k + 1) & ~1;
      const double ctas = std::ceil((double)nx / (kTileCols - 2 * ke)) * std::ceil((double)ny / (rows - 2 * k));
      const int64_t passes = pass_count(n, k, parity);  // of equal depth
      const double t = std::ceil(ctas / sms) * (c.fix[i] * passes + c.step[i] * n) / n;
      if (t < best) {
        best = t;
        *plan = TilePlan{nr, k};
      }
    }
  }
  // the pipeline's cut of n steps; beyond 48 its pattern repeats
  const int m = (int)std::min<int64_t>(n, 48);
  double us[SSLBM_MAX_DEPTH + 1] = {0.0}, pipe = 0.0;
  for (int left = m; left > 0;) {
    const int k = next_pass_depth(left, 4, deep, kAnyParity);
    if (us[k] == 0.0) us[k] = pipe_pass_us(c, nx, ny, k, sms);
    pipe += us[k] / m;
    left -= k;
  }
  return best <= pipe;
}

}  // namespace sslbm
