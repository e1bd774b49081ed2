// tile.cuh -- the register-tile pass of small grids (tile.cu).
#pragma once
#include "pass_plan.cuh"
#include "sslbm_internal.cuh"

namespace sslbm {

// K steps of the FP32 update (D2Q5 plain and deviation storage, D2Q9, varying diffusion) from `in`
// to `out`, regions of 64 x 16 nr cells; nr = 1, 2 or 4, 2 K < 16 nr and K < 31.
cudaError_t launch_tile(int lattice, int precision, const GridView& g, const void* coeffs, const void* in, void* out,
                        const void* kx, const void* ky, int nr, int K, cudaStream_t s);

// Steps per pipeline pass that the default blocking takes where n allows.  Measured at automatic
// segments, no-flux, us per step of 48 steps at depth 4 against the depth below, at 8192^2, 2048^2
// and 1700 x 1500: varying diffusion 350 -> 247, 25.3 -> 18.8, 16 -> 13; Kahan 478 -> 410, 34.6 ->
// 29.6, 23 -> 20.3; split 213 -> 192, 16.5 -> 15.1, 11.8 -> 10.6.  The plain storage gains 5% at
// depth 8 on 8192^2 and loses 13% on 3786 x 6055, D2Q9 is as uneven: those stay at 4.
inline int default_pass_depth(int lattice, int precision) {
  if (lattice == SSLBM_LATTICE_D2Q5_VARD) return 6;
  return lattice == SSLBM_LATTICE_D2Q5 && (precision == SSLBM_FP32_SPLIT || precision == SSLBM_FP32_KAHAN) ? 8 : 4;
}

// The tile passes' rows per warp and depth for n steps of this grid, or false where the row pipeline is
// expected to be faster (or the update has no tile pass).  parity: of the number of passes.
struct TilePlan {
  int nr, depth;
};
bool tile_plan(int lattice, int precision, const GridView& g, int64_t n, int parity, TilePlan* plan);

}  // namespace sslbm
