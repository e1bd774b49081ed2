// tile.cuh -- the register-tile pass of small grids (tile.cu).
#pragma once
#include "pass_plan.cuh"
#include "sslbm_internal.cuh"

namespace sslbm {

// K steps of the FP32 update (D2Q5 plain and deviation storage, D2Q9, varying diffusion) from `in`
// to `out`, regions of 64 x 16 nr cells; nr = 1, 2 or 4, 2 K < 16 nr and K < 31.
cudaError_t launch_tile(int lattice, int precision, const GridView& g, const void* coeffs, const void* in, void* out,
                        const void* kx, const void* ky, int nr, int K, cudaStream_t s);

}  // namespace sslbm
