// fno_bwd.cuh -- the surrogate's fused backward pass (fno_bwd.cu) for the shapes of fno_fused.cuh.
#pragma once
#include "fno_fused.cuh"

namespace sslbm {
namespace fno_fused {

enum BwdMode { BWD_LAST = 0, BWD_MID = 1, BWD_FIRST = 2 };

struct BwdArgs {
  int B;
  const float* x;      // [B][8][n][n] network input
  const bf16* F;       // [n][4m] Fx
  // last
  const float* dy;     // [B][5][n][n] dL/dy
  const float* y;      // [B][5][n][n] the cached prediction
  const float* seed;   // [B] sum(dy y) / sum y, then [B] sigma of E and I
  const float* ratio;  // [B] sum u / sum v
  const bf16* zp;      // [B][H][n][n]
  const bf16* p;       // [B][H][n][n]
  const bf16* hL;      // [B][W][n][n]
  const bf16* Q1;      // [H][W]
  const bf16* Q2;      // [5][H]
  float* gQ2;          // gradients (added to)
  float* gq2;
  float* gQ1;
  float* gq1;
  // mid, first
  const float* dzin;   // [B][W][n][n] dz_l
  const float* dH1;    // [B][n][W][4m]
  const bf16* Bl;      // [W][W] B_l
  const bf16* z;       // [B][W][n][n] z_{l-1} (mid)
  // the produced dz (last: dz_L, mid: dz_{l-1}, first: dh_0)
  const bf16* hprev;   // [B][W][n][n] the input of its layer (last, mid)
  float* dz;           // [B][W][n][n] (last, mid)
  float* dG1;          // [B][n][W][4m] dz Fx * scale (last, mid)
  float scale;
  float* gW;           // gradient of its layer's channel map (first: of A0) and bias (added to)
  float* gb;
};

struct BwdSpectral {
  const float* dG1;  // [B][n][W][4m]
  const bf16* Fy;    // [2m][n]
  const bf16* Fyi;   // [n][2m]
  const float* hat;  // [B][W][2m*m][2] the forward pass's modes
  const float* R;    // [W][W][2m*m][2]
  float* dG;         // [B][W][2m*m][2] scratch
  float* dhat;       // [B][W][2m*m][2] scratch
  float* dR;         // [W][W][2m*m][2]
  float* dH1;        // [B][n][W][4m] (may be dG1's memory)
};

cudaError_t launch_bwd_row(int mode, int W, int m, int H, int n, const BwdArgs& a, cudaStream_t s);
// dG1 -> dR, dH1 of one layer
cudaError_t launch_bwd_spectral(int W, int m, int H, int B, int n, const BwdSpectral& a, cudaStream_t s);

}  // namespace fno_fused
}  // namespace sslbm
