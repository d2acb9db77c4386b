// Interface between the proposal network's entry points (mlp.cu) and its tensor-core kernels (mlp_tc.cu).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>

#include "doa_internal.cuh"

namespace doa {

constexpr int kMlpGbCols = 3 * DOA_MLP_HIDDEN + 192;   // bias-gradient partial sums of one row group
constexpr int kMlpLossParts = 16;                      // loss partial sums of a 128-row tile
constexpr int kMlpDwTiles = 34;                        // 128 x 64 tiles of the four weight gradients

constexpr int kMlpOutPitch = 192;                      // row pitch of dZ_4 (181 columns, zero padding)

struct MlpMaps {
  CUtensorMap m[7];     // W_1 .. W_4 (out rows, K = in), then W_4^T, W_3^T, W_2^T (in rows, K = out)
  CUtensorMap store[8]; // training: X, A_1, A_2, A_3, dZ_4, dZ_3, dZ_2, dZ_1 as the passes' operands leave
};
struct MlpDwMaps {
  CUtensorMap a[4], b[4];   // dZ_l and the layer's input, both batch rows x features
};

struct MlpRowArgs {
  const float *X;           // B x 272 features
  int B;
  int x_vec, out_vec;       // the features / the forward outputs are 16-byte aligned
  const float *bias[4];
  float *logits, *probs;    // forward outputs (nullable)
  const float *Y;           // training: labels (B x 181)
  __nv_bfloat16 *X0, *A[3], *dZ[4];   // training: row-major copies for the weight gradients (dZ[l] of layer l + 1)
  float *gb_part;           // [row groups of 32][kMlpGbCols]
  float *loss_part;         // [tiles][kMlpLossParts]
  int *err;                 // set to 1 if a bounded wait ran out
};

struct MlpGrads {
  float *gW[4], *gb[4];
  float *loss;              // nullable
};

cudaError_t launch_mlp_rows(const doa_mlp *net, const MlpRowArgs &g, bool train, cudaStream_t s);
cudaError_t launch_mlp_dw(const MlpRowArgs &g, const MlpGrads &o, cudaStream_t s);

}  // namespace doa
