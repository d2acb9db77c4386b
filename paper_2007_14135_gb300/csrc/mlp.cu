// Learned angle proposal (not in the paper): a 272 -> 256 -> 256 -> 256 -> 181 MLP with ReLU hidden
// layers and a sigmoid occupancy output over 1-degree bins, trained with binary cross-entropy on
// logits and Adam. Weights are kept in FP32 (master) and used as BF16 in the tensor-core GEMMs
// (FP32 accumulation). The products and the elementwise work between them run in mlp_tc.cu:
//   forward  A_l = relu(A_{l-1} W_l^T + b_l), Z = A_3 W_4^T + b_4, a 128-row tile through all layers
//   backward dZ_4 = (sigmoid(Z) - Y) / B, dZ_l = (dZ_{l+1} W_{l+1}) * [A_l > 0] in the same tile, then
//            dW_l = dZ_l^T A_{l-1} over the batch
// Here: the entry points, the workspace, Adam and the BF16 weight refresh.
#include <cuda_bf16.h>

#include "doa_internal.cuh"
#include "mlp_tc.cuh"

namespace doa {
namespace {

constexpr int kIn = DOA_MLP_IN, kHid = DOA_MLP_HIDDEN, kOut = DOA_MLP_OUT;
constexpr int kDims[5] = {kIn, kHid, kHid, kHid, kOut};

__host__ __device__ inline int pitch8(int n) { return (n + 7) / 8 * 8; }

struct MlpWs {
  __nv_bfloat16 *X0, *A[3], *dZ[4];
  float *gb_part, *loss_part;
  int *err;
  size_t bytes;
};

MlpWs ws_layout(uint8_t *base, int B) {
  MlpWs w{};
  size_t at = 0;
  auto take = [&](size_t n) {
    uint8_t *p = base ? base + at : nullptr;
    at += (n + 255) / 256 * 256;
    return p;
  };
  const size_t tiles = ((size_t)B + 127) / 128;
  w.X0 = reinterpret_cast<__nv_bfloat16 *>(take((size_t)kIn * B * 2));
  for (int l = 0; l < 3; ++l) w.A[l] = reinterpret_cast<__nv_bfloat16 *>(take((size_t)kHid * B * 2));
  for (int l = 0; l < 4; ++l)
    w.dZ[l] = reinterpret_cast<__nv_bfloat16 *>(take((size_t)(l == 3 ? kMlpOutPitch : kHid) * B * 2));
  w.gb_part = reinterpret_cast<float *>(take(tiles * 4 * kMlpGbCols * 4));
  w.loss_part = reinterpret_cast<float *>(take(tiles * kMlpLossParts * 4));
  w.err = reinterpret_cast<int *>(take(4));
  w.bytes = at;
  return w;
}

struct LayerPtrs {
  float *W, *b, *mW, *vW, *mb, *vb, *gW, *gb;
  __nv_bfloat16 *Wh, *WhT;
  int out, in;
};

struct NetPtrs {
  LayerPtrs l[4];
};

// Adam on the FP32 masters, then the BF16 copies (row-major and transposed); grid.y = layer.
__global__ void adam_kernel(const __grid_constant__ NetPtrs net, float lr, float b1, float b2, float eps, float c1, float c2, int update) {
  start_after_previous();
  let_next_start();
  const LayerPtrs &p = net.l[blockIdx.y];
  const int nW = p.out * p.in;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nW + p.out; i += gridDim.x * blockDim.x) {
    float *w, *m, *v;
    const float *gp;
    if (i < nW) {
      w = p.W + i; m = p.mW + i; v = p.vW + i; gp = p.gW + i;
    } else {
      w = p.b + (i - nW); m = p.mb + (i - nW); v = p.vb + (i - nW); gp = p.gb + (i - nW);
    }
    if (update) {
      const float g = *gp;
      const float mm = b1 * *m + (1.f - b1) * g;
      const float vv = b2 * *v + (1.f - b2) * g * g;
      *m = mm;
      *v = vv;
      *w -= lr * (mm / c1) / (sqrtf(vv / c2) + eps);
    }
    if (i < nW) {
      const int r = i / p.in, c = i % p.in;
      const __nv_bfloat16 h = __float2bfloat16_rn(*w);
      p.Wh[(size_t)r * p.in + c] = h;
      p.WhT[(size_t)c * pitch8(p.out) + r] = h;
    }
  }
}

LayerPtrs layer(const doa_mlp *net, int l) {
  LayerPtrs p;
  p.W = net->W[l]; p.b = net->b[l]; p.mW = net->mW[l]; p.vW = net->vW[l];
  p.mb = net->mb[l]; p.vb = net->vb[l]; p.gW = net->gW[l]; p.gb = net->gb[l];
  p.Wh = reinterpret_cast<__nv_bfloat16 *>(net->Wh[l]);
  p.WhT = reinterpret_cast<__nv_bfloat16 *>(net->WhT[l]);
  p.out = kDims[l + 1];
  p.in = kDims[l];
  return p;
}

bool net_ok(const doa_mlp *net, bool train) {
  if (!net) return false;
  for (int l = 0; l < 4; ++l) {
    if (!net->Wh[l] || !net->WhT[l] || !net->b[l]) return false;
    if (train && (!net->W[l] || !net->mW[l] || !net->vW[l] || !net->mb[l] || !net->vb[l] || !net->gW[l] ||
                  !net->gb[l]))
      return false;
  }
  return true;
}

cudaError_t adam(const doa_mlp *net, float lr, float b1, float b2, float eps, float c1, float c2, int update,
                 cudaStream_t s) {
  NetPtrs n;
  for (int l = 0; l < 4; ++l) n.l[l] = layer(net, l);
  return launch_programmatic(true, adam_kernel, dim3(256, 4), 256, 0, s, n, lr, b1, b2, eps, c1, c2, update);
}

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

MlpRowArgs row_args(const doa_mlp *net, const float *features, int batch, const MlpWs &w) {
  MlpRowArgs g{};
  g.X = features;
  g.B = batch;
  g.x_vec = aligned16(features);
  for (int l = 0; l < 4; ++l) {
    g.bias[l] = net->b[l];
    g.dZ[l] = w.dZ[l];
    if (l < 3) g.A[l] = w.A[l];
  }
  g.X0 = w.X0;
  g.gb_part = w.gb_part;
  g.loss_part = w.loss_part;
  g.err = w.err;
  return g;
}

}  // namespace
}  // namespace doa

using namespace doa;

extern "C" size_t doa_mlp_workspace_bytes(int batch) {
  if (batch < 8 || (batch & 7)) return 0;
  return ws_layout(nullptr, batch).bytes;
}

extern "C" doa_status doa_mlp_refresh(const doa_mlp *net, void *stream) {
  if (!net_ok(net, false)) return DOA_EINVAL;
  for (int l = 0; l < 4; ++l)
    if (!net->W[l]) return DOA_EINVAL;
  return adam(net, 0.f, 0.f, 0.f, 0.f, 1.f, 1.f, 0, reinterpret_cast<cudaStream_t>(stream)) == cudaSuccess ? DOA_OK
                                                                                                          : DOA_ECUDA;
}

extern "C" doa_status doa_mlp_forward(const doa_mlp *net, const float *features, int batch, float *probs,
                                      float *logits, void *ws, size_t ws_bytes, void *stream) {
  if (!net_ok(net, false) || !features || batch < 8 || (batch & 7) || !ws) return DOA_EINVAL;
  MlpWs w = ws_layout(static_cast<uint8_t *>(ws), batch);
  if (ws_bytes < w.bytes) return DOA_ENOMEM;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  MlpRowArgs g = row_args(net, features, batch, w);
  g.logits = logits;
  g.probs = probs;
  g.out_vec = aligned16(logits) && aligned16(probs);
  return launch_mlp_rows(net, g, false, s) == cudaSuccess ? DOA_OK : DOA_ECUDA;
}

extern "C" doa_status doa_mlp_backward(const doa_mlp *net, const float *features, const float *labels, int batch,
                                       float *loss, void *ws, size_t ws_bytes, void *stream) {
  if (!net_ok(net, true) || !features || !labels || batch < 8 || (batch & 7) || !ws) return DOA_EINVAL;
  MlpWs w = ws_layout(static_cast<uint8_t *>(ws), batch);
  if (ws_bytes < w.bytes) return DOA_ENOMEM;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  MlpRowArgs g = row_args(net, features, batch, w);
  g.Y = labels;
  MlpGrads o{};
  for (int l = 0; l < 4; ++l) {
    o.gW[l] = net->gW[l];
    o.gb[l] = net->gb[l];
  }
  o.loss = loss;
  if (launch_mlp_rows(net, g, true, s) != cudaSuccess) return DOA_ECUDA;
  return launch_mlp_dw(g, o, s) == cudaSuccess ? DOA_OK : DOA_ECUDA;
}

extern "C" doa_status doa_mlp_adam(const doa_mlp *net, float lr, float beta1, float beta2, float eps, int t,
                                   void *stream) {
  if (!net_ok(net, true) || t < 1 || !(lr >= 0.f) || !(beta1 >= 0.f && beta1 < 1.f) || !(beta2 >= 0.f && beta2 < 1.f))
    return DOA_EINVAL;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const float c1 = 1.f - powf(beta1, (float)t), c2 = 1.f - powf(beta2, (float)t);
  return adam(net, lr, beta1, beta2, eps, c1, c2, 1, s) == cudaSuccess ? DOA_OK : DOA_ECUDA;
}
