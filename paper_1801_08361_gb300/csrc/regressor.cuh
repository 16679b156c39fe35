// regressor.cuh -- argument blocks and launchers of the regressor kernels (regressor.cu), used by
// the C ABI in api.cu.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "relo_internal.cuh"

namespace relo {

typedef __nv_bfloat16 bf16;

// Convolution (forward / backward-data): out[p, n] = sum_{tap, k} in[src(p, tap), k] W[tap, n, k]
struct ConvArgs {
  const bf16* in;      // [B][Hi][Wi][CIN] (or the real tensor behind a virtual upsampling)
  const bf16* w;       // [9][N][CIN]
  const float* bias;   // [N] or null
  const bf16* mask;    // [B][Ho][Wo][N]: output multiplied by (mask > 0), or null
  bf16* out;           // [B][Ho][Wo][N] or null
  float* out_f32;      // [B][Ho][Wo][N] or null
  int B, Hi, Wi;       // input grid as the convolution sees it (the upsampled grid when upsample)
  int Hs, Ws;          // real input size when upsample
  int Ho, Wo, stride;
  int relu, upsample;
};

// Backward-weight sums (see wgrad_kernel)
struct WgradArgs {
  const bf16* in;     // layer input [B][Hi][Wi][64], or (the first layer) the images
  const uint16_t* depth;  // [B][Hi][Wi] mm
  const uint32_t* rgba;   // [B][Hi][Wi]
  const bf16* g;      // gradient of the pre-activation output [B][Ho][Wo][GS] (first N channels used)
  float* partial;     // [wgrad_parts][wgrad_partial_floats]
  int B, Hi, Wi, Ho, Wo, stride, GS;
};

// Targets (see targets_kernel)
struct CellArgs {
  const uint16_t* depth;  // [n][H][W]
  const double* poses;    // [n][16] camera -> scene
  int n, W, H, Wc, Hc;
  double fx, fy, cx, cy;
  double ox, oy, oz;      // origin
};

// Cell forest (see cell_forest_kernel)
struct CellForestArgs {
  const float* out;        // [n][Hc][Wc][ostride]: head output (ostride 8) or given cells (4)
  int ostride = 8;
  const uint16_t* depth;   // [n][H][W] full-resolution depth
  int n, W, H, Wc, Hc, L;  // L = leaves per tree (power of two >= Wc Hc)
  float ox, oy, oz;
  float* modes;            // [n][L][1][12]
  uint8_t* n_modes;        // [n][L]
  float4* top;             // [n][L]
  uint16_t* leaves;        // [n][Hc][Wc]
  uint16_t* depth_lr;      // [n][Hc][Wc]
};

// The network's input per pixel: centred and scaled depth, (depth m - 3) / 2, and colour channels,
// (c / 255 - 1/2) x 4.
__device__ __forceinline__ bf16 input_depth(uint32_t mm) { return __float2bfloat16(((float)mm * 0.001f - 3.0f) * 0.5f); }
__device__ __forceinline__ bf16 input_colour(uint32_t c) { return __float2bfloat16(((float)c / 255.f - 0.5f) * 4.0f); }

constexpr int kRegLayers = 8;
constexpr int kRegStride[kRegLayers] = {2, 2, 2, 1, 1, 1, 1, 1};
constexpr int kRegCin[kRegLayers] = {4, 64, 64, 64, 64, 64, 64, 64};
constexpr int kRegCout[kRegLayers] = {64, 64, 64, 64, 64, 64, 64, 4};
constexpr int kRegCinPad[kRegLayers] = {16, 64, 64, 64, 64, 64, 64, 64};
constexpr int kRegCoutPad[kRegLayers] = {64, 64, 64, 64, 64, 64, 64, 8};
// Most CTAs (partial sums per weight) of a backward-weight launch, one an SM; first layer: four times that.  A
// constant, since the order of the sums, so the gradients' bits, and the workspace's size follow it.
constexpr int kWgradCtas = 152;

// Adam step of all parameters and the operands derived from them (see adam_kernel)
struct AdamArgs {
  float *p, *m, *v;
  const float* g;
  int n;
  int w_off[kRegLayers];   // first weight of each layer; its biases follow its weights
  bf16* wk[kRegLayers];
  bf16* wt[kRegLayers];
  float* bias[kRegLayers];
};

cudaError_t launch_conv(int cin, int nt, const ConvArgs& a, int n_sms, cudaStream_t s);
// Gradients gw [3][3][cin_real][cout_real] and gb [cout_real] of a layer (cin 4: the first, from the images).
int wgrad_parts(int cin, int B, int Ho, int Wo);
size_t wgrad_partial_floats(int cin, int cout_pad);
cudaError_t launch_wgrad(int cin, int cout_pad, const WgradArgs& a, int cin_real, int cout_real, float* gw, float* gb,
                         cudaStream_t s);
cudaError_t launch_pack(const float* w, int cin, int cout, int cin_pad, int cout_pad, bf16* wk, bf16* wt,
                        int cout_pad_t, cudaStream_t s);
cudaError_t launch_input(const uint16_t* depth, const uint32_t* rgba, long n_pix, bf16* x, cudaStream_t s);
// counters (2 words): [0] receives the scored cells, [1] is zeroed for launch_loss
cudaError_t launch_targets(const CellArgs& a, float4* tgt, int32_t* counters, cudaStream_t s);
int loss_blocks(int n_cells);  // floats of launch_loss's sums
cudaError_t launch_loss(const float* out, const float4* tgt, int n_cells, bf16* grad, int32_t* counters, float* sums,
                        float* loss, cudaStream_t s);
cudaError_t launch_adam(const AdamArgs& a, float lr, int t, cudaStream_t s);
cudaError_t launch_cell_forest(const CellForestArgs& a, cudaStream_t s);

// Forward 3x3 convolution of a cin -> 64-channel layer (cin 16 or 64) on the tcgen05 tensor cores
// (conv_tc.cu): in [B][Hi][Wi][cin], w [9][64][cin], bias [64] (nullable), mask [B][Ho][Wo][64]
// (nullable: outputs where mask <= 0 become 0), out [B][Ho][Wo][64] BF16 NHWC; stride 1 or 2,
// dilation 1-8, zero padding = dilation.  A bounded wait that runs out sets *status = RELO_ETIMEOUT.
// stall_tile >= 0 (test hook) withholds that tile's loads so that the wait for them runs out.
cudaError_t launch_conv_tc(int cin, const bf16* in, int B, int Hi, int Wi, const bf16* w, const float* bias,
                           const bf16* mask, bf16* out, int Ho, int Wo, int stride, int dil, int relu, int32_t* status,
                           int n_sms, cudaStream_t s, unsigned long long timeout_ns, int stall_tile);
// The first layer from the images (depth [B][H][W] mm, rgba): w [9][64][16], out [B][Ho][Wo][64], ReLU.
cudaError_t launch_conv_first(const uint16_t* depth, const uint32_t* rgba, int B, int H, int W, const bf16* w,
                              const float* bias, bf16* out, int Ho, int Wo, int32_t* status, int n_sms, cudaStream_t s,
                              unsigned long long timeout_ns, int stall_tile);
// Backward-data of a stride-2 layer: g [B][Hg][Wg][64], w [9][64][64] flipped and transposed, mask and out
// [B][2 Hg][2 Wg][64].
cudaError_t launch_conv_up(const bf16* g, int B, int Hg, int Wg, const bf16* w, const bf16* mask, bf16* out, int32_t* status,
                           int n_sms, cudaStream_t s, unsigned long long timeout_ns, int stall_tile);
// The head: 64 -> 8 channels (w [9][8][64], bias [8]), stride 1, FP32 out [B][H][W][8].
cudaError_t launch_conv_head(const bf16* in, int B, int H, int W, const bf16* w, const float* bias, float* out,
                             int32_t* status, int n_sms, cudaStream_t s, unsigned long long timeout_ns, int stall_tile);
cudaError_t launch_head_copy(const float* head, long n_cells, float* out4, cudaStream_t s);

}  // namespace relo
