// regressor.cu -- the learned scene-coordinate regressor: BF16 tensor-core 3x3 convolutions
// (forward, backward-data, backward-weight) with FP32 accumulation, the Gaussian-NLL loss, Adam,
// and the cell forest that hands its output to the preemptive RANSAC.
//
// The paper relocalises with a forest (Sec. 3.3 (b)); this network is the workload's alternative
// relocaliser for a scene, trained online on renders of the scene's own voxel map.  Readings
// (identical in the CPU oracle): 4 input channels ((depth m - 3) / 2, (RGB / 255 - 1/2) x 4), eight
// 3x3 convolutions with zero padding, 64 channels, strides 2, 2, 2, 1, 1, 1, 1, 1, ReLU after
// layers 1-7, 4 outputs per 8 x 8-pixel cell (scene coordinate - origin, log-variance s); the
// target of a cell is the scene coordinate of its centre pixel; loss = mean over scored cells of
// rho(e) + 1/2 e^2 exp(-s) + 3/2 s with e = |y - y_hat|, rho(e) = sqrt(e^2 + 1e-6), the error in the
// variance term held fixed for the gradient; Adam (0.9, 0.999, 1e-8).
//
// Layout: activations NHWC in BF16 (channels contiguous); layer 1's input is padded to 16
// channels and the head's output to 8 (its gradient to 16) so every contraction is a multiple
// of the mma.sync m16n8k16 shape.  A convolution is an implicit GEMM: output pixels x output
// channels, contracted over 9 taps x input channels; each CTA (4 warps) keeps all 9 taps of the
// weights in shared memory and loops over 64-pixel tiles, gathering one tap's input rows per
// step.  The backward-data pass of a stride-2 layer is the same kernel reading its input
// through a virtual zero-inserted upsampling, with the weights flipped and transposed.  That
// kernel (conv_kernel) is what the tcgen05 convolutions (conv_tc.cu), which run by default, are
// compared with bit for bit; the other kernels here serve both.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "regressor.cuh"

namespace relo {

// ---------------------------------------------------------------------------------------------
// Tensor-core primitive
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t ld32(const bf16* p) { return *reinterpret_cast<const uint32_t*>(p); }

// ldmatrix: four (or two) 8 x 8 b16 matrices from shared memory, rows addressed by lanes 8q..8q+7
__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], const bf16* p) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a));
}

__device__ __forceinline__ void ldsm_x2(uint32_t& r0, uint32_t& r1, const bf16* p) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];\n" : "=r"(r0), "=r"(r1) : "r"(a));
}

// Forward / backward-data convolution.  A CTA of 8 warps keeps all 9 taps of the weights in shared
// memory and loops over tiles of 128 output pixels (16 per warp, all N output channels per warp).
// Per tap the tile's input rows (one per output pixel) are gathered into shared memory; the next
// tap's rows are loaded into registers while the current tap's MMAs run, so the gathers overlap
// the tensor-core work.  Fragments come from shared memory by ldmatrix; rows are padded to
// CIN + 8 elements, which keeps every ldmatrix phase free of bank conflicts.
constexpr int kConvThreads = 256;
constexpr int kConvTile = 128;

template <int CIN>
struct ConvGather {
  static constexpr int CH = CIN / 8;                              // 16-B chunks per pixel
  static constexpr int PER = kConvTile * CH / kConvThreads;       // chunks per thread per tap
  static_assert(PER >= 1 && kConvTile * CH % kConvThreads == 0, "tile / channel split");
  int b[PER], oy[PER], ox[PER], m[PER], c8[PER];
  bool ok[PER];

  __device__ __forceinline__ void setup(const ConvArgs& a, long m0, long total, int tid) {
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const int v = tid + i * kConvThreads;
      m[i] = v / CH;
      c8[i] = v % CH;
      const long p = m0 + m[i];
      ok[i] = p < total;
      ox[i] = ok[i] ? (int)(p % a.Wo) : 0;
      oy[i] = ok[i] ? (int)((p / a.Wo) % a.Ho) : 0;
      b[i] = ok[i] ? (int)(p / ((long)a.Wo * a.Ho)) : 0;
    }
  }

  __device__ __forceinline__ void load(const ConvArgs& a, int tap, uint4 (&val)[PER]) const {
    const int ky = tap / 3, kx = tap % 3;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      val[i] = make_uint4(0u, 0u, 0u, 0u);
      const int iy = oy[i] * a.stride + ky - 1, ix = ox[i] * a.stride + kx - 1;
      if (ok[i] && iy >= 0 && ix >= 0 && iy < a.Hi && ix < a.Wi) {
        if (!a.upsample) {
          val[i] = __ldg(reinterpret_cast<const uint4*>(a.in + (((size_t)b[i] * a.Hi + iy) * a.Wi + ix) * CIN) + c8[i]);
        } else if (!(iy & 1) && !(ix & 1) && (iy >> 1) < a.Hs && (ix >> 1) < a.Ws) {
          val[i] = __ldg(reinterpret_cast<const uint4*>(a.in + (((size_t)b[i] * a.Hs + (iy >> 1)) * a.Ws + (ix >> 1)) *
                                                                  CIN) + c8[i]);
        }
      }
    }
  }
};

template <int CIN, int NT>
__global__ void __launch_bounds__(kConvThreads) conv_kernel(ConvArgs a) {
  constexpr int N = NT * 8;
  constexpr int RS = CIN + 8;  // padded row stride (bf16) of the shared tiles
  using G = ConvGather<CIN>;
  extern __shared__ __align__(16) unsigned char conv_smem[];
  bf16* sW = reinterpret_cast<bf16*>(conv_smem);   // [9][N][RS]
  bf16* sA = sW + 9 * N * RS;                       // [kConvTile][RS]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  for (int v = tid; v < 9 * N * (CIN / 8); v += kConvThreads) {
    const int row = v / (CIN / 8), c8 = v % (CIN / 8);
    *reinterpret_cast<uint4*>(sW + row * RS + c8 * 8) = __ldg(reinterpret_cast<const uint4*>(a.w + (size_t)row * CIN) + c8);
  }
  const long total = (long)a.B * a.Ho * a.Wo;
  const long n_tiles = (total + kConvTile - 1) / kConvTile;
  // ldmatrix row addresses of this lane: A rows warp * 16 + (lane & 7) + 8 * ((lane >> 3) & 1),
  // k half (lane >> 4); B rows (n) (lane & 7) + 8 * (lane >> 4), k half ((lane >> 3) & 1)
  const int a_row = warp * 16 + (lane & 7) + 8 * ((lane >> 3) & 1), a_k = 8 * (lane >> 4);
  const int b_row = (lane & 7) + 8 * (lane >> 4), b_k = 8 * ((lane >> 3) & 1);
  for (long tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const long m0 = tile * kConvTile;
    G gat;
    gat.setup(a, m0, total, tid);
    uint4 pre[G::PER];
    gat.load(a, 0, pre);
    float acc[NT][4];
#pragma unroll
    for (int j = 0; j < NT; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
    for (int tap = 0; tap < 9; ++tap) {
      __syncthreads();  // readers of the previous tap's rows (and, first, the weight stores) are done
#pragma unroll
      for (int i = 0; i < G::PER; ++i) *reinterpret_cast<uint4*>(sA + gat.m[i] * RS + gat.c8[i] * 8) = pre[i];
      __syncthreads();
      if (tap < 8) gat.load(a, tap + 1, pre);  // in flight during this tap's MMAs
      const bf16* Wt = sW + tap * N * RS;
#pragma unroll
      for (int ks = 0; ks < CIN / 16; ++ks) {
        uint32_t af[4];
        ldsm_x4(af, sA + a_row * RS + ks * 16 + a_k);
#pragma unroll
        for (int j = 0; j + 1 < NT; j += 2) {
          uint32_t bf[4];
          ldsm_x4(bf, Wt + (j * 8 + b_row) * RS + ks * 16 + b_k);
          mma_bf16(acc[j], af, bf[0], bf[1]);
          mma_bf16(acc[j + 1], af, bf[2], bf[3]);
        }
        if (NT & 1) {
          uint32_t b0, b1;
          ldsm_x2(b0, b1, Wt + ((NT - 1) * 8 + (lane & 7)) * RS + ks * 16 + 8 * ((lane >> 3) & 1));
          mma_bf16(acc[NT - 1], af, b0, b1);
        }
      }
    }
    // epilogue: bias, ReLU, mask, stores
#pragma unroll
    for (int j = 0; j < NT; ++j) {
      const int n0 = j * 8 + 2 * t;
      const float b0 = a.bias ? a.bias[n0] : 0.f, b1 = a.bias ? a.bias[n0 + 1] : 0.f;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const long p = m0 + warp * 16 + g + 8 * h;
        if (p >= total) continue;
        float v0 = acc[j][2 * h] + b0, v1 = acc[j][2 * h + 1] + b1;
        if (a.relu) {
          v0 = fmaxf(v0, 0.f);
          v1 = fmaxf(v1, 0.f);
        }
        if (a.mask) {
          const __nv_bfloat162 mk = *reinterpret_cast<const __nv_bfloat162*>(a.mask + (size_t)p * N + n0);
          if (!(__bfloat162float(mk.x) > 0.f)) v0 = 0.f;
          if (!(__bfloat162float(mk.y) > 0.f)) v1 = 0.f;
        }
        if (a.out) *reinterpret_cast<__nv_bfloat162*>(a.out + (size_t)p * N + n0) = __floats2bfloat162_rn(v0, v1);
        if (a.out_f32) {
          a.out_f32[(size_t)p * N + n0] = v0;
          a.out_f32[(size_t)p * N + n0 + 1] = v1;
        }
      }
    }
  }
}

template <int CIN, int NT>
cudaError_t launch_conv_t(const ConvArgs& a, int n_sms, cudaStream_t s) {
  constexpr int N = NT * 8, RS = CIN + 8;
  const size_t smem = (size_t)(9 * N + kConvTile) * RS * sizeof(bf16);
  static PerDevice resident;  // resident CTAs per SM on each device
  int per_sm = 0;
  const cudaError_t e = per_device(resident, &per_sm, [smem](int, int* v) {
    cudaError_t r = cudaFuncSetAttribute(conv_kernel<CIN, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (r == cudaSuccess) r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(v, conv_kernel<CIN, NT>, kConvThreads, smem);
    if (*v < 1) *v = 1;
    return r;
  });
  if (e != cudaSuccess) return e;
  const long total = (long)a.B * a.Ho * a.Wo;
  const long tiles = (total + kConvTile - 1) / kConvTile;
  const long slots = (long)n_sms * per_sm;
  const long grid = tiles < slots ? tiles : slots;
  if (grid <= 0) return cudaSuccess;
  conv_kernel<CIN, NT><<<(unsigned)grid, kConvThreads, smem, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_conv(int cin, int nt, const ConvArgs& a, int n_sms, cudaStream_t s) {
  if (cin == 16 && nt == 8) return launch_conv_t<16, 8>(a, n_sms, s);
  if (cin == 64 && nt == 8) return launch_conv_t<64, 8>(a, n_sms, s);
  if (cin == 64 && nt == 1) return launch_conv_t<64, 1>(a, n_sms, s);
  return cudaErrorInvalidValue;
}

// ---------------------------------------------------------------------------------------------
// Backward-weight: gw[tap][k][n] = sum over output pixels p of in[src(p, tap), k] g[p, n], and the bias
// gradient, the sum of g.  A persistent CTA (8 warps) walks tiles of 8 x 8 output pixels; a tile's
// input window and its gradients come into shared memory once, by asynchronous copies while the
// previous tile is multiplied, and serve all nine taps (a CTA per tap read both nine times over and
// left 75 to 1200 partial sums per weight: 1.2 ms of a 2.9 ms step with its sums and a bias pass of
// its own).  Contraction over the pixels with ldmatrix.trans fragments: M = input channels, N = output
// channels, K = the 16 pixels of two tile rows.  The tensor core sums the 64 pixels of a tile; tiles are
// added to the sums of all taps, in registers (144 a thread at 64 x 64 channels), by rounded FP32
// additions -- the tensor core's own additions drop bits, which a chain over hundreds of tiles shows --
// and one partial per CTA is left to sum.
// The bias is one more product, with a row of ones.  16 views of 640 x 480: 0.31 ms with the sums for
// all layers, the first's (wgrad_first_kernel) among them; bound by mma.sync (288 products a scheduler and
// tile of 64 channels, 17 cycles each).
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void ldsm_x4_t(uint32_t (&r)[4], const bf16* p) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a));
}

__device__ __forceinline__ void ldsm_x2_t(uint32_t& r0, uint32_t& r1, const bf16* p) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n" : "=r"(r0), "=r"(r1) : "r"(a));
}

// 16 bytes to shared memory, zeros where !ok (src is then not read)
__device__ __forceinline__ void copy_or_zero16(bf16* dst, const bf16* src, bool ok) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(dst);
  const int n = ok ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(a), "l"(src), "r"(n) : "memory");
}

constexpr int kWgradThreads = 256, kWgradW = 8, kWgradH = 8;  // a tile's output pixels
constexpr int kWgradK = kWgradW * kWgradH / 16;               // products' depth: pairs of tile rows

// CIN input channels (64), NW n8 tiles of output channels per warp: N = 16 NW channels of g rows
// of GS; STRIDE 1 or 2.
template <int CIN, int NW, int STRIDE>
struct WgradShape {
  static constexpr int kHaloW = (kWgradW - 1) * STRIDE + 3, kHaloH = (kWgradH - 1) * STRIDE + 3;
  static constexpr int kN = 16 * NW;
  static constexpr int kRowI = CIN + 8, kRowG = kN + 8;  // padded rows (bf16): conflict-free ldmatrix
  static constexpr int kInElems = kHaloW * kHaloH * kRowI, kGElems = kWgradW * kWgradH * kRowG;
  static constexpr int kStage = kInElems + kGElems;
  static constexpr int kStages = 4;
  static constexpr size_t kSmem = kStages * (size_t)kStage * sizeof(bf16);
  // warps: MG groups of 16 input channels x 2 halves of the output channels x TG groups of taps
  static constexpr int kMG = CIN / 16, kTG = 8 / (2 * kMG), kTaps = (9 + kTG - 1) / kTG;
};

template <int CIN, int NW, int STRIDE>
__global__ void __launch_bounds__(kWgradThreads, 1) wgrad_kernel(WgradArgs a) {
  using S = WgradShape<CIN, NW, STRIDE>;
  extern __shared__ __align__(16) unsigned char wgrad_smem[];
  bf16* smem = reinterpret_cast<bf16*>(wgrad_smem);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int mg = warp % S::kMG, nh = (warp / S::kMG) & 1, tg = warp / (2 * S::kMG);
  const int tap0 = tg * S::kTaps;
  const bool bias_warp = mg == 0 && tg == 0;
  float acc[S::kTaps][NW][4], accb[NW][2];
#pragma unroll
  for (int t = 0; t < S::kTaps; ++t)
#pragma unroll
    for (int j = 0; j < NW; ++j) acc[t][j][0] = acc[t][j][1] = acc[t][j][2] = acc[t][j][3] = 0.f;
#pragma unroll
  for (int j = 0; j < NW; ++j) accb[j][0] = accb[j][1] = 0.f;
  const uint32_t ones[4] = {0x3F803F80u, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u};
  const int tiles_x = (a.Wo + kWgradW - 1) / kWgradW, tiles_y = (a.Ho + kWgradH - 1) / kWgradH;
  const int n_tiles = a.B * tiles_x * tiles_y;

  auto load = [&](int tile, int stage) {
    bf16* sI = smem + stage * S::kStage;
    bf16* sG = sI + S::kInElems;
    const int b = tile / (tiles_x * tiles_y), q = tile % (tiles_x * tiles_y);
    const int oy0 = q / tiles_x * kWgradH, ox0 = q % tiles_x * kWgradW;
    constexpr int CI = CIN / 8, CG = S::kN / 8;
    for (int v = tid; v < S::kHaloW * S::kHaloH * CI; v += kWgradThreads) {
      const int px = v / CI, c = v % CI, hy = px / S::kHaloW, hx = px % S::kHaloW;
      const int iy = oy0 * STRIDE - 1 + hy, ix = ox0 * STRIDE - 1 + hx;
      const bool ok = iy >= 0 && ix >= 0 && iy < a.Hi && ix < a.Wi;
      copy_or_zero16(sI + px * S::kRowI + c * 8, ok ? a.in + (((size_t)b * a.Hi + iy) * a.Wi + ix) * CIN + c * 8 : a.in, ok);
    }
    for (int v = tid; v < kWgradW * kWgradH * CG; v += kWgradThreads) {
      const int px = v / CG, c = v % CG, oy = oy0 + px / kWgradW, ox = ox0 + px % kWgradW;
      const bool ok = oy < a.Ho && ox < a.Wo;
      copy_or_zero16(sG + px * S::kRowG + c * 8, ok ? a.g + (((size_t)b * a.Ho + oy) * a.Wo + ox) * a.GS + c * 8 : a.g, ok);
    }
  };

  // the next kStages - 1 tiles are on their way while one is multiplied (a group per tile, empty past the end)
#pragma unroll
  for (int k = 0; k < S::kStages - 1; ++k) {
    if ((int)(blockIdx.x + k * gridDim.x) < n_tiles) load(blockIdx.x + k * gridDim.x, k);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  int stage = 0;
  for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, stage = stage + 1 < S::kStages ? stage + 1 : 0) {
    asm volatile("cp.async.wait_group %0;" ::"n"(S::kStages - 2) : "memory");
    __syncthreads();  // the tile is here for all, and the one before is read
    const int next = tile + (S::kStages - 1) * gridDim.x;
    if (next < n_tiles) load(next, stage > 0 ? stage - 1 : S::kStages - 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const bf16* sI = smem + stage * S::kStage;
    const bf16* sG = sI + S::kInElems;
    const int q = lane >> 3, r = lane & 7;
    uint32_t bf[kWgradK][NW][2];
#pragma unroll
    for (int ks = 0; ks < kWgradK; ++ks) {
      if (NW == 1) {
        ldsm_x2_t(bf[ks][0][0], bf[ks][0][1], sG + (ks * 16 + r + 8 * (q & 1)) * S::kRowG + nh * 8);
      } else {
#pragma unroll
        for (int j = 0; j + 1 < NW; j += 2) {
          uint32_t b4[4];
          ldsm_x4_t(b4, sG + (ks * 16 + r + 8 * (q & 1)) * S::kRowG + (nh * NW + j) * 8 + 8 * (q >> 1));
          bf[ks][j][0] = b4[0];
          bf[ks][j][1] = b4[1];
          bf[ks][j + 1 < NW ? j + 1 : j][0] = b4[2];
          bf[ks][j + 1 < NW ? j + 1 : j][1] = b4[3];
        }
      }
    }
#pragma unroll
    for (int t = 0; t < S::kTaps; ++t) {
      const int tap = tap0 + t;
      if (S::kTG * S::kTaps > 9 && tap > 8) continue;
      const int ky = tap / 3, kx = tap - 3 * ky;
      float sum[NW][4];  // of this tile alone
#pragma unroll
      for (int j = 0; j < NW; ++j) sum[j][0] = sum[j][1] = sum[j][2] = sum[j][3] = 0.f;
#pragma unroll
      for (int ks = 0; ks < kWgradK; ++ks) {
        uint32_t af[4];
        ldsm_x4_t(af, sI + (((2 * ks + (q >> 1)) * STRIDE + ky) * S::kHaloW + r * STRIDE + kx) * S::kRowI + mg * 16 + 8 * (q & 1));
#pragma unroll
        for (int j = 0; j < NW; ++j) mma_bf16(sum[j], af, bf[ks][j][0], bf[ks][j][1]);
      }
#pragma unroll
      for (int j = 0; j < NW; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[t][j][e] += sum[j][e];
    }
    if (bias_warp) {
      float sum[NW][4];
#pragma unroll
      for (int j = 0; j < NW; ++j) {
        sum[j][0] = sum[j][1] = sum[j][2] = sum[j][3] = 0.f;
#pragma unroll
        for (int ks = 0; ks < kWgradK; ++ks) mma_bf16(sum[j], ones, bf[ks][j][0], bf[ks][j][1]);
        accb[j][0] += sum[j][0];
        accb[j][1] += sum[j][1];
      }
    }
  }
  float* out = a.partial + (size_t)blockIdx.x * (9 * S::kN * CIN + S::kN);
  const int g = lane >> 2, t2 = 2 * (lane & 3);
#pragma unroll
  for (int t = 0; t < S::kTaps; ++t) {
    const int tap = tap0 + t;
    if (tap > 8) continue;
#pragma unroll
    for (int j = 0; j < NW; ++j) {
      const int k = mg * 16 + g, n = (nh * NW + j) * 8 + t2;
      float* o = out + ((size_t)tap * S::kN + n) * CIN + k;
      o[0] = acc[t][j][0];
      o[CIN] = acc[t][j][1];
      o[8] = acc[t][j][2];
      o[CIN + 8] = acc[t][j][3];
    }
  }
  if (bias_warp && g == 0)
#pragma unroll
    for (int j = 0; j < NW; ++j) {
      float* o = out + 9 * S::kN * CIN + (nh * NW + j) * 8 + t2;
      o[0] = accb[j][0];
      o[1] = accb[j][1];
    }
}

template <int CIN, int NW, int STRIDE>
cudaError_t launch_wgrad_t(const WgradArgs& a, int grid, cudaStream_t s) {
  using S = WgradShape<CIN, NW, STRIDE>;
  static PerDevice configured;
  int dummy = 0;
  const cudaError_t e = per_device(configured, &dummy, [](int, int* v) {
    *v = 1;
    return cudaFuncSetAttribute(wgrad_kernel<CIN, NW, STRIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::kSmem);
  });
  if (e != cudaSuccess) return e;
  wgrad_kernel<CIN, NW, STRIDE><<<grid, kWgradThreads, S::kSmem, s>>>(a);
  return cudaGetLastError();
}

// The first layer's, straight from the depth and colour images: a CTA converts the 17 x 17 pixels under
// its tile of 8 x 8 outputs as it loads them (the next tile's are on their way meanwhile), 4 channels = 8
// bytes a pixel, so that 16 bytes hold two neighbouring taps and an operand row of a kernel row ky is
// its four columns' channels (the fourth column's products are dropped): three products a 16-pixel step
// where nine taps of 16 padded channels took nine.  A warp per 8 output channels, four CTAs an SM.
// 16 views of 640 x 480: 73 us; the padded operand's kernel took 127 us and making that
// operand another 31.  The gradient's 157 MB would take 23.
constexpr int kWgrad0Cols = 2 * kWgradW + 2, kWgrad0Rows = 2 * kWgradH + 1, kWgrad0Px = kWgrad0Cols * kWgrad0Rows;
constexpr int kWgrad0Stages = 3, kWgrad0RowG = 64 + 8;
__global__ void __launch_bounds__(kWgradThreads, 4) wgrad_first_kernel(WgradArgs a) {
  static_assert(kWgradThreads == 256 && kWgrad0Px <= 2 * kWgradThreads, "eight warps of 8 channels, two pixels a thread");
  __shared__ __align__(16) bf16 s_in[2][kWgrad0Px * 4];
  __shared__ __align__(16) bf16 s_g[kWgrad0Stages][kWgradW * kWgradH * kWgrad0RowG];
  __shared__ bf16 s_colour[256];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  s_colour[tid] = input_colour((uint32_t)tid);
  const uint32_t ones[4] = {0x3F803F80u, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u};
  const int tiles_x = (a.Wo + kWgradW - 1) / kWgradW, tiles_y = (a.Ho + kWgradH - 1) / kWgradH;
  const int n_tiles = a.B * tiles_x * tiles_y;

  uint32_t dep[2], col[2];
  auto fetch = [&](int tile) {
    const int b = tile / (tiles_x * tiles_y), q = tile % (tiles_x * tiles_y);
    const int iy0 = q / tiles_x * kWgradH * 2 - 1, ix0 = q % tiles_x * kWgradW * 2 - 1;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int p = tid + k * kWgradThreads, row = p / kWgrad0Cols, c = p - row * kWgrad0Cols;
      const int iy = iy0 + row, ix = ix0 + c;
      dep[k] = 0x10000u;  // outside the image (and the fourth column's last pixel): zeros
      col[k] = 0;
      if (p < kWgrad0Px && c < kWgrad0Cols - 1 && iy >= 0 && ix >= 0 && iy < a.Hi && ix < a.Wi) {
        const size_t px = ((size_t)b * a.Hi + iy) * a.Wi + ix;
        dep[k] = __ldg(&a.depth[px]);
        col[k] = __ldg(&a.rgba[px]);
      }
    }
  };
  auto load_g = [&](int tile, int stage) {
    const int b = tile / (tiles_x * tiles_y), q = tile % (tiles_x * tiles_y);
    const int oy0 = q / tiles_x * kWgradH, ox0 = q % tiles_x * kWgradW;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int v = tid + k * kWgradThreads, px = v >> 3, c = v & 7, oy = oy0 + px / kWgradW, ox = ox0 + px % kWgradW;
      const bool ok = oy < a.Ho && ox < a.Wo;
      copy_or_zero16(&s_g[stage][px * kWgrad0RowG + c * 8], ok ? a.g + (((size_t)b * a.Ho + oy) * a.Wo + ox) * a.GS + c * 8 : a.g, ok);
    }
  };

  float acc[3][4] = {}, accb[2] = {};
  if ((int)blockIdx.x < n_tiles) fetch(blockIdx.x);
#pragma unroll
  for (int k = 0; k < kWgrad0Stages - 1; ++k) {
    if ((int)(blockIdx.x + k * gridDim.x) < n_tiles) load_g(blockIdx.x + k * gridDim.x, k);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  __syncthreads();  // the colour table
  const int q = lane >> 3, r = lane & 7;
  int stage = 0, buf = 0;
  for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, buf ^= 1, stage = stage + 1 < kWgrad0Stages ? stage + 1 : 0) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int p = tid + k * kWgradThreads;
      if (p >= kWgrad0Px) continue;
      const bf16 d = input_depth(dep[k]);
      const uint16_t* lut = reinterpret_cast<const uint16_t*>(s_colour);
      uint2 v = make_uint2(*reinterpret_cast<const uint16_t*>(&d) | (uint32_t)lut[col[k] & 0xFF] << 16,
                           (uint32_t)lut[(col[k] >> 8) & 0xFF] | (uint32_t)lut[(col[k] >> 16) & 0xFF] << 16);
      if (dep[k] & 0x10000u) v = make_uint2(0u, 0u);
      *reinterpret_cast<uint2*>(&s_in[buf][p * 4]) = v;
    }
    asm volatile("cp.async.wait_group %0;" ::"n"(kWgrad0Stages - 2) : "memory");
    __syncthreads();  // the tile is here for all, and the one before is read
    if (tile + (int)gridDim.x < n_tiles) fetch(tile + gridDim.x);
    const int next = tile + (kWgrad0Stages - 1) * gridDim.x;
    if (next < n_tiles) load_g(next, stage > 0 ? stage - 1 : kWgrad0Stages - 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const bf16 *sI = s_in[buf], *sG = s_g[stage];
    uint32_t bf[kWgradK][2];
#pragma unroll
    for (int ks = 0; ks < kWgradK; ++ks)
      ldsm_x2_t(bf[ks][0], bf[ks][1], sG + (ks * 16 + r + 8 * (q & 1)) * kWgrad0RowG + warp * 8);
#pragma unroll
    for (int ky = 0; ky < 3; ++ky) {
      float sum[4] = {};
#pragma unroll
      for (int ks = 0; ks < kWgradK; ++ks) {
        uint32_t af[4];
        ldsm_x4_t(af, sI + ((2 * (2 * ks + (q >> 1)) + ky) * kWgrad0Cols + 2 * r + 2 * (q & 1)) * 4);
        mma_bf16(sum, af, bf[ks][0], bf[ks][1]);
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[ky][e] += sum[e];
    }
    float sum[4] = {};
#pragma unroll
    for (int ks = 0; ks < kWgradK; ++ks) mma_bf16(sum, ones, bf[ks][0], bf[ks][1]);
    accb[0] += sum[0];
    accb[1] += sum[1];
  }
  // rows of a product: channel m & 3 of column m >> 2
  float* out = a.partial + (size_t)blockIdx.x * (9 * 64 * 4 + 64);
  const int g = lane >> 2, n = warp * 8 + 2 * (lane & 3);
#pragma unroll
  for (int ky = 0; ky < 3; ++ky) {
    float* o = out + ((3 * ky + (g >> 2)) * 64 + n) * 4 + (g & 3);
    o[0] = acc[ky][0];
    o[4] = acc[ky][1];
    if (g < 4) {
      o = out + ((3 * ky + 2) * 64 + n) * 4 + g;
      o[0] = acc[ky][2];
      o[4] = acc[ky][3];
    }
  }
  if (g == 0) {
    out[9 * 64 * 4 + n] = accb[0];
    out[9 * 64 * 4 + n + 1] = accb[1];
  }
}

// Sum of the CTAs' partials into the master-layout gradients gw [3][3][cin][cout] and gb [cout] (only
// the real channels): 32 neighbouring weights per CTA, eight warps taking every eighth partial each,
// added in a fixed order.
__global__ void __launch_bounds__(256) wgrad_reduce_kernel(const float* __restrict__ partial, int n_parts, int N, int CIN,
                                                           int cin_real, int cout_real, float* __restrict__ gw,
                                                           float* __restrict__ gb) {
  __shared__ float part[8][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int per_tap = cin_real * cout_real, n_w = 9 * per_tap;
  const int i = blockIdx.x * 32 + lane;
  const size_t pitch = (size_t)9 * N * CIN + N;
  size_t src = 0;
  float* dst = nullptr;
  if (i < n_w) {
    const int tap = i / per_tap, r = i % per_tap, co = r / cin_real, ci = r % cin_real;
    src = ((size_t)tap * N + co) * CIN + ci;
    dst = gw + (size_t)tap * per_tap + (size_t)ci * cout_real + co;
  } else if (i < n_w + cout_real) {
    src = (size_t)9 * N * CIN + (i - n_w);
    dst = gb + (i - n_w);
  }
  float s = 0.f;
  if (dst) {
#pragma unroll 8
    for (int c = warp; c < n_parts; c += 8) s += partial[(size_t)c * pitch + src];
  }
  part[warp][lane] = s;
  __syncthreads();
  if (warp == 0 && dst) {
    float v = part[0][lane];
#pragma unroll
    for (int w = 1; w < 8; ++w) v += part[w][lane];
    *dst = v;
  }
}

int wgrad_parts(int cin, int B, int Ho, int Wo) {
  const long tiles = (long)B * ((Wo + kWgradW - 1) / kWgradW) * ((Ho + kWgradH - 1) / kWgradH);
  const int most = kWgradCtas * (cin == 4 ? 4 : 1);
  return (int)(tiles < most ? tiles : most);
}

size_t wgrad_partial_floats(int cin, int cout_pad) {
  const int n = cout_pad < 16 ? 16 : cout_pad;
  return (size_t)9 * n * cin + n;
}

cudaError_t launch_wgrad(int cin, int cout_pad, const WgradArgs& a, int cin_real, int cout_real, float* gw, float* gb,
                         cudaStream_t s) {
  const int parts = wgrad_parts(cin, a.B, a.Ho, a.Wo);
  if (parts <= 0) return cudaSuccess;
  cudaError_t e = cudaErrorInvalidValue;
  if (cin == 4 && cout_pad == 64 && a.stride == 2) {
    wgrad_first_kernel<<<parts, kWgradThreads, 0, s>>>(a);
    e = cudaGetLastError();
  }
  if (cin == 64 && cout_pad == 64 && a.stride == 2) e = launch_wgrad_t<64, 4, 2>(a, parts, s);
  else if (cin == 64 && cout_pad == 64 && a.stride == 1) e = launch_wgrad_t<64, 4, 1>(a, parts, s);
  else if (cin == 64 && cout_pad == 8 && a.stride == 1) e = launch_wgrad_t<64, 1, 1>(a, parts, s);
  if (e != cudaSuccess) return e;
  const int n = 9 * cin_real * cout_real + cout_real;
  wgrad_reduce_kernel<<<(n + 31) / 32, 256, 0, s>>>(a.partial, parts, cout_pad < 16 ? 16 : cout_pad, cin, cin_real, cout_real,
                                                    gw, gb);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// Weight packing from the FP32 master layout [3][3][cin][cout]:
//   forward:   wk[tap][n = cout_pad][k = cin_pad]
//   transpose: wt[tap][n = cin][k = cout_pad]  with tap -> 8 - tap (the backward-data kernel)
// ---------------------------------------------------------------------------------------------
__global__ void pack_forward_kernel(const float* __restrict__ w, int cin, int cout, int cin_pad, int cout_pad,
                                    bf16* __restrict__ wk) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 9 * cout_pad * cin_pad) return;
  const int tap = i / (cout_pad * cin_pad), r = i % (cout_pad * cin_pad), n = r / cin_pad, k = r % cin_pad;
  const float v = (n < cout && k < cin) ? w[((size_t)tap * cin + k) * cout + n] : 0.f;
  wk[i] = __float2bfloat16(v);
}

__global__ void pack_transpose_kernel(const float* __restrict__ w, int cin, int cout, int cout_pad,
                                      bf16* __restrict__ wt) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 9 * cin * cout_pad) return;
  const int tp = i / (cin * cout_pad), r = i % (cin * cout_pad), n = r / cout_pad, k = r % cout_pad;
  const int tap = 8 - tp;
  const float v = k < cout ? w[((size_t)tap * cin + n) * cout + k] : 0.f;
  wt[i] = __float2bfloat16(v);
}

cudaError_t launch_pack(const float* w, int cin, int cout, int cin_pad, int cout_pad, bf16* wk, bf16* wt,
                        int cout_pad_t, cudaStream_t s) {
  const int n1 = 9 * cout_pad * cin_pad;
  pack_forward_kernel<<<(n1 + 255) / 256, 256, 0, s>>>(w, cin, cout, cin_pad, cout_pad, wk);
  if (wt) {
    const int n2 = 9 * cin * cout_pad_t;
    pack_transpose_kernel<<<(n2 + 255) / 256, 256, 0, s>>>(w, cin, cout, cout_pad_t, wt);
  }
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// Input, targets, loss, Adam
// ---------------------------------------------------------------------------------------------
// [n][H][W] depth + colour -> [n][H][W][16] BF16: (depth m - 3) / 2, (R, G, B / 255 - 1/2) x 4, zeros.
__global__ void input_kernel(const uint16_t* __restrict__ depth, const uint32_t* __restrict__ rgba, long n_pix,
                             bf16* __restrict__ x) {
  const long p = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n_pix) return;
  const uint32_t c = rgba[p];
  __align__(16) bf16 v[16];
  v[0] = input_depth(depth[p]);
  for (int k = 0; k < 3; ++k) v[1 + k] = input_colour((c >> (8 * k)) & 0xFF);
  for (int k = 4; k < 16; ++k) v[k] = __float2bfloat16(0.f);
  uint4* dst = reinterpret_cast<uint4*>(x + (size_t)p * 16);
  dst[0] = *reinterpret_cast<uint4*>(&v[0]);
  dst[1] = *reinterpret_cast<uint4*>(&v[8]);
}

cudaError_t launch_input(const uint16_t* depth, const uint32_t* rgba, long n_pix, bf16* x, cudaStream_t s) {
  input_kernel<<<(unsigned)((n_pix + 255) / 256), 256, 0, s>>>(depth, rgba, n_pix, x);
  return cudaGetLastError();
}

// Targets: scene coordinate of each cell's centre pixel minus the origin; w = 1 if scored.  The scored
// cells are counted into *scored (zeroed before).
__global__ void __launch_bounds__(256) targets_kernel(CellArgs a, float4* __restrict__ tgt, int32_t* __restrict__ scored) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int per = a.Wc * a.Hc;
  bool on = false;
  if (i < a.n * per) {
    const int img = i / per, c = i % per;
    on = a.depth[((size_t)img * a.H + c / a.Wc * 8 + 4) * a.W + c % a.Wc * 8 + 4] != 0;
  }
  const int count = __syncthreads_count(on);
  if (threadIdx.x == 0 && count) atomicAdd(scored, count);
  if (i >= a.n * per) return;
  const int img = i / per, c = i % per, cx = c % a.Wc, cy = c / a.Wc;
  const int u = cx * 8 + 4, v = cy * 8 + 4;
  const int d = a.depth[((size_t)img * a.H + v) * a.W + u];
  if (d == 0) {
    tgt[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    return;
  }
  const double z = d / 1000.0;
  const double c0 = z * (u - a.cx) / a.fx, c1 = z * (v - a.cy) / a.fy;
  const double* P = a.poses + 16 * (size_t)img;
  const double y0 = P[0] * c0 + P[1] * c1 + P[2] * z + P[3] - a.ox;
  const double y1 = P[4] * c0 + P[5] * c1 + P[6] * z + P[7] - a.oy;
  const double y2 = P[8] * c0 + P[9] * c1 + P[10] * z + P[11] - a.oz;
  tgt[i] = make_float4((float)y0, (float)y1, (float)y2, 1.f);
}

cudaError_t launch_targets(const CellArgs& a, float4* tgt, int32_t* counters, cudaStream_t s) {
  const int n = a.n * a.Wc * a.Hc;
  const cudaError_t e = cudaMemsetAsync(counters, 0, 2 * sizeof(int32_t), s);
  if (e != cudaSuccess) return e;
  targets_kernel<<<(n + 255) / 256, 256, 0, s>>>(a, tgt, counters);
  return cudaGetLastError();
}

// Loss and its gradient with respect to the head output (stored [cell][8] FP32), written as the
// BF16 gradient [cell][16] (channels 4..15 zero).  counters: [0] scored cells (targets_kernel), [1]
// CTAs done.  Each CTA leaves its sum; the last one to finish adds them in order, so the loss does not
// depend on scheduling (one CTA over all cells took 118 us for 16 views).
constexpr int kLossThreads = 256;
__global__ void __launch_bounds__(kLossThreads) loss_kernel(const float* __restrict__ out, const float4* __restrict__ tgt,
                                                            int n_cells, bf16* __restrict__ grad,
                                                            int32_t* __restrict__ counters, float* __restrict__ sums,
                                                            float* __restrict__ loss) {
  __shared__ float red[kLossThreads / 32];
  __shared__ int s_last;
  const int scored = counters[0];
  const float inv = 1.0f / (float)(scored > 0 ? scored : 1);
  float acc = 0.f;
  const int i = blockIdx.x * kLossThreads + threadIdx.x;
  if (i < n_cells) {
    const float4 y = tgt[i];
    const float4 o = *reinterpret_cast<const float4*>(out + (size_t)i * 8);
    __align__(16) bf16 gv[16];
    for (int k = 0; k < 16; ++k) gv[k] = __float2bfloat16(0.f);
    if (y.w > 0.5f) {
      // rho(e) + 1/2 e^2 exp(-s) + 3/2 s, rho(e) = sqrt(e^2 + 1e-6): the coordinates follow d rho,
      // s the NLL's derivative with the error held fixed
      const float e0 = o.x - y.x, e1 = o.y - y.y, e2 = o.z - y.z, s = o.w;
      const float sq = e0 * e0 + e1 * e1 + e2 * e2, es = expf(-s), rho = sqrtf(sq + 1e-6f);
      acc += rho + 0.5f * sq * es + 1.5f * s;
      const float gc = inv / rho;
      gv[0] = __float2bfloat16(e0 * gc);
      gv[1] = __float2bfloat16(e1 * gc);
      gv[2] = __float2bfloat16(e2 * gc);
      gv[3] = __float2bfloat16((-0.5f * sq * es + 1.5f) * inv);
    }
    uint4* dst = reinterpret_cast<uint4*>(grad + (size_t)i * 16);
    dst[0] = *reinterpret_cast<uint4*>(&gv[0]);
    dst[1] = *reinterpret_cast<uint4*>(&gv[8]);
  }
  acc = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    float s = 0.f;
    for (int w = 0; w < kLossThreads / 32; ++w) s += red[w];
    sums[blockIdx.x] = s;
    __threadfence();
    s_last = atomicAdd(&counters[1], 1) == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last || threadIdx.x >= 32) return;
  __threadfence();
  float s = 0.f;
  for (int c = threadIdx.x; c < (int)gridDim.x; c += 32) s += __ldcg(&sums[c]);
  s = warp_sum(s);
  if (threadIdx.x == 0) *loss = s * inv;
}

int loss_blocks(int n_cells) { return (n_cells + kLossThreads - 1) / kLossThreads; }

cudaError_t launch_loss(const float* out, const float4* tgt, int n_cells, bf16* grad, int32_t* counters, float* sums,
                        float* loss, cudaStream_t s) {
  loss_kernel<<<loss_blocks(n_cells), kLossThreads, 0, s>>>(out, tgt, n_cells, grad, counters, sums, loss);
  return cudaGetLastError();
}

// One Adam step of every parameter, and the BF16 weights and padded biases that the convolutions
// read (their padding stays as launch_pack left it): one launch instead of an update and 23 small
// packing launches (65 us a step).
constexpr int kCinFirst = kRegCin[0], kCinFirstPad = kRegCinPad[0];
constexpr int kCoutHead = kRegCout[kRegLayers - 1], kCoutHeadPad = kRegCoutPad[kRegLayers - 1];
__global__ void __launch_bounds__(256) adam_kernel(AdamArgs a, float lr, float b1, float b2, float eps, float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.n) return;
  const float gi = a.g[i];
  const float mi = b1 * a.m[i] + (1.f - b1) * gi;
  const float vi = b2 * a.v[i] + (1.f - b2) * gi * gi;
  a.m[i] = mi;
  a.v[i] = vi;
  float p = a.p[i];
  p -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  a.p[i] = p;
  int l = 0;
#pragma unroll
  for (int k = 1; k < kRegLayers; ++k) l += i >= a.w_off[k];
  const int cin = l == 0 ? kCinFirst : 64, cout = l == kRegLayers - 1 ? kCoutHead : 64;
  const int cin_pad = l == 0 ? kCinFirstPad : 64, cout_pad = l == kRegLayers - 1 ? kCoutHeadPad : 64;
  const int r = i - a.w_off[l];
  if (r >= 9 * cin * cout) {
    a.bias[l][r - 9 * cin * cout] = p;
    return;
  }
  const int tap = r / (cin * cout), k = r / cout % cin, n = r % cout;
  const bf16 w = __float2bfloat16(p);
  a.wk[l][((size_t)tap * cout_pad + n) * cin_pad + k] = w;
  const int pad_t = l == kRegLayers - 1 ? 16 : 64;
  if (l > 0) a.wt[l][((size_t)(8 - tap) * cin + k) * pad_t + n] = w;
}

cudaError_t launch_adam(const AdamArgs& a, float lr, int t, cudaStream_t s) {
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
  adam_kernel<<<(unsigned)((a.n + 255) / 256), 256, 0, s>>>(a, lr, b1, b2, 1e-8f, c1, c2);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// Cell forest: the regressor output as a one-tree forest over the cell grid (leaf = cell, one
// Gaussian of mean y_hat + o and covariance exp(s) I per scored cell) plus the coarse view
// (centre-pixel depths) the RANSAC runs on.
// ---------------------------------------------------------------------------------------------


__global__ void cell_forest_kernel(CellForestArgs a) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int img = blockIdx.y;
  if (i >= a.L) return;
  const int n = a.Wc * a.Hc;
  float* m = a.modes + ((size_t)img * a.L + i) * kModeFloats;
  uint8_t* nm = a.n_modes + (size_t)img * a.L;
  float4* top = a.top + (size_t)img * a.L;
  if (i >= n) {
    nm[i] = 0;
    top[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    return;
  }
  const int cx = i % a.Wc, cy = i / a.Wc;
  const int d = a.depth[(size_t)img * a.W * a.H + (size_t)(cy * 8 + 4) * a.W + cx * 8 + 4];
  const float* o = a.out + ((size_t)img * n + i) * a.ostride;
  const float s = o[3], inv = expf(-s);
  const float mx = o[0] + a.ox, my = o[1] + a.oy, mz = o[2] + a.oz;
  m[0] = mx;
  m[1] = my;
  m[2] = mz;
  m[3] = inv;
  m[4] = 0.f;
  m[5] = 0.f;
  m[6] = inv;
  m[7] = 0.f;
  m[8] = inv;
  m[9] = -1.5f * 1.8378770664093453f - 1.5f * s;  // log w - 0.5 log det(2 pi exp(s) I), w = 1
  m[10] = 1.f;
  m[11] = 0.f;
  nm[i] = d > 0 ? 1 : 0;
  top[i] = make_float4(mx, my, mz, d > 0 ? 1.f : 0.f);
  a.leaves[(size_t)img * n + i] = (uint16_t)i;
  a.depth_lr[(size_t)img * n + i] = (uint16_t)d;
}

cudaError_t launch_cell_forest(const CellForestArgs& a, cudaStream_t s) {
  if (a.n <= 0) return cudaSuccess;
  cell_forest_kernel<<<dim3((a.L + 255) / 256, a.n), 256, 0, s>>>(a);
  return cudaGetLastError();
}

// Head output [cell][8] -> [cell][4] (scene coordinate - origin, log-variance).
__global__ void head_copy_kernel(const float* __restrict__ head, long n, float* __restrict__ out4) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  reinterpret_cast<float4*>(out4)[i] = make_float4(head[i * 8], head[i * 8 + 1], head[i * 8 + 2], head[i * 8 + 3]);
}

cudaError_t launch_head_copy(const float* head, long n_cells, float* out4, cudaStream_t s) {
  head_copy_kernel<<<(unsigned)((n_cells + 255) / 256), 256, 0, s>>>(head, n_cells, out4);
  return cudaGetLastError();
}

}  // namespace relo
