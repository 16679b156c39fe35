// conv_tc.cu -- the regressor's 3x3 convolutions on the fifth-generation tensor cores (tcgen05,
// sm_103a): the forward pass of every layer and the backward-data pass of every layer but the first.
// conv_tc_kernel (the stride-2 layers of 64 channels, and the head's backward-data pass), then
// conv_halo_kernel (stride 1), conv_first_kernel (layer 1 from the images) and conv_up_kernel
// (backward-data of stride 2).  All share the roles and bounded waits described here.
//
// conv_tc_kernel, an implicit GEMM: the 128 output pixels of a tile (M) times the 64 output channels (N), contracted
// over 9 taps x 64 input channels (K).  For each tap the tile's input rows arrive in one TMA load:
// a 4-D tensor map over the NHWC BF16 activations [B][H][W][64] whose box is 64 channels x Wt x Ht
// pixels (Wt Ht = 128), walked with element strides equal to the layer's stride and started at the
// tap's offset ((ky - 1), (kx - 1)) x dilation.  Rows outside the image are zero-filled by the TMA
// unit: the convolution's zero padding.  A row is 64 channels = 128 B and lands 128-B swizzled,
// which is the canonical K-major layout of the MMA's shared-memory operand (8-row atoms of
// 1024 B).  The 9 taps' weights [9][64 out][64 in] are stored once per CTA in the same layout.
//
// Roles (one persistent CTA per SM, 6 warps): warp 0 issues the TMA loads into a ring of kStages
// buffers; one thread of warp 1 issues the 4 MMAs (K = 16 each) of every tap into one of two TMEM
// accumulators (128 lanes x 64 FP32 columns each) and commits them to mbarriers; warps 2-5 read a
// finished accumulator back (tcgen05.ld: each warp its quarter of the 128 lanes), add the bias,
// apply ReLU and store BF16 NHWC rows while the next tile accumulates into the other buffer.
//
// Every mbarrier wait is bounded by a wall-clock limit (the global nanosecond timer): a wait that
// runs out records RELO_ETIMEOUT in *status, raises the CTA's abort flag (every other wait of the
// CTA then gives up too), the producer waits (bounded) for the loads it still has in flight, and
// the CTA frees its TMEM and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>
#include <stdint.h>

#include <mutex>

#include "regressor.cuh"

namespace relo {
namespace {

constexpr int kTcThreads = 192;             // 6 warps
constexpr int kTcM = 128, kTcN = 64;
constexpr int kTcAccCols = 64;              // FP32 columns of one accumulator
constexpr int kTcTmemCols = 2 * kTcAccCols;

// Per input-channel count CIN (64: the strided layers but the first; 16: the head's backward-data pass, whose
// gradients' 4 channels are padded): a pixel row is CIN x 2 bytes, which is also the swizzle span of the
// operand layout (128 B or 32 B; 8-row atoms of 1024 B or 256 B).
template <int CIN>
struct TcShape {
  static constexpr int kRowBytes = CIN * 2;
  static constexpr int kABytes = kTcM * kRowBytes;           // one tap's tile: 16 KB or 4 KB
  static constexpr int kWBytes = 9 * kTcN * kRowBytes;
  static constexpr int kAtomBytes = 8 * kRowBytes;           // stride between 8-row atoms
  static constexpr int kChunks = kRowBytes / 16;             // 16-byte chunks per row
  static constexpr uint64_t kLayout = CIN == 64 ? 2 : 6;     // descriptor swizzle: 128 B / 32 B
  // A-operand ring: what shared memory holds beside the weights (8 stages of 16 KB, or 40 of 4 KB).
  static constexpr int kStages = CIN == 64 ? 8 : 40;
  static constexpr size_t kSmem = 1024 + (size_t)kWBytes + (size_t)kStages * kABytes;
  static_assert(CIN == 16 || CIN == 64, "64 -> 64 and 16 -> 64 channels");
};

struct TcArgs {
  const float* bias;      // [64] or null
  const bf16* mask;       // [B][Ho][Wo][64]: outputs where mask <= 0 are zeroed (ReLU derivative), or null
  const bf16* w;          // [9][64 out][64 in]
  bf16* out;              // [B][Ho][Wo][64]
  int32_t* status;        // RELO_ETIMEOUT when a wait ran out (else untouched)
  int B, Ho, Wo, stride, dil, relu;
  int Wt, Ht;             // tile shape in output pixels, Wt * Ht = 128
  int tiles_x, tiles_y, n_tiles;
  unsigned long long timeout_ns;
  int stall_tile;         // test hook: the producer issues no load for this tile (-1: none)
};

// ---- PTX wrappers ------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait for the phase with the given parity to complete.  False: the limit ran out or
// another role of the CTA gave up first (abort); the caller then stops its role.
template <class Args>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort, const Args& a) {
  const unsigned long long t0 = global_ns();
  for (uint32_t i = 0;; ++i) {
    if (mbar_test(bar, parity)) return true;
    if ((i & 63) == 63) {
      if (*abort) return false;
      if (global_ns() - t0 > a.timeout_ns) {
        *abort = 1;
        atomicExch(a.status, RELO_ETIMEOUT);
        return false;
      }
    }
  }
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2,
                                            int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
      : "memory");
}

// Shared-memory matrix descriptor of a K-major operand in a swizzled layout whose span equals a
// row: start address, stride between 8-row atoms (the leading offset is unused with these
// swizzles), descriptor version 1 (bits 46-47), swizzle mode (bits 61-63: 2 = 128 B, 6 = 32 B).
template <int CIN>
__device__ __forceinline__ uint64_t operand_desc(uint32_t addr) {
  using S = TcShape<CIN>;
  return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(S::kAtomBytes >> 4) << 32) |
         ((uint64_t)1 << 46) | (S::kLayout << 61);
}

// Offset of 16-byte chunk j of row r in the swizzled layout: the chunk index XOR the row's position
// in its 8-row atom (128 B: 3 bits), or its bit 2 (32 B: 1 bit), as the TMA unit writes it.
template <int CIN>
__device__ __forceinline__ int swizzled(int r, int j) {
  using S = TcShape<CIN>;
  const int x = CIN == 64 ? (r & 7) : ((r >> 2) & 1);
  return r * S::kRowBytes + ((j ^ x) << 4);
}

// Instruction descriptor of kind::f16: D FP32 (bits 4-5 = 1), A and B BF16 (bits 7-9, 10-12 = 1),
// both K-major (bits 15, 16 = 0), N / 8 at bits 17-22, M / 16 at bits 24-28.
template <int N>
constexpr uint32_t kTcIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
                              ((uint32_t)(kTcM >> 4) << 24);

template <int N = kTcN>
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(kTcIdesc<N>), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// mbar_wait by lane 0 for the warp.
template <class Args>
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort, const Args& a, int lane) {
  const bool r = lane == 0 ? mbar_wait(bar, parity, abort, a) : false;
  return __shfl_sync(0xffffffffu, r, 0);
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 32 lanes x 32 consecutive FP32 columns: thread i of the warp gets lane (base + i), columns col..col+31
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,"
      "%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8]) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tile_origin(const TcArgs& a, int t, int& b, int& oy0, int& ox0) {
  const int per = a.tiles_x * a.tiles_y;
  b = t / per;
  const int r = t - b * per;
  oy0 = (r / a.tiles_x) * a.Ht;
  ox0 = (r % a.tiles_x) * a.Wt;
}

template <int CIN>
__global__ void __launch_bounds__(kTcThreads, 1) conv_tc_kernel(const __grid_constant__ CUtensorMap in_map, TcArgs a) {
  using S = TcShape<CIN>;
  constexpr int kTcStages = S::kStages;
  extern __shared__ uint8_t tc_smem_raw[];
  __shared__ uint64_t bars[2 * kTcStages + 5];     // full[s], empty[s], acc_full[2], acc_empty[2], drain
  __shared__ uint32_t tmem_base_sh;
  __shared__ int abort_sh;
  uint8_t* base = reinterpret_cast<uint8_t*>(((uintptr_t)tc_smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sW = base;                    // [9][64][row] swizzled
  uint8_t* sA = base + S::kWBytes;       // [kStages][128][row] swizzled
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t full0 = smem_u32(&bars[0]), empty0 = smem_u32(&bars[kTcStages]);
  const uint32_t accf0 = smem_u32(&bars[2 * kTcStages]), acce0 = smem_u32(&bars[2 * kTcStages + 2]);
  const uint32_t drain = smem_u32(&bars[2 * kTcStages + 4]);
  volatile int* abort = &abort_sh;

  // weights -> shared memory in the swizzled K-major layout
  for (int v = threadIdx.x; v < 9 * kTcN * S::kChunks; v += kTcThreads) {
    const int row = v / S::kChunks, j = v % S::kChunks;
    const uint4 x = __ldg(reinterpret_cast<const uint4*>(a.w) + v);
    *reinterpret_cast<uint4*>(sW + swizzled<CIN>(row, j)) = x;
  }
  if (threadIdx.x == 0) {
    abort_sh = 0;
    for (int s = 0; s < kTcStages; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(accf0 + 8 * b, 1);
      mbar_init(acce0 + 8 * b, 4);
    }
    mbar_init(drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // the generic-proxy stores of the weights must be visible to the tensor cores' async proxy
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_sh)),
                 "r"(kTcTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_sh;

  if (warp == 0) {
    // ---- producer: one TMA load per (tile, tap) ----
    if (lane == 0) {
      uint32_t q = 0;
      int issued[kTcStages];         // stage s holds a load not yet known to be consumed ...
      uint32_t phase[kTcStages];     // ... which completes the full barrier's phase of this parity
      for (int s = 0; s < kTcStages; ++s) issued[s] = 0, phase[s] = 0;
      bool ok = true;
      for (int t = blockIdx.x; ok && t < a.n_tiles; t += gridDim.x) {
        int b, oy0, ox0;
        tile_origin(a, t, b, oy0, ox0);
        for (int tap = 0; tap < 9; ++tap, ++q) {
          const int s = (int)(q % kTcStages);
          const uint32_t round = q / kTcStages;
          if (round > 0 && !mbar_wait(empty0 + 8 * s, (round - 1) & 1, abort, a)) {
            ok = false;
            break;
          }
          issued[s] = 0;
          if (t == a.stall_tile) continue;   // test hook: the consumer's wait for this stage runs out
          const int ky = tap / 3, kx = tap % 3;
          mbar_expect_tx(full0 + 8 * s, S::kABytes);
          tma_load_4d(smem_u32(sA + s * S::kABytes), &in_map, full0 + 8 * s, 0, ox0 * a.stride + (kx - 1) * a.dil,
                      oy0 * a.stride + (ky - 1) * a.dil, b);
          issued[s] = 1;
          phase[s] = round & 1;
        }
      }
      if (!ok || *abort) {
        // copies still in flight land before the CTA's shared memory is released
        for (int s = 0; s < kTcStages; ++s) {
          if (!issued[s]) continue;
          const unsigned long long t0 = global_ns();
          while (!mbar_test(full0 + 8 * s, phase[s]) && global_ns() - t0 < a.timeout_ns) {
          }
        }
      }
    }
  } else if (warp == 1) {
    // ---- MMA issuer ----
    if (lane == 0) {
      uint32_t q = 0, it = 0;
      bool ok = true;
      for (int t = blockIdx.x; ok && t < a.n_tiles; t += gridDim.x, ++it) {
        const int buf = (int)(it & 1);
        const uint32_t use = it >> 1;
        if (use > 0 && !mbar_wait(acce0 + 8 * buf, (use - 1) & 1, abort, a)) break;
        tc_fence_after();
        const uint32_t d = tmem + (uint32_t)(buf * kTcAccCols);
        for (int tap = 0; tap < 9; ++tap, ++q) {
          const int s = (int)(q % kTcStages);
          if (!mbar_wait(full0 + 8 * s, (q / kTcStages) & 1, abort, a)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t a0 = smem_u32(sA + s * S::kABytes), b0 = smem_u32(sW + tap * (kTcN * S::kRowBytes));
#pragma unroll
          for (int kk = 0; kk < CIN / 16; ++kk)
            umma_bf16(d, operand_desc<CIN>(a0 + 32 * kk), operand_desc<CIN>(b0 + 32 * kk), (tap > 0 || kk > 0) ? 1u : 0u);
          umma_commit(empty0 + 8 * s);      // the stage is free once these MMAs have read it
        }
        if (ok) umma_commit(accf0 + 8 * buf);
      }
      if (!ok || *abort) {
        // MMAs still in flight finish before the TMEM is released
        umma_commit(drain);
        const unsigned long long t0 = global_ns();
        while (!mbar_test(drain, 0) && global_ns() - t0 < a.timeout_ns) {
        }
      }
    }
  } else {
    // ---- epilogue: warps 2-5, TMEM lane quarter = warp % 4 ----
    const int quarter = warp & 3;
    uint32_t it = 0;
    for (int t = blockIdx.x; t < a.n_tiles; t += gridDim.x, ++it) {
      const int buf = (int)(it & 1);
      // lane 0 waits for the accumulator and tells the warp: tcgen05.ld needs the whole warp
      bool ready = lane == 0 ? mbar_wait(accf0 + 8 * buf, (it >> 1) & 1, abort, a) : false;
      ready = __shfl_sync(0xffffffffu, ready, 0);
      if (!ready) break;
      tc_fence_after();
      const int m = quarter * 32 + lane;
      float v0[32], v1[32];
      const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(buf * kTcAccCols);
      tmem_ld32(taddr, v0);
      tmem_ld32(taddr + 32, v1);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acce0 + 8 * buf);
      int b, oy0, ox0;
      tile_origin(a, t, b, oy0, ox0);
      const int oy = oy0 + m / a.Wt, ox = ox0 + m % a.Wt;
      if (oy < a.Ho && ox < a.Wo) {
        const size_t px = ((size_t)b * a.Ho + oy) * a.Wo + ox;
        uint4* dst = reinterpret_cast<uint4*>(a.out + px * kTcN);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          uint4 mk = make_uint4(0u, 0u, 0u, 0u);
          if (a.mask) mk = __ldg(reinterpret_cast<const uint4*>(a.mask + px * kTcN) + j);
          const uint32_t mw[4] = {mk.x, mk.y, mk.z, mk.w};
          uint32_t pk[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int n = 8 * j + 2 * e;
            const float* v = n < 32 ? v0 : v1;
            float x0 = v[n & 31], x1 = v[(n & 31) + 1];
            if (a.bias) {
              x0 += __ldg(&a.bias[n]);
              x1 += __ldg(&a.bias[n + 1]);
            }
            if (a.relu) {
              x0 = fmaxf(x0, 0.f);
              x1 = fmaxf(x1, 0.f);
            }
            if (a.mask) {
              const __nv_bfloat162 mm = *reinterpret_cast<const __nv_bfloat162*>(&mw[e]);
              if (!(__bfloat162float(mm.x) > 0.f)) x0 = 0.f;
              if (!(__bfloat162float(mm.y) > 0.f)) x1 = 0.f;
            }
            const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
            pk[e] = *reinterpret_cast<const uint32_t*>(&h);
          }
          dst[j] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcTmemCols) : "memory");
  }
}

// =============================================================================================
// Stride 1, 64 input channels: the layers at one cell per 8 x 8 pixels and their backward-data passes.
//
// The kernel above loads each tap's 128 x 64 operand on its own, 147 KB a tile of which 23 KB are
// distinct, and a layer's time was the loads' (58 us for 64 views of 640 x 480, the MMAs an eighth of
// it).  Here an output tile is 8 x 16 pixels and its input comes as three copies, one per kernel
// column kx: 18 rows of 8 pixels starting at column ox0 + kx - 1.  A row of 8 pixels is one 1024-B atom
// of the swizzled K-major layout, so the operand of tap (ky, kx) is 16 consecutive atoms of copy kx
// from atom ky on: 55 KB a tile serve all nine taps, with every operand on an atom boundary.  Two tiles
// are in flight.  The weights come by TMA too (a thread's loads took microseconds before the first
// MMA), and the outputs leave by TMA through a staging tile per epilogue warp, which also clips the
// image's ragged edge.  Taps and channels are multiplied in the same order as above: the same bits.
// N = 64 output channels, or 16 for the head (8 stored, FP32).
// 64 views: 33 us a layer.  The 36 MMAs of a tile bound it (2800 cycles of 3100, measured at the issuing
// thread): each takes about 70 cycles whether N is 16 or 64, the time of reading its 128 rows of A from
// shared memory, so 64 channels reach half the tensor core's rate at best.
// =============================================================================================
struct HaloArgs {
  const float* bias;      // [N] ([8] for the head) or null
  const bf16* mask;       // [B][Ho][Wo][64] or null (64 channels)
  float* out_f32;         // head: [B][Ho][Wo][8]
  int32_t* status;
  int Ho, Wo, relu;
  int tiles_x, tiles_y, n_tiles;
  unsigned long long timeout_ns;
  int stall_tile;
};

constexpr int kHaloThreads = 320;                             // loads, MMA, 4 epilogue warps per accumulator buffer
constexpr int kHaloW = 8, kHaloH = 16;                        // output pixels of a tile
constexpr int kHaloCopy = (kHaloH + 2) * kHaloW * 128;        // one column copy: 18 atoms
constexpr int kHaloStage = 3 * kHaloCopy, kHaloStages = 2;
constexpr int kHaloStaging = 32 * 128;                        // an epilogue warp's 32 output rows
template <int N>
struct HaloShape {
  static constexpr int kTap = N * 128;                        // one tap's weights
  static constexpr int kWeights = 9 * kTap;
  static constexpr int kCols = N < 16 ? 16 : N;               // accumulator columns
  static constexpr int kTmem = 2 * kCols;
  static constexpr int kStagings = N == 64 ? 2 * 4 : 0;
  static constexpr size_t kSmem = 1024 + kWeights + kHaloStages * kHaloStage + kStagings * kHaloStaging;
};

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void tma_store_4d(const CUtensorMap* map, uint32_t src, int c0, int c1, int c2, int c3) {
  asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(src), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
               : "memory");
}

__device__ __forceinline__ void halo_origin(const HaloArgs& a, int t, int& b, int& oy0, int& ox0) {
  const int per = a.tiles_x * a.tiles_y;
  b = t / per;
  const int r = t - b * per;
  oy0 = r / a.tiles_x * kHaloH;
  ox0 = r % a.tiles_x * kHaloW;
}

// One output channel: bias, ReLU.
__device__ __forceinline__ float finish(float x, float bias, int relu) {
  x += bias;
  return relu ? fmaxf(x, 0.f) : x;
}

// 32 channels (half 0 or 1) of a warp's 32 output pixels, finished, rounded and laid out in the warp's
// staging tile (128-B rows, swizzled), from which one lane's TMA store takes the rows.
__device__ __forceinline__ void stage_half(uint8_t* stage, int lane, int half, const float (&v)[32], const float* bias,
                                           int relu, const bf16* mask) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int c8 = 4 * half + j;
    uint4 mk = make_uint4(0x3F803F80u, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u);
    if (mask) mk = __ldg(reinterpret_cast<const uint4*>(mask) + c8);
    const uint32_t mw[4] = {mk.x, mk.y, mk.z, mk.w};
    uint32_t pk[4];
    float bb[8];
    if (bias) {
      const float4 lo = reinterpret_cast<const float4*>(bias)[2 * c8], hi = reinterpret_cast<const float4*>(bias)[2 * c8 + 1];
      bb[0] = lo.x, bb[1] = lo.y, bb[2] = lo.z, bb[3] = lo.w, bb[4] = hi.x, bb[5] = hi.y, bb[6] = hi.z, bb[7] = hi.w;
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      float x0 = v[8 * j + 2 * e], x1 = v[8 * j + 2 * e + 1];
      if (bias) {
        x0 = finish(x0, bb[2 * e], relu);
        x1 = finish(x1, bb[2 * e + 1], relu);
      }
      const __nv_bfloat162 mm = *reinterpret_cast<const __nv_bfloat162*>(&mw[e]);
      if (!(__bfloat162float(mm.x) > 0.f)) x0 = 0.f;
      if (!(__bfloat162float(mm.y) > 0.f)) x1 = 0.f;
      const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
      pk[e] = *reinterpret_cast<const uint32_t*>(&h);
    }
    *reinterpret_cast<uint4*>(stage + swizzled<64>(lane, c8)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
  }
}

// The staged rows are seen by the TMA store that one lane issues next.
__device__ __forceinline__ void stage_done() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncwarp();
}

template <int N>
__global__ void __launch_bounds__(kHaloThreads, 1)
    conv_halo_kernel(const __grid_constant__ CUtensorMap in_map, const __grid_constant__ CUtensorMap w_map,
                     const __grid_constant__ CUtensorMap out_map, const __grid_constant__ HaloArgs a) {
  using S = HaloShape<N>;
  extern __shared__ uint8_t tc_smem_raw[];
  __shared__ uint64_t bars[2 * kHaloStages + 6];  // full[s], empty[s], acc_full[2], acc_empty[2], weights, drain
  __shared__ uint32_t tmem_base_sh;
  __shared__ int abort_sh;
  __shared__ __align__(16) float s_bias[64];
  uint8_t* base = reinterpret_cast<uint8_t*>(((uintptr_t)tc_smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sA = base;                                    // [stage][kx][18][8][128 B], swizzled
  uint8_t* sW = base + kHaloStages * kHaloStage;         // [9][N][128 B], swizzled
  uint8_t* sOut = sW + S::kWeights;                      // [2][4 warps][32][128 B], swizzled
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t full0 = smem_u32(&bars[0]), empty0 = smem_u32(&bars[kHaloStages]);
  const uint32_t accf0 = smem_u32(&bars[2 * kHaloStages]), acce0 = smem_u32(&bars[2 * kHaloStages + 2]);
  const uint32_t wfull = smem_u32(&bars[2 * kHaloStages + 4]), drain = smem_u32(&bars[2 * kHaloStages + 5]);
  volatile int* abort = &abort_sh;
  if (threadIdx.x < 64) s_bias[threadIdx.x] = a.bias && (N == 64 || threadIdx.x < 8) ? a.bias[threadIdx.x] : 0.f;
  if (N == 16) {
    // the head's 8 output channels come by TMA; the other 8 rows of each tap's operand are zero
    for (int v = threadIdx.x; v < 9 * 64; v += kHaloThreads)
      *reinterpret_cast<uint4*>(sW + (v / 64) * S::kTap + 1024 + (v % 64) * 16) = make_uint4(0u, 0u, 0u, 0u);
  }
  if (threadIdx.x == 0) {
    abort_sh = 0;
    for (int s = 0; s < kHaloStages; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(accf0 + 8 * b, 1);
      mbar_init(acce0 + 8 * b, 4);
    }
    mbar_init(wfull, 1);
    mbar_init(drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_sh)),
                 "r"(S::kTmem)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_sh;

  if (warp == 0) {
    // ---- producer: the weights, then three column copies per tile ----
    if (lane == 0) {
      constexpr int kRows = N == 64 ? 64 : 8;  // weight rows of a tap
      mbar_expect_tx(wfull, 9 * kRows * 128);
      for (int tap = 0; tap < 9; ++tap) tma_load_2d(smem_u32(sW + tap * S::kTap), &w_map, wfull, 0, tap * kRows);
      uint32_t q = 0;
      int issued[kHaloStages] = {};
      uint32_t phase[kHaloStages] = {};
      bool ok = true;
      for (int t = blockIdx.x; t < a.n_tiles; t += gridDim.x, ++q) {
        const int s = (int)(q % kHaloStages);
        const uint32_t round = q / kHaloStages;
        if (round > 0 && !mbar_wait(empty0 + 8 * s, (round - 1) & 1, abort, a)) {
          ok = false;
          break;
        }
        issued[s] = 0;
        if (t == a.stall_tile) continue;  // test hook: the consumer's wait for this tile runs out
        int b, oy0, ox0;
        halo_origin(a, t, b, oy0, ox0);
        mbar_expect_tx(full0 + 8 * s, kHaloStage);
        for (int kx = 0; kx < 3; ++kx)
          tma_load_4d(smem_u32(sA + s * kHaloStage + kx * kHaloCopy), &in_map, full0 + 8 * s, 0, ox0 + kx - 1, oy0 - 1, b);
        issued[s] = 1;
        phase[s] = round & 1;
      }
      if (!ok || *abort) {
        // copies still in flight land before the CTA's shared memory is released
        const unsigned long long t0 = global_ns();
        while (!mbar_test(wfull, 0) && global_ns() - t0 < a.timeout_ns) {
        }
        for (int s = 0; s < kHaloStages; ++s) {
          if (!issued[s]) continue;
          const unsigned long long t1 = global_ns();
          while (!mbar_test(full0 + 8 * s, phase[s]) && global_ns() - t1 < a.timeout_ns) {
          }
        }
      }
    }
  } else if (warp == 1) {
    // ---- MMA issuer ----
    if (lane == 0) {
      uint32_t q = 0;
      const bool ok = mbar_wait(wfull, 0, abort, a);
      for (int t = blockIdx.x; ok && t < a.n_tiles; t += gridDim.x, ++q) {
        const int buf = (int)(q & 1), s = (int)(q % kHaloStages);
        const uint32_t use = q >> 1;
        if (use > 0 && !mbar_wait(acce0 + 8 * buf, (use - 1) & 1, abort, a)) break;
        if (!mbar_wait(full0 + 8 * s, (q / kHaloStages) & 1, abort, a)) break;
        tc_fence_after();
        const uint32_t d = tmem + (uint32_t)(buf * S::kCols);
        const uint64_t ad = operand_desc<64>(smem_u32(sA + s * kHaloStage)), bd = operand_desc<64>(smem_u32(sW));
#pragma unroll
        for (int tap = 0; tap < 9; ++tap) {
          const int ky = tap / 3, kx = tap % 3;
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            umma_bf16<N>(d, ad + ((kx * kHaloCopy + ky * 1024 + 32 * kk) >> 4), bd + ((tap * S::kTap + 32 * kk) >> 4),
                         (tap > 0 || kk > 0) ? 1u : 0u);
        }
        umma_commit(empty0 + 8 * s);
        umma_commit(accf0 + 8 * buf);
      }
      if (*abort) {
        // MMAs still in flight finish before the TMEM is released
        umma_commit(drain);
        const unsigned long long t0 = global_ns();
        while (!mbar_test(drain, 0) && global_ns() - t0 < a.timeout_ns) {
        }
      }
    }
  } else {
    // ---- epilogue: warps 2-9, four per accumulator buffer, TMEM lane quarter = warp % 4: rows
    // 4 quarter .. + 3 of the tile ----
    const int quarter = warp & 3, buf = (warp - 2) >> 2;
    uint32_t q = buf;
    for (int t = blockIdx.x + buf * gridDim.x; t < a.n_tiles; t += 2 * gridDim.x, q += 2) {
      if (!mbar_wait_warp(accf0 + 8 * buf, (q >> 1) & 1, abort, a, lane)) break;
      tc_fence_after();
      int b, oy0, ox0;
      halo_origin(a, t, b, oy0, ox0);
      const int oy = oy0 + quarter * 4 + (lane >> 3), ox = ox0 + (lane & 7);
      const bool inside = oy < a.Ho && ox < a.Wo;
      const size_t px = ((size_t)b * a.Ho + oy) * a.Wo + ox;
      const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(buf * S::kCols);
      if (N == 16) {
        float v[8];
        tmem_ld8(taddr, v);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acce0 + 8 * buf);
        if (inside) {
          float4* dst = reinterpret_cast<float4*>(a.out_f32 + px * 8);
#pragma unroll
          for (int j = 0; j < 2; ++j)
            dst[j] = make_float4(finish(v[4 * j], s_bias[4 * j], a.relu), finish(v[4 * j + 1], s_bias[4 * j + 1], a.relu),
                                 finish(v[4 * j + 2], s_bias[4 * j + 2], a.relu),
                                 finish(v[4 * j + 3], s_bias[4 * j + 3], a.relu));
        }
      } else {
        float v0[32], v1[32];
        tmem_ld32(taddr, v0);
        tmem_ld32(taddr + 32, v1);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acce0 + 8 * buf);
        uint8_t* stage = sOut + (buf * 4 + quarter) * kHaloStaging;
        // the last store has read this staging tile
        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        __syncwarp();
        const float* bias = a.bias ? s_bias : nullptr;
        const bf16* mask = a.mask && inside ? a.mask + px * kTcN : nullptr;
        stage_half(stage, lane, 0, v0, bias, a.relu, mask);
        stage_half(stage, lane, 1, v1, bias, a.relu, mask);
        stage_done();
        if (lane == 0) {
          if (oy0 + quarter * 4 < a.Ho) tma_store_4d(&out_map, smem_u32(stage), 0, ox0, oy0 + quarter * 4, b);
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
      }
    }
    // stores still in flight finish before the CTA's shared memory is released
    if (N == 64 && lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(S::kTmem) : "memory");
  }
}

// =============================================================================================
// The first layer (stride 2, 4 real input channels of 16, 64 output channels), straight from the depth
// and colour images.
//
// Its operand rows are 32 B, of which 8 are not zero; loading each tap's rows by TMA took 563 us for 64
// views of 640 x 480 (the unit's rate for short strided rows), and making the padded 16-channel input
// another 116 us.  Here sixteen warps convert the 33 x 17 pixels under a tile of 16 x 8 outputs and place
// them in shared memory as the MMA's K-major operand (32-B rows, whose zero channels are written once):
// three copies, one per kernel column kx, of 16 pixels a row, a copy's even input rows first, then its
// odd ones, so that the operand of tap (ky, kx) is 8 consecutive rows of one parity.  Taps in order, 16
// channels per MMA: the same products and sums as before.  246 us for 64 views.  The output's 629 MB
// would take 92; the rest is the nine MMAs a tile (1100 cycles) and the conversions, which eight warps
// had taken 330 us for: a warp alone issues one of its dependent instructions every few cycles.
// =============================================================================================
struct FirstArgs {
  const uint16_t* depth;  // [B][H][W] mm
  const uint32_t* rgba;   // [B][H][W]
  const float* bias;
  const bf16* w;          // [9][64][16]
  int32_t* status;
  int H, W, Ho, Wo;
  int tiles_x, tiles_y, n_tiles;
  unsigned long long timeout_ns;
  int stall_tile;
};

constexpr int kFirstW = 16, kFirstH = 8;
constexpr int kFirstRow = kFirstW * 32;                              // one input row of a copy
constexpr int kFirstCopy = (2 * kFirstH + 1) * kFirstRow;            // even rows (9), then odd rows (8)
constexpr int kFirstOdd = (kFirstH + 1) * kFirstRow;
constexpr int kFirstStage = 3 * kFirstCopy, kFirstStages = 4;
constexpr int kFirstConv = 16, kFirstGroup = kFirstConv / kFirstStages;  // converting warps, a group of four per stage
constexpr int kFirstThreads = 32 * (kFirstConv + 9);                 // ..., MMA, 2 x 4 epilogue warps
constexpr int kFirstPer = (2 * kFirstH + 1 + kFirstGroup - 1) / kFirstGroup;
static_assert(kFirstGroup == 4 && kFirstPer == 5 && kFirstW == 16, "17 rows of 33 pixels by 4 warps: see the converting warps");
constexpr int kFirstStaging = 2 * 4 * 32 * 128;
constexpr size_t kFirstSmem = 1024 + kFirstStaging + 9 * 64 * 32 + kFirstStages * kFirstStage;

__global__ void __launch_bounds__(kFirstThreads, 1)
    conv_first_kernel(const __grid_constant__ CUtensorMap out_map, const __grid_constant__ FirstArgs a) {
  extern __shared__ uint8_t tc_smem_raw[];
  __shared__ uint64_t bars[2 * kFirstStages + 5];
  __shared__ uint32_t tmem_base_sh;
  __shared__ int abort_sh;
  __shared__ __align__(16) float s_bias[64];
  __shared__ bf16 s_colour[256];
  uint8_t* base = reinterpret_cast<uint8_t*>(((uintptr_t)tc_smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sOut = base;                                  // [2][4 warps][32][128 B], swizzled
  uint8_t* sW = sOut + kFirstStaging;                    // [9][64][32 B], swizzled
  uint8_t* sA = sW + 9 * 64 * 32;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t full0 = smem_u32(&bars[0]), empty0 = smem_u32(&bars[kFirstStages]);
  const uint32_t accf0 = smem_u32(&bars[2 * kFirstStages]), acce0 = smem_u32(&bars[2 * kFirstStages + 2]);
  const uint32_t drain = smem_u32(&bars[2 * kFirstStages + 4]);
  volatile int* abort = &abort_sh;
  for (int v = threadIdx.x; v < 9 * 64 * 2; v += kFirstThreads)
    *reinterpret_cast<uint4*>(sW + swizzled<16>(v / 2, v % 2)) = __ldg(reinterpret_cast<const uint4*>(a.w) + v);
  for (int v = threadIdx.x; v < kFirstStages * kFirstStage / 16; v += kFirstThreads)
    reinterpret_cast<uint4*>(sA)[v] = make_uint4(0u, 0u, 0u, 0u);
  if (threadIdx.x < 64) s_bias[threadIdx.x] = a.bias[threadIdx.x];
  if (threadIdx.x < 256) s_colour[threadIdx.x] = input_colour((uint32_t)threadIdx.x);
  if (threadIdx.x == 0) {
    abort_sh = 0;
    for (int s = 0; s < kFirstStages; ++s) {
      mbar_init(full0 + 8 * s, kFirstGroup);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(accf0 + 8 * b, 1);
      mbar_init(acce0 + 8 * b, 4);
    }
    mbar_init(drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (warp == kFirstConv) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_sh)),
                 "r"(kTcTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_sh;
  const int per = a.tiles_x * a.tiles_y;

  if (warp < kFirstConv) {
    // ---- converting warps: a group's next pixels are on their way while it places these; the fence
    // waits for them too, so four groups take tiles in turn, each its own stage.  Warp w of a group takes
    // the window's rows w, w + 4, ..., a lane per column; column 32 is the fifth turn of warp 3 ----
    const int s = warp / kFirstGroup, w = warp % kFirstGroup;
    uint32_t dep[kFirstPer], col[kFirstPer];
    auto fetch = [&](int t) {
      const int b = t / per, r = t - b * per, iy0 = 2 * (r / a.tiles_x * kFirstH) - 1, ix0 = 2 * (r % a.tiles_x * kFirstW) - 1;
      const size_t image = (size_t)b * a.H * a.W;
#pragma unroll
      for (int k = 0; k < kFirstPer; ++k) {
        const bool last = k == 4 && w == 3;
        const int row = last ? lane : w + 4 * k, iy = iy0 + row, ix = ix0 + (last ? 32 : lane);
        dep[k] = 0x10000u;  // outside the image: zeros
        col[k] = 0;
        if (row < 2 * kFirstH + 1 && iy >= 0 && ix >= 0 && iy < a.H && ix < a.W) {
          const size_t px = image + (size_t)iy * a.W + ix;
          dep[k] = __ldg(&a.depth[px]);
          col[k] = __ldg(&a.rgba[px]);
        }
      }
    };
    const int first = blockIdx.x + s * gridDim.x, step = kFirstStages * gridDim.x;
    uint32_t round = 0;
    if (first < a.n_tiles) fetch(first);
    for (int t = first; t < a.n_tiles; t += step, ++round) {
      if (round > 0 && !mbar_wait_warp(empty0 + 8 * s, (round - 1) & 1, abort, a, lane)) break;
      uint2 v[kFirstPer];
#pragma unroll
      for (int k = 0; k < kFirstPer; ++k) {
        const bf16 d = input_depth(dep[k]);
        const uint32_t d16 = *reinterpret_cast<const uint16_t*>(&d);
        const uint16_t* lut = reinterpret_cast<const uint16_t*>(s_colour);
        v[k] = make_uint2(d16 | (uint32_t)lut[col[k] & 0xFF] << 16,
                          (uint32_t)lut[(col[k] >> 8) & 0xFF] | (uint32_t)lut[(col[k] >> 16) & 0xFF] << 16);
        if (dep[k] & 0x10000u) v[k] = make_uint2(0u, 0u);
      }
      if (t + step < a.n_tiles) fetch(t + step);
      uint8_t* st = sA + s * kFirstStage;
#pragma unroll
      for (int k = 0; k < kFirstPer; ++k) {
        const bool last = k == 4 && w == 3;
        const int row = last ? lane : w + 4 * k, j = last ? 32 : lane;
        if (row >= 2 * kFirstH + 1) continue;
        uint8_t* at = st + ((row & 1) ? kFirstOdd : 0) + (row >> 1) * kFirstRow;
        if (j & 1) {
          *reinterpret_cast<uint2*>(at + kFirstCopy + swizzled<16>(j >> 1, 0)) = v[k];
        } else {
          if (j < 2 * kFirstW) *reinterpret_cast<uint2*>(at + swizzled<16>(j >> 1, 0)) = v[k];
          if (j >= 2) *reinterpret_cast<uint2*>(at + 2 * kFirstCopy + swizzled<16>((j >> 1) - 1, 0)) = v[k];
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0 && t != a.stall_tile) mbar_arrive(full0 + 8 * s);  // (stall_tile: test hook, a wait that runs out)
    }
  } else if (warp == kFirstConv) {
    // ---- MMA issuer ----
    if (lane == 0) {
      uint32_t q = 0;
      for (int t = blockIdx.x; t < a.n_tiles; t += gridDim.x, ++q) {
        const int buf = (int)(q & 1), s = (int)(q % kFirstStages);
        const uint32_t use = q >> 1;
        if (use > 0 && !mbar_wait(acce0 + 8 * buf, (use - 1) & 1, abort, a)) break;
        if (!mbar_wait(full0 + 8 * s, (q / kFirstStages) & 1, abort, a)) break;
        tc_fence_after();
        const uint32_t d = tmem + (uint32_t)(buf * kTcAccCols);
        const uint32_t a0 = smem_u32(sA + s * kFirstStage);
        const uint64_t bd = operand_desc<16>(smem_u32(sW));
#pragma unroll
        for (int tap = 0; tap < 9; ++tap) {
          const int ky = tap / 3, kx = tap % 3;
          const uint32_t at = a0 + kx * kFirstCopy + ((ky & 1) ? kFirstOdd : 0) + (ky >> 1) * kFirstRow;
          umma_bf16<kTcN>(d, operand_desc<16>(at), bd + ((tap * (kTcN * 32)) >> 4), tap > 0 ? 1u : 0u);
        }
        umma_commit(empty0 + 8 * s);
        umma_commit(accf0 + 8 * buf);
      }
      if (*abort) {
        umma_commit(drain);
        const unsigned long long t0 = global_ns();
        while (!mbar_test(drain, 0) && global_ns() - t0 < a.timeout_ns) {
        }
      }
    }
  } else {
    // ---- epilogue: four warps per accumulator buffer, TMEM lane quarter = warp % 4: rows 2 quarter,
    // 2 quarter + 1 of the tile ----
    const int quarter = warp & 3, buf = (warp - kFirstConv - 1) >> 2;
    uint32_t q = buf;
    for (int t = blockIdx.x + buf * gridDim.x; t < a.n_tiles; t += 2 * gridDim.x, q += 2) {
      if (!mbar_wait_warp(accf0 + 8 * buf, (q >> 1) & 1, abort, a, lane)) break;
      tc_fence_after();
      const int b = t / per, r = t - b * per, oy = r / a.tiles_x * kFirstH + quarter * 2, ox0 = r % a.tiles_x * kFirstW;
      const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(buf * kTcAccCols);
      uint8_t* stage = sOut + (buf * 4 + quarter) * (32 * 128);
      if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
      __syncwarp();
      float v[32];  // a half of the channels at a time: 25 warps leave 80 registers a thread
      tmem_ld32(taddr, v);
      stage_half(stage, lane, 0, v, s_bias, 1, nullptr);
      tmem_ld32(taddr + 32, v);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acce0 + 8 * buf);
      stage_half(stage, lane, 1, v, s_bias, 1, nullptr);
      stage_done();
      if (lane == 0) {
        if (oy < a.Ho) tma_store_4d(&out_map, smem_u32(stage), 0, ox0, oy, b);
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
      }
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kFirstConv) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcTmemCols) : "memory");
  }
}

// =============================================================================================
// Backward-data of a stride-2 layer: the convolution of the zero-inserted output gradient g with the
// flipped, transposed weights.  Three of four inserted pixels are zero, so an input pixel (2 y + py,
// 2 x + px) sees one, two or four of the nine taps, on g at (y, x) to (y + 1, x + 1): the four parity
// classes are four convolutions of g itself, 9 tap products for 4 pixels instead of 36 (on mma.sync the
// virtual upsampling took 675 us of a 2.9 ms step).  A tile is 8 x 16 pixels of g, its window two
// copies (columns x and x + 1) of 17 rows; each class has an accumulator, and its outputs leave through
// a tensor map with twice the pixel strides.  A class's taps come in their order; the skipped ones
// added zeros: the same bits.
// =============================================================================================
struct UpArgs {
  const bf16* mask;       // [B][2 Hg][2 Wg][64]
  int32_t* status;
  int Hg, Wg;
  int tiles_x, tiles_y, n_tiles;
  unsigned long long timeout_ns;
  int stall_tile;
};
struct UpMaps {
  CUtensorMap g, w, out[4];
};
constexpr int kUpCopy = (kHaloH + 1) * kHaloW * 128;          // 17 atoms
constexpr int kUpStage = 2 * kUpCopy, kUpStages = 3;
constexpr int kUpWeights = 9 * 64 * 128;
constexpr int kUpTmem = 512;                                  // 2 buffers x 4 classes x 64 columns
constexpr size_t kUpSmem = 1024 + kUpWeights + kUpStages * kUpStage + 8 * kHaloStaging;

__global__ void __launch_bounds__(kHaloThreads, 1) conv_up_kernel(const __grid_constant__ UpMaps maps, const __grid_constant__ UpArgs a) {
  extern __shared__ uint8_t tc_smem_raw[];
  __shared__ uint64_t bars[2 * kUpStages + 6];
  __shared__ uint32_t tmem_base_sh;
  __shared__ int abort_sh;
  uint8_t* base = reinterpret_cast<uint8_t*>(((uintptr_t)tc_smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sA = base;
  uint8_t* sW = base + kUpStages * kUpStage;
  uint8_t* sOut = sW + kUpWeights;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t full0 = smem_u32(&bars[0]), empty0 = smem_u32(&bars[kUpStages]);
  const uint32_t accf0 = smem_u32(&bars[2 * kUpStages]), acce0 = smem_u32(&bars[2 * kUpStages + 2]);
  const uint32_t wfull = smem_u32(&bars[2 * kUpStages + 4]), drain = smem_u32(&bars[2 * kUpStages + 5]);
  volatile int* abort = &abort_sh;
  if (threadIdx.x == 0) {
    abort_sh = 0;
    for (int s = 0; s < kUpStages; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(accf0 + 8 * b, 1);
      mbar_init(acce0 + 8 * b, 4);
    }
    mbar_init(wfull, 1);
    mbar_init(drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_sh)),
                 "r"(kUpTmem)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_sh;
  const int per = a.tiles_x * a.tiles_y;

  if (warp == 0) {
    if (lane == 0) {
      mbar_expect_tx(wfull, kUpWeights);
      for (int tap = 0; tap < 9; ++tap) tma_load_2d(smem_u32(sW + tap * 8192), &maps.w, wfull, 0, tap * 64);
      uint32_t q = 0;
      int issued[kUpStages] = {};
      uint32_t phase[kUpStages] = {};
      bool ok = true;
      for (int t = blockIdx.x; t < a.n_tiles; t += gridDim.x, ++q) {
        const int s = (int)(q % kUpStages);
        const uint32_t round = q / kUpStages;
        if (round > 0 && !mbar_wait(empty0 + 8 * s, (round - 1) & 1, abort, a)) {
          ok = false;
          break;
        }
        issued[s] = 0;
        if (t == a.stall_tile) continue;  // test hook: the consumer's wait for this tile runs out
        const int b = t / per, r = t - b * per, y0 = r / a.tiles_x * kHaloH, x0 = r % a.tiles_x * kHaloW;
        mbar_expect_tx(full0 + 8 * s, kUpStage);
        for (int dx = 0; dx < 2; ++dx)
          tma_load_4d(smem_u32(sA + s * kUpStage + dx * kUpCopy), &maps.g, full0 + 8 * s, 0, x0 + dx, y0, b);
        issued[s] = 1;
        phase[s] = round & 1;
      }
      if (!ok || *abort) {
        const unsigned long long t0 = global_ns();
        while (!mbar_test(wfull, 0) && global_ns() - t0 < a.timeout_ns) {
        }
        for (int s = 0; s < kUpStages; ++s) {
          if (!issued[s]) continue;
          const unsigned long long t1 = global_ns();
          while (!mbar_test(full0 + 8 * s, phase[s]) && global_ns() - t1 < a.timeout_ns) {
          }
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      uint32_t q = 0;
      const bool ok = mbar_wait(wfull, 0, abort, a);
      for (int t = blockIdx.x; ok && t < a.n_tiles; t += gridDim.x, ++q) {
        const int buf = (int)(q & 1), s = (int)(q % kUpStages);
        const uint32_t use = q >> 1;
        if (use > 0 && !mbar_wait(acce0 + 8 * buf, (use - 1) & 1, abort, a)) break;
        if (!mbar_wait(full0 + 8 * s, (q / kUpStages) & 1, abort, a)) break;
        tc_fence_after();
        const uint64_t ad = operand_desc<64>(smem_u32(sA + s * kUpStage)), bd = operand_desc<64>(smem_u32(sW));
#pragma unroll
        for (int cls = 0; cls < 4; ++cls) {
          const int py = cls >> 1, px = cls & 1;
          const uint32_t d = tmem + (uint32_t)(buf * 256 + cls * 64);
          bool first = true;
#pragma unroll
          for (int tap = 0; tap < 9; ++tap) {
            const int ky = tap / 3, kx = tap % 3;
            // the tap reads the zero-inserted grid at 2 y + py + ky - 1: g's row y + (py + ky - 1) / 2
            if (((py + ky - 1) & 1) || ((px + kx - 1) & 1)) continue;
            const int dy = (py + ky - 1) >> 1, dx = (px + kx - 1) >> 1;
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              umma_bf16<64>(d, ad + ((dx * kUpCopy + dy * 1024 + 32 * kk) >> 4), bd + ((tap * 8192 + 32 * kk) >> 4),
                            (!first || kk > 0) ? 1u : 0u);
            first = false;
          }
        }
        umma_commit(empty0 + 8 * s);
        umma_commit(accf0 + 8 * buf);
      }
      if (*abort) {
        umma_commit(drain);
        const unsigned long long t0 = global_ns();
        while (!mbar_test(drain, 0) && global_ns() - t0 < a.timeout_ns) {
        }
      }
    }
  } else {
    const int quarter = warp & 3, buf = (warp - 2) >> 2;
    uint32_t q = buf;
    for (int t = blockIdx.x + buf * gridDim.x; t < a.n_tiles; t += 2 * gridDim.x, q += 2) {
      if (!mbar_wait_warp(accf0 + 8 * buf, (q >> 1) & 1, abort, a, lane)) break;
      tc_fence_after();
      const int b = t / per, r = t - b * per, y0 = r / a.tiles_x * kHaloH + quarter * 4, x0 = r % a.tiles_x * kHaloW;
      const int y = y0 + (lane >> 3), x = x0 + (lane & 7);
      const bool inside = y < a.Hg && x < a.Wg;
      for (int cls = 0; cls < 4; ++cls) {
        float v0[32], v1[32];
        const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(buf * 256 + cls * 64);
        tmem_ld32(taddr, v0);
        tmem_ld32(taddr + 32, v1);
        tc_fence_before();
        __syncwarp();
        if (cls == 3 && lane == 0) mbar_arrive(acce0 + 8 * buf);
        uint8_t* stage = sOut + (buf * 4 + quarter) * kHaloStaging;
        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        __syncwarp();
        const size_t pix = ((size_t)b * 2 * a.Hg + 2 * y + (cls >> 1)) * (2 * (size_t)a.Wg) + 2 * x + (cls & 1);
        const bf16* mask = inside ? a.mask + pix * 64 : nullptr;
        stage_half(stage, lane, 0, v0, nullptr, 0, mask);
        stage_half(stage, lane, 1, v1, nullptr, 0, mask);
        stage_done();
        if (lane == 0) {
          if (y0 < a.Hg) tma_store_4d(&maps.out[cls], smem_u32(stage), 0, x0, y0, b);
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
      }
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kUpTmem) : "memory");
  }
}

// ---- host ---------------------------------------------------------------------------------------
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static std::once_flag once;
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

int conv_tc_tile_width(int Wo) {
  // output tiles of Wt x (128 / Wt) pixels: the widest of 128, 64, 32, 16 that wastes no column,
  // else 16
  for (int wt : {128, 64, 32, 16})
    if (Wo % wt == 0) return wt;
  return 16;
}

template <int CIN>
cudaError_t launch_conv_tc_t(const bf16* in, int B, int Hi, int Wi, const bf16* w, const float* bias, const bf16* mask,
                             bf16* out, int Ho, int Wo, int stride, int dil, int relu, int32_t* status, int n_sms,
                             cudaStream_t s, unsigned long long timeout_ns, int stall_tile) {
  using S = TcShape<CIN>;
  if (B <= 0 || Ho <= 0 || Wo <= 0) return cudaSuccess;
  if ((stride != 1 && stride != 2) || dil < 1 || dil > 8 || !status) return cudaErrorInvalidValue;
  if (((uintptr_t)in & 15) || ((uintptr_t)out & 15) || ((uintptr_t)w & 15)) return cudaErrorMisalignedAddress;
  PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
  if (!enc) return cudaErrorNotSupported;
  if (mask && ((uintptr_t)mask & 15)) return cudaErrorMisalignedAddress;
  TcArgs a{};
  a.bias = bias;
  a.mask = mask;
  a.w = w;
  a.out = out;
  a.status = status;
  a.B = B;
  a.Ho = Ho;
  a.Wo = Wo;
  a.stride = stride;
  a.dil = dil;
  a.relu = relu;
  a.Wt = conv_tc_tile_width(Wo);
  a.Ht = kTcM / a.Wt;
  a.tiles_x = (Wo + a.Wt - 1) / a.Wt;
  a.tiles_y = (Ho + a.Ht - 1) / a.Ht;
  a.n_tiles = B * a.tiles_x * a.tiles_y;
  a.timeout_ns = timeout_ns;
  a.stall_tile = stall_tile;
  // 4-D map: (channel, x, y, image), box CIN x Wt*stride x Ht*stride x 1 walked with element strides
  // (1, stride, stride, 1): Wt x Ht pixel rows of CIN x 2 bytes
  CUtensorMap map;
  const cuuint64_t dims[4] = {(cuuint64_t)CIN, (cuuint64_t)Wi, (cuuint64_t)Hi, (cuuint64_t)B};
  const cuuint64_t strides[3] = {(cuuint64_t)CIN * 2, (cuuint64_t)Wi * CIN * 2, (cuuint64_t)Hi * Wi * CIN * 2};
  const cuuint32_t box[4] = {(cuuint32_t)CIN, (cuuint32_t)(a.Wt * stride), (cuuint32_t)(a.Ht * stride), 1};
  const cuuint32_t estr[4] = {1, (cuuint32_t)stride, (cuuint32_t)stride, 1};
  if (box[1] > 256 || box[2] > 256) return cudaErrorInvalidValue;
  const CUresult r = enc(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<bf16*>(in), dims, strides, box, estr,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CIN == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_32B,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
  static PerDevice configured;
  int dummy = 0;
  cudaError_t e = per_device(configured, &dummy, [](int, int* v) {
    *v = 1;
    return cudaFuncSetAttribute(conv_tc_kernel<CIN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::kSmem);
  });
  if (e != cudaSuccess) return e;
  const int grid = std::min(a.n_tiles, n_sms);
  conv_tc_kernel<CIN><<<grid, kTcThreads, S::kSmem, s>>>(map, a);
  return cudaGetLastError();
}

// A tiled map over bf16 values: dims (innermost first) d[rank], box b[rank], unit element strides.
CUresult encode_bf16(PFN_cuTensorMapEncodeTiled_v12000 enc, CUtensorMap* map, const void* p, int rank, const cuuint64_t* d,
                     const cuuint32_t* b) {
  cuuint64_t strides[4];
  cuuint64_t pitch = 2;
  for (int k = 0; k + 1 < rank; ++k) strides[k] = pitch *= d[k];
  const cuuint32_t ones[5] = {1, 1, 1, 1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void*>(p), d, strides, b, ones,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
}

template <int N>
cudaError_t launch_conv_halo_t(const bf16* in, int B, int H, int W, const bf16* w, const float* bias, const bf16* mask,
                               bf16* out, float* out_f32, int relu, int32_t* status, int n_sms, cudaStream_t s,
                               unsigned long long timeout_ns, int stall_tile) {
  using S = HaloShape<N>;
  PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
  if (!enc) return cudaErrorNotSupported;
  if (((uintptr_t)in & 15) || ((uintptr_t)w & 15) || ((uintptr_t)out & 15) || ((uintptr_t)out_f32 & 15) ||
      ((uintptr_t)mask & 15))
    return cudaErrorMisalignedAddress;
  HaloArgs a{};
  a.bias = bias;
  a.mask = mask;
  a.out_f32 = out_f32;
  a.status = status;
  a.Ho = H;
  a.Wo = W;
  a.relu = relu;
  a.tiles_x = (W + kHaloW - 1) / kHaloW;
  a.tiles_y = (H + kHaloH - 1) / kHaloH;
  a.n_tiles = B * a.tiles_x * a.tiles_y;
  a.timeout_ns = timeout_ns;
  a.stall_tile = stall_tile;
  CUtensorMap in_map, w_map, out_map;
  const cuuint64_t dims[4] = {64, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)B};
  const cuuint32_t in_box[4] = {64, kHaloW, kHaloH + 2, 1}, out_box[4] = {64, kHaloW, 4, 1};
  const cuuint32_t rows = N == 64 ? 64 : 8;
  const cuuint64_t w_dims[2] = {64, (cuuint64_t)9 * rows};
  const cuuint32_t w_box[2] = {64, rows};
  if (encode_bf16(enc, &in_map, in, 4, dims, in_box) != CUDA_SUCCESS ||
      encode_bf16(enc, &w_map, w, 2, w_dims, w_box) != CUDA_SUCCESS ||
      encode_bf16(enc, &out_map, N == 64 ? out : in, 4, dims, out_box) != CUDA_SUCCESS)  // (the head stores no BF16)
    return cudaErrorInvalidValue;
  static PerDevice configured;
  int dummy = 0;
  const cudaError_t e = per_device(configured, &dummy, [](int, int* v) {
    *v = 1;
    return cudaFuncSetAttribute(conv_halo_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::kSmem);
  });
  if (e != cudaSuccess) return e;
  conv_halo_kernel<N><<<std::min(a.n_tiles, n_sms), kHaloThreads, S::kSmem, s>>>(in_map, w_map, out_map, a);
  return cudaGetLastError();
}

template <class Kernel>
cudaError_t allow_smem(PerDevice& configured, Kernel k, size_t bytes) {
  int dummy = 0;
  return per_device(configured, &dummy, [k, bytes](int, int* v) {
    *v = 1;
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  });
}

}  // namespace

cudaError_t launch_conv_tc(int cin, const bf16* in, int B, int Hi, int Wi, const bf16* w, const float* bias,
                           const bf16* mask, bf16* out, int Ho, int Wo, int stride, int dil, int relu, int32_t* status,
                           int n_sms, cudaStream_t s, unsigned long long timeout_ns, int stall_tile) {
  if (cin == 64 && stride == 1 && dil == 1 && B > 0 && Ho == Hi && Wo == Wi && status)
    return launch_conv_halo_t<64>(in, B, Hi, Wi, w, bias, mask, out, nullptr, relu, status, n_sms, s, timeout_ns, stall_tile);
  if (cin == 64)
    return launch_conv_tc_t<64>(in, B, Hi, Wi, w, bias, mask, out, Ho, Wo, stride, dil, relu, status, n_sms, s,
                                timeout_ns, stall_tile);
  if (cin == 16)
    return launch_conv_tc_t<16>(in, B, Hi, Wi, w, bias, mask, out, Ho, Wo, stride, dil, relu, status, n_sms, s,
                                timeout_ns, stall_tile);
  return cudaErrorInvalidValue;
}

cudaError_t launch_conv_first(const uint16_t* depth, const uint32_t* rgba, int B, int H, int W, const bf16* w,
                              const float* bias, bf16* out, int Ho, int Wo, int32_t* status, int n_sms, cudaStream_t s,
                              unsigned long long timeout_ns, int stall_tile) {
  if (B <= 0 || Ho <= 0 || Wo <= 0) return cudaSuccess;
  PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
  if (!enc) return cudaErrorNotSupported;
  if (((uintptr_t)w & 15) || ((uintptr_t)out & 15)) return cudaErrorMisalignedAddress;
  FirstArgs a{};
  a.depth = depth;
  a.rgba = rgba;
  a.bias = bias;
  a.w = w;
  a.status = status;
  a.H = H;
  a.W = W;
  a.Ho = Ho;
  a.Wo = Wo;
  a.tiles_x = (Wo + kFirstW - 1) / kFirstW;
  a.tiles_y = (Ho + kFirstH - 1) / kFirstH;
  a.n_tiles = B * a.tiles_x * a.tiles_y;
  a.timeout_ns = timeout_ns;
  a.stall_tile = stall_tile;
  CUtensorMap out_map;
  const cuuint64_t dims[4] = {64, (cuuint64_t)Wo, (cuuint64_t)Ho, (cuuint64_t)B};
  const cuuint32_t box[4] = {64, kFirstW, 2, 1};
  if (encode_bf16(enc, &out_map, out, 4, dims, box) != CUDA_SUCCESS) return cudaErrorInvalidValue;
  static PerDevice configured;
  const cudaError_t e = allow_smem(configured, conv_first_kernel, kFirstSmem);
  if (e != cudaSuccess) return e;
  conv_first_kernel<<<std::min(a.n_tiles, n_sms), kFirstThreads, kFirstSmem, s>>>(out_map, a);
  return cudaGetLastError();
}

cudaError_t launch_conv_up(const bf16* g, int B, int Hg, int Wg, const bf16* w, const bf16* mask, bf16* out, int32_t* status,
                           int n_sms, cudaStream_t s, unsigned long long timeout_ns, int stall_tile) {
  if (B <= 0 || Hg <= 0 || Wg <= 0) return cudaSuccess;
  PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
  if (!enc) return cudaErrorNotSupported;
  if (((uintptr_t)g & 15) || ((uintptr_t)w & 15) || ((uintptr_t)mask & 15) || ((uintptr_t)out & 15))
    return cudaErrorMisalignedAddress;
  UpArgs a{};
  a.mask = mask;
  a.status = status;
  a.Hg = Hg;
  a.Wg = Wg;
  a.tiles_x = (Wg + kHaloW - 1) / kHaloW;
  a.tiles_y = (Hg + kHaloH - 1) / kHaloH;
  a.n_tiles = B * a.tiles_x * a.tiles_y;
  a.timeout_ns = timeout_ns;
  a.stall_tile = stall_tile;
  UpMaps m;
  const cuuint64_t dims[4] = {64, (cuuint64_t)Wg, (cuuint64_t)Hg, (cuuint64_t)B};
  const cuuint32_t g_box[4] = {64, kHaloW, kHaloH + 1, 1}, out_box[4] = {64, kHaloW, 4, 1}, ones[4] = {1, 1, 1, 1};
  const cuuint64_t w_dims[2] = {64, 9 * 64};
  const cuuint32_t w_box[2] = {64, 64};
  CUresult r = encode_bf16(enc, &m.g, g, 4, dims, g_box);
  if (r == CUDA_SUCCESS) r = encode_bf16(enc, &m.w, w, 2, w_dims, w_box);
  // class (py, px) of the output: pixels 2 apart in both directions from (py, px)
  const cuuint64_t row = (cuuint64_t)2 * Wg * 128, strides[3] = {256, 2 * row, (cuuint64_t)2 * Hg * row};
  for (int c = 0; c < 4 && r == CUDA_SUCCESS; ++c)
    r = enc(&m.out[c], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, out + ((size_t)(c >> 1) * 2 * Wg + (c & 1)) * 64, dims, strides,
            out_box, ones, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
  static PerDevice configured;
  const cudaError_t e = allow_smem(configured, conv_up_kernel, kUpSmem);
  if (e != cudaSuccess) return e;
  conv_up_kernel<<<std::min(a.n_tiles, n_sms), kHaloThreads, kUpSmem, s>>>(m, a);
  return cudaGetLastError();
}

cudaError_t launch_conv_head(const bf16* in, int B, int H, int W, const bf16* w, const float* bias, float* out,
                             int32_t* status, int n_sms, cudaStream_t s, unsigned long long timeout_ns, int stall_tile) {
  if (B <= 0 || H <= 0 || W <= 0) return cudaSuccess;
  return launch_conv_halo_t<16>(in, B, H, W, w, bias, nullptr, nullptr, out, 0, status, n_sms, s, timeout_ns, stall_tile);
}

}  // namespace relo
