// relo_internal.cuh -- device data layouts and helpers shared by the library's translation units.
//
// Everything here belongs to the CUDA path; nothing is shared with the CPU oracle.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "../../include/relo.h"

namespace relo {

// ---------------------------------------------------------------------------------------------
// A launch parameter that depends only on the device (its SM count, a kernel's resident CTAs per
// SM): computed once per device ordinal, with that device current, and shared by every host
// thread.  The lock makes a value and its "ready" mark appear together, so no thread launches
// with a half-published pair.
// ---------------------------------------------------------------------------------------------
struct PerDevice {
  static constexpr int kMaxDevices = 64;
  std::mutex m;
  int value[kMaxDevices] = {};
  bool ready[kMaxDevices] = {};
};

template <class F>
cudaError_t per_device(PerDevice& c, int* out, F&& compute) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= PerDevice::kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(c.m);
  if (!c.ready[dev]) {
    int v = 0;
    e = compute(dev, &v);
    if (e != cudaSuccess) return e;
    c.value[dev] = v;
    c.ready[dev] = true;
  }
  *out = c.value[dev];
  return cudaSuccess;
}

// SMs of the current device.
inline cudaError_t device_sms(int* out) {
  static PerDevice cache;
  return per_device(cache, out, [](int dev, int* v) {
    return cudaDeviceGetAttribute(v, cudaDevAttrMultiProcessorCount, dev);
  });
}

constexpr int kBlockSide = 8;
constexpr int kVoxelsPerBlock = 512;
constexpr int kMaxTrees = 16;
constexpr int kModeFloats = 12;
constexpr float kLogEps = 69.07755278982137f;  // -log(1e-30): energy of a pixel no mode explains
constexpr int kMaxMarchSamples = 100000;

// ---------------------------------------------------------------------------------------------
// Spatial hash of a voxel scene.  Entry = 16 bytes {int16 x, y, z, pad; int32 block; int32 next},
// loaded as one int4.  Bucket h holds the first block hashing to h; later ones are chained
// through the excess list (next = index into it, -1 ends the chain).
// ---------------------------------------------------------------------------------------------
struct SceneView {
  const int4* buckets;
  const int4* excess;
  const float* tsdf;      // [n_blocks][512]
  const uint32_t* rgba;   // [n_blocks][512] packed r | g << 8 | b << 16 | a << 24
  uint32_t mask;          // n_buckets - 1
  int32_t n_blocks;
  int32_t max_chain;      // longest chain at build time (bounds the walk)
  float voxel, inv_voxel, mu, block_size, inv_block;
  // Dense grid over the blocks' bounding box (null when the box is too large): per block
  // coordinate the block index, or -D for an unallocated block whose nearest allocated block is
  // D >= 1 blocks away in the Chebyshev metric (every block within D - 1 of it is unallocated).
  const int32_t* grid;
  int32_t ox, oy, oz;     // grid origin (block coordinates)
  int32_t gx, gy, gz;     // grid extent in blocks (multiples of 8)
  // Apron copy of the tsdf (null when not built or not in use): per block a 9 x 9 x 9 array
  // (x + 9 y + 81 z, padded to kApronStride floats) whose last plane along each axis repeats the
  // first voxels of the neighbouring block (+1 where that block is unallocated), so the eight
  // corners of every trilinear sample lie in the block holding the sample.
  const float* tsdf9;
  // Scenes that grow by fusion (null otherwise): one bit per block, 64-bit words of 4 x 4 x 4 blocks
  // indexed by the low kCellBits bits of the word's coordinates (cell_index), so that words 64 apart
  // share one.  A clear bit says that the block is not allocated, without a walk of the hash; a set
  // one, that it may be.
  const unsigned long long* cells;
};
constexpr int kApronStride = 736;  // 729 voxels padded to a multiple of 32 floats (128 bytes)
constexpr int kCellBits = 6;       // 64^3 words of 64 blocks, 2 MB: 10 m without sharing at 5 mm voxels

__device__ __forceinline__ int cell_index(int bx, int by, int bz) {
  constexpr int m = (1 << kCellBits) - 1;
  return ((bx >> 2) & m) | ((by >> 2) & m) << kCellBits | ((bz >> 2) & m) << (2 * kCellBits);
}
__device__ __forceinline__ int cell_bit(int bx, int by, int bz) { return (bx & 3) | (by & 3) << 2 | (bz & 3) << 4; }

// How a raycast launch reads its scenes: every scene through its apron copy, every scene a growing
// one through its cell words and hash, or each by what it has (grid or hash, the blocks' own tsdf).
enum SceneMode { kSceneAny = 0, kSceneApron = 1, kSceneCells = 2 };
__host__ __device__ inline int scene_mode(const SceneView& s) {
  return s.tsdf9 ? kSceneApron : (s.cells && !s.grid) ? kSceneCells : kSceneAny;
}

// Block index, or -D (see SceneView::grid), through the dense grid (caller checks s.grid).
// Outside the box D is the Chebyshev distance to the box, a lower bound of the distance to any
// allocated block.
__device__ __forceinline__ int grid_block(const SceneView& s, int x, int y, int z) {
  const int a = x - s.ox, b = y - s.oy, c = z - s.oz;
  if ((unsigned)a >= (unsigned)s.gx || (unsigned)b >= (unsigned)s.gy || (unsigned)c >= (unsigned)s.gz) {
    const int da = a < 0 ? -a : a - (s.gx - 1);
    const int db = b < 0 ? -b : b - (s.gy - 1);
    const int dc = c < 0 ? -c : c - (s.gz - 1);
    return -max(da, max(db, dc));
  }
  return __ldg(&s.grid[((size_t)c * s.gy + b) * s.gx + a]);
}

__host__ __device__ inline uint32_t block_hash(int x, int y, int z) {
  return ((uint32_t)x * 73856093u) ^ ((uint32_t)y * 19349669u) ^ ((uint32_t)z * 83492791u);
}

__host__ __device__ inline int4 pack_entry(int x, int y, int z, int block, int next) {
  int4 e;
  e.x = (int)((uint32_t)(uint16_t)(int16_t)x | ((uint32_t)(uint16_t)(int16_t)y << 16));
  e.y = (int)((uint32_t)(uint16_t)(int16_t)z);
  e.z = block;
  e.w = next;
  return e;
}

// Block index of block coordinate (x, y, z), -1 if absent; *err set if the chain walk exceeds
// its bound (a corrupted table).
__device__ __forceinline__ int lookup_block(const SceneView& s, int x, int y, int z, int* err) {
  if (x < -32768 || x > 32767 || y < -32768 || y > 32767 || z < -32768 || z > 32767) return -1;
  const int k0 = (int)((uint32_t)(uint16_t)(int16_t)x | ((uint32_t)(uint16_t)(int16_t)y << 16));
  const int k1 = (int)((uint32_t)(uint16_t)(int16_t)z);
  int4 e = __ldg(&s.buckets[block_hash(x, y, z) & s.mask]);
  for (int steps = 0; steps <= s.max_chain; ++steps) {
    if (e.z >= 0 && e.x == k0 && (e.y & 0xFFFF) == k1) return e.z;
    if (e.w < 0) return -1;
    e = __ldg(&s.excess[e.w]);
  }
  *err = 1;
  return -1;
}

// ---------------------------------------------------------------------------------------------
// Forest
// ---------------------------------------------------------------------------------------------
struct ForestView {
  const int4* nodes;        // [2^D][T] split nodes, 16 bytes each (numbered as forest.cu's descent takes them)
  const float* modes;       // [T][2^D][M][12]
  const uint8_t* n_modes;   // [T][2^D]
  const float4* top;        // [T][2^D]: mode 0 mean xyz, w = number of modes
  int32_t T, D, M;
  int32_t probe_reach;      // 1 + the largest |offset| of any node (0: not known, every probe clamped)
  int32_t offset_shift;     // the device nodes hold offset << offset_shift (7 when every |offset| <= 255, else 0)
};

// ---------------------------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC 2011): 10 rounds, multipliers 0xD2511F53 and
// 0xCD9E8D57, Weyl key increments 0x9E3779B9 and 0xBB67AE85.
// ---------------------------------------------------------------------------------------------
__host__ __device__ inline uint32_t mulhi32(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
  return __umulhi(a, b);
#else
  return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}

__host__ __device__ inline uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int i = 0; i < 10; ++i) {
    const uint32_t hi0 = mulhi32(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
    const uint32_t hi1 = mulhi32(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
    c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return c;
}

__host__ __device__ inline uint32_t uniform_below(uint32_t x, uint32_t n) { return mulhi32(x, n); }

// ---------------------------------------------------------------------------------------------
// Poses: 12 doubles, row-major [R | t], camera -> scene.
// ---------------------------------------------------------------------------------------------
struct PoseF {
  float r[9], t[3];
};

__device__ __forceinline__ PoseF pose_to_float(const double* p) {
  PoseF q;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
#pragma unroll
    for (int j = 0; j < 3; ++j) q.r[3 * i + j] = (float)p[4 * i + j];
    q.t[i] = (float)p[4 * i + 3];
  }
  return q;
}

__device__ __forceinline__ float3 apply(const PoseF& P, float3 c) {
  return make_float3(fmaf(P.r[0], c.x, fmaf(P.r[1], c.y, fmaf(P.r[2], c.z, P.t[0]))),
                     fmaf(P.r[3], c.x, fmaf(P.r[4], c.y, fmaf(P.r[5], c.z, P.t[1]))),
                     fmaf(P.r[6], c.x, fmaf(P.r[7], c.y, fmaf(P.r[8], c.z, P.t[2]))));
}

// Pose [R | t] (12 doubles) of the rotation (w, x, y, z), normalised here, that maps centroid cbar to
// wbar.  Every operation states its rounding, here and in the solves, so that both forms of a solve
// (horn_pose by a thread, horn_pose_group by 16 lanes) give the same bits.
__device__ __forceinline__ void quaternion_pose(double w, double x, double y, double z, const double cbar[3],
                                                const double wbar[3], double* out) {
  const double n = __dsqrt_rn(__fma_rn(z, z, __fma_rn(y, y, __fma_rn(x, x, __dmul_rn(w, w)))));
  w = __ddiv_rn(w, n);
  x = __ddiv_rn(x, n);
  y = __ddiv_rn(y, n);
  z = __ddiv_rn(z, n);
  const double yy = __dmul_rn(y, y), zz = __dmul_rn(z, z);
  const double R[9] = {__dsub_rn(1.0, 2 * __dadd_rn(yy, zz)),         2 * __fma_rn(x, y, -__dmul_rn(w, z)),
                       2 * __fma_rn(x, z, __dmul_rn(w, y)),           2 * __fma_rn(x, y, __dmul_rn(w, z)),
                       __dsub_rn(1.0, 2 * __fma_rn(x, x, zz)),        2 * __fma_rn(y, z, -__dmul_rn(w, x)),
                       2 * __fma_rn(x, z, -__dmul_rn(w, y)),          2 * __fma_rn(y, z, __dmul_rn(w, x)),
                       __dsub_rn(1.0, 2 * __fma_rn(x, x, yy))};
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    out[4 * i + 0] = R[3 * i + 0];
    out[4 * i + 1] = R[3 * i + 1];
    out[4 * i + 2] = R[3 * i + 2];
    out[4 * i + 3] = __dsub_rn(wbar[i], __fma_rn(R[3 * i + 2], cbar[2], __fma_rn(R[3 * i], cbar[0], __dmul_rn(R[3 * i + 1], cbar[1]))));
  }
}

// Rigid transform from centroids and cross-covariance by Horn's closed form (1987): the rotation is
// the unit quaternion of the largest eigenvalue of the symmetric 4x4 matrix N(S), S = sum of
// (c - cbar)(w - wbar)^T.  horn_refined solves the eigenproblem where the largest eigenvalue stands
// clear of the others, horn_jacobi, by cyclic Jacobi rotations in FP64 (stable for near-degenerate point
// sets), where it does not.

// The largest eigenvalue's eigenvector (near unit length) by FP32 Jacobi rotations and refinement in
// FP64: with approximate eigenvectors v_k and eigenvalues l_k, the residual r = N q - rho q in FP64
// gives the correction sum of v_k (v_k . r) / (l_max - l_k), which FP32 suffices for (iterative
// refinement; the first-order perturbation of an eigenvector).  Each turn leaves about kappa = 4e-7 / gap
// of the error, so two are usual, and what remains is the residual's own rounding: that of FP64
// rotations.  About 100 FP64 operations where the rotations take 700 a sweep and five sweeps, on a pipe
// that takes 16 cycles or more a warp.  False (the caller takes horn_jacobi): a relative gap under 5e-4
// (beyond, the residual's rounding would pass for a step; 0.4 to 1 % of a room's kept triples),
// no convergence, or entries FP32 cannot hold (zeros, infinities, NaN).
__device__ __forceinline__ bool horn_refined(const double S_in[9], double (&q)[4]) {
  int top = 0;
#pragma unroll
  for (int k = 0; k < 9; ++k) top = max(top, __double2hiint(S_in[k]) & 0x7FFFFFFF);
  const int e = top >> 20;  // biased exponent of the largest entry
  if (e < 64 || e > 1980) return false;
  const double scale = __hiloint2double((2046 - e) << 20, 0);  // 2^(1023 - e): exact
  double S[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) S[k] = __dmul_rn(S_in[k], scale);
  double N[4][4];
  N[0][0] = __dadd_rn(__dadd_rn(S[0], S[4]), S[8]);
  N[1][1] = __dsub_rn(__dsub_rn(S[0], S[4]), S[8]);
  N[2][2] = __dsub_rn(__dsub_rn(S[4], S[0]), S[8]);
  N[3][3] = __dsub_rn(__dsub_rn(S[8], S[0]), S[4]);
  N[0][1] = N[1][0] = __dsub_rn(S[5], S[7]);
  N[0][2] = N[2][0] = __dsub_rn(S[6], S[2]);
  N[0][3] = N[3][0] = __dsub_rn(S[1], S[3]);
  N[1][2] = N[2][1] = __dadd_rn(S[1], S[3]);
  N[1][3] = N[3][1] = __dadd_rn(S[6], S[2]);
  N[2][3] = N[3][2] = __dadd_rn(S[5], S[7]);
  float d[4], o[6], V[4][4];  // diagonal; (0,1) (0,2) (0,3) (1,2) (1,3) (2,3); columns: eigenvectors
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    d[i] = (float)N[i][i];
#pragma unroll
    for (int j = 0; j < 4; ++j) V[i][j] = i == j ? 1.f : 0.f;
  }
  o[0] = (float)N[0][1], o[1] = (float)N[0][2], o[2] = (float)N[0][3];
  o[3] = (float)N[1][2], o[4] = (float)N[1][3], o[5] = (float)N[2][3];
  // (x, y) <- (c x - s y, s x + c y)
  auto rotate = [](float& x, float& y, float c, float s) {
    const float a = __fmaf_rn(c, x, -__fmul_rn(s, y));
    y = __fmaf_rn(s, x, __fmul_rn(c, y));
    x = a;
  };
  auto angle = [](float& dp, float& dq, float& apq, float& c, float& s) {
    c = 1.f, s = 0.f;
    if (fabsf(apq) < 1e-30f) return;
    const float theta = __fdividef(__fsub_rn(dq, dp), __fmul_rn(2.f, apq));
    const float t = __fdividef(theta >= 0.f ? 1.f : -1.f, __fadd_rn(fabsf(theta), __fsqrt_rn(__fmaf_rn(theta, theta, 1.f))));
    c = rsqrtf(__fmaf_rn(t, t, 1.f));
    s = __fmul_rn(t, c);
    dp = __fmaf_rn(-t, apq, dp);
    dq = __fmaf_rn(t, apq, dq);
    apq = 0.f;
  };
  // disjoint pairs (p, q), (r, s) and the entries between them
  auto stage = [&](int p, int q_, int r, int s_, float& apq, float& ars, float& bpr, float& bps, float& bqr, float& bqs) {
    float c1, s1, c2, s2;
    angle(d[p], d[q_], apq, c1, s1);
    angle(d[r], d[s_], ars, c2, s2);
    rotate(bpr, bqr, c1, s1);
    rotate(bps, bqs, c1, s1);
    rotate(bpr, bps, c2, s2);
    rotate(bqr, bqs, c2, s2);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      rotate(V[k][p], V[k][q_], c1, s1);
      rotate(V[k][r], V[k][s_], c2, s2);
    }
  };
  for (int sweep = 0; sweep < 10; ++sweep) {
    float off = 0.f, diag = 0.f;
#pragma unroll
    for (int k = 0; k < 6; ++k) off = __fmaf_rn(o[k], o[k], off);
#pragma unroll
    for (int k = 0; k < 4; ++k) diag = __fmaf_rn(d[k], d[k], diag);
    if (off <= __fmul_rn(1e-13f, diag)) break;
    stage(0, 1, 2, 3, o[0], o[5], o[1], o[2], o[3], o[4]);
    stage(0, 2, 1, 3, o[1], o[4], o[0], o[2], o[3], o[5]);
    stage(0, 3, 1, 2, o[2], o[3], o[0], o[1], o[4], o[5]);
  }
  float best = d[0], size = fabsf(d[0]);
  float b[4] = {V[0][0], V[1][0], V[2][0], V[3][0]};
  int at = 0;
#pragma unroll
  for (int k = 1; k < 4; ++k) {
    size = fmaxf(size, fabsf(d[k]));
    if (d[k] > best) {
      best = d[k];
      at = k;
#pragma unroll
      for (int i = 0; i < 4; ++i) b[i] = V[i][k];
    }
  }
  float gap = INFINITY, inv[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float g = __fsub_rn(best, d[k]);
    if (k != at) gap = fminf(gap, g);
    inv[k] = k != at ? __fdividef(1.f, g) : 0.f;
  }
  if (!(gap > __fmul_rn(5e-4f, size))) return false;
  const float kappa = __fdividef(__fmul_rn(4e-7f, size), gap);
#pragma unroll
  for (int i = 0; i < 4; ++i) q[i] = (double)b[i];
  for (int it = 0; it < 6; ++it) {
    double y[4], nn = 0.0, rho = 0.0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      y[i] = __fma_rn(N[i][3], q[3], __fma_rn(N[i][2], q[2], __fma_rn(N[i][1], q[1], __dmul_rn(N[i][0], q[0]))));
      nn = __fma_rn(q[i], q[i], nn);
      rho = __fma_rn(q[i], y[i], rho);
    }
    const double t = __dsub_rn(2.0, nn);  // rho / nn by two Newton steps: nn is 1 + (an error of q)^2
    rho = __dmul_rn(rho, __dmul_rn(t, __fma_rn(-nn, t, 2.0)));
    float r[4], c[4], s2 = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) r[i] = (float)__fma_rn(-rho, q[i], y[i]);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float dot = __fmaf_rn(V[3][k], r[3], __fmaf_rn(V[2][k], r[2], __fmaf_rn(V[1][k], r[1], __fmul_rn(V[0][k], r[0]))));
      c[k] = __fmul_rn(dot, inv[k]);
      s2 = __fmaf_rn(c[k], c[k], s2);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      q[i] = __dadd_rn(q[i], (double)__fmaf_rn(V[i][3], c[3], __fmaf_rn(V[i][2], c[2], __fmaf_rn(V[i][1], c[1], __fmul_rn(V[i][0], c[0])))));
    const float step = __fsqrt_rn(s2);
    if (__fmul_rn(__fadd_rn(kappa, step), step) <= 1e-16f) return true;
  }
  return false;
}

__device__ inline void horn_jacobi(const double S[9], const double cbar[3], const double wbar[3], double* out) {
  const double Sxx = S[0], Sxy = S[1], Sxz = S[2], Syx = S[3], Syy = S[4], Syz = S[5], Szx = S[6], Szy = S[7],
               Szz = S[8];
  double A[4][4] = {{Sxx + Syy + Szz, Syz - Szy, Szx - Sxz, Sxy - Syx},
                    {Syz - Szy, Sxx - Syy - Szz, Sxy + Syx, Szx + Sxz},
                    {Szx - Sxz, Sxy + Syx, -Sxx + Syy - Szz, Syz + Szy},
                    {Sxy - Syx, Szx + Sxz, Syz + Szy, -Sxx - Syy + Szz}};
  double V[4][4] = {{1, 0, 0, 0}, {0, 1, 0, 0}, {0, 0, 1, 0}, {0, 0, 0, 1}};
  // Cyclic Jacobi in the parallel ordering: each sweep is three stages of two rotations on
  // disjoint index pairs, ((0,1),(2,3)), ((0,2),(1,3)), ((0,3),(1,2)), whose angles are computed
  // independently (two divide / square-root chains in flight instead of one).  Every index is a
  // compile-time constant after unrolling, so A and V stay in registers.
  constexpr int kPairs[3][2][2] = {{{0, 1}, {2, 3}}, {{0, 2}, {1, 3}}, {{0, 3}, {1, 2}}};
  for (int sweep = 0; sweep < 30; ++sweep) {
    double off = 0.0, diag = 0.0;
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      diag = __fma_rn(A[p][p], A[p][p], diag);
#pragma unroll
      for (int q = p + 1; q < 4; ++q) off = __fma_rn(A[p][q], A[p][q], off);
    }
    if (off <= 1e-30 * (diag + 1e-300)) break;
#pragma unroll
    for (int st = 0; st < 3; ++st) {
      double cs[2], sn[2];
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int p = kPairs[st][r][0], q = kPairs[st][r][1];
        const double apq = A[p][q];
        cs[r] = 1.0;
        sn[r] = 0.0;
        if (fabs(apq) >= 1e-300) {
          const double theta = __ddiv_rn(__dsub_rn(A[q][q], A[p][p]), 2.0 * apq);
          const double t = __ddiv_rn(theta >= 0.0 ? 1.0 : -1.0,
                                     __dadd_rn(fabs(theta), __dsqrt_rn(__fma_rn(theta, theta, 1.0))));
          cs[r] = rsqrt(__fma_rn(t, t, 1.0));
          sn[r] = __dmul_rn(t, cs[r]);
        }
      }
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int p = kPairs[st][r][0], q = kPairs[st][r][1];
        const double c = cs[r], s = sn[r];
#pragma unroll
        for (int k = 0; k < 4; ++k) {  // A <- J^T A J
          const double akp = A[k][p], akq = A[k][q];
          A[k][p] = __fma_rn(c, akp, -__dmul_rn(s, akq));
          A[k][q] = __fma_rn(s, akp, __dmul_rn(c, akq));
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const double apk = A[p][k], aqk = A[q][k];
          A[p][k] = __fma_rn(c, apk, -__dmul_rn(s, aqk));
          A[q][k] = __fma_rn(s, apk, __dmul_rn(c, aqk));
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const double vkp = V[k][p], vkq = V[k][q];
          V[k][p] = __fma_rn(c, vkp, -__dmul_rn(s, vkq));
          V[k][q] = __fma_rn(s, vkp, __dmul_rn(c, vkq));
        }
      }
    }
  }
  double best_d = A[0][0], w = V[0][0], x = V[1][0], y = V[2][0], z = V[3][0];
#pragma unroll
  for (int k = 1; k < 4; ++k)
    if (A[k][k] > best_d) {
      best_d = A[k][k];
      w = V[0][k];
      x = V[1][k];
      y = V[2][k];
      z = V[3][k];
    }
  quaternion_pose(w, x, y, z, cbar, wbar, out);
}

// Writes 12 doubles [R | t].
__device__ __forceinline__ void horn_pose(const double S[9], const double cbar[3], const double wbar[3], double* out) {
  double q[4];
  if (horn_refined(S, q)) quaternion_pose(q[0], q[1], q[2], q[3], cbar, wbar, out);
  else horn_jacobi(S, cbar, wbar, out);
}

// Warp-wide sum (all lanes get the result).
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ int warp_sum_i(int v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Round half up of a non-negative float to an integer in [lo, hi].
__device__ __forceinline__ int round_half_up_clamp(float x, int lo, int hi) {
  float r = floorf(x + 0.5f);
  r = fminf(fmaxf(r, (float)lo), (float)hi);
  return (int)r;
}

// ---------------------------------------------------------------------------------------------
// Raycast jobs (query renders, training renders, verification renders)
// ---------------------------------------------------------------------------------------------
struct RayJob {
  SceneView scene;
  float R[9], t[3];            // camera -> scene (ignored when pose_dev is set)
  const double* pose_dev;      // device pose (12 doubles, row-major R | t) overriding R, t
  const int32_t* status_dev;   // when set, the job is skipped unless *status_dev == RELO_OK
  float fx, fy, cx, cy, dmin, dmax;
  int32_t W, H;
  const float* noise;          // nullable
  uint16_t* depth;             // nullable in compare mode
  uint32_t* rgba;              // nullable
  const uint16_t* depth_ref;   // compare mode: reference depth (D_b)
  unsigned long long* counts;  // compare mode: {omega_a, omega_b, omega_ab, sum |D_a - D_b|}
  int32_t* err;                // device error flag (nullable)
  uint16_t* tiled;             // nullable, colour renders: the image as the forest reads it (see ForestJob)
  int32_t tile_begin;          // first 16 x 16 tile of this job in the flattened launch
  int32_t pad;                 // size: a multiple of 16 bytes (staged in shared memory)
};
static_assert(sizeof(RayJob) % 16 == 0, "RayJob is staged in shared memory as 16-byte words");

// ---------------------------------------------------------------------------------------------
// Forest jobs (one image through one forest)
// ---------------------------------------------------------------------------------------------
// Passed to the kernel by value, an array of them for a batch: read at every node visit, a job's fields
// come from the constant bank as operands, not through registers or shared memory.
struct ForestJob {
  const int4* nodes;           // as ForestView
  const uint16_t* depth;
  const uint32_t* rgba;
  const uint16_t* tiled;       // nullable (null for a forest that reads alpha): the same image in 8 x 8 tiles,
                               // row-major, each [depth, r, g, b][8][8] u16
  uint16_t* leaves;            // [T][H][W]
  const int32_t* skip;         // when set and non-zero the job does nothing (fallback not needed)
  int32_t W, H;
  int32_t T, D;
  int32_t probe_reach, offset_shift;
  int32_t tile_begin;          // first 32 x 8 pixel tile of this job in the flattened launch
  int32_t pad;
};
constexpr int kMaxForestJobs = 256;  // per launch (kernel parameters: 80 bytes a job, 20 KB)
inline ForestJob make_forest_job(const ForestView& f, const uint16_t* depth, const uint32_t* rgba, uint16_t* leaves, int W,
                                 int H) {
  ForestJob j{};
  j.nodes = f.nodes;
  j.depth = depth;
  j.rgba = rgba;
  j.leaves = leaves;
  j.W = W;
  j.H = H;
  j.T = f.T;
  j.D = f.D;
  j.probe_reach = f.probe_reach;
  j.offset_shift = f.offset_shift;
  return j;
}

// ---------------------------------------------------------------------------------------------
// RANSAC jobs (one query view, one forest) and their workspace
// ---------------------------------------------------------------------------------------------
struct RansacJob {
  ForestView forest;
  const uint16_t* depth;
  const uint16_t* leaves;      // [T][H][W]
  int32_t W, H;
  double fx, fy, cx, cy;       // FP64 intrinsics: exact re-checks match the oracle bit for bit
  int32_t K, B, max_tries, n_rounds;
  double rigidity, min_area, inlier_dist;
  uint32_t key0, key1;
  // workspace
  uint4* table;                // [W*H][nv] valid pixels in raster order, packed u16 {u, v, depth, leaf[T]}
  int32_t nv;                  // uint4 words per table entry: ceil((3 + T) / 8)
  int32_t pad1;
  int32_t* chunk_count;        // [n_chunks]
  int32_t* n_valid;            // [1]
  double* poses;               // [K][12]
  int32_t* hyp_ok;             // [K]
  int32_t* tries;              // [K]
  double* energy;              // [K]
  int32_t* alive_a;            // [K]
  int32_t* alive_b;            // [K]
  int32_t* drawn;              // [n_rounds * B] positions in the valid-pixel table
  int32_t* inliers;            // [K]
  float2* refit;               // [K][refit_parts][16] per-survivor inlier sums as compensated (high,
                               // low) FP32 pairs, one block per part of kRefinePixels drawn pixels
                               // (summed in order by the FP64 re-fit)
  float* refit_ref;            // [K][8] reference correspondence of those sums: c_ref (3), w_ref (3)
  int4* pix;                   // [n_rounds * B][hs] drawn pixels: camera point (FP32 bits), then
                               // (first mode, mode count) of the pixel's leaf in each tree, two per word
  int32_t hs;                  // int4 words per drawn-pixel record: 1 + ceil(T / 2)
  int32_t refit_parts;         // blocks per hypothesis in refit: ceil(n_rounds * B / kRefinePixels)
  int32_t* err;                // [1]
  const int32_t* upstream;     // nullable: status of the stage that made this job's input (the
                               // learned path's network); when nonzero it becomes the result's status
  relo_pose_result* result;    // device
  int32_t chunk_begin;         // flattened compaction chunks
  int32_t hyp_begin;           // flattened hypotheses
  int32_t has_pose_b;          // finalise also writes a_T_b = P_a P_b^-1
  int32_t vW, vH;              // size of the view the pose is verified on (the full image)
  int32_t pad2;
  double pose_b[16];           // camera -> scene b pose of the query
  const int32_t* skip;         // when set and non-zero every stage skips the job (fallback not needed)
};

__device__ __forceinline__ bool job_skipped(const int32_t* skip) { return skip != nullptr && *skip != 0; }

constexpr int kCompactChunk = 4096;
constexpr int kRefinePixels = 64;  // drawn pixels per part of the re-fit sums

// Workspace carving helper (256-byte aligned sub-buffers).
struct Carver {
  char* base;
  size_t off;
  template <class T>
  T* take(size_t count) {
    off = (off + 255) & ~(size_t)255;
    T* p = base ? reinterpret_cast<T*>(base + off) : nullptr;
    off += count * sizeof(T);
    return p;
  }
};

// ---------------------------------------------------------------------------------------------
// Launchers (defined in the .cu files)
// ---------------------------------------------------------------------------------------------
// Launch schedule of a batch's kernels (relo_schedule): work-to-thread mappings and grid sizes
// only, so every schedule computes the same results.
struct Schedule {
  int ray_warp_log2w = 3;    // raycast: each warp covers a (1 << w) x (32 >> w) footprint of its 16 x 16 tile
  int forest_threads = 256;  // forest: CTA size (128 or 256)
  int forest_tiles = 0;      // forest: each warp takes 8 x 4 pixels (0) or a row of 32 (1) of a 32 x 8 tile
  int forest_smem_levels = 0;  // forest: top levels of the trees each CTA copies to shared memory (0: none)
  int search_ctas_per_sm = 0;  // hypothesis search: persistent CTAs per SM (0: occupancy maximum)
  int refit_per = 0;         // re-fit: survivors per one-warp CTA (0: spread over twice the SM count)
  int persistent = 0;        // RANSAC of a batch: 0 = one launch per stage, 1 = one persistent launch
};
constexpr int kMaxSmemLevels = 10;
// 32 x 8 pixel tiles of a W x H image.
inline int forest_job_tiles(int W, int H) { return ((W + 31) / 32) * ((H + 7) / 8); }
// u16 values of a W x H image in 8 x 8 tiles (ForestJob::tiled).
inline size_t tiled_values(int W, int H) { return (size_t)((W + 7) / 8) * ((H + 7) / 8) * 256; }

// jobs_dev == nullptr: the single job is passed by value.  mode: the scene_mode that all scenes of
// jobs_dev share, or kSceneAny (a single job's own scene decides for itself).  tiled: jobs have tiled
// images to write (RayJob::tiled), which the launch ignores otherwise.
cudaError_t launch_raycast(const RayJob* jobs_dev, int n_jobs, const RayJob* single, int total_tiles,
                           bool with_colour, bool compare, cudaStream_t s, const Schedule& sched = Schedule(),
                           int mode = kSceneAny, bool tiled = false);
// n jobs (host array, tile_begin ascending from 0), forest_launches(n) launches.
inline int forest_launches(int n) { return (n + kMaxForestJobs - 1) / kMaxForestJobs; }
cudaError_t launch_forest(const ForestJob* jobs, int n, cudaStream_t s, const Schedule& sched = Schedule());
int ray_tiles(int W, int H);
// Global map rendering over n scene jobs sharing one image size (owner, rgba, err_flag nullable).
cudaError_t launch_render_global(const RayJob* jobs_dev, int n, int W, int H, uint16_t* depth, uint32_t* rgba,
                                 int8_t* owner, int32_t* err_flag, cudaStream_t s, int mode);
cudaError_t launch_verify_decide(const RansacJob* jobs, int n_jobs, cudaStream_t s);
cudaError_t launch_verify_decide_one(relo_pose_result* res, uint64_t omega, cudaStream_t s);
// Learned batches: mark fallback results not run, then pick each attempt's final result.
cudaError_t launch_init_results(relo_pose_result* res, int n, cudaStream_t s);
cudaError_t launch_merge_results(const relo_pose_result* learned, const relo_pose_result* fallback,
                                 const int32_t* kind, int n, relo_pose_result* out, cudaStream_t s);
// Builds SceneView::tsdf9 for n blocks with coordinates coords_dev (n x int32 xyz) from the
// scene's tsdf and hash table.
cudaError_t launch_build_apron(const SceneView& sv, const int32_t* coords_dev, int64_t n, float* out, cudaStream_t s);
cudaError_t launch_scene_lookup(SceneView sv, const int32_t* keys, int64_t n, int64_t* out, int32_t* err,
                                cudaStream_t s);

// RANSAC stages over a device array of jobs.
inline int table_words(int T) { return (3 + T + 7) / 8; }
cudaError_t launch_compact(const RansacJob* jobs, int n_jobs, int total_chunks, cudaStream_t s);
// counter_dev: one int of device scratch the search's warps take hypotheses from (zeroed here);
// max_draws > 0: every job's drawn pixels too (all its rounds), max_draws the most of any job
cudaError_t launch_hypotheses(const RansacJob* jobs, int n_jobs, int total_hyps, int32_t* counter_dev, cudaStream_t s,
                              const Schedule& sched = Schedule(), int max_draws = 0);
// the drawn pixels of one round
cudaError_t launch_draw(const RansacJob* jobs, int n_jobs, int round, const int32_t* alive_prefix_dev, cudaStream_t s);
// round r, its pixels drawn: prefix[n_jobs + 1] = flattened alive-hypothesis offsets of the jobs still
// running.  It takes round_launches(n_jobs, max_alive, B) launches.
int round_launches(int n_jobs, int max_alive, int B);
cudaError_t launch_round(const RansacJob* jobs, int n_jobs, int round, const int32_t* alive_prefix_dev,
                         int total_alive, int max_alive, const int32_t* surv_prefix_dev, int total_surv, int max_surv,
                         int B, cudaStream_t s, const Schedule& sched = Schedule(), bool after_draw = false);
cudaError_t launch_finalise(const RansacJob* jobs, int n_jobs, cudaStream_t s);

// One persistent launch for a pass's search, fit, rounds and finalise (ransac.cu): items in
// dependency order, per-(stage, job) completion counters, bounded waits.
enum PItemKind { kItemFit = 0, kItemDraw, kItemEnergy, kItemSelect, kItemRefine, kItemRefit, kItemFinal };
constexpr int kPersistThreadsHost = 256;  // threads of a persistent CTA (fit and re-fit chunk sizes)
struct PItem {
  int32_t kind, job, sub, part, round;
  int32_t dep, need;  // wait until done[dep] >= need
  int32_t done;       // then add one to done[done]
};
struct PersistArgs {
  const RansacJob* jobs;
  int n_jobs, total_hyps;
  int32_t* ctrl;                  // [0] search counter, [1] item counter, [2] abort flag
  const PItem* items;
  int n_items;
  int32_t* done;                  // completion counters; done[j] = job j's searched hypotheses
  int final_base;                 // done[final_base + j] = job j finalised
  const int32_t* alive_prefix;    // [rounds][n_jobs + 1], as launch_round
  const int32_t* surv_prefix;
  unsigned long long timeout_ns;
};
// ctrl_words: words zeroed from ctrl (ctrl[0..2] and the done counters that follow them)
cudaError_t launch_persistent(const PersistArgs& a, int ctrl_words, cudaStream_t s);
cudaError_t persistent_grid(int* grid);


// Training
// Leaves of the pixels (u, v) = stride * (grid column, grid row): out [T][ceil(H / stride)][ceil(W / stride)].
cudaError_t launch_forest_grid(const ForestJob& job, int stride, cudaStream_t s);
// One frame's offers to the reservoirs of `trees` trees from tree0 (training.cu).
constexpr int kSortItems = 2048, kSortBlocks = 64;  // the sort's CTAs per tree: at least so many items each, at most so many CTAs
struct ReservoirFrame {
  const uint16_t* depth;       // [H][W]
  const uint16_t* leaves;      // [trees][n] leaf of each grid pixel
  const float* coords;         // [n][3] scene coordinates of the grid pixels
  int W, stride, gw;
  int64_t n;                   // grid pixels
  int trees, tree0, D;
  int blocks, per_block;       // CTAs of the sort per tree, items of each (a multiple of 256)
  // scratch
  uint64_t* items[2];          // [trees][n] leaf << 32 | grid pixel, after each pass
  uint32_t* hist;              // [trees][blocks][256]
  int32_t* n_valid;            // [trees] valid pixels
  // by global leaf id
  int32_t* start;              // run of each leaf in its tree's sorted items
  int32_t* end;
  float* samples;              // [T][2^D][capacity][3]
  int32_t* count;
  int64_t* seen;
  int capacity;
  uint32_t key0, key1;
};
cudaError_t launch_reservoirs(const ReservoirFrame& f, cudaStream_t s);
cudaError_t launch_scene_coords(const uint16_t* depth, int W, int H, int stride, double fx, double fy, double cx,
                                double cy, const double* P /*16 host values passed by value*/, float* out,
                                cudaStream_t s);
cudaError_t launch_mean_shift(const float* samples, const int32_t* count, int capacity, int n_leaves_total,
                              float bandwidth, float tol, int max_iter, float merge_dist, float cov_floor,
                              int max_modes, float* modes, uint8_t* n_modes, cudaStream_t s);
cudaError_t launch_top_modes(const float* modes, const uint8_t* n_modes, int n_leaves_total, int max_modes,
                             float4* top, cudaStream_t s);

// Helpers for ray jobs
RayJob make_ray_job(const SceneView& sv, const relo_intrinsics& in, const double* pose_host);

// Checked builds (built with RELO_CHECKED=1): guarded accesses first check their index; a failed
// check is counted, once per translation unit, and the access is skipped.  The stand-in for a
// device memory checker.  In normal builds a check is the constant true and costs nothing.
#ifdef RELO_CHECKED
static __device__ unsigned int g_check_failures;
#define RELO_CHECK(cond) ((cond) ? true : (atomicAdd(&g_check_failures, 1u), false))
#define RELO_DEFINE_CHECK_READER(name)                                    \
  unsigned long long name() {                                             \
    unsigned int v = 0;                                                   \
    if (cudaMemcpyFromSymbol(&v, g_check_failures, sizeof v) != cudaSuccess) return ~0ull; \
    return v;                                                             \
  }
#else
#define RELO_CHECK(cond) true
#define RELO_DEFINE_CHECK_READER(name) \
  unsigned long long name() { return 0; }
#endif
unsigned long long check_failures_scene();
unsigned long long check_failures_forest();
unsigned long long check_failures_ransac();
unsigned long long check_failures_fusion();

// Every device allocation of the library goes through here: from cudaMalloc, or from the
// caller's allocator (relo_set_allocator); tests can make the next allocations fail
// (relo_debug_fail_allocations) and check the error paths.  dev_free returns a block to
// whichever of the two gave it (null is ignored).
cudaError_t dev_malloc(void** p, size_t bytes);
void dev_free(void* p);

// TSDF fusion of one frame into a growing scene (fusion.cu).
struct FuseJob {
  int4* buckets;
  int4* excess;
  float* tsdf;
  uint32_t* rgba;
  uint16_t* weight;
  int4* coords;                 // [capacity] block coordinates (w unused)
  int32_t* counters;            // [0] blocks in use, [1] excess entries in use
  int32_t* status;              // RELO_OK, or RELO_ENOMEM once the pool, the chain or the set ran out
  uint32_t bucket_mask;
  int32_t capacity, max_weight;
  const uint16_t* depth;        // frame [H][W] mm
  const uint32_t* frame_rgba;   // frame [H][W] or null
  int32_t W, H;
  float fx, fy, cx, cy, dmin, dmax;
  float R[9], t[3];             // camera -> scene
  float voxel, mu;
  unsigned long long* set;      // per-frame block set, set_mask + 1 slots
  uint32_t set_mask;
  unsigned long long* new_keys; // set_mask + 1
  unsigned long long* keys;     // set_mask + 1: the frame's distinct block keys, in insertion order
  int32_t* visible;             // set_mask + 1 block indices
  int32_t* n_visible;           // n_visible[0], then n_new, then n_keys
  int32_t* n_new;
  int32_t* n_keys;
  unsigned long long* updates;  // the scene's running count of block updates
  unsigned long long* cells;    // SceneView::cells
};
cudaError_t launch_fuse_frame(const FuseJob& j, cudaStream_t s);
cudaError_t launch_fuse_init(float* tsdf, int64_t n, cudaStream_t s);

}  // namespace relo

// Opaque handles (C ABI)
struct relo_scene {
  relo::SceneView view;
  void* d_buckets;
  void* d_excess;
  void* d_tsdf;
  void* d_rgba;
  void* d_grid;
  void* d_tsdf9;       // apron copy of the tsdf (SceneView::tsdf9), static scenes only
  int64_t n_blocks;
  // scenes that grow by fusion (relo_create_fusion_scene): capacity > 0
  int64_t capacity;
  void* d_weight;      // uint16 [capacity][512]
  void* d_coords;      // int4 [capacity]
  void* d_cells;       // SceneView::cells
  void* d_counters;    // int32 [4]: blocks in use, excess entries in use, status, pad; then uint64 block updates
  int32_t max_weight;
  int64_t n_excess;    // excess entries allocated (the chains' storage)
};

struct relo_forest {
  relo::ForestView view;
  void* d_nodes;
  void* d_modes;
  void* d_n_modes;
  void* d_top;
  int32_t T, D, M;
  bool reads_alpha;  // some node compares colour channel 3
  // training state
  relo_train_params train;
  bool training;
  // reservoirs on the device, allocated and zeroed by the first frame after train_begin (res_ready: that
  // frame has run)
  bool res_ready;
  float* res_samples;   // [T][L][cap][3]
  int32_t* res_count;   // [T][L]
  int64_t* res_seen;    // [T][L]
  int32_t* res_runs;    // [2][T][L] a frame's runs (ReservoirFrame::start, end)
  size_t res_slots;     // capacity of res_samples (T L cap)
  void* d_scratch;      // a frame's scratch, kept between frames
  size_t scratch_bytes;
};
