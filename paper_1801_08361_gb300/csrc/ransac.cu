// ransac.cu -- preemptive RANSAC over forest correspondences (the relocaliser's pose solver,
// after Cavallari et al. as used in Sec. 3.3.1; every rule is a stated reading, see relo.h).
//
// Stages, each one launch over all jobs of a batch:
//   compact    : ordered table of valid pixels, each entry packing {u, v, depth, leaf per tree}
//                in 16-byte words so that one load serves a correspondence (two passes: chunk
//                counts, then an ordered scatter with warp ballots);
//   search     : one warp per hypothesis evaluates 32 tries at a time and keeps the first passing
//                try, so the result equals a sequential scan of the tries.  The rigidity / area
//                tests run in FP32 with a guard band; a try inside the band is settled in FP64 in
//                the oracle's operation order;
//   fit        : one thread per hypothesis: 3-point Kabsch in FP64 (Horn's quaternion form);
//   per round  : draw B pixels; energies (warp per hypothesis, lanes over pixels, FP32 with an
//                FP64 running total); halving (CTA per job, bitonic sort of (energy, index));
//                re-fit sums (warp per survivor, one pass of shifted FP32 sums reduced with
//                shuffles); re-fit solve (thread per survivor, FP64 Horn).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cfloat>
#include <climits>

#include "relo_internal.cuh"

namespace relo {

__device__ __forceinline__ int find_job_by(const int32_t* prefix, int n_jobs, int gid) {
  int lo = 0, hi = n_jobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (prefix[mid] <= gid) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// u16 number k (0..7) of a 16-byte word
__device__ __forceinline__ uint32_t u16_of(uint4 q, int k) {
  const uint32_t w = (k < 4) ? ((k < 2) ? q.x : q.y) : ((k < 6) ? q.z : q.w);
  return (k & 1) ? (w >> 16) : (w & 0xFFFFu);
}

struct TableEntry {
  int u, v, depth;
  uint4 w0;  // first word (u, v, depth, leaf[0..4])
};

__device__ __forceinline__ TableEntry load_entry(const RansacJob& job, int idx) {
  TableEntry e;
  if (!RELO_CHECK(idx >= 0 && idx < *job.n_valid)) idx = 0;
  e.w0 = __ldg(&job.table[(size_t)idx * job.nv]);
  e.u = (int)(e.w0.x & 0xFFFFu);
  e.v = (int)(e.w0.x >> 16);
  e.depth = (int)(e.w0.y & 0xFFFFu);
  return e;
}

// Leaf of tree t for a table entry (field 3 + t of the packed entry).
__device__ __forceinline__ int entry_leaf(const RansacJob& job, int idx, const TableEntry& e, int t) {
  const int f = 3 + t;
  if (f < 8) return (int)u16_of(e.w0, f);
  return (int)u16_of(__ldg(&job.table[(size_t)idx * job.nv + (f >> 3)]), f & 7);
}

// FP32 camera point with reciprocal focal lengths ifx = 1 / fx, ify = 1 / fy (a few ulp from the
// FP64 point; the FP32 tests and scores that use it tolerate that).
__device__ __forceinline__ float3 cam_point_f(int u, int v, int d, float ifx, float ify, float cx, float cy) {
  const float z = (float)d * 0.001f;
  return make_float3(z * ((float)u - cx) * ifx, z * ((float)v - cy) * ify, z);
}

// FP64 camera point in the oracle's operation order: z = d / 1000; x = (z (u - cx)) / fx.
__device__ __forceinline__ void cam_point_d(int u, int v, int d, double fx, double fy, double cx, double cy,
                                            double out[3]) {
  const double z = __ddiv_rn((double)d, 1000.0);
  out[0] = __ddiv_rn(__dmul_rn(z, __dsub_rn((double)u, cx)), fx);
  out[1] = __ddiv_rn(__dmul_rn(z, __dsub_rn((double)v, cy)), fy);
  out[2] = z;
}

// ---------------------------------------------------------------------------------------------
// horn_pose (relo_internal.cuh) by 16 lanes, two solves per warp.  Every lane of a group runs
// horn_refined on the same matrix (a warp's instruction costs the same for 2 lanes and 32); where a group
// has to take the FP64 rotations, lane 4 i + j of it holds entries (i, j) of A and V.  The FP64 pipe
// takes many cycles per warp instruction however few lanes are active, so one thread's rotations (about
// 700 FP64 instructions a sweep) are bound by that pipe's latency: 84-105 us whether one hypothesis or two
// thousand are re-fitted.  Sharing the entries among lanes leaves about 200 a sweep, most of them the two
// rotations' angles, which both halves of the columns take at once.  Every entry goes through
// horn_jacobi's operations in its order and rounding, so both forms give the same bits.  Used where a
// launch has at most kGroupSolves solves; beyond, the 32 solves a warp of the other form advances per
// instruction win.  A house frame's re-fit: 95 us a round by single threads, 35 with the rotations
// shared, 18 now.
// ---------------------------------------------------------------------------------------------
#ifndef RELO_GROUP_SOLVES
#define RELO_GROUP_SOLVES 2048
#endif
constexpr int kGroupSolves = RELO_GROUP_SOLVES;
constexpr int kSolvesPerWarp = 2;

__device__ __forceinline__ double group_get(double v, int from) { return __shfl_sync(0xffffffffu, v, from, 16); }

// S: the cross-covariance's entry `lane & 15` (0..8) in lanes 0..8 of the group; cbar, wbar: all
// lanes.  active: the group has a solve (the warp's other group may not).  Lane 0 of the group
// writes out.  All 32 lanes call it together.
__device__ __forceinline__ void horn_pose_group(double S_lane, const double cbar[3], const double wbar[3], bool active,
                                                double* out) {
  const int l = threadIdx.x & 15, i = l >> 2, j = l & 3;
  double S[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) S[k] = group_get(S_lane, k);
  double q[4];
  if (active && horn_refined(S, q)) {
    if (l == 0) quaternion_pose(q[0], q[1], q[2], q[3], cbar, wbar, out);
    active = false;
  }
  if (!__any_sync(0xffffffffu, active)) return;
  const double Sxx = S[0], Sxy = S[1], Sxz = S[2], Syx = S[3], Syy = S[4], Syz = S[5], Szx = S[6], Szy = S[7],
               Szz = S[8];
  double A, V = i == j ? 1.0 : 0.0;
  {
    const int u = min(i, j), v = max(i, j);
    double x = Syz, y = -Szy;                                   // (0, 1)
    if (u == 0 && v == 2) x = Szx, y = -Sxz;
    if (u == 0 && v == 3) x = Sxy, y = -Syx;
    if (u == 1 && v == 2) x = Sxy, y = Syx;
    if (u == 1 && v == 3) x = Szx, y = Sxz;
    if (u == 2 && v == 3) x = Syz, y = Szy;
    if (u == v) {
      x = u < 2 ? Sxx : -Sxx;
      y = (u == 0 || u == 2) ? Syy : -Syy;
    }
    A = __dadd_rn(x, y);
    if (u == v) A = __dadd_rn(A, (u == 0 || u == 3) ? Szz : -Szz);
  }
  bool busy = active;
  for (int sweep = 0; sweep < 30; ++sweep) {
    double off = 0.0, diag = 0.0;
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const double d = group_get(A, 5 * p);
      diag = __fma_rn(d, d, diag);
#pragma unroll
      for (int q = p + 1; q < 4; ++q) {
        const double o = group_get(A, 4 * p + q);
        off = __fma_rn(o, o, off);
      }
    }
    if (off <= 1e-30 * (diag + 1e-300)) busy = false;
    if (!__any_sync(0xffffffffu, busy)) break;
#pragma unroll
    for (int st = 0; st < 3; ++st) {
      // stage st rotates the pairs (0, st + 1) and the two other indices, in that order
      const int flip = st + 1;
      const int jp = j ^ flip, ip = i ^ flip;                   // partners
      const bool j_first = j < jp, i_first = i < ip;            // first index of its pair
      const bool j0 = j == 0 || j == flip, i0 = i == 0 || i == flip;  // in pair (0, flip)
      // angle of the pair holding j: p = min(j, jp), q = max(j, jp)
      const int p = min(j, jp), q = max(j, jp);
      const double apq = group_get(A, 4 * p + q), aqq = group_get(A, 5 * q), app = group_get(A, 5 * p);
      double c = 1.0, s = 0.0;
      if (fabs(apq) >= 1e-300) {
        const double theta = __ddiv_rn(__dsub_rn(aqq, app), 2.0 * apq);
        const double t = __ddiv_rn(theta >= 0.0 ? 1.0 : -1.0, __dadd_rn(fabs(theta), __dsqrt_rn(__fma_rn(theta, theta, 1.0))));
        c = rsqrt(__fma_rn(t, t, 1.0));
        s = __dmul_rn(t, c);
      }
      const double ci = group_get(c, i), si = group_get(s, i);  // lane i (row 0) holds column i's angle
      // x' = c x - s y for the pair's first index, y' = s x + c y for its second
      auto rotate = [](double mine, double other, bool first, double cc, double ss) {
        const double x = first ? mine : other, y = first ? other : mine;
        return __fma_rn(first ? cc : ss, x, __dmul_rn(first ? -ss : cc, y));
      };
      // horn_jacobi rotates pair 0's columns, its rows, then pair 1's columns and rows: entries in
      // pair 0's rows and pair 1's columns see the row rotation first, all others the column's
      const bool row_first = i0 && !j0;
      double other = group_get(A, row_first ? 4 * ip + j : 4 * i + jp);
      double B = rotate(A, other, row_first ? i_first : j_first, row_first ? ci : c, row_first ? si : s);
      other = group_get(B, row_first ? 4 * i + jp : 4 * ip + j);
      B = rotate(B, other, row_first ? j_first : i_first, row_first ? c : ci, row_first ? s : si);
      other = group_get(V, 4 * i + jp);
      const double U = rotate(V, other, j_first, c, s);
      if (busy) {
        A = B;
        V = U;
      }
    }
  }
  double best_d = group_get(A, 0);
  int bk = 0;
#pragma unroll
  for (int k = 1; k < 4; ++k) {
    const double d = group_get(A, 5 * k);
    if (d > best_d) {
      best_d = d;
      bk = k;
    }
  }
  const double w = group_get(V, bk), x = group_get(V, 4 + bk), y = group_get(V, 8 + bk), z = group_get(V, 12 + bk);
  if (!active || l != 0) return;
  quaternion_pose(w, x, y, z, cbar, wbar, out);
}

// ---------------------------------------------------------------------------------------------
// Chained launches: a kernel of the sequence starts while the one before it runs its last CTAs, and
// begins with chain_begin, which waits until that one has completed and its writes are visible; its own
// successor may be launched from then on.  A lone attempt is up to fifty launches of 5 to 30 us, and the
// gaps between them were a tenth of it (a house frame's RANSAC: 848 us unchained, 784 chained).  Every
// thread calls chain_begin before anything else, so a kernel never completes before those in front of it.
// Data written by the kernel in front is read with plain loads only (not __ldg, whose data may not change
// while a kernel is resident): hence no chaining from the draws, whose records are read so.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void chain_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <class... Params, class... Args>
cudaError_t launch_chained(bool chained, void (*kernel)(Params...), dim3 grid, unsigned threads, size_t smem, cudaStream_t s,
                           Args... args) {
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = dim3(threads);
  c.dynamicSmemBytes = smem;
  c.stream = s;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  c.attrs = &attr;
  c.numAttrs = chained ? 1 : 0;
  return cudaLaunchKernelEx(&c, kernel, Params(args)...);
}

// ---------------------------------------------------------------------------------------------
// Valid-pixel table
// ---------------------------------------------------------------------------------------------
constexpr int kCompactThreads = 256;
constexpr int kIters = kCompactChunk / kCompactThreads;  // 16 coalesced passes of 256 pixels

__device__ __forceinline__ int chunk_job(const RansacJob* jobs, int n_jobs, int gid) {
  int lo = 0, hi = n_jobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].chunk_begin <= gid) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

__global__ void __launch_bounds__(kCompactThreads) compact_count_kernel(const RansacJob* __restrict__ jobs,
                                                                       int n_jobs) {
  chain_begin();
  const RansacJob& job = jobs[chunk_job(jobs, n_jobs, blockIdx.x)];
  if (job_skipped(job.skip)) return;
  const int chunk = blockIdx.x - job.chunk_begin;
  const int n_pix = job.W * job.H;
  int c = 0;
  for (int it = 0; it < kIters; ++it) {
    const int p = chunk * kCompactChunk + it * kCompactThreads + threadIdx.x;
    if (p < n_pix && job.depth[p] > 0) ++c;
  }
  c = warp_sum_i(c);
  __shared__ int part[kCompactThreads / 32];
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    int s = 0;
    for (int w = 0; w < kCompactThreads / 32; ++w) s += part[w];
    job.chunk_count[chunk] = s;
  }
}

__global__ void __launch_bounds__(kCompactThreads) compact_scatter_kernel(const RansacJob* __restrict__ jobs,
                                                                         int n_jobs) {
  chain_begin();
  const RansacJob& job = jobs[chunk_job(jobs, n_jobs, blockIdx.x)];
  if (job_skipped(job.skip)) return;
  const int chunk = blockIdx.x - job.chunk_begin;
  const int n_pix = job.W * job.H;
  const int n_chunks = (n_pix + kCompactChunk - 1) / kCompactChunk;
  const int T = job.forest.T, nv = job.nv;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int kWarps = kCompactThreads / 32;
  __shared__ int s_off;
  __shared__ int s_count[kIters * kWarps];  // valid pixels per 32, in raster order; then those before them
  // All of the chunk's depths at once, and two barriers in all: with a barrier pair per 256 pixels a
  // chunk was 16 dependent rounds (38 us for a lone 640 x 480 view).
  int d[kIters];
#pragma unroll
  for (int it = 0; it < kIters; ++it) {
    const int p = chunk * kCompactChunk + it * kCompactThreads + threadIdx.x;
    d[it] = p < n_pix ? job.depth[p] : 0;
  }
  if (warp == 0) {
    int s = 0;
    for (int c = lane; c < chunk; c += 32) s += job.chunk_count[c];
    s = warp_sum_i(s);
    if (lane == 0) s_off = s;
  }
  unsigned ball[kIters];
#pragma unroll
  for (int it = 0; it < kIters; ++it) {
    ball[it] = __ballot_sync(0xffffffffu, d[it] > 0);
    if (lane == 0) s_count[it * kWarps + warp] = __popc(ball[it]);
  }
  __syncthreads();
  if (warp == 0) {
    constexpr int kPer = kIters * kWarps / 32;
    int c[kPer], sum = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) sum += c[k] = s_count[lane * kPer + k];
    int before = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, before, o);
      if (lane >= o) before += y;
    }
    int at = s_off + before - sum;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      s_count[lane * kPer + k] = at;
      at += c[k];
    }
    if (chunk == n_chunks - 1 && lane == 31) *job.n_valid = at;
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < kIters; ++it) {
    if (d[it] == 0) continue;
    const int p = chunk * kCompactChunk + it * kCompactThreads + threadIdx.x;
    const int pos = s_count[it * kWarps + warp] + __popc(ball[it] & ((1u << lane) - 1u));
    // fields u, v, depth, leaf[T], packed two to a word and eight to an entry
    uint4* dst = job.table + (size_t)pos * nv;
    const uint16_t* leaves = job.leaves + p;
    auto field = [&](int k) -> uint32_t {
      return k == 0 ? (uint32_t)(p % job.W) : k == 1 ? (uint32_t)(p / job.W) : k == 2 ? (uint32_t)d[it]
             : k < 3 + T ? (uint32_t)leaves[(size_t)(k - 3) * n_pix] : 0u;
    };
    for (int q = 0; q < nv; ++q)
      dst[q] = make_uint4(field(8 * q) | field(8 * q + 1) << 16, field(8 * q + 2) | field(8 * q + 3) << 16,
                          field(8 * q + 4) | field(8 * q + 5) << 16, field(8 * q + 6) | field(8 * q + 7) << 16);
  }
}

cudaError_t launch_compact(const RansacJob* jobs, int n_jobs, int total_chunks, cudaStream_t s) {
  if (total_chunks <= 0) return cudaSuccess;
  compact_count_kernel<<<total_chunks, kCompactThreads, 0, s>>>(jobs, n_jobs);
  const cudaError_t e = launch_chained(true, compact_scatter_kernel, total_chunks, kCompactThreads, 0, s, jobs, n_jobs);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// Hypothesis search
// ---------------------------------------------------------------------------------------------
constexpr float kGuardRigid = 1e-4f;  // FP32 error of a distance difference stays below 2e-5 m here
constexpr float kGuardArea = 2e-4f;   // and that of |cross| below 2e-5 m^2

__device__ __forceinline__ double dist_d(const double* a, const double* b) {
  const double d0 = __dsub_rn(a[0], b[0]), d1 = __dsub_rn(a[1], b[1]), d2 = __dsub_rn(a[2], b[2]);
  return __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(d0, d0), __dmul_rn(d1, d1)), __dmul_rn(d2, d2)));
}

__device__ __forceinline__ double cross_norm_d(const double* p0, const double* p1, const double* p2) {
  const double e1[3] = {__dsub_rn(p1[0], p0[0]), __dsub_rn(p1[1], p0[1]), __dsub_rn(p1[2], p0[2])};
  const double e2[3] = {__dsub_rn(p2[0], p0[0]), __dsub_rn(p2[1], p0[1]), __dsub_rn(p2[2], p0[2])};
  const double x = __dsub_rn(__dmul_rn(e1[1], e2[2]), __dmul_rn(e1[2], e2[1]));
  const double y = __dsub_rn(__dmul_rn(e1[2], e2[0]), __dmul_rn(e1[0], e2[2]));
  const double z = __dsub_rn(__dmul_rn(e1[0], e2[1]), __dmul_rn(e1[1], e2[0]));
  return __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(x, x), __dmul_rn(y, y)), __dmul_rn(z, z)));
}

// Distance through the hardware reciprocal square root (relative error about 2^-22, i.e. below
// 1e-5 m on the few-metre distances here and inside the guard band of the tests using it).
__device__ __forceinline__ float dist_f(float3 a, float3 b) {
  const float x = a.x - b.x, y = a.y - b.y, z = a.z - b.z;
  const float s = x * x + y * y + z * z;
  return s > 0.f ? s * rsqrtf(s) : 0.f;
}

// |cross(p1 - p0, p2 - p0)|^2 (compared against squared area bounds).
__device__ __forceinline__ float cross_norm2_f(float3 p0, float3 p1, float3 p2) {
  const float ax = p1.x - p0.x, ay = p1.y - p0.y, az = p1.z - p0.z;
  const float bx = p2.x - p0.x, by = p2.y - p0.y, bz = p2.z - p0.z;
  const float x = ay * bz - az * by, y = az * bx - ax * bz, z = ax * by - ay * bx;
  return x * x + y * y + z * z;
}

struct Corr {
  int idx[3], tree[3], leaf[3];
  TableEntry e[3];
};

__device__ __forceinline__ Corr draw_try(const RansacJob& job, int h, int j, int n_valid) {
  const uint4 x = philox4x32_10(make_uint4(1u, (uint32_t)h, (uint32_t)j, 0u), job.key0, job.key1);
  Corr c;
  const uint32_t w[3] = {x.x, x.y, x.z};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    c.idx[k] = (int)uniform_below(w[k], (uint32_t)n_valid);
    c.tree[k] = (int)((((x.w >> (8 * k)) & 0xFFu) * (uint32_t)job.forest.T) >> 8);
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) c.e[k] = load_entry(job, c.idx[k]);
#pragma unroll
  for (int k = 0; k < 3; ++k) c.leaf[k] = entry_leaf(job, c.idx[k], c.e[k], c.tree[k]);
  return c;
}

// Exact decision of the rigidity and area tests in FP64, in the oracle's operation order.
__device__ __noinline__ bool exact_geometry(const RansacJob& job, int h, int j, int n_valid) {
  const Corr c = draw_try(job, h, j, n_valid);
  const int L = 1 << job.forest.D;
  double cp[3][3], wp[3][3];
  for (int k = 0; k < 3; ++k) {
    cam_point_d(c.e[k].u, c.e[k].v, c.e[k].depth, job.fx, job.fy, job.cx, job.cy, cp[k]);
    const float4 m = __ldg(&job.forest.top[(size_t)c.tree[k] * L + c.leaf[k]]);
    wp[k][0] = (double)m.x;
    wp[k][1] = (double)m.y;
    wp[k][2] = (double)m.z;
  }
  const int pr[3][2] = {{0, 1}, {0, 2}, {1, 2}};
  bool ok = true;
  for (int q = 0; q < 3; ++q) {
    const double dc = dist_d(cp[pr[q][0]], cp[pr[q][1]]), dw = dist_d(wp[pr[q][0]], wp[pr[q][1]]);
    ok = ok && (fabs(__dsub_rn(dc, dw)) <= job.rigidity);
  }
  return ok && (cross_norm_d(cp[0], cp[1], cp[2]) >= job.min_area) &&
         (cross_norm_d(wp[0], wp[1], wp[2]) >= job.min_area);
}

// Mode-0 mean of a correspondence's leaf (w = its count; w < 0.5: empty leaf), or w = -1 when the
// leaf id is outside the forest.
__device__ __forceinline__ float4 corr_mode(const RansacJob& job, int tree, int leaf, int L) {
  return leaf < L ? __ldg(&job.forest.top[(size_t)tree * L + leaf]) : make_float4(0.f, 0.f, 0.f, -1.f);
}

// Rigidity of one pair: 0 fails, 1 passes, 2 inside the guard band.
__device__ __forceinline__ int pair_status(float3 pa, float3 pb, float3 qa, float3 qb, float rig) {
  const float diff = fabsf(dist_f(pa, pb) - dist_f(qa, qb));
  if (diff > rig + kGuardRigid) return 0;
  return diff >= rig - kGuardRigid ? 2 : 1;
}

// The draws of one try: three table positions and three trees.
struct TryDraw {
  int i0, i1, i2, t0, t1, t2;
};

__device__ __forceinline__ TryDraw draw_indices(const RansacJob& job, int h, int j, int n_valid) {
  const uint4 x = philox4x32_10(make_uint4(1u, (uint32_t)h, (uint32_t)j, 0u), job.key0, job.key1);
  const uint32_t T = (uint32_t)job.forest.T;
  TryDraw d;
  d.i0 = (int)uniform_below(x.x, (uint32_t)n_valid);
  d.i1 = (int)uniform_below(x.y, (uint32_t)n_valid);
  d.i2 = (int)uniform_below(x.z, (uint32_t)n_valid);
  d.t0 = (int)(((x.w & 0xFFu) * T) >> 8);
  d.t1 = (int)((((x.w >> 8) & 0xFFu) * T) >> 8);
  d.t2 = (int)((((x.w >> 16) & 0xFFu) * T) >> 8);
  return d;
}

// The first pair of a try, loaded: entries and mode-0 means of correspondences 0 and 1.
struct TryPair {
  TableEntry e0, e1;
  float4 m0, m1;
};

__device__ __forceinline__ TryPair load_pair(const RansacJob& job, const TryDraw& d, int L) {
  TryPair p;
  p.e0 = load_entry(job, d.i0);
  p.e1 = load_entry(job, d.i1);
  p.m0 = corr_mode(job, d.t0, entry_leaf(job, d.i0, p.e0, d.t0), L);
  p.m1 = corr_mode(job, d.t1, entry_leaf(job, d.i1, p.e1, d.t1), L);
  return p;
}

// 0: the try fails; 1: it passes; 2: a test lies inside the FP32 guard band (settle in FP64).
// The tests are a conjunction of pure conditions, so their order does not change the outcome:
// the pair (0, 1) (already loaded) is tested before the third correspondence is loaded, which
// most tries never reach.
__device__ __forceinline__ int try_status(const RansacJob& job, const TryDraw& d, const TryPair& pr, int L, float rig,
                                          float area_lo2, float area_hi2, float ifx, float ify, float cx, float cy) {
  if (d.i0 == d.i1 || d.i0 == d.i2 || d.i1 == d.i2) return 0;
  if (pr.m0.w < 0.5f || pr.m1.w < 0.5f) return 0;
  const float3 p0 = cam_point_f(pr.e0.u, pr.e0.v, pr.e0.depth, ifx, ify, cx, cy);
  const float3 p1 = cam_point_f(pr.e1.u, pr.e1.v, pr.e1.depth, ifx, ify, cx, cy);
  const float3 q0 = make_float3(pr.m0.x, pr.m0.y, pr.m0.z), q1 = make_float3(pr.m1.x, pr.m1.y, pr.m1.z);
  const int s01 = pair_status(p0, p1, q0, q1, rig);
  if (s01 == 0) return 0;
  const TableEntry e2 = load_entry(job, d.i2);
  const float4 m2 = corr_mode(job, d.t2, entry_leaf(job, d.i2, e2, d.t2), L);
  if (m2.w < 0.5f) return 0;
  const float3 p2 = cam_point_f(e2.u, e2.v, e2.depth, ifx, ify, cx, cy);
  const float3 q2 = make_float3(m2.x, m2.y, m2.z);
  const int s02 = pair_status(p0, p2, q0, q2, rig);
  if (s02 == 0) return 0;
  const int s12 = pair_status(p1, p2, q1, q2, rig);
  if (s12 == 0) return 0;
  bool ambiguous = s01 == 2 || s02 == 2 || s12 == 2;
  const float ac2 = cross_norm2_f(p0, p1, p2), aw2 = cross_norm2_f(q0, q1, q2);
  if (ac2 < area_lo2 || aw2 < area_lo2) return 0;
  if (ac2 <= area_hi2 || aw2 <= area_hi2) ambiguous = true;
  return ambiguous ? 2 : 1;
}

// Each warp step evaluates 64 tries, two per lane (tries base + lane and base + 32 + lane, whose loads
// are issued together), and keeps the first one not failing in try order, settling guard-band tries in
// FP64 in order.  What bounds it is the L1: a gather takes about one cycle per lane, four a try (84 % of
// the data pipe's peak over a batch).  Tried: queueing the tries that pass their first pair for a dense
// second stage (slower: house batch 19.2 -> 21.3 ms with the fits and compaction).  Testing first pairs
// from 16-bit position codes in the table, two gathers a try, with such a queue for the one in six that
// those let through, was faster at four CTAs an SM (18.2 ms of that 19.2, 2 % of the batch; 21.2 ms at
// five, its second stage a chain of six dependent loads): not kept for a gain that small and a larger table.
constexpr int kSearchWarps = 4;

// first try of mask (bits = lanes) that passes, settling guard-band statuses in FP64; -1 if none
__device__ __forceinline__ int first_passing(const RansacJob& job, int h, int n_valid, unsigned mask, int st,
                                             int j, int lane) {
  while (mask) {
    const int w = __ffs(mask) - 1;
    const int sw = __shfl_sync(0xffffffffu, st, w);
    int ok = sw == 1;
    if (!ok) {
      int e = 0;
      if (lane == w) e = exact_geometry(job, h, j, n_valid) ? 1 : 0;
      ok = __shfl_sync(0xffffffffu, e, w);
    }
    if (ok) return w;
    mask &= mask - 1;  // rejected in FP64: consider the next try of this step
  }
  return -1;
}

// CTAs per SM for the search (5 x 128 threads: 96 registers for the two tries in flight per lane,
// with about 60 bytes spilled): on the house batch the hypotheses stage takes 18.68 ms at 5, 18.98
// at 4 (128 registers, no spills) and 21.89 at 6 (80 registers, 128-byte spills)
#ifndef RELO_SEARCH_MIN_BLOCKS
#define RELO_SEARCH_MIN_BLOCKS 5
#endif
__device__ __forceinline__ int hypothesis_job(const RansacJob* __restrict__ jobs, int n_jobs, int gid) {
  int lo = 0, hi = n_jobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].hyp_begin <= gid) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// First passing try of hypothesis h among those of warp `part` of `parts` (steps of 64 tries in turn);
// INT_MAX if none.  *found (shared by the parts, null for one): the lowest passing try so far, beyond
// which no part needs to look.
__device__ __forceinline__ int search_part(const RansacJob& job, int h, int lane, int part, int parts,
                                           volatile int* found) {
  const int n_valid = *job.n_valid;
  if (n_valid <= 0) return INT_MAX;
  const float rig = (float)job.rigidity, area = (float)job.min_area;
  // the area test |cross| >= area with its guard band, on squares (both sides non-negative)
  const float area_lo = fmaxf(area - kGuardArea, 0.f), area_hi = area + kGuardArea;
  const float area_lo2 = area_lo * area_lo, area_hi2 = area_hi * area_hi;
  const float ifx = (float)(1.0 / job.fx), ify = (float)(1.0 / job.fy), cx = (float)job.cx, cy = (float)job.cy;
  const int L = 1 << job.forest.D;
  for (int base = part * 64; base < job.max_tries; base += 64 * parts) {
    if (found && __shfl_sync(0xffffffffu, *found, 0) < base) break;
    const int ja = base + lane, jb = base + 32 + lane;
    const TryDraw da = draw_indices(job, h, ja, n_valid), db = draw_indices(job, h, jb, n_valid);
    const TryPair pa = load_pair(job, da, L), pb = load_pair(job, db, L);
    const int sa = ja < job.max_tries ? try_status(job, da, pa, L, rig, area_lo2, area_hi2, ifx, ify, cx, cy) : 0;
    const int sb = jb < job.max_tries ? try_status(job, db, pb, L, rig, area_lo2, area_hi2, ifx, ify, cx, cy) : 0;
    int w = first_passing(job, h, n_valid, __ballot_sync(0xffffffffu, sa != 0), sa, ja, lane);
    if (w >= 0) return base + w;
    w = first_passing(job, h, n_valid, __ballot_sync(0xffffffffu, sb != 0), sb, jb, lane);
    if (w >= 0) return base + 32 + w;
  }
  return INT_MAX;
}

__device__ __forceinline__ void store_search(const RansacJob& job, int h, int found) {
  job.hyp_ok[h] = found != INT_MAX;
  job.tries[h] = found != INT_MAX ? found : job.max_tries;
}

// The search of hypothesis gw (flattened over the jobs) by one warp.
__device__ __forceinline__ int search_one(const RansacJob* __restrict__ jobs, int n_jobs, int gw, int lane) {
  const int jid = hypothesis_job(jobs, n_jobs, gw);
  const RansacJob& job = jobs[jid];
  const int h = gw - job.hyp_begin;
  if (h >= job.K || job_skipped(job.skip)) return jid;
  const int found = search_part(job, h, lane, 0, 1, nullptr);
  if (lane == 0) store_search(job, h, found);
  return jid;
}

#ifndef RELO_SEARCH_WIDE
#define RELO_SEARCH_WIDE 3
#endif
#ifndef RELO_SEARCH_SHARED
#define RELO_SEARCH_SHARED 3
#endif
// Persistent: hypotheses need from one try to max_tries, so each warp takes its next hypothesis
// from a counter when it finishes one (which warp computes a hypothesis does not change its result).
__global__ void __launch_bounds__(kSearchWarps * 32, RELO_SEARCH_MIN_BLOCKS)
    search_kernel(const RansacJob* __restrict__ jobs, int n_jobs, int total, int32_t* __restrict__ counter) {
  chain_begin();
  const int lane = threadIdx.x & 31;
  for (;;) {
    int gw = 0;
    if (lane == 0) gw = atomicAdd(counter, 1);
    gw = __shfl_sync(0xffffffffu, gw, 0);
    if (gw >= total) return;
    search_one(jobs, n_jobs, gw, lane);
  }
}

// Few hypotheses: the warps of a CTA share one, each taking every kWarps-th step (a hypothesis that uses
// up its 10 000 tries is a chain of 157 dependent steps for one warp, which set the time of a lone
// attempt: 247 us of a house frame's search, 242 of a room's).
template <int kWarps>
__global__ void __launch_bounds__(kWarps * 32, RELO_SEARCH_MIN_BLOCKS * kSearchWarps / kWarps)
    search_shared_kernel(const RansacJob* __restrict__ jobs, int n_jobs, int total, int32_t* __restrict__ counter) {
  chain_begin();
  __shared__ int s_found, s_next;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (;;) {
    if (threadIdx.x == 0) {
      s_next = atomicAdd(counter, 1);
      s_found = INT_MAX;
    }
    __syncthreads();
    const int gw = s_next;
    if (gw >= total) return;
    const RansacJob& job = jobs[hypothesis_job(jobs, n_jobs, gw)];
    const int h = gw - job.hyp_begin;
    const bool mine = h < job.K && !job_skipped(job.skip);
    if (mine) {
      const int r = search_part(job, h, lane, warp, kWarps, &s_found);
      if (lane == 0 && r != INT_MAX) atomicMin(&s_found, r);
    }
    __syncthreads();
    if (mine && threadIdx.x == 0) store_search(job, h, s_found);
    __syncthreads();
  }
}

// (first mode, mode count) of an entry's leaf in tree t: its modes are f.modes[first ..
// first + count) in units of kModeFloats; count 0 for a leaf id outside the forest.
__device__ __forceinline__ int2 tree_modes(const RansacJob& job, int idx, const TableEntry& e, int t, int L) {
  const ForestView& f = job.forest;
  const int leaf = entry_leaf(job, idx, e, t);
  if (leaf >= L || !RELO_CHECK(t >= 0 && t < f.T)) return make_int2(0, 0);
  const int node = t * L + leaf;
  return make_int2(node * f.M, min((int)__ldg(&f.n_modes[node]), f.M));
}

// Draws pixel i of round r (a position in the valid table) and writes its record (camera point and
// where its modes are), which every hypothesis then reads.
__device__ __forceinline__ void draw_pixel(const RansacJob& job, int r, int i, int n_valid) {
  const float ifx = (float)(1.0 / job.fx), ify = (float)(1.0 / job.fy), cx = (float)job.cx, cy = (float)job.cy;
  const int T = job.forest.T, L = 1 << job.forest.D;
  const uint4 x = philox4x32_10(make_uint4(2u, (uint32_t)r, (uint32_t)i, 0u), job.key0, job.key1);
  const int idx = (int)uniform_below(x.x, (uint32_t)n_valid);
  job.drawn[(size_t)r * job.B + i] = idx;
  const TableEntry e = load_entry(job, idx);
  const float3 c = cam_point_f(e.u, e.v, e.depth, ifx, ify, cx, cy);
  int4* rec = job.pix + ((size_t)r * job.B + i) * job.hs;
  rec[0] = make_int4(__float_as_int(c.x), __float_as_int(c.y), __float_as_int(c.z), 0);
  for (int t = 0; t < T; t += 2) {
    const int2 a = tree_modes(job, idx, e, t, L);
    const int2 b = t + 1 < T ? tree_modes(job, idx, e, t + 1, L) : make_int2(0, 0);
    rec[1 + t / 2] = make_int4(a.x, a.y, b.x, b.y);
  }
}

// FP64 Kabsch of hypothesis h's kept try; also initialises its round state.
__device__ __forceinline__ void fit_one(const RansacJob& job, int h) {
  double* pose = job.poses + 12 * (size_t)h;
  const bool ok = job.hyp_ok[h] != 0;
  if (ok) {
    const Corr c = draw_try(job, h, job.tries[h], *job.n_valid);
    const int L = 1 << job.forest.D;
    double cp[3][3], wp[3][3], cb[3] = {0, 0, 0}, wb[3] = {0, 0, 0};
    for (int k = 0; k < 3; ++k) {
      cam_point_d(c.e[k].u, c.e[k].v, c.e[k].depth, job.fx, job.fy, job.cx, job.cy, cp[k]);
      const float4 m = job.forest.top[(size_t)c.tree[k] * L + c.leaf[k]];
      wp[k][0] = m.x;
      wp[k][1] = m.y;
      wp[k][2] = m.z;
      for (int a = 0; a < 3; ++a) {
        cb[a] = __dadd_rn(cb[a], __ddiv_rn(cp[k][a], 3.0));
        wb[a] = __dadd_rn(wb[a], __ddiv_rn(wp[k][a], 3.0));
      }
    }
    double S[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    for (int k = 0; k < 3; ++k)
      for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b)
          S[3 * a + b] = __fma_rn(__dsub_rn(cp[k][a], cb[a]), __dsub_rn(wp[k][b], wb[b]), S[3 * a + b]);
    horn_pose(S, cb, wb, pose);
  } else {
    for (int q = 0; q < 12; ++q) pose[q] = (q % 5 == 0) ? 1.0 : 0.0;
  }
  job.energy[h] = ok ? 0.0 : (double)INFINITY;
  job.alive_a[h] = h;
  job.inliers[h] = 0;
}

// fit_one of two hypotheses by a warp (hypothesis h by the group of 16 lanes; h < 0: none).
__device__ __forceinline__ void fit_group(const RansacJob& job, int h) {
  const int l = threadIdx.x & 15;
  const bool ok = h >= 0 && job.hyp_ok[h] != 0;
  double cb[3] = {0, 0, 0}, wb[3] = {0, 0, 0}, S = 0.0;
  if (ok) {
    // every lane takes the three points (the loads are broadcasts); lane 3 a + b sums S(a, b)
    const Corr c = draw_try(job, h, job.tries[h], *job.n_valid);
    const int L = 1 << job.forest.D;
    double cp[3][3], wp[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      cam_point_d(c.e[k].u, c.e[k].v, c.e[k].depth, job.fx, job.fy, job.cx, job.cy, cp[k]);
      const float4 m = job.forest.top[(size_t)c.tree[k] * L + c.leaf[k]];
      wp[k][0] = m.x;
      wp[k][1] = m.y;
      wp[k][2] = m.z;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        cb[a] = __dadd_rn(cb[a], __ddiv_rn(cp[k][a], 3.0));
        wb[a] = __dadd_rn(wb[a], __ddiv_rn(wp[k][a], 3.0));
      }
    }
    const int a = min(l / 3, 2), b = l - 3 * (l / 3);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const double ca = a == 0 ? cp[k][0] : a == 1 ? cp[k][1] : cp[k][2], ma = a == 0 ? cb[0] : a == 1 ? cb[1] : cb[2];
      const double wv = b == 0 ? wp[k][0] : b == 1 ? wp[k][1] : wp[k][2], mb = b == 0 ? wb[0] : b == 1 ? wb[1] : wb[2];
      S = __fma_rn(__dsub_rn(ca, ma), __dsub_rn(wv, mb), S);
    }
  }
  __syncwarp();
  horn_pose_group(S, cb, wb, ok, h >= 0 ? job.poses + 12 * (size_t)h : nullptr);
  if (h < 0) return;
  if (!ok && l < 12) job.poses[12 * (size_t)h + l] = (l % 5 == 0) ? 1.0 : 0.0;
  if (l == 0) {
    job.energy[h] = ok ? 0.0 : (double)INFINITY;
    job.alive_a[h] = h;
    job.inliers[h] = 0;
  }
}

// The kept tries' poses, and the draws of every round (both need only the table and the search's
// result, and a round's draws are the same whoever is alive): CTAs below fit_blocks take the fits,
// draw_blocks CTAs per job after them the job's drawn pixels.  kGroup: two hypotheses per warp
// (fit_group) instead of 32.
constexpr int kFitThreads = 128;
template <bool kGroup>
__global__ void __launch_bounds__(kFitThreads) fit_kernel(const RansacJob* __restrict__ jobs, int n_jobs, int total,
                                                          int fit_blocks, int draw_blocks) {
  chain_begin();
  if ((int)blockIdx.x >= fit_blocks) {
    const int q = (int)blockIdx.x - fit_blocks, jid = q / draw_blocks;
    const RansacJob& job = jobs[jid];
    if (job_skipped(job.skip)) return;
    const int i = (q - jid * draw_blocks) * kFitThreads + threadIdx.x;
    if (i < job.n_rounds * job.B && *job.n_valid > 0) draw_pixel(job, i / job.B, i % job.B, *job.n_valid);
    return;
  }
  if (kGroup) {
    const int gid = ((int)blockIdx.x * kFitThreads + (int)threadIdx.x) >> 4;
    // the groups of a warp may serve different jobs; an idle group takes part with h = -1
    const RansacJob& job = jobs[hypothesis_job(jobs, n_jobs, min(gid, total - 1))];
    const int h = gid - job.hyp_begin;
    fit_group(job, gid < total && h < job.K && !job_skipped(job.skip) ? h : -1);
    return;
  }
  const int gid = blockIdx.x * blockDim.x + threadIdx.x;
  if (gid >= total) return;
  const RansacJob& job = jobs[hypothesis_job(jobs, n_jobs, gid)];
  const int h = gid - job.hyp_begin;
  if (h >= job.K || job_skipped(job.skip)) return;
  fit_one(job, h);
}

cudaError_t launch_hypotheses(const RansacJob* jobs, int n_jobs, int total_hyps, int32_t* counter, cudaStream_t s,
                              const Schedule& sched, int max_draws) {
  if (total_hyps <= 0) return cudaSuccess;
  static PerDevice resident;  // resident search CTAs per SM on each device
  int sms = 0, per_sm = 0;
  cudaError_t e = device_sms(&sms);
  if (e == cudaSuccess)
    e = per_device(resident, &per_sm, [](int, int* v) {
      cudaError_t r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(v, search_kernel, kSearchWarps * 32, 0);
      *v = std::max(1, *v);
      return r;
    });
  if (e != cudaSuccess) return e;
  if (sched.search_ctas_per_sm < 0) return cudaErrorInvalidValue;
  const int ctas = sched.search_ctas_per_sm == 0 ? per_sm : std::min(per_sm, sched.search_ctas_per_sm);
  e = cudaMemsetAsync(counter, 0, sizeof(int32_t), s);
  if (e != cudaSuccess) return e;
  // warps resident at once against the hypotheses: share each hypothesis among 16 or 4 warps while
  // that keeps to about one and a half rounds of them
  const int slots = sms * ctas * kSearchWarps;
  if (total_hyps <= RELO_SEARCH_WIDE * slots / 32)
    search_shared_kernel<16><<<std::min(total_hyps, std::max(1, slots / 16)), 512, 0, s>>>(jobs, n_jobs, total_hyps, counter);
  else if (total_hyps <= RELO_SEARCH_SHARED * slots / 8)
    search_shared_kernel<4><<<std::min(total_hyps, std::max(1, slots / 4)), 128, 0, s>>>(jobs, n_jobs, total_hyps, counter);
  else
    search_kernel<<<std::min(sms * ctas, (total_hyps + kSearchWarps - 1) / kSearchWarps), kSearchWarps * 32, 0, s>>>(
        jobs, n_jobs, total_hyps, counter);
  const bool group = total_hyps <= kGroupSolves;
  const int per_block = group ? kSolvesPerWarp * kFitThreads / 32 : kFitThreads;
  const int fit_blocks = (total_hyps + per_block - 1) / per_block, draw_blocks = (max_draws + kFitThreads - 1) / kFitThreads;
  const unsigned fit_grid = (unsigned)fit_blocks + (unsigned)draw_blocks * (unsigned)n_jobs;
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_chained(true, group ? fit_kernel<true> : fit_kernel<false>, fit_grid, kFitThreads, 0, s, jobs, n_jobs,
                        total_hyps, fit_blocks, draw_blocks);
}

// ---------------------------------------------------------------------------------------------
// Rounds
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ const int32_t* alive_in(const RansacJob& j, int r) { return (r & 1) ? j.alive_b : j.alive_a; }
__device__ __forceinline__ int32_t* alive_out(const RansacJob& j, int r) { return (r & 1) ? j.alive_a : j.alive_b; }

// Draw round r's B pixels, one CTA per job.
__device__ __forceinline__ void draw_block(const RansacJob* __restrict__ jobs, const int32_t* __restrict__ alive_prefix,
                                           int r, int jid) {
  if (alive_prefix[jid + 1] - alive_prefix[jid] == 0) return;
  const RansacJob& job = jobs[jid];
  if (job_skipped(job.skip)) return;
  const int n_valid = *job.n_valid;
  if (n_valid == 0) return;
  for (int i = threadIdx.x; i < job.B; i += blockDim.x) draw_pixel(job, r, i, n_valid);
}

__global__ void draw_kernel(const RansacJob* __restrict__ jobs, const int32_t* __restrict__ alive_prefix, int r) {
  draw_block(jobs, alive_prefix, r, blockIdx.x);
}

// A pixel's modes, staged by its warp in shared memory: the warp copies every mode of the pixel's
// leaves (trees in order, modes in order), then every lane scores them from there, instead of each
// mode being a dependent global load in turn.  A pixel's staging is two dependent L2 round trips
// (its record's mode ranges, then the modes), which is what bound the round kernels: the copies are
// asynchronous into two slots per warp, so that the next pixel's modes arrive while this one is
// scored, and the ranges are read a pixel earlier still.
constexpr int kStageModes = 64;  // modes per warp slot (two slots of 8 warps take 48 KB, what a static array may);
                                 // a pixel with more is scored from global memory, which takes two to three times
                                 // as long (4 trees of 16 modes, 64 hypotheses, 500 pixels: 270 us staged, 731 not)

struct ModeSlot {
  float4 m[kStageModes * 3];
};
struct ModeSlots {
  ModeSlot s[2];
};

__device__ __forceinline__ void copy_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// (first mode, mode count) of a pixel record's leaf in tree `lane` (lanes below T; 0 elsewhere).
__device__ __forceinline__ int2 mode_range(const int4* __restrict__ rec, int T, int lane) {
  return lane < T ? __ldg(reinterpret_cast<const int2*>(rec + 1) + lane) : make_int2(0, 0);
}

// Starts the copies of the modes of a pixel with ranges `range` into slot (all lanes of the warp
// take part); returns their number, or -1 if they do not fit (then nothing is staged).
__device__ __forceinline__ int stage_modes(const RansacJob& job, int2 range, ModeSlot& slot, int lane) {
  const ForestView& f = job.forest;
  const int total = warp_sum_i(range.y);
  if (total > kStageModes) return -1;
  int off = 0;
  for (int t = 0; t < f.T; ++t) {
    const int first = __shfl_sync(0xffffffffu, range.x, t), nm = __shfl_sync(0xffffffffu, range.y, t);
    const float4* src = reinterpret_cast<const float4*>(f.modes + (size_t)first * kModeFloats);
    for (int i = lane; i < 3 * nm; i += 32) copy_async16(&slot.m[3 * off + i], src + i);
    off += nm;
  }
  return total;
}

// Gaussian score of one mode (a, b, c: its 3 float4) at x.
__device__ __forceinline__ float mode_score(float4 a, float4 b, float4 c, float3 x) {
  const float dx = x.x - a.x, dy = x.y - a.y, dz = x.z - a.z;
  // a.w = inv_xx, b = (inv_xy, inv_xz, inv_yy, inv_yz), c = (inv_zz, logw - 0.5 log det, w, pad)
  const float q = dx * (a.w * dx + b.x * dy + b.y * dz) + dy * (b.x * dx + b.z * dy + b.w * dz) +
                  dz * (b.y * dx + b.w * dy + c.x * dz);
  return c.y - 0.5f * q;
}

// Best mode of a drawn pixel (its record) under x = P c, over trees then modes in order (the first
// of equal scores wins), read from global memory: its score (-inf if none) and mean.
__device__ __forceinline__ float record_best_global(const RansacJob& job, const int4* __restrict__ rec, float3 x,
                                                    float3* mu_best) {
  float best = -INFINITY;
  const ForestView& f = job.forest;
  for (int t = 0; t < f.T; ++t) {
    const int4 w = __ldg(&rec[1 + t / 2]);
    const int first = (t & 1) ? w.z : w.x, nm = (t & 1) ? w.w : w.y;
    const float4* m = reinterpret_cast<const float4*>(f.modes + (size_t)first * kModeFloats);
    for (int k = 0; k < nm; ++k) {
      const float4 a = __ldg(&m[3 * k]), b = __ldg(&m[3 * k + 1]), c = __ldg(&m[3 * k + 2]);
      const float sc = mode_score(a, b, c, x);
      if (sc > best) {
        best = sc;
        if (mu_best) *mu_best = make_float3(a.x, a.y, a.z);
      }
    }
  }
  return best;
}

__device__ __forceinline__ float3 record_point(const int4* __restrict__ rec) {
  const int4 w = __ldg(&rec[0]);
  return make_float3(__int_as_float(w.x), __int_as_float(w.y), __int_as_float(w.z));
}

// record_best over staged modes by a group of 1 << g lanes (aligned; every lane of it passes the
// same x): lane `sub` of the group scores modes sub, sub + (1 << g), ..., then the group keeps the
// largest score and, among equal ones, the lowest index -- the mode that the scan in order with a
// strict comparison keeps (a NaN score never wins in either).  Returns the score (-inf if none) and,
// in every lane of the group, the mode's mean.
__device__ __forceinline__ float group_best_staged(const ModeSlot& slot, int n_staged, float3 x, int sub, int g,
                                                   float3* mu_best) {
  float best = -INFINITY;
  int bi = -1;
  for (int k = sub; k < n_staged; k += 1 << g) {
    const float sc = mode_score(slot.m[3 * k], slot.m[3 * k + 1], slot.m[3 * k + 2], x);
    if (sc > best) {
      best = sc;
      bi = k;
    }
  }
  for (int o = 1 << g >> 1; o > 0; o >>= 1) {
    const float ob = __shfl_xor_sync(0xffffffffu, best, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (ob > best || (ob == best && oi >= 0 && (bi < 0 || oi < bi))) {
      best = ob;
      bi = oi;
    }
  }
  if (mu_best && bi >= 0) {
    const float4 a = slot.m[3 * bi];
    *mu_best = make_float3(a.x, a.y, a.z);
  }
  return best;
}

// Lanes per hypothesis of a chunk with n of them, as a power of two: a chunk of 32 gives each lane
// one hypothesis; the last rounds, where a job keeps few survivors, share a hypothesis's modes among
// the lanes that would otherwise idle.
__host__ __device__ __forceinline__ int group_log2(int n) { return n > 16 ? 0 : n > 8 ? 1 : n > 4 ? 2 : n > 2 ? 3 : n > 1 ? 4 : 5; }

// Round kernels: a CTA takes up to 32 hypotheses of one job and its warps split the pixels, each
// warp walking every kRoundWarps-th pixel; per-warp partial sums are combined in warp order, so the
// result does not depend on scheduling.
constexpr int kRoundWarps = 8;

// Calls score(i, point, slot, n_staged) for pixels i = first, first + step, ... below end in turn,
// with the pixel's modes staged (n_staged as stage_modes) and the next one's on their way.  rec0:
// record of pixel 0, hs: its int4 words.
template <class F>
__device__ __forceinline__ void for_staged_pixels(const RansacJob& job, const int4* __restrict__ rec0, int hs, int first,
                                                  int end, int step, ModeSlots& slots, int lane, F&& score) {
  const int T = job.forest.T;
  if (first >= end) return;
  const int4* rec = rec0 + (size_t)first * hs;
  int4 point = __ldg(rec);
  int n_staged = stage_modes(job, mode_range(rec, T, lane), slots.s[0], lane);
  copy_commit();
  int2 range = make_int2(0, 0);
  int4 next_point = point;
  if (first + step < end) {
    rec = rec0 + (size_t)(first + step) * hs;
    next_point = __ldg(rec);
    range = mode_range(rec, T, lane);
  }
  int which = 0;
  for (int i = first; i < end; i += step, which ^= 1) {
    int next_staged = 0;
    const int4 c = point;
    __syncwarp();  // the other slot's pixel is scored
    if (i + step < end) next_staged = stage_modes(job, range, slots.s[which ^ 1], lane);
    copy_commit();
    point = next_point;
    if (i + 2 * step < end) {
      rec = rec0 + (size_t)(i + 2 * step) * hs;
      next_point = __ldg(rec);
      range = mode_range(rec, T, lane);
    }
    copy_wait<1>();
    __syncwarp();  // every lane's copies of pixel i have landed
    score(i, make_float3(__int_as_float(c.x), __int_as_float(c.y), __int_as_float(c.z)), slots.s[which], n_staged);
    n_staged = next_staged;
  }
  copy_wait<0>();
}

// Whether a split launch's energies of the job go through its score buffer: the per-pixel scores
// take the re-fit sums' buffer, whose 128 ceil(R B / 64) bytes per hypothesis hold 4 B for R >= 2
// rounds (a job of two hypotheses has one).
__device__ __forceinline__ bool split_scores(const RansacJob& job, int n_split) { return n_split > 1 && job.K > 2; }

// Shared memory of the energies: the warps' mode slots, then (the pixels all scored) their sums.
union EnergyShared {
  ModeSlots slots[kRoundWarps];
  float part[kRoundWarps][32];
};

// Energies of round r for hypotheses chunk * 32 .. + 31 of job jid.  n_split > 1: only the pixels of
// part `split`, whose scores go to the job's score buffer [pixel][alive hypothesis] instead, for
// sum_scores to add in the same order.
__device__ __forceinline__ void energy_block(const RansacJob* __restrict__ jobs, const int32_t* __restrict__ alive_prefix,
                                             int r, int chunk, int jid, int split, int n_split, EnergyShared& sh) {
  const int n_alive = alive_prefix[jid + 1] - alive_prefix[jid];
  if (chunk * 32 >= n_alive) return;
  const RansacJob& job = jobs[jid];
  if (job_skipped(job.skip) || *job.n_valid == 0) return;
  const bool to_scores = split_scores(job, n_split);
  if (!to_scores && split > 0) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n_here = min(32, n_alive - chunk * 32);
  const int g = group_log2(n_here), sub = lane & ((1 << g) - 1);
  const int a = chunk * 32 + (lane >> g);
  const int h = a < n_alive ? alive_in(job, r)[a] : 0;
  const PoseF P = pose_to_float(job.poses + 12 * (size_t)h);
  float sum = 0.f;
  const int rows = (job.B + kRoundWarps - 1) / kRoundWarps, per = (rows + n_split - 1) / n_split;
  const int row0 = to_scores ? split * per : 0, row1 = to_scores ? min(rows, row0 + per) : rows;
  float* scores = reinterpret_cast<float*>(job.refit);
  for_staged_pixels(job, job.pix + (size_t)r * job.B * job.hs, job.hs, row0 * kRoundWarps + warp,
                    min(row1 * kRoundWarps, job.B), kRoundWarps, sh.slots[warp], lane,
                    [&](int i, float3 c, const ModeSlot& slot, int n_staged) {
                      const float3 x = apply(P, c);
                      const float best =
                          n_staged >= 0 ? group_best_staged(slot, n_staged, x, sub, g, nullptr)
                                        : record_best_global(job, job.pix + ((size_t)r * job.B + i) * job.hs, x, nullptr);
                      const float e = fminf(kLogEps, -best);
                      if (to_scores) {
                        if (sub == 0 && a < n_alive) scores[(size_t)i * n_alive + a] = e;
                      } else {
                        sum += e;
                      }
                    });
  if (to_scores) return;
  __syncthreads();  // the slots are read
  if (sub == 0) sh.part[warp][lane >> g] = sum;
  __syncthreads();
  if (warp == 0 && chunk * 32 + lane < n_alive) {
    const int hl = alive_in(job, r)[chunk * 32 + lane];
    if (job.hyp_ok[hl]) {
      float e = 0.f;
#pragma unroll
      for (int w = 0; w < kRoundWarps; ++w) e += sh.part[w][lane];
      job.energy[hl] += (double)e;
    }
  }
}

// Energies of round r: grid (hypothesis chunks, jobs, pixel splits).
// CTAs per SM the compiler must fit for the energies, when set (otherwise the compiler's choice)
#ifdef RELO_ENERGY_MIN_BLOCKS
#define RELO_ENERGY_BOUNDS __launch_bounds__(kRoundWarps * 32, RELO_ENERGY_MIN_BLOCKS)
#else
#define RELO_ENERGY_BOUNDS __launch_bounds__(kRoundWarps * 32)
#endif
__global__ void RELO_ENERGY_BOUNDS energy_kernel(const RansacJob* __restrict__ jobs,
                                                                  const int32_t* __restrict__ alive_prefix, int r) {
  __shared__ EnergyShared sh;
  chain_begin();
  energy_block(jobs, alive_prefix, r, blockIdx.x, blockIdx.y, blockIdx.z, gridDim.z, sh);
}

// The energies of a split round from its per-pixel scores: eight lanes per hypothesis take the sums
// that energy_block's eight warps take (every eighth pixel in turn), added in warp order.
__global__ void __launch_bounds__(256) sum_scores_kernel(const RansacJob* __restrict__ jobs,
                                                         const int32_t* __restrict__ alive_prefix, int r, int n_split) {
  static_assert(kRoundWarps == 8, "eight lanes stand for the warps");
  chain_begin();
  const int jid = blockIdx.y, n_alive = alive_prefix[jid + 1] - alive_prefix[jid];
  const int a = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 3), w = threadIdx.x & 7, lane = threadIdx.x & 31;
  const RansacJob& job = jobs[jid];
  if (n_alive == 0 || !split_scores(job, n_split) || job_skipped(job.skip) || *job.n_valid == 0) return;
  const float* scores = reinterpret_cast<const float*>(job.refit);
  float sum = 0.f;
  if (a < n_alive) {
#pragma unroll 8
    for (int i = w; i < job.B; i += kRoundWarps) sum += scores[(size_t)i * n_alive + a];
  }
  float e = 0.f;
#pragma unroll
  for (int q = 0; q < kRoundWarps; ++q) e += __shfl_sync(0xffffffffu, sum, (lane & 24) + q);
  if (w == 0 && a < n_alive) {
    const int h = alive_in(job, r)[a];
    if (job.hyp_ok[h]) job.energy[h] += (double)e;
  }
}

__device__ __forceinline__ unsigned long long order_key(double e) {
  unsigned long long b = (unsigned long long)__double_as_longlong(e);
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

// Whether (ka, ia) sorts after (kb, ib).
__device__ __forceinline__ bool sorts_after(unsigned long long ka, int ia, unsigned long long kb, int ib) {
  return ka > kb || (ka == kb && ia > ib);
}

// Halving: CTA per job, bitonic sort of (energy key, index) ascending; keep ceil(n/2).  Up to one
// hypothesis per thread the pairs stay in registers: the network's strides below 32 are shuffles, and
// only the larger ones (15 of the 55 steps at 1024) go through shared memory with barriers.
__device__ __forceinline__ void select_block(const RansacJob* __restrict__ jobs, const int32_t* __restrict__ alive_prefix,
                                             int r, int jid, unsigned long long* skey) {
  const int n = alive_prefix[jid + 1] - alive_prefix[jid];
  if (n == 0) return;
  const RansacJob& job = jobs[jid];
  if (job_skipped(job.skip)) return;
  int npow = 32;
  while (npow < n) npow <<= 1;
  int* sidx = reinterpret_cast<int*>(skey + npow);
  const int32_t* in = alive_in(job, r);
  const int keep = (n + 1) / 2;
  int32_t* out = alive_out(job, r);
  if (npow <= (int)blockDim.x) {
    const int i = threadIdx.x;
    const bool on = i < npow;  // whole warps: npow is a multiple of 32
    unsigned long long key = ~0ull;
    int idx = INT_MAX;
    if (i < n) {
      idx = in[i];
      key = order_key(job.energy[idx]);
    }
    for (int k = 2; k <= npow; k <<= 1) {
      for (int jj = k >> 1; jj > 0; jj >>= 1) {
        unsigned long long ok = 0;
        int oi = 0;
        if (jj >= 32) {
          __syncthreads();  // the step before has read
          if (on) {
            skey[i] = key;
            sidx[i] = idx;
          }
          __syncthreads();
          if (on) {
            ok = skey[i ^ jj];
            oi = sidx[i ^ jj];
          }
        } else if (on) {
          ok = __shfl_xor_sync(0xffffffffu, key, jj);
          oi = __shfl_xor_sync(0xffffffffu, idx, jj);
        }
        // the lower of the two places keeps the smaller pair in an ascending run, the larger in a descending one
        const bool lower = (i & jj) == 0, up = (i & k) == 0;
        const bool after = sorts_after(key, idx, ok, oi);
        if (on && after == (lower == up)) {
          key = ok;
          idx = oi;
        }
      }
    }
    if (i < keep) out[i] = idx;
    return;
  }
  for (int i = threadIdx.x; i < npow; i += blockDim.x) {
    if (i < n) {
      const int h = in[i];
      skey[i] = order_key(job.energy[h]);
      sidx[i] = h;
    } else {
      skey[i] = ~0ull;
      sidx[i] = INT_MAX;
    }
  }
  __syncthreads();
  for (int k = 2; k <= npow; k <<= 1) {
    for (int jj = k >> 1; jj > 0; jj >>= 1) {
      for (int i = threadIdx.x; i < npow; i += blockDim.x) {
        const int l = i ^ jj;
        if (l > i) {
          const bool up = (i & k) == 0;
          const bool gt = sorts_after(skey[i], sidx[i], skey[l], sidx[l]);
          if (gt == up) {
            const unsigned long long tk = skey[i];
            skey[i] = skey[l];
            skey[l] = tk;
            const int ti = sidx[i];
            sidx[i] = sidx[l];
            sidx[l] = ti;
          }
        }
      }
      __syncthreads();
    }
  }
  for (int i = threadIdx.x; i < keep; i += blockDim.x) out[i] = sidx[i];
}

__global__ void __launch_bounds__(1024) select_kernel(const RansacJob* __restrict__ jobs,
                                                      const int32_t* __restrict__ alive_prefix, int r) {
  extern __shared__ unsigned long long skey[];
  chain_begin();
  select_block(jobs, alive_prefix, r, blockIdx.x, skey);
}

// Re-fit sums over all pixels drawn in rounds 0..r: grid (survivor chunks, parts of kRefinePixels
// pixels, jobs).  Sums are taken about a reference correspondence (the first drawn pixel and its
// predicted scene point) so one FP32 pass gives well-conditioned centroids and cross-covariance:
//   refit[h][part] = {n, sum dc (3), sum dw (3), sum dc dw^T (9)},  refit_ref[h] = {c_ref, w_ref}.
// s + e accumulates x: the rounding error of each addition is carried in e (Neumaier 1974), with
// explicitly rounded operations so that no contraction changes the error terms.
__device__ __forceinline__ void comp_add(float& s, float& e, float x) {
  const float t = __fadd_rn(s, x);
  const float err = fabsf(s) >= fabsf(x) ? __fadd_rn(__fsub_rn(s, t), x) : __fadd_rn(__fsub_rn(x, t), s);
  e = __fadd_rn(e, err);
  s = t;
}

// Squared distance with explicitly rounded operations, so that every kernel taking the inlier
// decision takes it on the same bits.
__device__ __forceinline__ float dist2_rn(float3 a, float3 b) {
  const float dx = __fsub_rn(a.x, b.x), dy = __fsub_rn(a.y, b.y), dz = __fsub_rn(a.z, b.z);
  return __fmaf_rn(dx, dx, __fmaf_rn(dy, dy, __fmul_rn(dz, dz)));
}

// Shared memory of the re-fit sums: the warps' mode slots, then (the pixels all scored) their sums.
union RefineShared {
  ModeSlots slots[kRoundWarps];
  float red[kRoundWarps][16][32];
};

// LG: a hypothesis's modes and its sixteen sums are shared among 1 << LG lanes (lane `sub` carries
// sums sub, sub + (1 << LG), ...), so a CTA takes 32 >> LG survivors.  Every sum sees the same
// additions in the same order whatever LG is.
template <int LG>
__device__ __forceinline__ void refine_block(const RansacJob* __restrict__ jobs, const int32_t* __restrict__ surv_prefix,
                                             int r, int chunk, int part, int jid, RefineShared& sh) {
  constexpr int kHere = 32 >> LG, kGroup = 1 << LG, kSums = LG < 4 ? 16 >> LG : 1;
  const int n_surv = surv_prefix[jid + 1] - surv_prefix[jid];
  if (chunk * kHere >= n_surv) return;
  const RansacJob& job = jobs[jid];
  const int n_drawn = (r + 1) * job.B;
  const int p0 = part * kRefinePixels;
  if (p0 >= n_drawn || job_skipped(job.skip) || *job.n_valid == 0) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int sub = lane & (kGroup - 1), slot_h = lane >> LG;
  const int a = chunk * kHere + slot_h;
  const int h = a < n_surv ? alive_out(job, r)[a] : 0;
  const PoseF P = pose_to_float(job.poses + 12 * (size_t)h);
  const float r2 = (float)(job.inlier_dist * job.inlier_dist);
  const float3 cref = record_point(job.pix);
  const float3 wref = apply(P, cref);
  // Each sum is carried as hi + lo in FP32, compensated: products are split exactly into their
  // rounded value and its error (fmaf), and every addition's rounding error is kept (Neumaier's
  // variant of Kahan summation), so the sums hold about twice FP32's precision.  The sums are taken
  // relative to the first drawn pixel; with plain FP32 sums their cancellation against the small
  // spread of a few inliers moved ill-conditioned re-fits by ~1e-4 rad.
  float acc[kSums], lo[kSums];
#pragma unroll
  for (int q = 0; q < kSums; ++q) acc[q] = lo[q] = 0.f;
  for_staged_pixels(
      job, job.pix, job.hs, p0 + warp, min(p0 + kRefinePixels, n_drawn), kRoundWarps, sh.slots[warp], lane,
      [&](int i, float3 c, const ModeSlot& slot, int n_staged) {
        const float3 x = apply(P, c);
        float3 mu = make_float3(0.f, 0.f, 0.f);
        const float best = n_staged >= 0 ? group_best_staged(slot, n_staged, x, sub, LG, &mu)
                                         : record_best_global(job, job.pix + (size_t)i * job.hs, x, &mu);
        if (best == -INFINITY || !(dist2_rn(x, mu) < r2)) return;
        const float u[3] = {c.x - cref.x, c.y - cref.y, c.z - cref.z};
        const float w[3] = {mu.x - wref.x, mu.y - wref.y, mu.z - wref.z};
#pragma unroll
        for (int k = 0; k < kSums; ++k) {
          const int q = LG == 0 ? k : sub + k * kGroup;  // 0: count, 1..3: u, 4..6: w, 7..15: u w^T
          if (LG > 4 && q > 15) continue;
          float first = 1.f, second = 1.f;
          if (q >= 7) {
            const int p = (q - 7) / 3, m = (q - 7) - 3 * p;
            first = p == 0 ? u[0] : p == 1 ? u[1] : u[2];
            second = m == 0 ? w[0] : m == 1 ? w[1] : w[2];
          } else if (q > 0) {
            first = q == 1 ? u[0] : q == 2 ? u[1] : q == 3 ? u[2] : q == 4 ? w[0] : q == 5 ? w[1] : w[2];
          }
          // (a product with 1 is exact and its error is 0)
          const float pr = __fmul_rn(first, second);
          comp_add(acc[k], lo[k], pr);
          if (LG > 0 || q >= 7) lo[k] = __fadd_rn(lo[k], __fmaf_rn(first, second, -pr));
        }
      });
  // warps w then write sums q = w, w + kRoundWarps: the kRoundWarps partials added in warp order,
  // compensated as above (first their high parts, then their low parts: one shared buffer, two
  // passes), kept as a (high, low) pair that the re-fit adds in FP64
  constexpr int kPer = (16 + kRoundWarps - 1) / kRoundWarps;
  float s_hi[kPer], s_lo[kPer];
#pragma unroll
  for (int i = 0; i < kPer; ++i) s_hi[i] = s_lo[i] = 0.f;
#pragma unroll
  for (int pass = 0; pass < 2; ++pass) {
    __syncthreads();  // the slots, then the first pass's partials, are read
#pragma unroll
    for (int k = 0; k < kSums; ++k)
      if (LG <= 4 || sub + k * kGroup < 16) sh.red[warp][sub + k * kGroup][slot_h] = pass ? lo[k] : acc[k];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int q = warp + i * kRoundWarps;
      if (q < 16 && lane < kHere)
#pragma unroll
        for (int w = 0; w < kRoundWarps; ++w) {
          if (pass == 0) comp_add(s_hi[i], s_lo[i], sh.red[w][q][lane]);
          else s_lo[i] = __fadd_rn(s_lo[i], sh.red[w][q][lane]);
        }
    }
  }
  if (part == 0 && warp == 0 && sub == 0 && a < n_surv && job.hyp_ok[h]) {
    float* ref = job.refit_ref + (size_t)h * 8;
    ref[0] = cref.x;
    ref[1] = cref.y;
    ref[2] = cref.z;
    ref[3] = wref.x;
    ref[4] = wref.y;
    ref[5] = wref.z;
  }
  if (lane >= kHere || chunk * kHere + lane >= n_surv) return;
  const int hl = alive_out(job, r)[chunk * kHere + lane];
  if (!job.hyp_ok[hl]) return;
#pragma unroll
  for (int i = 0; i < kPer; ++i) {
    const int q = warp + i * kRoundWarps;
    if (q < 16) job.refit[((size_t)hl * job.refit_parts + part) * 16 + q] = make_float2(s_hi[i], s_lo[i]);
  }
}

// CTAs per SM the compiler must fit for the re-fit sums of one lane per survivor (the 16 compensated
// sums per lane take registers); with more lanes per survivor a lane holds fewer and more CTAs fit
#ifndef RELO_REFINE_MIN_BLOCKS
#define RELO_REFINE_MIN_BLOCKS 2
#endif
#ifndef RELO_REFINE_FEW_MIN_BLOCKS
#define RELO_REFINE_FEW_MIN_BLOCKS 4
#endif
template <int LG>
__global__ void __launch_bounds__(kRoundWarps * 32, LG == 0 ? RELO_REFINE_MIN_BLOCKS : LG == 1 ? 3 : RELO_REFINE_FEW_MIN_BLOCKS)
    refine_kernel(const RansacJob* __restrict__ jobs, const int32_t* __restrict__ surv_prefix, int r) {
  __shared__ RefineShared sh;
  chain_begin();
  refine_block<LG>(jobs, surv_prefix, r, blockIdx.x, blockIdx.y, blockIdx.z, sh);
}

// Re-fit solve: thread per survivor; the parts' sums are added in order in FP64, then FP64 Horn on
// the centroids and cross-covariance (>= 3 inliers, else the pose is kept).  CTAs of one warp take
// `per` survivors each: with few survivors (late rounds) they spread over the SMs, whose FP64 pipes
// would otherwise run one warp's solves in series.
// Re-fit of survivor k of job `job` after round r.
__device__ __forceinline__ void refit_one(const RansacJob& job, int k, int r) {
  if (job_skipped(job.skip)) return;
  const int h = alive_out(job, r)[k];
  if (!job.hyp_ok[h] || *job.n_valid == 0) return;
  const int parts = ((r + 1) * job.B + kRefinePixels - 1) / kRefinePixels;
  double f[16];
  for (int q = 0; q < 16; ++q) f[q] = 0.0;
  for (int p = 0; p < parts; ++p) {
    const float2* src = job.refit + ((size_t)h * job.refit_parts + p) * 16;
    for (int q = 0; q < 16; ++q) f[q] += (double)src[q].x + (double)src[q].y;
  }
  job.inliers[h] = (int)f[0];
  const double n = f[0];
  if (n < 3.0) return;
  const float* ref = job.refit_ref + (size_t)h * 8;
  double mc[3], mw[3], cb[3], wb[3], S[9];
  for (int k = 0; k < 3; ++k) {
    mc[k] = f[1 + k] / n;
    mw[k] = f[4 + k] / n;
    cb[k] = (double)ref[k] + mc[k];
    wb[k] = (double)ref[3 + k] + mw[k];
  }
  for (int p = 0; p < 3; ++p)
    for (int q = 0; q < 3; ++q) S[3 * p + q] = __fma_rn(-__dmul_rn(n, mc[p]), mw[q], f[7 + 3 * p + q]);
  horn_pose(S, cb, wb, job.poses + 12 * (size_t)h);
}

// refit_one of two survivors by a warp (survivor k by the group of 16 lanes; k < 0: none): lane q of
// the group adds up sum q.
__device__ __forceinline__ void refit_group(const RansacJob& job, int k, int r) {
  const int l = threadIdx.x & 15;
  int h = -1;
  if (k >= 0 && !job_skipped(job.skip) && *job.n_valid != 0) {
    h = alive_out(job, r)[k];
    if (!job.hyp_ok[h]) h = -1;
  }
  double f = 0.0, ref = 0.0;
  if (h >= 0) {
    const int parts = ((r + 1) * job.B + kRefinePixels - 1) / kRefinePixels;
    const float2* src = job.refit + (size_t)h * job.refit_parts * 16 + l;
#pragma unroll 16
    for (int p = 0; p < parts; ++p) {
      const float2 v = src[16 * p];
      f = __dadd_rn(f, __dadd_rn((double)v.x, (double)v.y));
    }
    if (l >= 1 && l < 7) ref = (double)job.refit_ref[(size_t)h * 8 + l - 1];
  }
  __syncwarp();
  const double n = group_get(f, 0);
  if (h >= 0 && l == 0) job.inliers[h] = (int)n;
  const bool solve = h >= 0 && !(n < 3.0);
  const double mean = __ddiv_rn(f, n);  // lanes 1..3: of the camera points, 4..6: of the scene points
  const double centre = __dadd_rn(ref, mean);
  double cb[3], wb[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    cb[q] = group_get(centre, 1 + q);
    wb[q] = group_get(centre, 4 + q);
  }
  // lane 3 p + q: S(p, q) = f[7 + 3 p + q] - n mc[p] mw[q]
  const int p = min(l / 3, 2), q = l - 3 * (l / 3);
  const double sum = group_get(f, min(7 + l, 15)), mc = group_get(mean, 1 + p), mw = group_get(mean, 4 + q);
  horn_pose_group(__fma_rn(-__dmul_rn(n, mc), mw, sum), cb, wb, solve, h >= 0 ? job.poses + 12 * (size_t)h : nullptr);
}

__global__ void __launch_bounds__(32) refit_group_kernel(const RansacJob* __restrict__ jobs, int n_jobs,
                                                         const int32_t* __restrict__ surv_prefix, int total, int r) {
  chain_begin();
  const int gid = (int)blockIdx.x * kSolvesPerWarp + ((int)threadIdx.x >> 4);
  const int jid = find_job_by(surv_prefix, n_jobs, min(gid, total - 1));
  refit_group(jobs[jid], gid < total ? gid - surv_prefix[jid] : -1, r);
}

__global__ void __launch_bounds__(32) refit_kernel(const RansacJob* __restrict__ jobs, int n_jobs,
                                                   const int32_t* __restrict__ surv_prefix, int total, int r,
                                                   int per) {
  chain_begin();
  const int gid = blockIdx.x * per + threadIdx.x;
  if ((int)threadIdx.x >= per || gid >= total) return;
  const int jid = find_job_by(surv_prefix, n_jobs, gid);
  refit_one(jobs[jid], gid - surv_prefix[jid], r);
}

template <int LG>
cudaError_t launch_refine(const RansacJob* jobs, int n_jobs, const int32_t* surv_prefix, int max_surv, int parts, int round,
                          cudaStream_t s) {
  constexpr int kHere = 32 >> LG;
  return launch_chained(true, refine_kernel<LG>, dim3((max_surv + kHere - 1) / kHere, parts, n_jobs), kRoundWarps * 32, 0, s,
                        jobs, surv_prefix, round);
}

int energy_splits(int n_jobs, int max_alive, int B) {
  int sms = 0;
  if (device_sms(&sms) != cudaSuccess) sms = 152;
  const int ctas = (max_alive + 31) / 32 * n_jobs, rows = (B + kRoundWarps - 1) / kRoundWarps;
  return std::max(1, std::min(rows, 2 * sms / std::max(1, ctas)));
}

int round_launches(int n_jobs, int max_alive, int B) { return energy_splits(n_jobs, max_alive, B) > 1 ? 5 : 4; }

cudaError_t launch_draw(const RansacJob* jobs, int n_jobs, int round, const int32_t* alive_prefix_dev, cudaStream_t s) {
  draw_kernel<<<n_jobs, 256, 0, s>>>(jobs, alive_prefix_dev, round);
  return cudaGetLastError();
}

cudaError_t launch_round(const RansacJob* jobs, int n_jobs, int round, const int32_t* alive_prefix_dev,
                         int total_alive, int max_alive, const int32_t* surv_prefix_dev, int total_surv, int max_surv,
                         int B, cudaStream_t s, const Schedule& sched, bool after_draw) {
  if (total_alive <= 0) return cudaSuccess;
  if (sched.refit_per < 0 || sched.refit_per > 32) return cudaErrorInvalidValue;
  // few jobs: their pixels are split over more CTAs than the hypothesis chunks make
  const int n_split = energy_splits(n_jobs, max_alive, B);
  // (round 0 follows the draws, which are read with __ldg)
  cudaError_t e = launch_chained(round > 0 && !after_draw, energy_kernel, dim3((max_alive + 31) / 32, n_jobs, n_split), kRoundWarps * 32, 0, s,
                                 jobs, alive_prefix_dev, round);
  if (e == cudaSuccess && n_split > 1)
    e = launch_chained(true, sum_scores_kernel, dim3((max_alive * 8 + 255) / 256, n_jobs), 256, 0, s, jobs, alive_prefix_dev,
                       round, n_split);
  if (e != cudaSuccess) return e;
  int npow = 32;
  while (npow < max_alive) npow <<= 1;
  e = launch_chained(true, select_kernel, n_jobs, std::min(npow, 1024), (size_t)npow * (sizeof(unsigned long long) + sizeof(int)),
                     s, jobs, alive_prefix_dev, round);
  if (e != cudaSuccess) return e;
  const int parts = ((round + 1) * B + kRefinePixels - 1) / kRefinePixels;
  int n_sms = 0;
  e = device_sms(&n_sms);
  if (e != cudaSuccess) return e;
  // Few survivors in all: a hypothesis is shared by more lanes, up to sixteen, while the CTAs leave SMs
  // idle (a house frame's first round: 16 chunks of 32 survivors, one part of 64 pixels).  Re-fit sums of a
  // frame's ten rounds: 320 -> 275 us; batches of 32 attempts and more keep one survivor a lane.
  int lg = group_log2(max_surv);
  while (lg < 4 && (long)((max_surv + (32 >> lg) - 1) / (32 >> lg)) * parts * n_jobs < 2 * n_sms) ++lg;
  switch (lg) {
    case 0: e = launch_refine<0>(jobs, n_jobs, surv_prefix_dev, max_surv, parts, round, s); break;
    case 1: e = launch_refine<1>(jobs, n_jobs, surv_prefix_dev, max_surv, parts, round, s); break;
    case 2: e = launch_refine<2>(jobs, n_jobs, surv_prefix_dev, max_surv, parts, round, s); break;
    case 3: e = launch_refine<3>(jobs, n_jobs, surv_prefix_dev, max_surv, parts, round, s); break;
    case 4: e = launch_refine<4>(jobs, n_jobs, surv_prefix_dev, max_surv, parts, round, s); break;
    default: e = launch_refine<5>(jobs, n_jobs, surv_prefix_dev, max_surv, parts, round, s); break;
  }
  if (e != cudaSuccess) return e;
  if (sched.refit_per == 0 && total_surv <= kGroupSolves)
    return launch_chained(true, refit_group_kernel, (unsigned)((total_surv + kSolvesPerWarp - 1) / kSolvesPerWarp), 32, 0, s,
                          jobs, n_jobs, surv_prefix_dev, total_surv, round);
  const int per = sched.refit_per > 0 ? sched.refit_per
                                     : std::max(1, std::min(32, (total_surv + 2 * n_sms - 1) / (2 * n_sms)));
  return launch_chained(true, refit_kernel, (unsigned)((total_surv + per - 1) / per), 32, 0, s, jobs, n_jobs, surv_prefix_dev,
                        total_surv, round, per);
}

// Tries of every hypothesis of the job (a kept try j counts j + 1, a failed hypothesis max_tries),
// summed by the 32 lanes of a warp; every lane returns the total.
__device__ __forceinline__ unsigned long long job_tries(const RansacJob& job, int lane) {
  unsigned long long tries = 0;
#pragma unroll 8
  for (int q = lane; q < job.K; q += 32)
    tries += job.hyp_ok[q] ? (unsigned long long)job.tries[q] + 1 : job.max_tries;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tries += __shfl_xor_sync(0xffffffffu, tries, o);
  return tries;
}

// Final hypothesis -> result (one thread per job; tries from job_tries).
__device__ __forceinline__ void finalise_one(const RansacJob& job, unsigned long long tries) {
  if (job_skipped(job.skip)) return;
  const int32_t* fin = (job.n_rounds & 1) ? job.alive_b : job.alive_a;
  const int h = fin[0];
  relo_pose_result* res = job.result;
  // everything is loaded before the first store, which would hold the loads back
  double p[12];
#pragma unroll
  for (int q = 0; q < 12; ++q) p[q] = job.poses[12 * (size_t)h + q];
  const double energy = job.energy[h];
  const int32_t inliers = job.inliers[h], up = job.upstream ? *job.upstream : 0, err = *job.err, ok = job.hyp_ok[h];
  const int32_t n_valid = *job.n_valid;
#pragma unroll
  for (int q = 0; q < 12; ++q) res->pose_c2s[q] = p[q];
  res->pose_c2s[12] = res->pose_c2s[13] = res->pose_c2s[14] = 0.0;
  res->pose_c2s[15] = 1.0;
  res->energy = energy;
  res->n_inliers = inliers;
  res->status = up ? up : (err ? RELO_EDEVICE : (ok ? RELO_OK : RELO_ENOTFOUND));
  res->verified = 0;
  res->n_valid = n_valid;
  res->hypothesis = h;
  res->n_rounds = job.n_rounds;
  res->omega = res->omega_a = res->omega_b = res->omega_ab = res->sum_absdiff_mm = 0;
  res->tries = tries;
  res->path = RELO_PATH_FOREST;
  res->pad = 0;
  for (int q = 0; q < 16; ++q) res->rel_a_b[q] = (q % 5 == 0) ? 1.0 : 0.0;
  if (job.has_pose_b) {
    // a_T_b = P_a P_b^-1 with P_b^-1 = [R_b^T | -R_b^T t_b]
    const double* b = job.pose_b;
    double inv[12];
    for (int i = 0; i < 3; ++i) {
      for (int q = 0; q < 3; ++q) inv[4 * i + q] = b[4 * q + i];
      inv[4 * i + 3] = -(b[i] * b[3] + b[4 + i] * b[7] + b[8 + i] * b[11]);
    }
    for (int i = 0; i < 3; ++i)
      for (int q = 0; q < 4; ++q) {
        double acc = (q == 3) ? p[4 * i + 3] : 0.0;
        for (int k = 0; k < 3; ++k) acc += p[4 * i + k] * inv[4 * k + q];
        res->rel_a_b[4 * i + q] = acc;
      }
  }
}

// Warp per job.
__global__ void __launch_bounds__(128) finalise_kernel(const RansacJob* __restrict__ jobs, int n_jobs) {
  chain_begin();
  const int jid = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (jid >= n_jobs) return;
  const RansacJob& job = jobs[jid];
  if (job_skipped(job.skip)) return;
  const unsigned long long tries = job_tries(job, lane);
  if (lane == 0) finalise_one(job, tries);
}

// ---------------------------------------------------------------------------------------------
// One persistent launch for a pass's hypotheses, rounds and results (schedule option).  Warps
// first search hypotheses taken from a counter (as search_kernel); a CTA whose warps find the
// search queue empty then takes items -- (fit | round stage | finalise) x job x chunk -- from a
// host-built list in dependency order.  Before an item runs, one thread waits until the counter of
// the item it depends on (same job) reaches the number of that item's chunks; after it, the CTA
// adds one to its own counter.  An item depends only on items earlier in the list, which threads
// that have started took, so the waits always end -- unless a counter never reaches its target:
// the wait is bounded in time, and one that runs out raises an abort flag that stops every CTA
// (persist_timeout_kernel then reports RELO_ETIMEOUT for the jobs not finalised).  Each item runs
// the same device code as the per-stage kernels, so results are bit-identical.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ int ld_acquire_gpu(const int32_t* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

constexpr int kPersistThreads = kRoundWarps * 32;
static_assert(kPersistThreads == kPersistThreadsHost, "the host's item chunks match the CTA size");
constexpr size_t kPersistSmem = 4096 * (sizeof(unsigned long long) + sizeof(int));  // the largest sort
static_assert(sizeof(EnergyShared) <= kPersistSmem && sizeof(RefineShared) <= kPersistSmem,
              "round stages fit the persistent kernel's shared memory");

__global__ void __launch_bounds__(kPersistThreads, 2) persistent_kernel(PersistArgs a) {
  extern __shared__ __align__(16) unsigned char psm[];
  __shared__ int s_item, s_go;
  const int lane = threadIdx.x & 31;
  volatile int32_t* abort = a.ctrl + 2;
  // phase 1: hypothesis search, one warp per hypothesis
  for (;;) {
    int gw = 0;
    if (lane == 0) gw = *abort ? a.total_hyps : atomicAdd(a.ctrl + 0, 1);
    gw = __shfl_sync(0xffffffffu, gw, 0);
    if (gw >= a.total_hyps) break;
    const int jid = search_one(a.jobs, a.n_jobs, gw, lane);
    __threadfence();
    __syncwarp();
    if (lane == 0) atomicAdd(a.done + jid, 1);
  }
  __syncthreads();
  // phase 2: CTA items
  for (;;) {
    if (threadIdx.x == 0) {
      const int it = atomicAdd(a.ctrl + 1, 1);
      int go = it < a.n_items && !*abort;
      if (go) {
        const PItem pi = a.items[it];
        const unsigned long long t0 = global_ns();
        for (unsigned n = 1; ld_acquire_gpu(a.done + pi.dep) < pi.need; ++n) {
          if ((n & 63) == 0) {
            if (*abort) {
              go = 0;
              break;
            }
            if (global_ns() - t0 > a.timeout_ns) {
              atomicExch(a.ctrl + 2, 1);
              go = 0;
              break;
            }
          }
        }
      }
      s_item = it;
      s_go = go;
    }
    __syncthreads();
    if (!s_go) break;
    __threadfence();
    const PItem it = a.items[s_item];
    const RansacJob& job = a.jobs[it.job];
    const int np = a.n_jobs + 1;
    switch (it.kind) {
      case kItemFit: {
        const int h = it.sub * kPersistThreads + threadIdx.x;
        if (h < job.K && !job_skipped(job.skip)) fit_one(job, h);
        break;
      }
      case kItemDraw:
        draw_block(a.jobs, a.alive_prefix + (size_t)it.round * np, it.round, it.job);
        break;
      case kItemEnergy:
        energy_block(a.jobs, a.alive_prefix + (size_t)it.round * np, it.round, it.sub, it.job, 0, 1,
                     *reinterpret_cast<EnergyShared*>(psm));
        break;
      case kItemSelect:
        select_block(a.jobs, a.alive_prefix + (size_t)it.round * np, it.round, it.job,
                     reinterpret_cast<unsigned long long*>(psm));
        break;
      case kItemRefine:
        refine_block<0>(a.jobs, a.surv_prefix + (size_t)it.round * np, it.round, it.sub, it.part, it.job,
                        *reinterpret_cast<RefineShared*>(psm));
        break;
      case kItemRefit: {
        const int32_t* sp = a.surv_prefix + (size_t)it.round * np;
        const int k = it.sub * kPersistThreads + threadIdx.x;
        if (k < sp[it.job + 1] - sp[it.job]) refit_one(job, k, it.round);
        break;
      }
      default:
        if (threadIdx.x < 32 && !job_skipped(job.skip)) {
          const unsigned long long tries = job_tries(job, threadIdx.x);
          if (threadIdx.x == 0) finalise_one(job, tries);
        }
        break;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) atomicAdd(a.done + it.done, 1);
  }
}

// After an aborted persistent launch: the jobs it did not finalise report RELO_ETIMEOUT.
__global__ void persist_timeout_kernel(const RansacJob* __restrict__ jobs, int n_jobs, const int32_t* __restrict__ ctrl,
                                       const int32_t* __restrict__ final_done) {
  const int jid = blockIdx.x * blockDim.x + threadIdx.x;
  if (jid >= n_jobs || !ctrl[2]) return;
  const RansacJob& job = jobs[jid];
  if (job_skipped(job.skip) || final_done[jid] != 0) return;
  job.result->status = RELO_ETIMEOUT;
  job.result->verified = 0;
}

// The persistent kernel's CTAs: as many as are resident on the device at once (its shared-memory
// limit is raised here, once per device; batches call this when they are prepared, so that a
// launch inside a stream capture finds it done).
cudaError_t persistent_grid(int* grid) {
  static PerDevice resident;  // resident persistent CTAs per SM on each device
  int sms = 0, per_sm = 0;
  cudaError_t e = device_sms(&sms);
  if (e == cudaSuccess)
    e = per_device(resident, &per_sm, [](int, int* v) {
      cudaError_t r = cudaFuncSetAttribute(persistent_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)kPersistSmem);
      if (r == cudaSuccess)
        r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(v, persistent_kernel, kPersistThreads, kPersistSmem);
      *v = std::max(1, *v);
      return r;
    });
  *grid = sms * per_sm;
  return e;
}

cudaError_t launch_persistent(const PersistArgs& a, int ctrl_words, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(a.ctrl, 0, (size_t)ctrl_words * sizeof(int32_t), s);
  if (e != cudaSuccess) return e;
  int grid = 0;
  e = persistent_grid(&grid);
  if (e != cudaSuccess) return e;
  persistent_kernel<<<grid, kPersistThreads, kPersistSmem, s>>>(a);
  persist_timeout_kernel<<<(a.n_jobs + 127) / 128, 128, 0, s>>>(a.jobs, a.n_jobs, a.ctrl, a.done + a.final_base);
  return cudaGetLastError();
}

// Verification decision (Sec. 3.3.1) from the counts the compare raycast accumulated:
// accept iff |Omega_a| / |Omega| > 1/2 and the mean |D_a - D_b| over Omega_ab is below 50 mm
// (an empty Omega_ab rejects), in integers.
__device__ __forceinline__ void decide(relo_pose_result* res, unsigned long long omega) {
  res->omega = omega;
  res->verified = (res->status == RELO_OK && 2 * res->omega_a > res->omega && res->omega_ab > 0 &&
                   res->sum_absdiff_mm < 50ull * res->omega_ab)
                      ? 1
                      : 0;
}

__global__ void verify_decide_kernel(const RansacJob* __restrict__ jobs, int n_jobs) {
  const int jid = blockIdx.x * blockDim.x + threadIdx.x;
  if (jid >= n_jobs || job_skipped(jobs[jid].skip)) return;
  // a bound failure in the verification raycast (it reports into the job's word) voids the result
  if (jobs[jid].err && *jobs[jid].err) jobs[jid].result->status = RELO_EDEVICE;
  decide(jobs[jid].result, (unsigned long long)jobs[jid].vW * jobs[jid].vH);
}

__global__ void verify_decide_one_kernel(relo_pose_result* res, unsigned long long omega) { decide(res, omega); }

cudaError_t launch_verify_decide(const RansacJob* jobs, int n_jobs, cudaStream_t s) {
  verify_decide_kernel<<<(n_jobs + 127) / 128, 128, 0, s>>>(jobs, n_jobs);
  return cudaGetLastError();
}

cudaError_t launch_verify_decide_one(relo_pose_result* res, uint64_t omega, cudaStream_t s) {
  verify_decide_one_kernel<<<1, 1, 0, s>>>(res, (unsigned long long)omega);
  return cudaGetLastError();
}

cudaError_t launch_finalise(const RansacJob* jobs, int n_jobs, cudaStream_t s) {
  if (n_jobs <= 0) return cudaSuccess;
  return launch_chained(true, finalise_kernel, (n_jobs + 3) / 4, 128, 0, s, jobs, n_jobs);
}

// Fallback results start as "not run" (a skipped job writes nothing).
__global__ void init_results_kernel(relo_pose_result* res, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  res[i].status = RELO_ENOTFOUND;
  res[i].verified = 0;
}

cudaError_t launch_init_results(relo_pose_result* res, int n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  init_results_kernel<<<(n + 127) / 128, 128, 0, s>>>(res, n);
  return cudaGetLastError();
}

// kind[i]: 0 forest only (fallback[i] holds the result), 1 learned without forest, 2 learned with
// a forest fallback.  A learned attempt keeps its learned result when it verified.
__global__ void merge_results_kernel(const relo_pose_result* learned, const relo_pose_result* fallback,
                                     const int32_t* kind, int n, relo_pose_result* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int k = kind[i];
  if (k == 0) {
    out[i] = fallback[i];
    out[i].path = RELO_PATH_FOREST;
  } else if (k == 1 || learned[i].verified) {
    out[i] = learned[i];
    out[i].path = RELO_PATH_LEARNED;
  } else {
    out[i] = fallback[i];
    out[i].path = RELO_PATH_FALLBACK;
  }
}

cudaError_t launch_merge_results(const relo_pose_result* learned, const relo_pose_result* fallback,
                                 const int32_t* kind, int n, relo_pose_result* out, cudaStream_t s) {
  merge_results_kernel<<<(n + 127) / 128, 128, 0, s>>>(learned, fallback, kind, n, out);
  return cudaGetLastError();
}

RELO_DEFINE_CHECK_READER(check_failures_ransac)

}  // namespace relo
