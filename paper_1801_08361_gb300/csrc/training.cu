// training.cu -- leaf reservoirs of the relocaliser's online training (Sec. 3.3 (b)), on the device.
//
// A training frame offers each valid grid pixel's scene coordinate to its leaf in every tree, in
// raster order; a leaf's n-th offer replaces reservoir slot floor(word * (n + 1) / 2^32) of a
// counter-based draw (Algorithm R), so an offer's fate depends only on its rank among its leaf's
// offers.  Ranks come from a stable sort of the pixels by leaf (least significant digit first, 8 bits
// a pass: two passes for up to 65536 leaves): equal leaves end up adjacent and in raster order.  Each
// leaf's run is then applied by one warp, 32 offers at a time, the last of equal slots winning, which
// leaves what offering them one by one would leave.
//
// The sort moves 16 B per pixel, tree and pass (a 320 x 240 frame of five trees: 25 MB in all, in the
// L2), so a frame is bound by its eight short launches: about 0.13 ms, against 4.7 ms when the leaves
// went to the host and its reservoirs.
#include <cuda_runtime.h>
#include <stdint.h>

#include "relo_internal.cuh"

namespace relo {

namespace {

constexpr int kSortThreads = 256, kSortWarps = kSortThreads / 32;

// Item i of tree t in pass 0 (grid pixel i, raster order): false where the pixel has no depth.
__device__ __forceinline__ bool first_item(const ReservoirFrame& f, int t, int64_t i, uint64_t* item) {
  const int v = (int)(i / f.gw) * f.stride, u = (int)(i % f.gw) * f.stride;
  if (__ldg(&f.depth[(size_t)v * f.W + u]) == 0) return false;
  *item = ((uint64_t)__ldg(&f.leaves[(size_t)t * f.n + i]) << 32) | (uint64_t)i;
  return true;
}

// Item i of tree t entering the given pass; false beyond the tree's items.
__device__ __forceinline__ bool load_item(const ReservoirFrame& f, int pass, int t, int64_t i, uint64_t* item) {
  if (pass == 0) return i < f.n && first_item(f, t, i, item);
  if (i >= f.n || i >= f.n_valid[t]) return false;
  *item = f.items[0][(size_t)t * f.n + i];
  return true;
}

__device__ __forceinline__ int digit_of(uint64_t item, int pass) { return (int)(item >> (32 + 8 * pass)) & 0xFF; }

// Digit counts per block: hist[t][block][digit].
__global__ void __launch_bounds__(kSortThreads) sort_count_kernel(ReservoirFrame f, int pass) {
  __shared__ uint32_t h[256];
  const int t = blockIdx.y;
  h[threadIdx.x] = 0;
  __syncthreads();
  for (int r = 0; r < f.per_block; r += kSortThreads) {
    uint64_t item;
    if (load_item(f, pass, t, (int64_t)blockIdx.x * f.per_block + r + threadIdx.x, &item))
      atomicAdd(&h[digit_of(item, pass)], 1u);
  }
  __syncthreads();
  f.hist[((size_t)t * f.blocks + blockIdx.x) * 256 + threadIdx.x] = h[threadIdx.x];
}

// Stable scatter by the pass's digit: each warp takes an eighth of its block's items, in order.  The
// blocks are few (kSortBlocks at most), so each one adds up the counts before its own items by itself
// (a kernel that scanned them took 16 us a pass, most of it its barriers).
__global__ void __launch_bounds__(kSortThreads) sort_scatter_kernel(ReservoirFrame f, int pass) {
  __shared__ uint32_t at[kSortWarps][256];
  __shared__ uint32_t s_warp[kSortWarps];
  const int t = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int w = 0; w < kSortWarps; ++w) at[w][threadIdx.x] = 0;
  // thread d: digit d's items in the tree, and those of the blocks before this one
  const uint32_t* h = f.hist + (size_t)t * f.blocks * 256 + threadIdx.x;
  uint32_t all = 0, before = 0;
#pragma unroll 8
  for (int b = 0; b < f.blocks; ++b) {
    const uint32_t c = h[(size_t)b * 256];
    all += c;
    before += b < (int)blockIdx.x ? c : 0;
  }
  uint32_t scan = all;  // inclusive over the digits
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, scan, o);
    if (lane >= o) scan += y;
  }
  if (lane == 31) s_warp[warp] = scan;
  __syncthreads();
  uint32_t lower = 0, total = 0;
#pragma unroll
  for (int w = 0; w < kSortWarps; ++w) {
    lower += w < warp ? s_warp[w] : 0;
    total += s_warp[w];
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) f.n_valid[t] = (int32_t)total;
  const int per_warp = f.per_block / kSortWarps;
  const int64_t first = (int64_t)blockIdx.x * f.per_block + (int64_t)warp * per_warp;
  for (int r = 0; r < per_warp; r += 32) {
    uint64_t item;
    const int digit = load_item(f, pass, t, first + r + lane, &item) ? digit_of(item, pass) : 256;
    const unsigned same = __match_any_sync(0xffffffffu, digit);
    if (digit < 256 && lane == __ffs(same) - 1) at[warp][digit] += __popc(same);
    __syncwarp();
  }
  __syncthreads();
  {
    uint32_t pos = lower + scan - all + before;
    for (int w = 0; w < kSortWarps; ++w) {
      const uint32_t c = at[w][threadIdx.x];
      at[w][threadIdx.x] = pos;
      pos += c;
    }
  }
  __syncthreads();
  uint64_t* out = f.items[pass] + (size_t)t * f.n;
  for (int r = 0; r < per_warp; r += 32) {
    uint64_t item;
    const int digit = load_item(f, pass, t, first + r + lane, &item) ? digit_of(item, pass) : 256;
    const unsigned same = __match_any_sync(0xffffffffu, digit);
    if (digit < 256) out[at[warp][digit] + __popc(same & ((1u << lane) - 1u))] = item;
    __syncwarp();
    if (digit < 256 && lane == __ffs(same) - 1) at[warp][digit] += __popc(same);
    __syncwarp();
  }
}

// Runs of equal leaves in the sorted items: [start, end) per leaf (end is zero before and after a frame).
__global__ void __launch_bounds__(256) leaf_runs_kernel(ReservoirFrame f, int last_pass) {
  const int t = blockIdx.y;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t n = f.n_valid[t];
  if (i >= n) return;
  const uint64_t* items = f.items[last_pass] + (size_t)t * f.n;
  const uint32_t leaf = (uint32_t)(items[i] >> 32);
  const size_t id = ((size_t)(f.tree0 + t) << f.D) + leaf;
  if (i == 0 || (uint32_t)(items[i - 1] >> 32) != leaf) f.start[id] = (int32_t)i;
  if (i == n - 1 || (uint32_t)(items[i + 1] >> 32) != leaf) f.end[id] = (int32_t)(i + 1);
}

// Slot of a leaf's n-th offer, -1 if it is not kept.
__device__ __forceinline__ int offer_slot(const ReservoirFrame& f, int64_t id, int64_t n) {
  if (n < f.capacity) return (int)n;
  const uint4 x = philox4x32_10(make_uint4(3u, (uint32_t)id, (uint32_t)(n & 0xFFFFFFFF), (uint32_t)(n >> 32)), f.key0,
                                f.key1);
  const uint64_t j = ((uint64_t)x.x * (uint64_t)(n + 1)) >> 32;
  return j < (uint64_t)f.capacity ? (int)j : -1;
}

__device__ __forceinline__ void store_sample(const ReservoirFrame& f, float* res, int slot, uint64_t item) {
  const float* w = f.coords + 3 * (size_t)(uint32_t)item;
#pragma unroll
  for (int k = 0; k < 3; ++k) res[3 * (size_t)slot + k] = w[k];
}

// Algorithm R over each leaf's run: a warp per leaf, in steps of 32 offers, for runs up to kWarpRun;
// a longer run (a wall can send thousands of pixels to one leaf) by its whole CTA afterwards, which
// notes each slot's last offer in shared memory and then stores those.  With warps alone the longest
// run set the kernel's time (90 to 620 us a 320 x 240 frame).
constexpr int kWarpRun = 256;
__global__ void __launch_bounds__(256) reservoir_kernel(ReservoirFrame f, int last_pass) {
  extern __shared__ int s_last[];  // [capacity] 1 + the run's last offer to each slot, 0: none
  __shared__ int s_long[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t first = (int64_t)blockIdx.x * 8, n_leaves = (int64_t)f.trees << f.D;
  const int64_t mine = first + warp;
  int s = 0, e = 0;
  const int64_t base_id = (int64_t)f.tree0 << f.D;
  if (mine < n_leaves) {
    e = f.end[base_id + mine];
    s = e > 0 ? f.start[base_id + mine] : 0;
  }
  if (lane == 0) s_long[warp] = e - s > kWarpRun;
  if (e > s && e - s <= kWarpRun) {
    const int64_t id = base_id + mine, seen = f.seen[id];
    const uint64_t* items = f.items[last_pass] + (size_t)(mine >> f.D) * f.n;
    float* res = f.samples + (size_t)id * f.capacity * 3;
    for (int base = s; base < e; base += 32) {
      const int i = base + lane;
      const int slot = i < e ? offer_slot(f, id, seen + (i - s)) : -1;
      // of the offers to one slot the last stays
      const unsigned same = __match_any_sync(0xffffffffu, slot >= 0 ? slot : -1 - lane);
      if (slot >= 0 && lane == 31 - __clz(same)) store_sample(f, res, slot, items[i]);
      __syncwarp();  // this step's stores come before the next step's
    }
  }
  __syncthreads();
  for (int w = 0; w < 8; ++w) {
    if (!s_long[w]) continue;
    const int64_t id = base_id + first + w, seen = f.seen[id];
    const int ls = f.start[id], le = f.end[id];
    const uint64_t* items = f.items[last_pass] + (size_t)((first + w) >> f.D) * f.n;
    float* res = f.samples + (size_t)id * f.capacity * 3;
    for (int k = threadIdx.x; k < f.capacity; k += blockDim.x) s_last[k] = 0;
    __syncthreads();
    for (int i = ls + threadIdx.x; i < le; i += blockDim.x) {
      const int slot = offer_slot(f, id, seen + (i - ls));
      if (slot >= 0) atomicMax(&s_last[slot], i - ls + 1);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < f.capacity; k += blockDim.x)
      if (s_last[k] > 0) store_sample(f, res, k, items[ls + s_last[k] - 1]);
    __syncthreads();
  }
  if (lane == 0 && e > s) {
    const int64_t id = base_id + mine, all = f.seen[id] + (e - s);
    f.seen[id] = all;
    f.count[id] = (int32_t)(all < f.capacity ? all : f.capacity);
    f.end[id] = 0;  // for the next frame
  }
}

}  // namespace

cudaError_t launch_reservoirs(const ReservoirFrame& f, cudaStream_t s) {
  if (f.n <= 0 || f.trees <= 0) return cudaSuccess;
  const dim3 grid((unsigned)f.blocks, (unsigned)f.trees);
  const int passes = f.D > 8 ? 2 : 1;
  for (int pass = 0; pass < passes; ++pass) {
    sort_count_kernel<<<grid, kSortThreads, 0, s>>>(f, pass);
    sort_scatter_kernel<<<grid, kSortThreads, 0, s>>>(f, pass);
  }
  const size_t leaves = (size_t)f.trees << f.D;
  leaf_runs_kernel<<<dim3((unsigned)((f.n + 255) / 256), (unsigned)f.trees), 256, 0, s>>>(f, passes - 1);
  reservoir_kernel<<<(unsigned)((leaves + 7) / 8), 256, (size_t)f.capacity * sizeof(int), s>>>(f, passes - 1);
  return cudaGetLastError();
}

}  // namespace relo
