// Binning of very long tile lists (more than the per-tile sort holds) by their
// nearest entries.  Compositing stops at T < t_eps, so of a list of 100k large
// splats a few dozen entries are ever read; sorting 793M (tile, Gaussian) pairs
// for 38M blended ones took 78 of the 94 ms of an iteration (1752 x 1168, 1M
// Gaussians, a fifth of them large).  Instead:
//   1. the items are depth-sorted once (sort.cu) and split by rank into slabs
//      whose ends grow by sqrt(2), so that a tile's count over the first k
//      slabs grows about as finely;
//   2. every item adds its rectangle to its slab's difference grid (four
//      atomics whatever its size), and a 2D prefix sum turns the grids into
//      (slab, tile) counts;
//   3. each tile keeps the fewest slabs that give it `target` entries, never
//      more than the per-tile sort holds;
//   4. the kept pairs are scattered into per-tile lists, which the per-tile sort
//      then orders by (depth, id) like any other.
// A kept list is a prefix of the tile's full list, so every pixel that stops
// within it gets the full list's result bit for bit, and the backward pass
// never looks further.  A pixel that does not stop before the end of a cut list
// raises its tile's level, and the binning is repeated: level 1 keeps as many
// entries as the per-tile sort holds, level 2 all of them.  A level-2 tile's
// list is gathered by one block that walks the items in depth order, so it
// needs no sort; where so many tiles are left that this would take longer, all
// pairs are binned in full.
#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace gs {

namespace {

constexpr int kThreads = 256;

// An item's id and rectangle, checked in the bounds-checked build.
__device__ __forceinline__ bool item_ok(const PrefixArgs& a, uint32_t id) { return in_bounds(id < a.n); }
__device__ __forceinline__ bool rect_ok(const PrefixArgs& a, int v, ushort4 q) {
  return in_bounds(q.x <= q.z && q.y <= q.w && (int)q.z <= a.map.tiles_x[v] && (int)q.w <= a.tiles_y[v]);
}

__global__ void __launch_bounds__(kThreads) slab_count_kernel(const __grid_constant__ PrefixArgs a) {
  const uint32_t r = blockIdx.x * kThreads + threadIdx.x;
  const uint32_t id = r < a.ranks ? a.sorted[r] : 0u;
  bool live = r < a.ranks && item_ok(a, id) && a.tiles[id] != 0u;
  const int v = a.map.views == 1 || !live ? 0 : (int)(id / (uint32_t)a.map.n_per_view);
  const ushort4 q = live ? a.rects[id] : make_ushort4(0, 0, 0, 0);
  live = live && rect_ok(a, v, q);
  const unsigned act = __ballot_sync(0xFFFFFFFFu, live);
  if (!live) return;
  int s = 0;
  while (r >= a.bound[s]) ++s;
  const int w = a.map.tiles_x[v] + 1;
  int* g = a.diff + (size_t)s * a.grid_cells + a.grid_base[v];
  warp_agg_add(g + q.y * w + q.x, 1, act);
  warp_agg_add(g + q.y * w + q.z, -1, act);
  warp_agg_add(g + q.w * w + q.x, -1, act);
  warp_agg_add(g + q.w * w + q.z, 1, act);
}

// one block per (slab, view)
__global__ void __launch_bounds__(kThreads) slab_integrate_kernel(const __grid_constant__ PrefixArgs a) {
  const int v = blockIdx.y;
  integrate_grid<kThreads>(a.diff + (size_t)blockIdx.x * a.grid_cells + a.grid_base[v], a.map.tiles_x[v],
                           a.tiles_y[v], [](int, int*, int) {});
}

__global__ void __launch_bounds__(kThreads) prefix_choose_kernel(const __grid_constant__ PrefixArgs a) {
  const uint32_t t = blockIdx.x * kThreads + threadIdx.x;
  uint32_t lim = 0u;
  if (t < a.map.tile_base[a.map.views]) {
    int v = 0;
    for (int k = 1; k < a.map.views; ++k)
      if (t >= a.map.tile_base[k]) v = k;
    const uint32_t lt = t - a.map.tile_base[v], tx = (uint32_t)a.map.tiles_x[v];
    const size_t cell = a.grid_base[v] + (size_t)(lt / tx) * (tx + 1) + lt % tx;
    const int level = a.level[t];
    const uint32_t want = level ? (uint32_t)kTileSortCap : a.target, full = a.full[t];
    uint32_t kept = 0u;
    for (int s = 0; level < 2 && s < a.slabs && kept < want; ++s) {
      const uint32_t c = (uint32_t)a.diff[(size_t)s * a.grid_cells + cell];
      if (kept + c > (uint32_t)kTileSortCap) break;
      kept += c;
      lim = a.bound[s];
    }
    if (level >= 2) {
      kept = full;
      a.gather[atomicAdd(a.n_gather, 1ull)] = t;
    }
    a.lim[t] = lim;
    a.kept[t] = kept;
    a.cut[t] = kept < full ? 1 : 0;
  }
  lim = __reduce_max_sync(0xFFFFFFFFu, lim);
  if ((threadIdx.x & 31) == 0 && lim) atomicMax(a.max_lim, (unsigned long long)lim);
}

// one block per item of the first max_lim ranks: large rectangles are spread
// over the block
__global__ void __launch_bounds__(128) prefix_scatter_kernel(const __grid_constant__ PrefixArgs a,
                                                             uint32_t* __restrict__ cursors,
                                                             uint32_t* __restrict__ ids, uint32_t capacity) {
  const uint32_t r = blockIdx.x;
  const uint32_t id = a.sorted[r];
  if (!item_ok(a, id)) return;
  const uint32_t n = a.tiles[id];
  if (n == 0u) return;
  const int v = a.map.views == 1 ? 0 : (int)(id / (uint32_t)a.map.n_per_view);
  const ushort4 q = a.rects[id];
  const uint32_t w = (uint32_t)(q.z - q.x);
  for (uint32_t k = threadIdx.x; k < n; k += 128) {
    const uint32_t t = a.map.tile_base[v] + (q.y + k / w) * (uint32_t)a.map.tiles_x[v] + q.x + k % w;
    if (!in_bounds(t < a.map.tile_base[a.map.views]) || r >= a.lim[t]) continue;
    const uint32_t pos = atomicAdd(&cursors[t], 1u);
    if (pos < capacity) ids[pos] = id;
  }
}

__global__ void __launch_bounds__(kThreads) sort_rects_kernel(const __grid_constant__ PrefixArgs a,
                                                              ushort4* __restrict__ out) {
  const uint32_t r = blockIdx.x * kThreads + threadIdx.x;
  if (r >= a.n) return;
  const uint32_t id = a.sorted[r];
  out[r] = item_ok(a, id) ? a.rects[id] : make_ushort4(0, 0, 0, 0);
}

// One block per level-2 tile: its items in depth order, kGatherItems
// consecutive ranks per thread and round, their places by a block scan.
constexpr int kGatherThreads = 512, kGatherItems = 4;
__global__ void __launch_bounds__(kGatherThreads) prefix_gather_kernel(const __grid_constant__ PrefixArgs a,
                                                                       const ushort4* __restrict__ srects,
                                                                       const uint32_t* __restrict__ offsets,
                                                                       uint32_t* __restrict__ ids, uint32_t capacity) {
  __shared__ uint32_t s_w[2][kGatherThreads / 32];
  const uint32_t t = a.gather[blockIdx.x], n = a.n;
  if (!in_bounds(t < a.map.tile_base[a.map.views])) return;
  int v = 0;
  for (int k = 1; k < a.map.views; ++k)
    if (t >= a.map.tile_base[k]) v = k;
  const uint32_t lt = t - a.map.tile_base[v], tx = lt % (uint32_t)a.map.tiles_x[v], ty = lt / (uint32_t)a.map.tiles_x[v];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t at = offsets[t];
  int buf = 0;
  for (uint32_t r0 = 0; r0 < n; r0 += kGatherThreads * kGatherItems, buf ^= 1) {
    const uint32_t r = r0 + threadIdx.x * kGatherItems;
    unsigned hit = 0u;
    uint32_t id[kGatherItems];
#pragma unroll
    for (int k = 0; k < kGatherItems; ++k) {
      id[k] = 0u;
      if (r + k < n) {
        const ushort4 q = srects[r + k];
        id[k] = a.sorted[r + k];
        const bool view = a.map.views == 1 || (int)(id[k] / (uint32_t)a.map.n_per_view) == v;
        if (view && tx >= q.x && tx < q.z && ty >= q.y && ty < q.w) hit |= 1u << k;
      }
    }
    const uint32_t c = (uint32_t)__popc(hit);
    uint32_t incl = c;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, off);
      if (lane >= off) incl += y;
    }
    if (lane == 31) s_w[buf][warp] = incl;
    __syncthreads();  // (the next round writes the other buffer)
    uint32_t before = 0u, total = 0u;
#pragma unroll
    for (int k = 0; k < kGatherThreads / 32; ++k) {
      const uint32_t x = s_w[buf][k];
      before += k < warp ? x : 0u;
      total += x;
    }
    uint32_t pos = at + before + incl - c;
#pragma unroll
    for (int k = 0; k < kGatherItems; ++k)
      if (hit >> k & 1u) {
        if (pos < capacity) ids[pos] = id[k];
        ++pos;
      }
    at += total;
  }
}

__global__ void full_ranges_kernel(const uint32_t* __restrict__ offsets, const uint32_t* __restrict__ full, int n,
                                   uint2* __restrict__ out) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  out[t] = full[t] ? make_uint2(offsets[t], offsets[t] + full[t]) : make_uint2(0u, 0u);
}

}  // namespace

void prefix_slabs(PrefixArgs& a, uint32_t ranks) {
  a.ranks = ranks;
  a.slabs = 0;
  double b = 256.0;
  do {
    a.bound[a.slabs++] = b < (double)ranks ? (uint32_t)b : ranks;
    b *= 1.4142135623730951;
  } while (a.bound[a.slabs - 1] < ranks && a.slabs < kPrefixSlabs);
  a.bound[a.slabs - 1] = ranks;
}

void launch_prefix_choose(const PrefixArgs& a, cudaStream_t s, int64_t* launches) {
  const int T = (int)a.map.tile_base[a.map.views];
  cudaMemsetAsync(a.diff, 0, sizeof(int) * (size_t)a.slabs * a.grid_cells, s);
  cudaMemsetAsync(a.max_lim, 0, sizeof(unsigned long long), s);
  cudaMemsetAsync(a.n_gather, 0, sizeof(unsigned long long), s);
  slab_count_kernel<<<(a.ranks + kThreads - 1) / kThreads, kThreads, 0, s>>>(a);
  slab_integrate_kernel<<<dim3(a.slabs, a.map.views), kThreads, 0, s>>>(a);
  prefix_choose_kernel<<<(T + kThreads - 1) / kThreads, kThreads, 0, s>>>(a);
  if (launches) *launches += 3;
}

void launch_prefix_scatter(const PrefixArgs& a, uint32_t max_lim, uint32_t* cursors, uint32_t* ids, uint32_t capacity,
                           cudaStream_t s, int64_t* launches) {
  if (max_lim == 0) return;
  prefix_scatter_kernel<<<max_lim, 128, 0, s>>>(a, cursors, ids, capacity);
  if (launches) *launches += 1;
}

void launch_prefix_gather(const PrefixArgs& a, uint32_t n_gather, ushort4* srects, const uint32_t* offsets,
                          uint32_t* ids, uint32_t capacity, cudaStream_t s, int64_t* launches) {
  if (n_gather == 0 || a.n == 0) return;
  sort_rects_kernel<<<(a.n + kThreads - 1) / kThreads, kThreads, 0, s>>>(a, srects);
  prefix_gather_kernel<<<n_gather, kGatherThreads, 0, s>>>(a, srects, offsets, ids, capacity);
  if (launches) *launches += 2;
}

void launch_full_ranges(const uint32_t* offsets, const uint32_t* full, int n, uint2* out, cudaStream_t s) {
  if (n > 0) full_ranges_kernel<<<(n + 255) / 256, 256, 0, s>>>(offsets, full, n, out);
}

cudaError_t prefix_bind_bounds(uint32_t* word) { return bind_bounds_word(word); }

}  // namespace gs
