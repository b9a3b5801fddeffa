// Tile binning by counting scatter and per-tile sort (Sec. III-B.3: screen
// tiles, Gaussians sorted by depth in each tile):
//   1. count:   every (Gaussian, tile) pair of a Gaussian's tile rectangle adds
//               one to its tile's counter,
//   2. scan:    exclusive scan of the tile counters -> list offsets (and the
//               total pair count and the longest list),
//   3. scatter: every pair takes a slot of its tile's list with an atomic
//               cursor and writes its Gaussian id,
//   4. sort:    each tile's list is sorted by (float32 depth bits, id) with a
//               bitonic network: by one warp in registers up to 1024 entries,
//               by a CTA beyond.
// The per-tile keys are unique, so the result is exactly the (tile, depth, id)
// order of a stable sort and does not depend on the scatter's atomic order.
// Counting and scattering expand the rectangles warp-cooperatively, so a
// Gaussian covering thousands of tiles is spread over the whole warp.
#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace gs {

namespace {

constexpr int kBinThreads = 256;
constexpr int kScatterItems = 64;  // items per block of the scatter into lists of few items
constexpr int kScanThreads = 1024;
constexpr int kSortThreads = 128;
constexpr int kSortWarps = kSortThreads / 32;  // tiles per CTA of the per-tile sort
constexpr int kWarpSortMax = 1024;             // lists up to this length are sorted by one warp (32-bit keys)
constexpr int kWarpSort64 = 512;               // ... by their 64-bit keys

// Global tile of tile (tx, ty) of the view that item `it` belongs to.
struct ItemTiles {
  uint32_t base, stride;  // tile_base[v], tiles_x[v]
};
__device__ __forceinline__ ItemTiles item_tiles(const TileMap& map, uint32_t it) {
  if (map.views == 1) return ItemTiles{0u, (uint32_t)map.tiles_x[0]};
  const int v = (int)(it / (uint32_t)map.n_per_view);
  return ItemTiles{map.tile_base[v], (uint32_t)map.tiles_x[v]};
}

// Calls f(item, global tile, active) for every tile of every item's
// rectangle.  Items with more than kBigTiles tiles come from the queue
// the projection built (see the end); the others are expanded by their
// block, ITEMS consecutive items at a time: a block scan of their tile counts
// gives each item's first pair, and the block's threads take consecutive
// pairs (owner found by binary search over the prefix in shared memory), so
// one large splat is spread over the whole block and large splats clustered
// in one region are averaged over ITEMS items.
// f's third argument is the mask of lanes of the calling warp that call f
// together, or Distinct{} when their tiles are known to differ.
struct Distinct {};
constexpr uint32_t kHugeSpread = 256;
template <int ITEMS = kBinThreads, class F>
__device__ __forceinline__ void for_each_pair(int n, const ushort4* __restrict__ rects,
                                              const uint32_t* __restrict__ tiles, const TileMap& map,
                                              const uint32_t* __restrict__ big_queue,
                                              const uint32_t* __restrict__ big_len, F f) {
  __shared__ uint32_t s_excl[ITEMS];
  __shared__ ushort4 s_rect[ITEMS];
  __shared__ ItemTiles s_map[ITEMS];
  __shared__ uint32_t s_wsum[ITEMS / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int base = blockIdx.x * ITEMS; base < n; base += gridDim.x * ITEMS) {
    const bool item = (int)threadIdx.x < ITEMS;
    const int g = base + threadIdx.x;
    uint32_t cnt = item && g < n ? tiles[g] : 0u;
    if (cnt > kBigTiles) cnt = 0;  // expanded from the queue below
    const ushort4 r = item && g < n ? rects[g] : make_ushort4(0, 0, 0, 0);
    uint32_t incl = cnt;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, off);
      if (lane >= off) incl += y;
    }
    __syncthreads();  // previous round done with the shared arrays
    if (item && lane == 31) s_wsum[w] = incl;
    __syncthreads();
    uint32_t wpre = 0, total = 0;
#pragma unroll
    for (int k = 0; k < ITEMS / 32; ++k) {
      const uint32_t sk = s_wsum[k];
      wpre += k < w ? sk : 0u;
      total += sk;
    }
    if (item) {
      s_excl[threadIdx.x] = wpre + incl - cnt;
      s_rect[threadIdx.x] = r;
      s_map[threadIdx.x] = item_tiles(map, (uint32_t)min(g, n - 1));
    }
    __syncthreads();
    for (uint32_t k0 = 0; k0 < total; k0 += kBinThreads) {
      const uint32_t k = k0 + threadIdx.x;
      const unsigned active = __ballot_sync(0xFFFFFFFFu, k < total);
      if (k >= total) break;
      int o = 0;
#pragma unroll
      for (int step = ITEMS / 2; step > 0; step >>= 1)
        if (s_excl[o + step] <= k) o += step;
      const ushort4 ro = s_rect[o];
      const ItemTiles mt = s_map[o];
      const uint32_t local = k - s_excl[o];
      const uint32_t width = (uint32_t)(ro.z - ro.x);
      const uint32_t ty = ro.y + local / width, tx = ro.x + local % width;
      f(base + o, mt.base + ty * mt.stride + tx, active);
    }
  }
  // large splats: warp w of the grid expands queued items w, w + W, ...
  // spreading each one's tiles over its lanes (no shared cursor: one address
  // hit by every warp would serialise)
  const uint32_t nbig = *big_len;
  const uint32_t gwarp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t item = gwarp; item < nbig; item += nwarps) {
    const uint32_t g = big_queue[item];
    const ushort4 ro = rects[g];
    const uint32_t cnt = tiles[g];
    const ItemTiles mt = item_tiles(map, g);
    const uint32_t width = (uint32_t)(ro.z - ro.x);
    auto tile = [&](uint32_t k) { return mt.base + (ro.y + k / width) * mt.stride + ro.x + k % width; };
    if (cnt > kHugeSpread) {
      for (uint32_t k = lane; k < cnt; k += 32) f((int)g, tile(k), Distinct{});
    } else {
      for (uint32_t k0 = 0; k0 < cnt; k0 += 32) {
        const uint32_t k = k0 + lane;
        const unsigned active = __ballot_sync(0xFFFFFFFFu, k < cnt);
        if (k >= cnt) break;
        f((int)g, tile(k), active);
      }
    }
  }
}

// One more at tile t's counter: its value before.  Neighbouring items meet the
// same tiles, so a warp's equal tiles go in one atomic (2.3M pairs: 19 us, 65
// us with an atomic each).  The lanes of a large rectangle never share one, and
// from kHugeSpread tiles on go without the matching (8.6M pairs, most of
// rectangles of 1400 tiles: 206 -> 131 us; below, where queued rectangles of a
// few rounds crowd the same tiles, it was slower: 175 -> 203 us for 12.6M pairs
// of 8 views).
__device__ __forceinline__ uint32_t count_tile(uint32_t* __restrict__ counter, uint32_t t, unsigned active) {
  return warp_agg_inc(counter, t, active);
}
__device__ __forceinline__ uint32_t count_tile(uint32_t* __restrict__ counter, uint32_t t, Distinct) {
  return atomicAdd(&counter[t], 1u);
}

// Every (item, tile) pair adds one to its tile's counter (when the
// projection has not counted them itself, as for gs_bin_tiles).
__global__ void __launch_bounds__(kBinThreads) tile_count_kernel(const __grid_constant__ TileBinArgs a) {
  pdl_enter();
  for_each_pair(a.n, a.rects, a.tiles, a.map, a.big_queue, a.big_len,
                [&](int, uint32_t t, auto active) {
                  // (the checked build counts a tile beyond the grid into tile 0, reported)
                  count_tile(a.counts, in_bounds(t < (uint32_t)a.n_tiles) ? t : 0u, active);
                });
}

// Difference grids of the huge rectangles (TileBinArgs::big_diff).
struct BigGrids {
  int* diff;
  const uint32_t* big_len;
  int views;
  int tiles_x[kMaxViews], tiles_y[kMaxViews];
  uint32_t base[kMaxViews], tile_base[kMaxViews];
};

// Length class of a tile list for the visit order, four per octave: 0 for
// an empty list, else 4 floor(log2 c) + (the two bits after c's leading one)
// + 1, so classes grow with the length and tiles within 19% of each other's
// length share one.  kLenClasses classes (kLenClasses is also the "no tile"
// sentinel; the raster passes' bucket-mode visit order uses the same classes).
__device__ __forceinline__ int length_class(uint32_t c) {
  if (!c) return 0;
  const int lead = 31 - __clz(c);
  const int frac = lead >= 2 ? (int)((c >> (lead - 2)) & 3u) : (int)((c << (2 - lead)) & 3u);
  return 4 * lead + frac + 1;
}

// Adds view v's huge rectangles to the tile counts and leaves its difference
// grid zero (every thread of the block calls it).
template <int THREADS>
__device__ __forceinline__ void add_big_rects(const BigGrids& b, int v, uint32_t* __restrict__ counts) {
  const int TX = b.tiles_x[v], TY = b.tiles_y[v];
  int* g = b.diff + b.base[v];
  integrate_grid<THREADS>(g, TX, TY, [&](int t, int* cell, int n) {
    if (n) counts[b.tile_base[v] + t] += (uint32_t)n;
    *cell = 0;
  });
  for (int x = threadIdx.x; x <= TX; x += THREADS) g[(size_t)TY * (TX + 1) + x] = 0;
  for (int y = threadIdx.x; y < TY; y += THREADS) g[(size_t)y * (TX + 1) + TX] = 0;
}

// one block per view; nothing to do without huge rectangles
__global__ void __launch_bounds__(kScanThreads) big_rects_kernel(const __grid_constant__ BigGrids b,
                                                                 uint32_t* __restrict__ counts) {
  pdl_enter();
  if (b.big_len[kHugeFlag] == 0u) return;
  add_big_rects<kScanThreads>(b, blockIdx.x, counts);
}

// offsets = exclusive scan of counts (clamped to 32 bits), cursors = offsets;
// stats[0] = total pairs, stats[1] = longest list; n_pairs = min(total, capacity).
// order (if non-null) = the tiles by descending length class, the order in
// which the raster passes visit them (longest lists first, so that the
// slowest tiles do not start last).
__global__ void __launch_bounds__(kScanThreads) tile_scan_kernel(int T, uint32_t* counts,
                                                                 uint32_t* __restrict__ offsets,
                                                                 uint32_t* __restrict__ cursors, uint32_t capacity,
                                                                 uint32_t* __restrict__ n_pairs,
                                                                 unsigned long long* __restrict__ stats,
                                                                 uint32_t* __restrict__ order,
                                                                 const __grid_constant__ BigGrids big) {
  pdl_enter();
  if (big.diff && big.big_len[kHugeFlag]) {
    for (int v = 0; v < big.views; ++v) add_big_rects<kScanThreads>(big, v, counts);
    __syncthreads();
  }
  __shared__ unsigned long long s[kScanThreads];
  __shared__ uint32_t s_max[32];
  const int per = (T + kScanThreads - 1) / kScanThreads;
  const int beg = min(T, (int)threadIdx.x * per), end = min(T, beg + per);
  unsigned long long sum = 0;
  uint32_t mx = 0;
  for (int i = beg; i < end; ++i) {
    const uint32_t c = counts[i];
    sum += c;
    mx = max(mx, c);
  }
  s[threadIdx.x] = sum;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) mx = max(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, off));
  if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = mx;
  __syncthreads();
  for (int off = 1; off < kScanThreads; off <<= 1) {
    const unsigned long long v = threadIdx.x >= (unsigned)off ? s[threadIdx.x - off] : 0ull;
    __syncthreads();
    s[threadIdx.x] += v;
    __syncthreads();
  }
  unsigned long long run = s[threadIdx.x] - sum;
  for (int i = beg; i < end; ++i) {
    const uint32_t o = (uint32_t)(run < 0xFFFFFFFFull ? run : 0xFFFFFFFFull);
    offsets[i] = o;
    cursors[i] = o;
    run += counts[i];
  }
  if (threadIdx.x == 0) {
    uint32_t m = 0;
    for (int k = 0; k < kScanThreads / 32; ++k) m = max(m, s_max[k]);
    const unsigned long long tot = s[kScanThreads - 1];
    stats[0] = tot;
    stats[1] = m;
    *n_pairs = (uint32_t)(tot < (unsigned long long)capacity ? tot : (unsigned long long)capacity);
  }
  if (!order) return;
  // counting sort of the tiles by length class, descending; lanes of a warp
  // with the same class are aggregated into one atomic
  __shared__ uint32_t s_cls[kLenClasses];
  const int lane = threadIdx.x & 31;
  if (threadIdx.x < kLenClasses) s_cls[threadIdx.x] = 0;
  __syncthreads();
  for (int i0 = 0; i0 < T; i0 += kScanThreads) {
    const int i = i0 + threadIdx.x;
    const int c = i < T ? length_class(counts[i]) : kLenClasses;
    const unsigned peers = __match_any_sync(0xFFFFFFFFu, c);
    if (c < kLenClasses && lane == __ffs(peers) - 1) atomicAdd(&s_cls[c], (uint32_t)__popc(peers));
  }
  __syncthreads();
  if (threadIdx.x < 32) class_starts_desc(s_cls);
  __syncthreads();
  for (int i0 = 0; i0 < T; i0 += kScanThreads) {
    const int i = i0 + threadIdx.x;
    const int c = i < T ? length_class(counts[i]) : kLenClasses;
    const unsigned peers = __match_any_sync(0xFFFFFFFFu, c);
    const int leader = __ffs(peers) - 1;
    uint32_t base = 0;
    if (c < kLenClasses && lane == leader) base = atomicAdd(&s_cls[c], (uint32_t)__popc(peers));
    base = __shfl_sync(peers, base, leader);
    if (c < kLenClasses) order[base + __popc(peers & ((1u << lane) - 1u))] = (uint32_t)i;
  }
}

// Multi-block form of tile_scan_kernel for many tiles (batches of views):
//   up:   block b sums the counts of its kScanTiles tiles, takes their
//         maximum and the histogram of their length classes;
//   mid:  one block: the total (stats, n_pairs), the longest list and the
//         start of each length class in the visit order (descending);
//   down: block b adds up the earlier blocks' sums and class histograms (in
//         block order) for its bases, then writes offsets, cursors and the
//         visit order of its tiles.
// aux per block: {sum lo, sum hi, max, hist[kLenClasses]}; aux_tail: class starts[kLenClasses].
constexpr int kScanTiles = 1024;
constexpr int kScanAux = 3 + kLenClasses;

__global__ void __launch_bounds__(256) tile_scan_up_kernel(int T, const uint32_t* __restrict__ counts,
                                                           uint32_t* __restrict__ aux) {
  pdl_enter();
  __shared__ uint32_t s_hist[kLenClasses];
  __shared__ unsigned long long s_sum[8];
  __shared__ uint32_t s_max[8];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (threadIdx.x < kLenClasses) s_hist[threadIdx.x] = 0;
  __syncthreads();
  unsigned long long sum = 0;
  uint32_t mx = 0;
  const int i0 = blockIdx.x * kScanTiles;
#pragma unroll
  for (int j = 0; j < kScanTiles / 256; ++j) {
    const int i = i0 + j * 256 + threadIdx.x;
    const uint32_t c = i < T ? counts[i] : 0u;
    sum += c;
    mx = max(mx, c);
    const int cls = i < T ? length_class(c) : kLenClasses;
    const unsigned peers = __match_any_sync(0xFFFFFFFFu, cls);
    if (cls < kLenClasses && lane == __ffs(peers) - 1) atomicAdd(&s_hist[cls], (uint32_t)__popc(peers));
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    sum += __shfl_xor_sync(0xFFFFFFFFu, sum, off);
    mx = max(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, off));
  }
  if (lane == 0) {
    s_sum[wid] = sum;
    s_max[wid] = mx;
  }
  __syncthreads();
  uint32_t* out = aux + (size_t)kScanAux * blockIdx.x;
  if (threadIdx.x == 0) {
    unsigned long long t = 0;
    uint32_t m = 0;
    for (int w = 0; w < 8; ++w) {
      t += s_sum[w];
      m = max(m, s_max[w]);
    }
    out[0] = (uint32_t)t;
    out[1] = (uint32_t)(t >> 32);
    out[2] = m;
  }
  if (threadIdx.x < kLenClasses) out[3 + threadIdx.x] = s_hist[threadIdx.x];
}

__global__ void __launch_bounds__(64) tile_scan_mid_kernel(int nb, const uint32_t* __restrict__ aux,
                                                           uint32_t* __restrict__ aux_tail, uint32_t capacity,
                                                           uint32_t* __restrict__ n_pairs,
                                                           unsigned long long* __restrict__ stats) {
  pdl_enter();
  __shared__ uint32_t s_tot[kLenClasses];
  for (int c = threadIdx.x; c < kLenClasses; c += blockDim.x) {
    uint32_t t = 0;
    for (int b = 0; b < nb; ++b) t += aux[(size_t)kScanAux * b + 3 + c];
    s_tot[c] = t;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long tot = 0;
    uint32_t m = 0;
    for (int b = 0; b < nb; ++b) {
      const uint32_t* a = aux + (size_t)kScanAux * b;
      tot += (unsigned long long)a[0] | ((unsigned long long)a[1] << 32);
      m = max(m, a[2]);
    }
    stats[0] = tot;
    stats[1] = m;
    *n_pairs = (uint32_t)(tot < (unsigned long long)capacity ? tot : (unsigned long long)capacity);
  }
  if (threadIdx.x < 32) {  // longest class first
    class_starts_desc(s_tot);
    __syncwarp();
    for (int c = threadIdx.x; c < kLenClasses; c += 32) aux_tail[c] = s_tot[c];
  }
}

__global__ void __launch_bounds__(256) tile_scan_down_kernel(int T, const uint32_t* __restrict__ counts,
                                                             const uint32_t* __restrict__ aux,
                                                             const uint32_t* __restrict__ aux_tail,
                                                             uint32_t* __restrict__ offsets,
                                                             uint32_t* __restrict__ cursors,
                                                             uint32_t* __restrict__ order) {
  pdl_enter();
  constexpr int PER = kScanTiles / 256;  // consecutive tiles per thread
  __shared__ unsigned long long s_scan[256];
  __shared__ unsigned long long s_base;
  __shared__ uint32_t s_cls[kLenClasses];
  const int b = blockIdx.x, lane = threadIdx.x & 31;
  static_assert(kLenClasses < 255, "thread 255 sums the bases");
  if (threadIdx.x < kLenClasses) {  // start of this block's tiles within each length class
    uint32_t o = aux_tail[threadIdx.x];
    for (int k = 0; k < b; ++k) o += aux[(size_t)kScanAux * k + 3 + threadIdx.x];
    s_cls[threadIdx.x] = o;
  } else if (threadIdx.x == 255) {
    unsigned long long o = 0;
    for (int k = 0; k < b; ++k) {
      const uint32_t* a = aux + (size_t)kScanAux * k;
      o += (unsigned long long)a[0] | ((unsigned long long)a[1] << 32);
    }
    s_base = o;
  }
  const int i0 = b * kScanTiles + threadIdx.x * PER;
  uint32_t c[PER];
  unsigned long long sum = 0;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    c[j] = i0 + j < T ? counts[i0 + j] : 0u;
    sum += c[j];
  }
  s_scan[threadIdx.x] = sum;
  __syncthreads();
  for (int off = 1; off < 256; off <<= 1) {
    const unsigned long long v = threadIdx.x >= (unsigned)off ? s_scan[threadIdx.x - off] : 0ull;
    __syncthreads();
    s_scan[threadIdx.x] += v;
    __syncthreads();
  }
  unsigned long long run = s_base + s_scan[threadIdx.x] - sum;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    if (i0 + j < T) {
      const uint32_t o = (uint32_t)(run < 0xFFFFFFFFull ? run : 0xFFFFFFFFull);
      offsets[i0 + j] = o;
      cursors[i0 + j] = o;
    }
    run += c[j];
  }
  if (!order) return;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const int i = i0 + j;
    const int cls = i < T ? length_class(c[j]) : kLenClasses;
    const unsigned peers = __match_any_sync(0xFFFFFFFFu, cls);
    const int leader = __ffs(peers) - 1;
    uint32_t base = 0;
    if (cls < kLenClasses && lane == leader) base = atomicAdd(&s_cls[cls], (uint32_t)__popc(peers));
    base = __shfl_sync(peers, base, leader);
    if (cls < kLenClasses) order[base + __popc(peers & ((1u << lane) - 1u))] = (uint32_t)i;
  }
}

template <int ITEMS>
__global__ void __launch_bounds__(kBinThreads) tile_scatter_kernel(const __grid_constant__ TileBinArgs a) {
  pdl_enter();
  bool over = false;
  for_each_pair<ITEMS>(a.n, a.rects, a.tiles, a.map, a.big_queue, a.big_len,
                       [&](int g, uint32_t t, auto active) {
                         const uint32_t pos = count_tile(a.cursors, in_bounds(t < (uint32_t)a.n_tiles) ? t : 0u, active);
                         if (pos < a.capacity)
                           a.ids[pos] = (uint32_t)g;
                         else
                           over = true;
                       });
  if (over) atomicOr(a.overflow, 1u);
}

// Bitonic network over the 32 KEYS keys of one warp, sorted ascending.
// Blocked layout: lane l holds elements KEYS l .. KEYS l + KEYS - 1, so the
// compare-exchanges of partner distance j < KEYS stay inside a lane (no
// shuffle) and only the log2(32) largest distances of each merge level cross
// lanes.  Element e is the lower index of its pair when (e & j) == 0 and its
// block ascends when (e & k) == 0.
template <int KEYS>
__device__ __forceinline__ void warp_bitonic(unsigned long long (&x)[KEYS], int lane) {
  constexpr int M = 32 * KEYS;
#pragma unroll
  for (int k = 2; k <= M; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      if (j < KEYS) {
#pragma unroll
        for (int i = 0; i < KEYS; ++i) {
          if ((i & j) == 0) {
            const int p = i | j;
            // (e & k) for e = KEYS lane + i: i's bit when k < KEYS, else the lane's
            const bool up = k < KEYS ? ((i & k) == 0) : (((lane * KEYS) & k) == 0);
            const unsigned long long a = x[i], b = x[p];
            const bool sw = (a > b) == up;
            x[i] = sw ? b : a;
            x[p] = sw ? a : b;
          }
        }
      } else {
        const int d = j / KEYS;  // partner lane distance
        const bool keep_min = ((lane & d) == 0) == (((lane * KEYS) & k) == 0);
#pragma unroll
        for (int i = 0; i < KEYS; ++i) {
          const unsigned long long y = __shfl_xor_sync(0xFFFFFFFFu, x[i], d);
          x[i] = ((x[i] < y) == keep_min) ? x[i] : y;
        }
      }
    }
  }
}

// One warp sorts the list of n <= 32 KEYS ids at ids[off ..] by the key
// (depth bits << 32 | id), padded with all-ones keys to 32 KEYS.
template <int KEYS>
__device__ __forceinline__ void warp_sort_list(uint32_t* __restrict__ ids, const uint32_t* __restrict__ zkey,
                                               uint32_t off, uint32_t n, uint32_t n_items, int lane) {
  unsigned long long x[KEYS];
#pragma unroll
  for (int i = 0; i < KEYS; ++i) {
    const uint32_t e = (uint32_t)(lane * KEYS + i);
    x[i] = ~0ull;
    if (e < n) {
      const uint32_t g = ids[off + e];
      x[i] = in_bounds(g < n_items) ? ((unsigned long long)zkey[g] << 32) | g : ~0ull;
    }
  }
  warp_bitonic<KEYS>(x, lane);
#pragma unroll
  for (int i = 0; i < KEYS; ++i) {
    const uint32_t e = (uint32_t)(lane * KEYS + i);
    if (e < n) ids[off + e] = (uint32_t)x[i];
  }
}

// ---------------------------------------------------------------------------
// The usual sort of a list: 32-bit keys (depth rounded down) << B | place in the
// unsorted list, B bits for n places and the depth in what remains of the bits,
// offset by the list's smallest: a compare-exchange is a minimum and a maximum
// instead of a 64-bit compare and four selects, and half the shuffles.  Entries
// whose rounded depths are equal come out in the order of their places.  Equal
// depths are common (a level camera sees a horizontal plane at one depth per
// pixel row), so in a list that has any the runs of equal rounded depths are
// put in order by (the depth's bits that were rounded off, id): by neighbour
// exchanges within the runs, if these take long by a second sort with the run
// in front, and where the keys do not fit into 32 bits by the 64-bit keys.
//
// The networks' merges start by comparing mirrored places (e with e ^ (k - 1)),
// so every compare-exchange puts the smaller key at the smaller place.  Blocked
// layout as in warp_bitonic.
// ---------------------------------------------------------------------------
template <int KEYS>
__device__ __forceinline__ void lane_merge(uint32_t (&x)[KEYS]) {  // partner distances KEYS / 2 .. 1
#pragma unroll
  for (int j = KEYS / 2; j > 0; j >>= 1)
#pragma unroll
    for (int i = 0; i < KEYS; ++i)
      if ((i & j) == 0) {
        const uint32_t a = x[i], b = x[i | j];
        x[i] = min(a, b);
        x[i | j] = max(a, b);
      }
}

template <int KEYS>
__device__ __forceinline__ void lane_sort(uint32_t (&x)[KEYS]) {
#pragma unroll
  for (int k = 2; k <= KEYS; k <<= 1) {
#pragma unroll
    for (int i = 0; i < KEYS; ++i)
      if ((i & (k >> 1)) == 0) {
        const int p = i ^ (k - 1);
        const uint32_t a = x[i], b = x[p];
        x[i] = min(a, b);
        x[p] = max(a, b);
      }
#pragma unroll
    for (int j = k >> 2; j > 0; j >>= 1)
#pragma unroll
      for (int i = 0; i < KEYS; ++i)
        if ((i & j) == 0) {
          const uint32_t a = x[i], b = x[i | j];
          x[i] = min(a, b);
          x[i | j] = max(a, b);
        }
  }
}

// distances of d lanes down to one lane, then within the lane
template <int KEYS>
__device__ __forceinline__ void warp_merge_from(uint32_t (&x)[KEYS], int lane, int d) {
  for (; d > 0; d >>= 1) {
    const bool lower = (lane & d) == 0;
#pragma unroll
    for (int i = 0; i < KEYS; ++i) {
      const uint32_t y = __shfl_xor_sync(0xFFFFFFFFu, x[i], d);
      x[i] = lower ? min(x[i], y) : max(x[i], y);
    }
  }
  lane_merge(x);
}

// Sorts the first n of the warp's 32 KEYS keys (the others are all ones).
template <int KEYS>
__device__ __forceinline__ void warp_sort32(uint32_t (&x)[KEYS], int lane, uint32_t n) {
  lane_sort(x);
  for (int m = 1; m < 32 && (uint32_t)(KEYS * (m + 1) / 2) < n; m = 2 * m + 1) {
    const bool lower = (lane & ((m + 1) >> 1)) == 0;
#pragma unroll
    for (int i = 0; i < KEYS / 2; ++i) {
      const uint32_t a = __shfl_xor_sync(0xFFFFFFFFu, x[KEYS - 1 - i], m);
      const uint32_t b = __shfl_xor_sync(0xFFFFFFFFu, x[i], m);
      x[i] = lower ? min(x[i], a) : max(x[i], a);
      x[KEYS - 1 - i] = lower ? min(x[KEYS - 1 - i], b) : max(x[KEYS - 1 - i], b);
    }
    warp_merge_from(x, lane, (m + 1) >> 2);
  }
}

// How a list's depths become keys.
struct KeyMap {
  uint32_t zmin;
  int shift, bits;  // (z - zmin) >> shift, then << bits
  __device__ __forceinline__ uint32_t rounded(uint32_t z) const { return (z - zmin) >> shift; }
  __device__ __forceinline__ uint32_t place(uint32_t key) const { return key & ((1u << bits) - 1u); }
  __device__ __forceinline__ bool tie(uint32_t a, uint32_t b) const { return ((a ^ b) >> bits) == 0u; }
};
__device__ __forceinline__ KeyMap key_map(uint32_t n, uint32_t zmin, uint32_t zmax) {
  KeyMap k;
  k.zmin = zmin;
  k.bits = n > 1 ? 32 - __clz(n - 1) : 1;
  const int need = 32 - __clz(zmax - zmin);  // (__clz(0) = 32)
  k.shift = max(0, need - (32 - k.bits));
  return k;
}

// The places' entries: ids[off + place], and whether an entry's rounded depth
// equals that of the one before it (bit i: entry e0 + i); prev: the key before
// the lane's first one.
template <int KEYS>
__device__ __forceinline__ uint32_t sorted_ids_ties(const uint32_t (&x)[KEYS], const uint32_t* ids, uint32_t off,
                                                    uint32_t n, uint32_t e0, const KeyMap& k, uint32_t prev,
                                                    uint32_t (&id)[KEYS]) {
  uint32_t ties = 0u;
#pragma unroll
  for (int i = 0; i < KEYS; ++i) {
    const uint32_t e = e0 + i;
    id[i] = e < n ? ids[off + k.place(x[i])] : 0u;
    if (e > 0 && e < n && k.tie(x[i], i ? x[(i + KEYS - 1) % KEYS] : prev)) ties |= 1u << i;
  }
  return ties;
}

// Second keys of the entries: the depth's bits that were rounded off, id.
struct IdMap {
  uint32_t imin;
  int bits;
  __device__ __forceinline__ uint32_t id(uint32_t key) const {
    return imin + (key & (bits == 32 ? 0xFFFFFFFFu : (1u << bits) - 1u));
  }
};
__device__ __forceinline__ IdMap id_map(uint32_t imin, uint32_t imax) { return IdMap{imin, 32 - __clz(imax - imin)}; }
template <int KEYS>
__device__ __forceinline__ void second_keys(uint32_t (&id)[KEYS], const uint32_t* __restrict__ zkey, uint32_t n,
                                            uint32_t e0, const KeyMap& k, const IdMap& m, uint32_t n_items) {
#pragma unroll
  for (int i = 0; i < KEYS; ++i) {
    uint32_t low = 0u;
    if (k.shift && e0 + i < n && in_bounds(id[i] < n_items)) low = (zkey[id[i]] - k.zmin) & ((1u << k.shift) - 1u);
    id[i] = e0 + i < n ? (k.shift ? low << m.bits : 0u) | (id[i] - m.imin) : 0xFFFFFFFFu;
  }
}
// ... led by the run, counted from `run` on
template <int KEYS>
__device__ __forceinline__ void run_keys(uint32_t (&x)[KEYS], uint32_t n, uint32_t e0, uint32_t ties, uint32_t run,
                                         int low_bits) {
#pragma unroll
  for (int i = 0; i < KEYS; ++i) {
    if (!(ties >> i & 1u)) ++run;
    if (e0 + i < n) x[i] |= (run - 1u) << low_bits;
  }
}

// A pass of neighbour exchanges within the runs (odd-even transposition; every
// other pair of neighbours, then the rest), and whether each run is in order.
// Runs are short (1.5 entries on average) and nearly in order, so a few
// passes do what another sort would.
constexpr int kSettleRounds = 8, kSettlePasses = 2;
template <int KEYS>
__device__ __forceinline__ void settle_pass(uint32_t (&x)[KEYS], uint32_t ties, int lane) {
#pragma unroll
  for (int first = 0; first < 2; ++first)
#pragma unroll
    for (int i = first; i + 1 < KEYS; i += 2) {
      const uint32_t a = x[i], b = x[i + 1];
      const bool sw = (ties >> (i + 1) & 1u) && b < a;
      x[i] = sw ? b : a;
      x[i + 1] = sw ? a : b;
    }
  const uint32_t next = __shfl_down_sync(0xFFFFFFFFu, x[0], 1), prev = __shfl_up_sync(0xFFFFFFFFu, x[KEYS - 1], 1);
  const bool tie = __shfl_down_sync(0xFFFFFFFFu, ties, 1) & 1u;
  if (lane < 31 && tie) x[KEYS - 1] = min(x[KEYS - 1], next);
  if (lane > 0 && (ties & 1u)) x[0] = max(x[0], prev);
}
template <int KEYS>
__device__ __forceinline__ bool settled(const uint32_t (&x)[KEYS], uint32_t ties, int lane) {
  const uint32_t prev = __shfl_up_sync(0xFFFFFFFFu, x[KEYS - 1], 1);
  bool ok = lane == 0 || !(ties & 1u) || prev <= x[0];
#pragma unroll
  for (int i = 0; i + 1 < KEYS; ++i) ok = ok && (!(ties >> (i + 1) & 1u) || x[i] <= x[i + 1]);
  return __all_sync(0xFFFFFFFFu, ok);
}

// One warp sorts the list of n <= 32 KEYS ids at ids[off ..]; true: it has to
// be sorted by its 64-bit keys (and is as it was).
template <int KEYS>
__device__ __forceinline__ bool warp_sort_list32(uint32_t* ids, const uint32_t* __restrict__ zkey, uint32_t off,
                                                 uint32_t n, uint32_t n_items, int lane) {
  // up to 256 entries, consecutive ones per lane, so that short lists fill the
  // lower lanes only and need fewer merges
  auto place = [lane](int i) { return (uint32_t)(KEYS == 8 ? KEYS * lane + i : 32 * i + lane); };
  uint32_t x[KEYS];
  uint32_t zmin = 0xFFFFFFFFu, zmax = 0u, imin = 0xFFFFFFFFu, imax = 0u;
#pragma unroll
  for (int i = 0; i < KEYS; ++i) {
    const uint32_t e = place(i);
    x[i] = 0u;
    if (e < n) {
      const uint32_t g = ids[off + e];
      x[i] = in_bounds(g < n_items) ? zkey[g] : 0xFFFFFFFFu;
      zmin = min(zmin, x[i]);
      zmax = max(zmax, x[i]);
      imin = min(imin, g);
      imax = max(imax, g);
    }
  }
  const KeyMap k = key_map(n, __reduce_min_sync(0xFFFFFFFFu, zmin), __reduce_max_sync(0xFFFFFFFFu, zmax));
#pragma unroll
  for (int i = 0; i < KEYS; ++i) {
    const uint32_t e = place(i);
    x[i] = e < n ? (k.rounded(x[i]) << k.bits) | e : 0xFFFFFFFFu;
  }
  warp_sort32<KEYS>(x, lane, n);
  const uint32_t e0 = (uint32_t)(lane * KEYS);
  uint32_t id[KEYS];
  const uint32_t ties = sorted_ids_ties<KEYS>(x, ids, off, n, e0, k, __shfl_up_sync(0xFFFFFFFFu, x[KEYS - 1], 1), id);
  IdMap m{0u, 32};
  if (__any_sync(0xFFFFFFFFu, ties != 0u)) {
    m = id_map(__reduce_min_sync(0xFFFFFFFFu, imin), __reduce_max_sync(0xFFFFFFFFu, imax));
    if (k.shift + m.bits > 32) return true;
    second_keys<KEYS>(id, zkey, n, e0, k, m, n_items);
    int round = 0;
    for (; round < kSettleRounds && !settled<KEYS>(id, ties, lane); ++round)
#pragma unroll 1
      for (int p = 0; p < kSettlePasses; ++p) settle_pass<KEYS>(id, ties, lane);
    if (round == kSettleRounds) {
      if (k.bits + k.shift + m.bits > 32) return true;
      const uint32_t runs = (uint32_t)(KEYS - __popc(ties));
      uint32_t incl = runs;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (lane >= d) incl += y;
      }
      run_keys<KEYS>(id, n, e0, ties, incl - runs, k.shift + m.bits);
      warp_sort32<KEYS>(id, lane, n);
    }
  }
  __syncwarp();  // every place has been read
#pragma unroll
  for (int i = 0; i < KEYS; ++i)
    if (e0 + i < n) ids[off + e0 + i] = m.id(id[i]);
  return false;
}

// A CTA of kLongWarps warps sorts its 256 keys per warp: each warp its own, then
// levels of merges whose first exchanges go through shared memory (s: a word
// per key), as many as n keys need.
constexpr int kLongKeys = 8, kLongWarps = kTileSortCap / (32 * kLongKeys), kLongThreads = 32 * kLongWarps;
__device__ __forceinline__ void cta_sort32(uint32_t (&x)[kLongKeys], int lane, int warp, uint32_t n, uint32_t* s) {
  constexpr int KEYS = kLongKeys, W = 32 * KEYS;
  warp_sort32<KEYS>(x, lane, W);
  // exchange with warp ^ m: mirrored places (flip) or equal ones; word i of the
  // warp's lane l at s[W warp + 32 i + l], so neither side conflicts
  auto exchange = [&](int m, int high, bool flip) {
#pragma unroll
    for (int i = 0; i < KEYS; ++i) s[W * warp + 32 * i + lane] = x[i];
    __syncthreads();
    const bool lower = (warp & high) == 0;
    const uint32_t* o = s + W * (warp ^ m) + (flip ? 31 - lane : lane);
#pragma unroll
    for (int i = 0; i < KEYS; ++i) {
      const uint32_t y = o[32 * (flip ? KEYS - 1 - i : i)];
      x[i] = lower ? min(x[i], y) : max(x[i], y);
    }
    __syncthreads();
  };
  for (int m = 1; m < kLongWarps && (uint32_t)(W * (m + 1) / 2) < n; m = 2 * m + 1) {
    exchange(m, (m + 1) >> 1, true);
    for (int d = (m + 1) >> 2; d > 0; d >>= 1) exchange(d, d, false);
    warp_merge_from(x, lane, 16);
  }
}

// The CTA sorts a list of at most kTileSortCap ids; true as for warp_sort_list32.
__device__ __forceinline__ bool cta_sort_list32(uint32_t* ids, const uint32_t* __restrict__ zkey, uint32_t off,
                                                uint32_t n, uint32_t n_items, uint32_t* s) {
  constexpr int KEYS = kLongKeys, W = 32 * KEYS;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t e0 = (uint32_t)(W * warp + lane * KEYS);
  uint32_t x[KEYS];
  uint32_t zmin = 0xFFFFFFFFu, zmax = 0u, imin = 0xFFFFFFFFu, imax = 0u;
#pragma unroll
  for (int i = 0; i < KEYS; ++i) {
    x[i] = 0u;
    if (e0 + i < n) {
      const uint32_t g = ids[off + e0 + i];
      x[i] = in_bounds(g < n_items) ? zkey[g] : 0xFFFFFFFFu;
      zmin = min(zmin, x[i]);
      zmax = max(zmax, x[i]);
      imin = min(imin, g);
      imax = max(imax, g);
    }
  }
  zmin = __reduce_min_sync(0xFFFFFFFFu, zmin);
  zmax = __reduce_max_sync(0xFFFFFFFFu, zmax);
  imin = __reduce_min_sync(0xFFFFFFFFu, imin);
  imax = __reduce_max_sync(0xFFFFFFFFu, imax);
  if (lane == 0) {
    s[4 * warp] = zmin;
    s[4 * warp + 1] = zmax;
    s[4 * warp + 2] = imin;
    s[4 * warp + 3] = imax;
  }
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kLongWarps; ++w) {
    zmin = min(zmin, s[4 * w]);
    zmax = max(zmax, s[4 * w + 1]);
    imin = min(imin, s[4 * w + 2]);
    imax = max(imax, s[4 * w + 3]);
  }
  __syncthreads();
  const KeyMap k = key_map(n, zmin, zmax);
#pragma unroll
  for (int i = 0; i < KEYS; ++i) x[i] = e0 + i < n ? (k.rounded(x[i]) << k.bits) | (e0 + i) : 0xFFFFFFFFu;
  cta_sort32(x, lane, warp, n, s);
  if (lane == 31) s[warp] = x[KEYS - 1];
  __syncthreads();
  uint32_t prev = __shfl_up_sync(0xFFFFFFFFu, x[KEYS - 1], 1);
  if (lane == 0 && warp > 0) prev = s[warp - 1];
  uint32_t id[KEYS];
  const uint32_t ties = sorted_ids_ties<KEYS>(x, ids, off, n, e0, k, prev, id);
  if (lane == 0) s[kLongWarps + warp] = ties & 1u;
  IdMap m{0u, 32};
  if (__syncthreads_or(ties != 0u)) {  // (also: every place has been read)
    m = id_map(imin, imax);
    if (k.shift + m.bits > 32) return true;
    second_keys<KEYS>(id, zkey, n, e0, k, m, n_items);
    const bool tie_next = warp + 1 < kLongWarps && s[kLongWarps + warp + 1] != 0u;  // of the next warp's first entry
    __syncthreads();
    bool open = true;
    for (int round = 0; round < kSettleRounds && open; ++round) {
#pragma unroll 1
      for (int p = 0; p < kSettlePasses; ++p) settle_pass<KEYS>(id, ties, lane);
      if (lane == 0) s[warp] = id[0];
      if (lane == 31) s[kLongWarps + warp] = id[KEYS - 1];
      __syncthreads();
      if (lane == 0 && warp > 0 && (ties & 1u)) id[0] = max(id[0], s[kLongWarps + warp - 1]);
      if (lane == 31 && tie_next) id[KEYS - 1] = min(id[KEYS - 1], s[warp + 1]);
      open = __syncthreads_or(!settled<KEYS>(id, ties, lane));
    }
    if (open) {
      if (k.bits + k.shift + m.bits > 32) return true;
      const uint32_t runs = (uint32_t)(KEYS - __popc(ties));
      uint32_t incl = runs;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (lane >= d) incl += y;
      }
      if (lane == 31) s[kLongWarps + warp] = incl;
      __syncthreads();
      uint32_t run = incl - runs;
      for (int w = 0; w < warp; ++w) run += s[kLongWarps + w];
      __syncthreads();
      run_keys<KEYS>(id, n, e0, ties, run, k.shift + m.bits);
      cta_sort32(id, lane, warp, n, s);
    }
  }
#pragma unroll
  for (int i = 0; i < KEYS; ++i)
    if (e0 + i < n) ids[off + e0 + i] = m.id(id[i]);
  __syncthreads();  // s is reused by the next long list
  return false;
}

// A CTA of THREADS threads sorts a list by its 64-bit keys in shared memory.
template <int THREADS>
__device__ __forceinline__ void cta_sort_list64(uint32_t* __restrict__ ids, const uint32_t* __restrict__ zkey,
                                                uint32_t off, uint32_t n, uint32_t n_items,
                                                unsigned long long* __restrict__ s) {
  uint32_t m = 2;
  while (m < n) m <<= 1;
  for (uint32_t i = threadIdx.x; i < m; i += THREADS) {
    unsigned long long key = ~0ull;
    if (i < n) {
      const uint32_t g = ids[off + i];
      key = in_bounds(g < n_items) ? ((unsigned long long)zkey[g] << 32) | g : ~0ull;
    }
    s[i] = key;
  }
  __syncthreads();
  for (uint32_t k = 2; k <= m; k <<= 1) {
    for (uint32_t j = k >> 1; j > 0; j >>= 1) {
      for (uint32_t i = threadIdx.x; i < m; i += THREADS) {
        const uint32_t ixj = i ^ j;
        if (ixj > i) {
          const unsigned long long a = s[i], b = s[ixj];
          const bool up = (i & k) == 0;
          if ((a > b) == up) {
            s[i] = b;
            s[ixj] = a;
          }
        }
      }
      __syncthreads();
    }
  }
  for (uint32_t i = threadIdx.x; i < n; i += THREADS) ids[off + i] = (uint32_t)s[i];
  __syncthreads();  // s is reused by the next long list
}

// Per-tile sort of the lists by (depth bits, id).  A CTA takes kSortWarps
// consecutive tiles, one warp each: lists of up to kWarpSortMax entries are
// sorted by that warp in registers (no barriers), the few of those whose 32-bit
// keys do not suffice by the whole CTA; longer ones go to long_list, which
// tile_sort_long_kernel sorts.  The kernel also zeroes each tile's counter (and
// block 0 the large-splat queue length, the flag of the difference grids and
// the two raster job counters),
// leaving them zero for the next passes.  In bucket mode each warp also files
// its tile under its length class (see TileBinArgs).
//
// Bound by latency (one wave of warps, each a chain of loads and exchanges).
// 64-bit keys throughout, and long lists by the CTA that met them: 25.3 us for
// 3225 lists of 207 entries (1200 x 680), 503 us for 16125 of 494, 167 us for
// 8030 of 284, 941 us for 31360 of 398 (up to 4 lists of 4000 in one CTA).  With
// a second sort (by 64 bits for the longer lists of a million Gaussians, where
// the second keys with the run do not fit) in place of the neighbour exchanges
// 21, 224, 52 and 435 us; now 18.3, 155, 41 and 222 us.
__global__ void __launch_bounds__(kSortThreads, 6) tile_sort_kernel(const uint32_t* __restrict__ offsets,
                                                                 uint32_t* __restrict__ counts, uint32_t* ids,
                                                                 const uint32_t* __restrict__ zkey,
                                                                 uint2* __restrict__ ranges, uint32_t n_tiles,
                                                                 uint32_t capacity, uint32_t* __restrict__ overflow,
                                                                 uint32_t* __restrict__ big_len,
                                                                 uint32_t* __restrict__ raster_work,
                                                                 uint32_t n_items, uint32_t bucket_cap,
                                                                 uint32_t* __restrict__ cls_count,
                                                                 uint32_t* __restrict__ cls_tiles,
                                                                 uint32_t cls_stride, bool long_sorted,
                                                                 uint2* __restrict__ long_list,
                                                                 uint32_t* __restrict__ long_len) {
  pdl_enter();
  const bool buckets = cls_count != nullptr;  // the lists are per-tile buckets (see TileBinArgs)
  constexpr uint32_t CAP = kTileSortCap;
  __shared__ unsigned long long s[kWarpSortMax];
  __shared__ uint2 s_long[kSortWarps];  // (offset, length) of the CTA's lists that it sorts as a whole
  __shared__ uint32_t s_nlong;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    s_nlong = 0u;
    if (blockIdx.x == 0) {
      big_len[0] = big_len[kHugeFlag] = 0u;  // (the scan has used the grids up)
      raster_work[0] = raster_work[1] = 0u;  // the raster passes' job counters
    }
  }
  __syncthreads();
  const uint32_t t = blockIdx.x * kSortWarps + warp;
  if (t < n_tiles) {
    uint32_t n = counts[t];
    const uint32_t off = buckets ? t * bucket_cap : offsets[t];
    __syncwarp();  // every lane has read counts[t]
    if (buckets && n > bucket_cap) n = bucket_cap;  // its bucket overflowed (flagged by the projection)
    const bool fits = buckets || (unsigned long long)off + n <= (unsigned long long)capacity;
    if (lane == 0) {
      counts[t] = 0u;
      if (buckets) {  // file the tile under its length class (empty ones too: their pixels are composited)
        const int c = length_class(n);
        cls_tiles[(size_t)c * cls_stride + atomicAdd(&cls_count[c], 1u)] = t;
      }
      uint2 rg = (n && fits) ? make_uint2(off, off + n) : make_uint2(0u, 0u);
      if (fits && n > CAP && !long_sorted) {
        atomicOr(overflow, 2u);
        rg = make_uint2(0u, 0u);
      }
      ranges[t] = rg;
      if (fits && n > (uint32_t)kWarpSortMax && n <= CAP) long_list[atomicAdd(long_len, 1u)] = make_uint2(off, n);
    }
    bool whole = false;
    if (fits && n > 1 && n <= (uint32_t)kWarpSortMax) {
      if (n <= 256) whole = warp_sort_list32<8>(ids, zkey, off, n, n_items, lane);
      else if (n <= 512) whole = warp_sort_list32<16>(ids, zkey, off, n, n_items, lane);
      else whole = warp_sort_list32<32>(ids, zkey, off, n, n_items, lane);
    }
    if (whole && n <= (uint32_t)kWarpSort64) {
      if (n <= 256) warp_sort_list<8>(ids, zkey, off, n, n_items, lane);
      else warp_sort_list<16>(ids, zkey, off, n, n_items, lane);
    } else if (whole && lane == 0) {
      s_long[atomicAdd(&s_nlong, 1u)] = make_uint2(off, n);
    }
  }
  __syncthreads();
  const uint32_t n_long = s_nlong;
  for (uint32_t q = 0; q < n_long; ++q) cta_sort_list64<kSortThreads>(ids, zkey, s_long[q].x, s_long[q].y, n_items, s);
}

// The lists of more than kWarpSortMax entries, a CTA each.
__global__ void __launch_bounds__(kLongThreads) tile_sort_long_kernel(uint32_t* ids, const uint32_t* __restrict__ zkey,
                                                                      uint32_t n_items,
                                                                      const uint2* __restrict__ long_list,
                                                                      const uint32_t* __restrict__ long_len) {
  pdl_enter();
  __shared__ unsigned long long s[kTileSortCap];
  const uint32_t count = *long_len;
  for (uint32_t q = blockIdx.x; q < count; q += gridDim.x) {
    const uint2 l = long_list[q];
    if (cta_sort_list32(ids, zkey, l.x, l.y, n_items, reinterpret_cast<uint32_t*>(s)))
      cta_sort_list64<kLongThreads>(ids, zkey, l.x, l.y, n_items, s);
  }
}

int bin_grid(int n, int num_sms) {
  const int blocks = (n + kBinThreads - 1) / kBinThreads;
  return max(1, min(blocks, 16 * max(num_sms, 1)));
}

}  // namespace

int tile_sort_capacity() { return kTileSortCap; }

int64_t tile_scan_aux_size(int64_t n_tiles) { return (int64_t)kScanAux * ((n_tiles + kScanTiles - 1) / kScanTiles + 2); }

void launch_tile_count_scan(const TileBinArgs& a, cudaStream_t s, int64_t* launches) {
  if (!a.counted) {
    cudaMemsetAsync(a.counts, 0, sizeof(uint32_t) * (size_t)a.n_tiles, s);
    if (a.n > 0) {
      launch_pdl(tile_count_kernel, bin_grid(a.n, a.num_sms), kBinThreads, 0, s, a);
      if (launches) *launches += 1;
    }
  }
  BigGrids big{};
  big.diff = a.big_diff;
  big.big_len = a.big_len;
  big.views = a.map.views;
  for (int v = 0; v < a.map.views; ++v) {
    big.tiles_x[v] = a.map.tiles_x[v];
    big.tiles_y[v] = a.tiles_y[v];
    big.base[v] = a.big_base[v];
    big.tile_base[v] = a.map.tile_base[v];
  }
  if (a.n_tiles <= 4 * kScanThreads || !a.scan_aux) {  // one block is enough
    launch_pdl(tile_scan_kernel, 1, kScanThreads, 0, s, a.n_tiles, a.counts, a.offsets, a.cursors, a.capacity,
               a.n_pairs, a.stats, a.order, big);
    if (launches) *launches += 1;
  } else {
    if (a.big_diff) {
      launch_pdl(big_rects_kernel, a.map.views, kScanThreads, 0, s, big, a.counts);
      if (launches) *launches += 1;
    }
    const int nb = (a.n_tiles + kScanTiles - 1) / kScanTiles;
    uint32_t* tail = a.scan_aux + (size_t)kScanAux * nb;
    launch_pdl(tile_scan_up_kernel, nb, 256, 0, s, a.n_tiles, a.counts, a.scan_aux);
    launch_pdl(tile_scan_mid_kernel, 1, 64, 0, s, nb, a.scan_aux, tail, a.capacity, a.n_pairs, a.stats);
    launch_pdl(tile_scan_down_kernel, nb, 256, 0, s, a.n_tiles, a.counts, a.scan_aux, tail, a.offsets, a.cursors,
               a.order);
    if (launches) *launches += 3;
  }
}

void launch_tile_scatter(const TileBinArgs& a, cudaStream_t s, int64_t* launches) {
  if (a.n > 0) {
    // 64 items a block while that gives every block one round: more pairs in
    // flight, fewer rounds (25.7 -> 20.6 us with the scan for 100k items, 25.0
    // -> 20.1 us for 50k); with more items the blocks of 256 have enough of
    // them, and fewer scans (1M items: 37 against 46 us)
    if (a.n <= kScatterItems * 16 * max(a.num_sms, 1))
      launch_pdl(tile_scatter_kernel<kScatterItems>, (a.n + kScatterItems - 1) / kScatterItems, kBinThreads, 0, s, a);
    else
      launch_pdl(tile_scatter_kernel<kBinThreads>, bin_grid(a.n, a.num_sms), kBinThreads, 0, s, a);
    if (launches) *launches += 1;
  }
}

void launch_tile_sort(const TileBinArgs& a, cudaStream_t s, int64_t* launches) {
  const int grid = (a.n_tiles + kSortWarps - 1) / kSortWarps;
  const bool buckets = a.bucket_ids != nullptr;
  launch_pdl(tile_sort_kernel, grid, kSortThreads, 0, s, a.offsets, a.counts,
             buckets ? a.bucket_ids : a.ids, a.zkey, a.ranges, (uint32_t)a.n_tiles, a.capacity, a.overflow,
             const_cast<uint32_t*>(a.big_len), a.raster_work, (uint32_t)a.n, a.bucket_cap,
             buckets ? a.cls_count : nullptr,
             a.cls_tiles, a.cls_stride, a.long_sorted, a.long_list, a.long_len);
  if (launches) *launches += 1;
  if (a.longest > (uint32_t)kWarpSortMax) {
    launch_pdl(tile_sort_long_kernel, std::min(a.n_tiles, 3 * std::max(a.num_sms, 1)), kLongThreads, 0, s,
               buckets ? a.bucket_ids : a.ids, a.zkey, (uint32_t)a.n, (const uint2*)a.long_list,
               (const uint32_t*)a.long_len);
    if (launches) *launches += 1;
  }
}

cudaError_t tilebin_bind_bounds(uint32_t* word) { return bind_bounds_word(word); }

}  // namespace gs
