// Tile rasterizer, forward (Eq. 11, front to back with early stop on
// transmittance) and backward (back to front from the stored last
// contributor, transmittance recomputed from the stored final T).
//
// A warp owns a region of a tile's 256 pixels and its lanes form groups, each
// with a small block of the region (WarpMap).  The warp walks the tile's
// depth-sorted list with the records of the next 32 entries already in flight,
// converts them to tile-local coordinates (so per-pixel offsets keep float32
// precision) and finds which entries' support boxes meet which group's block;
// every group then takes its own next entry, so one warp iteration evaluates
// up to 32 (forward) or 16 (backward) different Gaussians, each on a block of
// the size of a small splat.  The backward pass sums a Gaussian's gradient over
// the group with shuffles and adds it to the global record with vector atomics.
//
// Both passes are bound by instruction issue (72% and 70% of cycles issue, the
// ALU pipe 50% and 42% busy, the FMA pipe 39% and 43%, DRAM 6%; one launch at
// 1200 x 680).  With one 8 x 8 block per warp and one list for all 32 lanes, a
// splat of 4-5 px met 2.95 evaluated pixels per blended one and each (warp,
// entry) hit paid its list handling and its reduction for 16 blended pixels;
// lists per group evaluate 1.69 (forward), and one reduction serves 16
// Gaussians: 85 -> 63 us and 168 -> 102 us at 1200 x 680 with 300k Gaussians, an
// iteration of five such views 1927 -> 1302 us.
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "internal.h"

namespace gs {

namespace {

constexpr int kThreads = 128;  // 4 independent warps per CTA
constexpr unsigned kFull = 0xFFFFFFFFu;
// Lanes per group (see WarpMap).  Forward: each lane by itself, its 1 x PPL
// pixels need no sums over lanes (65.3 -> 64.0 us at 1200 x 680, 675 -> 654 us
// for five such views with longer lists, against groups of two).  Backward:
// smaller blocks evaluate fewer pixels that take no part, larger ones make
// fewer atomics: 2 lanes x 4 pixels (104 us; 4 lanes 112, 1 lane 121 us), and
// 4 lanes x 2 or 1 pixels (2 x 2 would make too many: 92 us instead of 59 us
// on a map of large splats, 28.0 instead of 29.9 us on one of small ones).
constexpr int kFwdLanes = 1;
template <int PPL>
constexpr int kBwdLanes = PPL == 4 ? 2 : 4;
// CTAs per SM (registers: 80 and 96 per thread)
constexpr int kFwdCtas = 6, kBwdCtas = 5;

// Pixels of a warp: a region of RW x RH pixels, lane l with the PPL pixels of
// column l % RW from row PPL (l / RW) on (one column: dx, t0 and the column's
// constants are computed once per entry for PPL pixels).  LPG neighbouring
// lanes are a group, its LPG x PPL pixels a block.  A tile has JOBS regions
// (warp jobs).
template <int TW, int TH, int PPL, int LPG_>
struct WarpMap {
  static constexpr int LPG = LPG_;
  static constexpr int ROWS = PPL;  // rows of a block
  static constexpr int RW = PPL == 4 && TW >= 16 ? 16 : 8;
  static constexpr int RH = 32 * PPL / RW;
  static constexpr int JOBS = TW * TH / (RW * RH);
  static_assert(TW * TH == 256 && TW % RW == 0 && TH % RH == 0 && JOBS == 8 / PPL, "regions tile the tile");
};

// Flag in a pixel's stored list position: it did not stop before the list's end.
constexpr int kOpen = (int)0x80000000u;

// One list entry in tile-local coordinates:
//   a = {mu_x, mu_y, i0, -k}, b = {i1, log2 opacity, z, support radius r2},
//   c = {r, g, b, item id}
struct Entry {
  float4 a, b, c;
};

// Shared memory of a warp: the converted entries of four chunks of 32 (slot
// kRing is an entry that no pixel accepts, read by groups that have none), and
// the raw records of the next chunk.
constexpr int kRing = 128;
struct WarpSmem {
  Entry e[kRing + 1];
  float4 raw[32][3];
};

// A list entry's item id; the checked build redirects an id beyond the
// records to record 0 (and reports it), the normal build passes it through.
__device__ __forceinline__ uint32_t checked_id(uint32_t g, uint32_t n_items) {
  return in_bounds(g < n_items) ? g : 0u;
}

// Asynchronous copy of one 48 B record into shared memory (3 x 16 B cp.async).
__device__ __forceinline__ void cp_record(float4* dst, const float4* __restrict__ feat, uint32_t g) {
  const float4* src = feat + 3 * (size_t)g;
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
#pragma unroll
  for (int k = 0; k < 3; ++k)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d + 16u * k), "l"(src + k) : "memory");
}
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Support boxes of more than 512 tiles (half-extents' product): so many blocks
// add to such a splat's gradient record that they queue up at its address, at
// about 5 ns an addition (32 per tile).
constexpr float kWide = 512.f * 256.f / 4.f;

// log2 opacity in place of a NaN (others are at most 0): alpha is over alpha_max
// up to the support's edge, where q' = 6.5.
constexpr float kNanOpacity = 64.f;

// Converts a gathered record to tile-local coordinates and tests the splat's
// support bounding box against the blocks of the warp's region, whose first
// pixel is (bx, by): bit l of the result is set when the box meets the pixel
// centres of lane l's block.  The box holds every pixel the per-pixel test can
// accept: q' <= min(qmax, log2 o - log2 alpha_min) is the ellipse
// (i0 dx)^2 + (i1 (dy - k dx))^2 <= R2, with half-extents sqrt(R2) / i0 and
// sqrt(R2) sqrt(k^2 / i0^2 + 1 / i1^2), and in each half of the region's rows
// only the ellipse's extent over their pixel centres counts: the box of a thin
// slanted splat holds many times the pixels that it reaches (300k faint needles
// of 100 px: backward 23 -> 4.9 ms, forward 2.3, with one list per warp 13.7 and
// 12.4; 20000 random splats of up to 20:1 179 -> 150 and 291 -> 236 us; 300k
// seeded ones as before; per row of blocks instead of per half: 0.5% slower over
// 34 maps).  The widening covers float32 rounding of the test and of the hardware
// square roots and reciprocals.  `wide`: the
// box has more than 4 kWide pixels.  A NaN opacity (fminf passes it over in R2
// and here) becomes one that is clamped wherever the splat reaches: the raster
// loops multiply alpha by 0 outside the support, which a NaN would survive.
template <class M>
__device__ __forceinline__ unsigned make_entry(float4 f0, float4 f1, float4 f2, float ox, float oy, float bx, float by,
                                               const RasterParams& rp, uint32_t id, Entry& e, bool& wide) {
  wide = false;
  const float mlx = __fadd_rn(__fsub_rn(f0.x, ox), f0.z);
  const float mly = __fadd_rn(__fsub_rn(f0.y, oy), f0.w);
  const float R2 = fminf(rp.qmax_s, __fsub_rn(f1.w, rp.log2_alpha_min));
  e.a = make_float4(mlx, mly, f1.x, -f1.y);
  e.b = make_float4(f1.z, fminf(f1.w, kNanOpacity), f2.w, R2);
  e.c = make_float4(f2.x, f2.y, f2.z, __uint_as_float(id));
  if (!(R2 > 0.f && f1.x > 0.f && f1.z > 0.f)) return 0u;
  const float Rr = sqrt_approx(R2) * 1.0001f + 1e-4f;
  const float inv0 = rcp_approx(f1.x), inv1 = rcp_approx(f1.z);
  const float kw = f1.y * inv0, h2 = fmaxf(kw * kw + inv1 * inv1, 1e-30f), rs = rsqrt_approx(h2);
  const float ex = Rr * inv0 + 1e-3f, ey = Rr * (h2 * rs) + 1e-3f;
  wide = ex * ey > kWide;
  // at height y from its centre the ellipse's x is within kx y +- hx
  const float u = inv0 * rs;
  const float kx = f1.y * u * u, hx = u * Rr * inv1 + 1e-3f + 4e-6f * ex;
  // per half of the region's rows, the first and last column of blocks with
  // centres in that range and in the box (fmaxf and fminf pass a NaN of extreme
  // ratios over: the box alone), then the rows that the box meets
  constexpr int NR = M::RH / M::ROWS, RPH = NR / 2;  // rows of blocks, of a half
  constexpr float BW = M::LPG, BH = M::ROWS, HH = M::RH / 2, NC = M::RW / M::LPG;
  constexpr unsigned kRow = (1u << M::RW) - 1u;
  const float rx = mlx - bx, ry = mly - by;
  const float box0 = fmaxf((rx - ex + 0.5f) / BW - 1.f, 0.f), box1 = fminf((rx + ex - 0.5f) / BW, NC - 1.f);
  const float mid = rx + kx * (0.5f - ry), span = kx * (HH - 1.f), step = kx * (HH / BW);
  const float lo = (mid + fminf(span, 0.f) - hx + 0.5f) / BW - 1.f, hi = (mid + fmaxf(span, 0.f) + hx - 0.5f) / BW;
  const int r0 = __float2int_ru(fmaxf((ry - ey + 0.5f) / BH - 1.f, 0.f));
  const int r1 = __float2int_rd(fminf((ry + ey - 0.5f) / BH, NR - 1.f));
  unsigned m = 0u;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int c0 = __float2int_ru(fmaxf(lo + h * step, box0)), c1 = __float2int_rd(fminf(hi + h * step, box1));
    unsigned xm = (kRow >> (M::RW - M::LPG * (c1 - c0 + 1))) << (M::LPG * c0);
    if (RPH == 2) xm |= xm << M::RW;
    m |= c0 <= c1 ? xm << (M::RW * RPH * h) : 0u;
  }
  m = r0 <= r1 ? m & ((kFull >> (32 - M::RW * (r1 - r0 + 1))) << (M::RW * r0)) : 0u;
  return m;
}

// Transposes the 32 x 32 bit matrix whose row l is lane l's x: bit i of lane
// l's result is bit l of lane i's x (32 ballots' worth in five exchanges).
__device__ __forceinline__ unsigned warp_transpose(unsigned x, int lane) {
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) {
    const unsigned m = s == 16 ? 0x0000FFFFu : s == 8 ? 0x00FF00FFu : s == 4 ? 0x0F0F0F0Fu : s == 2 ? 0x33333333u : 0x55555555u;
    const unsigned y = __shfl_xor_sync(kFull, x, s);
    x = lane & s ? (x & ~m) | ((y >> s) & m) : (x & m) | ((y << s) & ~m);
  }
  return x;
}

// The walk of a tile's list, DIR = 1 from its front, DIR = -1 from its entry
// n - 1 backwards, in aligned chunks of 32 entries.  Offsets count entries of
// whole chunks from the walk's first chunk on.  Up to four chunks are held
// converted in shared memory (a ring), [base, top); each group has a bit per
// held entry that meets its block, and takes its own next one whatever the
// others do, up to four chunks ahead of the slowest: the groups of a warp meet
// different numbers of entries per chunk, and these even out over the window
// (with every group waiting at each chunk's end, a third of them idled).  A
// chunk is converted when a group runs dry; its records are in flight
// (cp.async) since the chunk before, the ids of one more in a register.
template <class M, int DIR>
struct Walk {
  const uint32_t* __restrict__ ids;  // of the list's entry 0
  const float4* __restrict__ feat;
  WarpSmem* sm;
  int n, lane;
  uint32_t n_items;
  float ox, oy, bx, by;
  uint32_t g_raw, g_next;     // ids of the chunk in flight and of the one after
  int first;                  // first entry of the walk's first chunk
  int end;                    // offset behind the last chunk
  int base, top;              // held chunks
  int off;                    // the group's chunk; off = top: waiting for the next one
  unsigned cur, w1, w2, w3;   // its remaining entries there and in the three chunks after (first one highest)
  int met = 0;                // one past the last entry met so far (DIR > 0)

  __device__ __forceinline__ int chunk(int o) const { return DIR > 0 ? o : first - o; }
  __device__ __forceinline__ uint32_t id_at(int o) const {
    const int i = chunk(o) + lane;
    return o < end && i < n ? checked_id(__ldg(&ids[i]), n_items) : 0u;
  }
  __device__ __forceinline__ void fetch(int o) {  // the chunk at o into flight
    g_raw = g_next;
    if (o < end && chunk(o) + lane < n) cp_record(sm->raw[lane], feat, g_raw);
    g_next = id_at(o + 32);
  }
  __device__ __forceinline__ void begin() {
    first = DIR > 0 ? 0 : ((n - 1) >> 5) << 5;
    end = (n + 31) & ~31;
    base = top = off = 0;
    cur = w1 = w2 = w3 = 0u;
    g_next = id_at(0);
    fetch(0);
  }
  // Converts the chunk at `top` and puts the following one into flight: in m the
  // blocks that the lane's entry meets, in wide whether it is wide.
  __device__ __forceinline__ void convert(const RasterParams& rp, unsigned& m, bool& wide) {
    cp_wait_all();
    Entry e;
    m = 0u;
    wide = false;
    if (chunk(top) + lane < n) {
      const float4* raw = sm->raw[lane];
      m = make_entry<M>(raw[0], raw[1], raw[2], ox, oy, bx, by, rp, g_raw, e, wide);
    }
    __syncwarp();  // every lane has read its last entry of the chunk that is overwritten
    if (m) sm->e[(top & (kRing - 1)) + lane] = e;
    fetch(top + 32);
    __syncwarp();  // the entries are stored before any lane reads them
  }
  // The same; returns the entries that meet the lane's group (bit i: entry i).
  __device__ __forceinline__ unsigned stage(const RasterParams& rp, unsigned& m, bool& wide) {
    convert(rp, m, wide);
    return warp_transpose(m, lane);
  }
  __device__ __forceinline__ void push(unsigned mine) {  // the staged chunk's entries
    if (DIR > 0) {
      if (mine) met = top + 32 - __clz(mine);
      mine = __brev(mine);
    }
    const int r = top - off;
    cur = r == 0 ? mine : cur;
    w1 = r == 32 ? mine : w1;
    w2 = r == 64 ? mine : w2;
    w3 = r == 96 ? mine : w3;
    top += 32;
  }
  __device__ __forceinline__ bool can_stage() const { return top < end && top - base < kRing; }
  __device__ __forceinline__ bool any_up_to(int lim) const { return __any_sync(kFull, cur != 0u && off <= lim); }
  // What the warp does next when no group is dry or no chunk can be staged
  // (`can`): >= 0: take entries, without `can` while a group has one at an
  // offset up to the result (everything is staged: anywhere; the ring is full:
  // in the oldest chunk); kAgain: the oldest chunk was given up, kEnd: done.
  static constexpr int kAgain = -1, kEnd = -2;
  __device__ __forceinline__ int limit(bool can) {
    if (can) return 0;
    if (top >= end) return __any_sync(kFull, cur != 0u) ? end : kEnd;
    if (any_up_to(base)) return base;
    base += 32;
    return kAgain;
  }
  __device__ __forceinline__ void drop() {  // the group takes no more entries
    cur = w1 = w2 = w3 = 0u;
    off = top;
  }
  __device__ __forceinline__ void step() {  // to the group's next chunk when it is done with this one
    if (cur == 0u && off < top) {
      cur = w1;
      w1 = w2;
      w2 = w3;
      w3 = 0u;
      off += 32;
    }
  }
  // The group's next entry: its slot in sm->e (kRing: none), idx = its place in the list.
  __device__ __forceinline__ int take(int& idx) {
    const int z = __clz(cur);  // 32: none
    const int j = DIR > 0 ? z : 31 - z;
    const int slot = cur ? (off & (kRing - 1)) + j : kRing;
    idx = chunk(off) + j;
    cur &= ~(0x80000000u >> (z & 31));
    step();
    return slot;
  }
};

// Backward passes with one or two pixels per lane take entries by all lanes
// together, with one addition to a Gaussian's record per region instead of one
// per block.  With four or eight pixels an addition the gradients' errors against
// 64 bits were up to 1.75 times those with 64 (200 x 150, 2000 large splats; 1.03
// to 1.07 for a seeded map; means over 24 to 50 maps); now they are 0.92 to 1.04
// times, with a spread of 0.03 (64 x 48 to 500 x 400).  With one pixel per lane
// every chunk is taken so, in a walk without lists, two entries at a time, since
// the few warps wait for each other's exchanges: the pass 45 -> 33 us for the
// former (with the ellipse's test), an iteration 98 -> 85; seeded maps 60 -> 58 us
// (200 x 150) and 54 -> 55 (66 x 38).  With two pixels per lane the chunks in which
// three quarters of the entries that meet the region meet every block of it, the
// groups' lists being nearly the same there: 64 -> 48 us for 5000 large splats at
// 320 x 240 (seven eighths: errors up to 1.25 at 280 x 210; half: 79 instead of 75
// us an iteration for 20000 seeded ones at 320 x 240).  Not with four, whose
// additions are of eight pixels in large images (errors as with 64): 294 -> 295 us
// for 300k Gaussians, 1327 -> 1340 for five views.
template <int PPL>
constexpr bool kTogether = PPL <= 2;

// Slot kRing of a warp's entries: support radius -1, accepted by no pixel.
__device__ __forceinline__ void init_warp_smem(WarpSmem& sm) {
  if ((threadIdx.x & 31) == 0) {
    sm.e[kRing].a = make_float4(0.f, 0.f, 1.f, 0.f);
    sm.e[kRing].b = make_float4(1.f, -126.f, 0.f, -1.f);
    sm.e[kRing].c = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __syncwarp();
}

// Tile, view and pixel origin of visit k: k indexes the tile visit order (or
// the tiles directly), global tiles map to views by tile_base.
struct TileJob {
  int v;          // view
  int ox, oy;     // pixel origin of the tile within the view
  uint2 range;
  uint32_t tile;  // global tile id
};
template <int TW, int TH>
__device__ __forceinline__ TileJob tile_job_of(const RasterArgs& a, uint32_t tile) {
  int v = 0;
  for (int k = 1; k < a.views; ++k)
    if (tile >= a.v[k].tile_base) v = k;
  const int lt = (int)(tile - a.v[v].tile_base);
  const int tx = lt % a.v[v].tiles_x, ty = lt / a.v[v].tiles_x;
  uint2 r = __ldg(&a.ranges[tile]);
  if (!in_bounds(r.x <= r.y && r.y <= a.n_ids)) r = make_uint2(0u, 0u);  // checked build: an empty list
  return TileJob{v, tx * TW, ty * TH, r, tile};
}
template <int TW, int TH>
__device__ __forceinline__ TileJob tile_job(const RasterArgs& a, uint32_t k) {
  return tile_job_of<TW, TH>(a, a.order ? __ldg(&a.order[k]) : k);
}

// Bucket mode: loads the class counts into s_start (kLenClasses + 1 words)
// as s_start[c] = tiles of class c or longer (s_start[kLenClasses] = 0);
// called by every thread of the CTA (it synchronises the CTA).
__device__ __forceinline__ void load_class_starts(const RasterArgs& a, uint32_t* __restrict__ s_start) {
  if (threadIdx.x < 32) {
    constexpr int PER = (kLenClasses + 31) / 32;
    uint32_t cnt[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const int c = (int)threadIdx.x + 32 * i;
      cnt[i] = c < kLenClasses ? __ldg(&a.cls_count[c]) : 0u;
    }
#pragma unroll
    for (int i = 0; i < PER; ++i)
      if ((int)threadIdx.x + 32 * i < kLenClasses) s_start[threadIdx.x + 32 * i] = cnt[i];
    __syncwarp();
    class_starts_desc(s_start);  // s_start[c] = tiles of the classes above c
    __syncwarp();
#pragma unroll
    for (int i = 0; i < PER; ++i)
      if ((int)threadIdx.x + 32 * i < kLenClasses) s_start[threadIdx.x + 32 * i] += cnt[i];
    if (threadIdx.x == 0) s_start[kLenClasses] = 0u;
  }
  __syncthreads();
}

// Bucket mode: the tile of visit k, the (k - tiles of longer classes)-th of
// its class, c the largest class with s_start[c] > k (s_start is
// non-increasing and s_start[0] is the tile count, which exceeds k).
__device__ __forceinline__ uint32_t class_visit_tile(const RasterArgs& a, const uint32_t* __restrict__ s_start,
                                                     uint32_t k) {
  int c = 0;
#pragma unroll
  for (int step = 128; step > 0; step >>= 1)
    if (c + step < kLenClasses && s_start[c + step] > k) c += step;
  return __ldg(&a.cls_tiles[(size_t)c * a.cls_stride + (k - s_start[c + 1])]);
}

// Two floats in one 64-bit register pair, for the packed FP32 instructions
// add / sub / mul / fma .rn.f32x2: each rounds both halves exactly as the
// scalar instruction would, and takes one issue slot for two operations per
// lane (the FMA pipe itself does not get wider: 124 FMA lanes per SM per
// clock either way, measured; the gain is issue slots in issue-bound code).
typedef unsigned long long f2x;
__device__ __forceinline__ f2x f2_pack(float lo, float hi) {
  f2x r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ f2x f2_bcast(float x) { return f2_pack(x, x); }
// 1 if a <= b, else 0 (also for NaN)
__device__ __forceinline__ float one_if_le(float a, float b) {
  float d;
  asm("set.le.f32.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}
// 1 if a <= b and i < n, else 0
__device__ __forceinline__ float one_if_le_and(float a, float b, int i, int n) {
  float d;
  asm("{\n .reg .pred p;\n setp.lt.s32 p, %3, %4;\n set.le.and.f32.f32 %0, %1, %2, p;\n}" : "=f"(d) : "f"(a), "f"(b), "r"(i), "r"(n));
  return d;
}
__device__ __forceinline__ float f2_lo(f2x r) { return __uint_as_float((unsigned)(r & 0xFFFFFFFFull)); }
__device__ __forceinline__ float f2_hi(f2x r) { return __uint_as_float((unsigned)(r >> 32)); }
template <int N>
__device__ __forceinline__ float f2_at(const f2x (&x)[N], int s) {
  return s & 1 ? f2_hi(x[s / 2]) : f2_lo(x[s / 2]);
}
__device__ __forceinline__ f2x f2_add(f2x a, f2x b) {
  f2x d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2x f2_sub(f2x a, f2x b) {
  f2x d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2x f2_mul(f2x a, f2x b) {
  f2x d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2x f2_fma(f2x a, f2x b, f2x c) {
  f2x d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

// x * s + y with the scalar s on both halves, as two scalar FMAs: they take the
// FMA pipe as long as the packed one does, which would need s in both halves of
// a register pair (raster_fwd 70.7 -> 65.3 us at 1200 x 680; the exponent's
// scalars are better broadcast, since each serves two pairs).
__device__ __forceinline__ f2x f2_fma_s(f2x x, float s, f2x y) {
  return f2_pack(__fmaf_rn(f2_lo(x), s, f2_lo(y)), __fmaf_rn(f2_hi(x), s, f2_hi(y)));
}

// Forward pass of region `quad` of global tile `tile` by one warp.  Every
// pixel's arithmetic is the scalar definition's, element for element (packed
// f32x2 instructions on pairs of a lane's pixels).  The ALU pipe (compares,
// selects, minima) has half the FMA pipe's rate, so per pixel it gets one
// compare whose 0 / 1 result multiplies alpha: alpha = 0 leaves T and the sums
// unchanged bit for bit.  A pixel that is done (or outside the image) has its
// row coordinate set to infinity, so that no entry accepts it; the clamp and
// the stop of a pixel are branches that most entries do not take.  Stored per
// pixel: the final T and the number of list entries in front of the one that
// it stopped at (of the last entry that meets its block, and the flag kOpen,
// if it did not stop).
template <int TW, int TH, int PPL, bool COUNT, bool LOSS>
__device__ __forceinline__ void fwd_job(const RasterArgs& a, const RasterParams& rp, uint32_t tile, int quad,
                                        WarpSmem& sm, float* __restrict__ T_final_all,
                                        int32_t* __restrict__ last_all, unsigned long long* __restrict__ counters) {
  using M = WarpMap<TW, TH, PPL, kFwdLanes>;
  constexpr int NP = (PPL + 1) / 2;  // pairs of pixels per lane
  const TileJob job = tile_job_of<TW, TH>(a, tile);
  const RasterView& vw = a.v[job.v];
  const int width = vw.width, height = vw.height;
  const int lane = threadIdx.x & 31;
  const int bxi = (quad % (TW / M::RW)) * M::RW, byi = (quad / (TW / M::RW)) * M::RH;
  const int lx = bxi + lane % M::RW, ly = byi + PPL * (lane / M::RW);
  const int px = job.ox + lx, py = job.oy + ly;
  const float plx = (float)lx + 0.5f;
  const float kInf = __int_as_float(0x7f800000);
  __syncwarp();  // the warp's previous job is done with sm

  Walk<M, 1> walk;
  walk.ids = a.ids + job.range.x;
  walk.feat = a.feat;
  walk.sm = &sm;
  walk.n = (int)(job.range.y - job.range.x);
  walk.lane = lane;
  walk.n_items = a.n_items;
  walk.ox = (float)job.ox;
  walk.oy = (float)job.oy;
  walk.bx = (float)bxi;
  walk.by = (float)byi;

  float ply[2 * NP];
  f2x T[NP], R[NP], G[NP], B[NP], D[NP];
  int stop[2 * NP];  // list entries in front of the one that the pixel stopped at
#pragma unroll
  for (int s = 0; s < 2 * NP; ++s) {
    ply[s] = s < PPL && px < width && py + s < height ? (float)(ly + s) + 0.5f : kInf;
    stop[s] = 0x7fffffff;
  }
  const f2x ONE2 = f2_pack(1.f, 1.f);
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    T[p] = ONE2;
    R[p] = G[p] = B[p] = D[p] = 0;
  }
  uint32_t n_blend = 0, n_visit = 0;

  if (walk.n > 0) {
    walk.begin();
    unsigned gone = 0u;  // 1: every pixel of the lane is done
    for (;;) {
      while (__any_sync(kFull, walk.cur == 0u && walk.off < walk.top)) walk.step();
      const bool can = walk.can_stage();
      if (can && __any_sync(kFull, (walk.cur | gone) == 0u)) {  // a lane is dry
        bool out = true;
#pragma unroll
        for (int s = 0; s < PPL; ++s) out = out && ply[s] == kInf;
        if (__all_sync(kFull, out)) break;
        static_assert(M::LPG == 1, "a lane by itself");
        gone = out ? 1u : 0u;
        unsigned m;
        bool wide;
        walk.push(walk.stage(rp, m, wide));
        if (out) walk.drop();
        continue;
      }
      const int lim = walk.limit(can);
      if (lim == walk.kEnd) break;
      if (lim == walk.kAgain) continue;
      do {
        int idx;
        const Entry& en = sm.e[walk.take(idx)];
        const float4 ea = en.a, eb = en.b, ec = en.c;
        const float dx = __fsub_rn(plx, ea.x);
        const float t0 = __fmul_rn(ea.z, dx);
        float al[2 * NP], in[2 * NP];
#pragma unroll
        for (int p = 0; p < NP; ++p) {
          const f2x DY = f2_sub(f2_pack(ply[2 * p], ply[2 * p + 1]), f2_bcast(ea.y));
          const f2x WQ = f2_fma(f2_bcast(ea.w), f2_bcast(dx), DY);
          const f2x TQ = f2_mul(WQ, f2_bcast(eb.x));
          const f2x Q = f2_fma(f2_bcast(t0), f2_bcast(t0), f2_mul(TQ, TQ));
          const f2x ARG = f2_sub(f2_bcast(eb.y), Q);
          al[2 * p] = ex2_approx(f2_lo(ARG));
          al[2 * p + 1] = ex2_approx(f2_hi(ARG));
          in[2 * p] = one_if_le(f2_lo(Q), eb.w);
          in[2 * p + 1] = one_if_le(f2_hi(Q), eb.w);
        }
        if (eb.y > rp.log2_clamp) {
#pragma unroll
          for (int s = 0; s < 2 * NP; ++s) al[s] = fminf(rp.alpha_max, al[s]);
        }
        f2x AL[NP], TEST[NP];
        float low = 1.f;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
          // alpha, exactly 0 (so that T, R, G, B and D stay as they are) outside the support
          AL[p] = f2_mul(f2_pack(al[2 * p], al[2 * p + 1]), f2_pack(in[2 * p], in[2 * p + 1]));
          TEST[p] = f2_mul(T[p], f2_sub(ONE2, AL[p]));
          low = fminf(low, fminf(f2_lo(TEST[p]), f2_hi(TEST[p])));
        }
        if (COUNT) {
#pragma unroll
          for (int s = 0; s < PPL; ++s) {
            n_visit += eb.w > 0.f && ply[s] != kInf ? 1u : 0u;
            n_blend += in[s] > 0.f && (s & 1 ? f2_hi(TEST[s / 2]) : f2_lo(TEST[s / 2])) >= rp.t_eps ? 1u : 0u;
          }
        }
        if (low < rp.t_eps) {  // a pixel stops in front of this entry
#pragma unroll
          for (int p = 0; p < NP; ++p) {
            const bool s0 = f2_lo(TEST[p]) < rp.t_eps, s1 = f2_hi(TEST[p]) < rp.t_eps;
            AL[p] = f2_pack(s0 ? 0.f : f2_lo(AL[p]), s1 ? 0.f : f2_hi(AL[p]));
            TEST[p] = f2_pack(s0 ? f2_lo(T[p]) : f2_lo(TEST[p]), s1 ? f2_hi(T[p]) : f2_hi(TEST[p]));
            ply[2 * p] = s0 ? kInf : ply[2 * p];
            ply[2 * p + 1] = s1 ? kInf : ply[2 * p + 1];
            stop[2 * p] = s0 ? idx : stop[2 * p];
            stop[2 * p + 1] = s1 ? idx : stop[2 * p + 1];
          }
        }
#pragma unroll
        for (int p = 0; p < NP; ++p) {
          const f2x W = f2_mul(AL[p], T[p]);
          T[p] = TEST[p];
          R[p] = f2_fma_s(W, ec.x, R[p]);
          G[p] = f2_fma_s(W, ec.y, G[p]);
          B[p] = f2_fma_s(W, ec.z, B[p]);
          D[p] = f2_fma_s(W, eb.z, D[p]);
        }
      } while (can ? !__any_sync(kFull, (walk.cur | gone) == 0u) : walk.any_up_to(lim));
    }
    cp_wait_all();
  }
  if (COUNT) {
    unsigned long long vb = n_blend, vv = n_visit;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      vb += __shfl_xor_sync(kFull, vb, off);
      vv += __shfl_xor_sync(kFull, vv, off);
    }
    if (lane == 0) {
      atomicAdd(&counters[0], vb);
      atomicAdd(&counters[1], vv);
    }
  }
  const size_t HW = (size_t)width * height;
  float* __restrict__ color = vw.color;
  float* __restrict__ depth = vw.depth;
  float* __restrict__ alpha = vw.alpha;
  float* __restrict__ T_final = T_final_all + vw.pix_base;
  int32_t* __restrict__ last_out = last_all + vw.pix_base;
  // L1 loss epilogue (Eq. 12 plus the depth term): the same residuals,
  // signs and colour scale as the separate loss kernels, per-region sums
  const float gscale_c = LOSS ? a.w_color / (3.f * (float)HW) : 0.f;
  float sc = 0.f, sd = 0.f, nv = 0.f;
#pragma unroll
  for (int s = 0; s < PPL; ++s) {
    if (!(px < width && py + s < height)) continue;
    const size_t p = (size_t)(py + s) * width + px;
    const float Tf = f2_at(T, s), Df = f2_at(D, s);
    const float col[3] = {f2_at(R, s) + Tf * rp.bg[0], f2_at(G, s) + Tf * rp.bg[1], f2_at(B, s) + Tf * rp.bg[2]};
    if (color) {
#pragma unroll
      for (int c = 0; c < 3; ++c) color[(size_t)c * HW + p] = col[c];
    }
    if (depth) depth[p] = Df;
    if (alpha) alpha[p] = 1.f - Tf;
    T_final[p] = Tf;
    last_out[p] = stop[s] == 0x7fffffff ? walk.met | kOpen : stop[s];
    if constexpr (LOSS) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float r = col[c] - __ldg(&vw.trgb[(size_t)c * HW + p]);
        sc += fabsf(r);
        vw.loss_dc[(size_t)c * HW + p] = gscale_c * (float)((r > 0.f) - (r < 0.f));
      }
      const float td = __ldg(&vw.tdep[p]);
      const bool valid = td > 0.f;
      const float rd = Df - td;
      sd += valid ? fabsf(rd) : 0.f;
      nv += valid ? 1.f : 0.f;
      vw.loss_dd[p] = valid ? (float)((rd > 0.f) - (rd < 0.f)) : 0.f;
    }
  }
  if constexpr (LOSS) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      sc += __shfl_xor_sync(kFull, sc, off);
      sd += __shfl_xor_sync(kFull, sd, off);
      nv += __shfl_xor_sync(kFull, nv, off);
    }
    if (lane == 0) {
      float* part = a.loss_partials + 3 * (M::JOBS * (size_t)job.tile + quad);
      part[0] = sc;
      part[1] = sd;
      part[2] = nv;
      if (a.nvalid) atomicAdd(&a.nvalid[job.v], (uint32_t)nv);  // an integer: exact in any order
    }
  }
}

// Pulls the next (tile visit, region) job for the calling warp from the
// device counter `work`: a visit's JOBS regions are consecutive jobs, so warps
// take the tiles in visit order (longest lists first) and a warp that
// finishes early takes new work instead of waiting for the other regions of
// its tile.  Returns false when all jobs are taken.
__device__ __forceinline__ bool next_job(uint32_t* __restrict__ work, uint32_t n_jobs, uint32_t& job) {
  uint32_t j = 0;
  if ((threadIdx.x & 31) == 0) j = atomicAdd(work, 1u);
  job = __shfl_sync(kFull, j, 0);
  return job < n_jobs;
}

// The tile of forward visit k: from the class lists in bucket mode (the warp
// on block 0 of the visit also records it in the flat order the backward
// pass reads), else from the flat order, else tile k.
__device__ __forceinline__ uint32_t fwd_visit_tile(const RasterArgs& a, const uint32_t* __restrict__ s_start,
                                                   uint32_t k, int quad) {
  if (!a.cls_count) return a.order ? a.order[k] : k;
  const uint32_t tile = class_visit_tile(a, s_start, k);
  if (quad == 0 && (threadIdx.x & 31) == 0) a.order_out[k] = tile;
  return tile;
}

// The warps of the grid (a persistent one, or one warp per job) pull jobs from
// `work` with next_job.
template <int TW, int TH, int PPL, bool COUNT, bool LOSS>
__global__ void __launch_bounds__(kThreads, kFwdCtas) raster_fwd_kernel(const __grid_constant__ RasterArgs a, RasterParams rp,
                                                              float* __restrict__ T_final_all,
                                                              int32_t* __restrict__ last_all,
                                                              unsigned long long* __restrict__ counters,
                                                              uint32_t* __restrict__ work) {
  pdl_enter();
  constexpr uint32_t JOBS = 8 / PPL;
  __shared__ __align__(16) WarpSmem s_w[kThreads / 32];
  __shared__ uint32_t s_start[kLenClasses + 1];  // bucket mode: tiles of class c or longer
  const int warp = threadIdx.x >> 5;
  if (a.cls_count) load_class_starts(a, s_start);  // CTA-uniform
  init_warp_smem(s_w[warp]);
  const uint32_t n_jobs = JOBS * a.n_tiles;
  uint32_t job;
  while (next_job(work, n_jobs, job)) {
    const int quad = (int)(job % JOBS);
    fwd_job<TW, TH, PPL, COUNT, LOSS>(a, rp, fwd_visit_tile(a, s_start, job / JOBS, quad), quad, s_w[warp], T_final_all,
                                      last_all, counters);
  }
}

// Adds x to the record's float4 `part` unless it is all zeros (a group without
// a contribution, or without an entry).
__device__ __forceinline__ void add_part(float* __restrict__ rec, int part, float a, float b, float c, float d) {
  const unsigned bits = (__float_as_uint(a) | __float_as_uint(b) | __float_as_uint(c) | __float_as_uint(d)) & 0x7fffffffu;
  if (bits) atomicAdd(reinterpret_cast<float4*>(rec) + part, make_float4(a, b, c, d));
}

// Sums the ten values v over the lanes of each group and adds the totals to
// the group's record (12 floats: {s0 .. s3}, {s4, s5, depth, -}, {r, g, b, -})
// with 16-byte vector atomics: four lanes exchange at distance 2 (v[0..6] to
// the lower two, v[7..9] to the upper) and 1, after which lane l has float4 l
// (11 shuffles for all groups of the warp at once); two lanes at distance 1
// (float4 0 to the first lane, 1 and 2 to the second).
template <int LPG>
__device__ __forceinline__ void group_reduce_add10(const float (&v)[10], int lane, float* __restrict__ rec) {
  if constexpr (LPG == 4) {
    const bool b1 = lane & 2, l0 = (lane & 3) == 0, l1 = (lane & 3) == 1;
    float u[7];
#pragma unroll
    for (int i = 0; i < 3; ++i) u[i] = (b1 ? v[7 + i] : v[i]) + __shfl_xor_sync(kFull, b1 ? v[i] : v[7 + i], 2);
#pragma unroll
    for (int i = 3; i < 7; ++i) u[i] = v[i] + __shfl_xor_sync(kFull, v[i], 2);
    float x[4];
#pragma unroll
    for (int i = 0; i < 3; ++i) x[i] = (l1 ? u[4 + i] : u[i]) + __shfl_xor_sync(kFull, l0 ? u[4 + i] : u[i], 1);
    x[3] = u[3] + __shfl_xor_sync(kFull, u[3], 1);
    if ((lane & 3) < 3) add_part(rec, lane & 3, x[0], x[1], x[2], l0 ? x[3] : 0.f);
  } else {
    static_assert(LPG == 2, "groups of 4 or 2 lanes");
    const bool l1 = lane & 1;
    float x[6];
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = (l1 ? v[4 + i] : v[i]) + __shfl_xor_sync(kFull, l1 ? v[i] : v[4 + i], 1);
    x[4] = v[8] + __shfl_xor_sync(kFull, v[8], 1);
    x[5] = v[9] + __shfl_xor_sync(kFull, v[9], 1);
    add_part(rec, l1 ? 1 : 0, x[0], x[1], x[2], l1 ? 0.f : x[3]);
    if (l1) add_part(rec, 2, x[3], x[4], x[5], 0.f);
  }
}

// float offset of gradient value k in the record
__device__ __forceinline__ int rec_off(int k) { return k < 7 ? k : k + 1; }

// Sums v[0..9] over the warp with exchanges that halve the number of values
// each lane carries (xor 16: 10 -> 5, xor 8: 5 -> 3, xor 4: 3 -> 2, xor 2: 2
// -> 1) and a final xor-1 step (12 shuffles instead of 50), then adds the
// totals to the record: even lanes hold distinct values, so this is one
// warp-wide scalar atomic add.
struct WarpSum {
  float x;   // the lane's total
  int off;   // its float of the record, -1: none
};
__device__ __forceinline__ WarpSum warp_sum10(const float (&v)[10], int lane) {
  const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4, b1 = lane & 2;
  float u[5];
#pragma unroll
  for (int i = 0; i < 5; ++i)  // keep v[i] (b4 = 0) or v[i + 5] (b4 = 1)
    u[i] = (b4 ? v[i + 5] : v[i]) + __shfl_xor_sync(kFull, b4 ? v[i] : v[i + 5], 16);
  float w3[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {  // keep u[0..2] (b3 = 0) or u[3..4], 0 (b3 = 1)
    const float hi = i < 2 ? u[i + 3] : 0.f;
    w3[i] = (b3 ? hi : u[i]) + __shfl_xor_sync(kFull, b3 ? u[i] : hi, 8);
  }
  float w2[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {  // keep w3[0..1] (b2 = 0) or w3[2], 0 (b2 = 1)
    const float hi = i < 1 ? w3[i + 2] : 0.f;
    w2[i] = (b2 ? hi : w3[i]) + __shfl_xor_sync(kFull, b2 ? w3[i] : hi, 4);
  }
  float x = (b1 ? w2[1] : w2[0]) + __shfl_xor_sync(kFull, b1 ? w2[0] : w2[1], 2);
  x += __shfl_xor_sync(kFull, x, 1);
  // value held: 5 b4 + i3 with i3 = 3 b3 + 2 b2 + b1 among the five kept at
  // xor 16; lanes with b2 and (b3 or b1) hold the zero pads
  const int i3 = (b3 ? 3 : 0) + (b2 ? 2 : 0) + (b1 ? 1 : 0);
  const bool valid = !(b2 && (b3 || b1));
  return WarpSum{x, !(lane & 1) && valid ? rec_off((b4 ? 5 : 0) + i3) : -1};
}
__device__ __forceinline__ void warp_reduce_add10(const float (&v)[10], int lane, float* __restrict__ rec) {
  const WarpSum s = warp_sum10(v, lane);
  if (s.off >= 0 && s.x != 0.f) atomicAdd(&rec[s.off], s.x);
}
// ... of two entries, whose exchanges do not wait for one another
__device__ __forceinline__ void warp_reduce_add10(const float (&v)[10], const float (&u)[10], int lane,
                                                  float* __restrict__ rec_v, float* __restrict__ rec_u) {
  const WarpSum s = warp_sum10(v, lane), t = warp_sum10(u, lane);
  if (s.off >= 0 && s.x != 0.f) atomicAdd(&rec_v[s.off], s.x);
  if (t.off >= 0 && t.x != 0.f) atomicAdd(&rec_u[t.off], t.x);
}

// Backward pass of region `quad` of the tile of visit k by one warp: back to
// front, from the pixels' last contributors.  Per pixel, the running
// transmittance T is recovered by division and U is the colour (and depth)
// behind, minus the alpha image's term.  With ga = dL/dalpha * alpha
// (unclamped alpha) the exponent and opacity gradients of a Gaussian are
// linear in
//   v[0] = sum ga t0, v[1] = sum ga t1, v[2] = sum ga t0 dx,
//   v[3] = sum ga t1 dx, v[4] = sum ga t1 w, v[5] = sum ga
// (t0 = i0 dx, t1 = i1 w, w = dy - k dx): the Gaussian's constants (i0, i1,
// k, ln 2, 1 / opacity) are applied once per Gaussian in the projection
// backward pass.  v[6] = sum w dD (depth), v[7..9] = sum w dC (colour).
// A lane's pixels share dx and t0, so v[0], v[2], v[3] follow from its sums
// of ga and ga t1.
template <int TW, int TH, int PPL>
__device__ __forceinline__ void bwd_job(const RasterArgs& a, const RasterParams& rp, uint32_t k, int quad,
                                        WarpSmem& sm, const float* __restrict__ T_final_all,
                                        const int32_t* __restrict__ last_all, float* __restrict__ g2d) {
  using M = WarpMap<TW, TH, PPL, kBwdLanes<PPL>>;
  constexpr int NP = (PPL + 1) / 2;  // pairs of pixels per lane
  const TileJob job = tile_job<TW, TH>(a, k);
  const RasterView& vw = a.v[job.v];
  const int width = vw.width, height = vw.height;
  const float* __restrict__ T_final = T_final_all + vw.pix_base;
  const int32_t* __restrict__ last_in = last_all + vw.pix_base;
  const float* __restrict__ dLdc = vw.dLdc;
  const float* __restrict__ dLdd = vw.dLdd;
  const float* __restrict__ dLda = vw.dLda;
  const float dscale = a.nvalid ? a.w_depth / (float)max(a.nvalid[job.v], 1u)
                                : (a.depth_scale ? a.depth_scale[job.v] : 1.f);
  const int lane = threadIdx.x & 31;
  const int bxi = (quad % (TW / M::RW)) * M::RW, byi = (quad / (TW / M::RW)) * M::RH;
  const int lx = bxi + lane % M::RW, ly = byi + PPL * (lane / M::RW);
  const int px = job.ox + lx, py = job.oy + ly;
  const float plx = (float)lx + 0.5f;
  const size_t HW = (size_t)width * height;
  __syncwarp();  // the warp's previous job is done with sm

  f2x PLY[NP], T[NP], U[NP], C0[NP], C1[NP], C2[NP], DD[NP];
  int last[2 * NP];
  int glast = 0;
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    float t[2], c0[2], c1[2], c2[2], d[2], u[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int s = 2 * p + h;
      t[h] = 1.f;
      c0[h] = c1[h] = c2[h] = d[h] = u[h] = 0.f;
      last[s] = 0;
      if (s < PPL && px < width && py + s < height) {
        const size_t q = (size_t)(py + s) * width + px;
        t[h] = T_final[q];
        last[s] = last_in[q] & ~kOpen;
        c0[h] = dLdc[q];
        c1[h] = dLdc[HW + q];
        c2[h] = dLdc[2 * HW + q];
        d[h] = dLdd[q] * dscale;
        // sum over Gaussians behind of w_j (c_j . dC + z_j dD) + T_final (bg . dC - dA)
        u[h] = t[h] * (rp.bg[0] * c0[h] + rp.bg[1] * c1[h] + rp.bg[2] * c2[h]) - (dLda ? dLda[q] * t[h] : 0.f);
      }
      glast = max(glast, last[s]);
    }
    PLY[p] = f2_pack((float)(ly + 2 * p) + 0.5f, (float)(ly + 2 * p + 1) + 0.5f);
    T[p] = f2_pack(t[0], t[1]);
    U[p] = f2_pack(u[0], u[1]);
    C0[p] = f2_pack(c0[0], c0[1]);
    C1[p] = f2_pack(c1[0], c1[1]);
    C2[p] = f2_pack(c2[0], c2[1]);
    DD[p] = f2_pack(d[0], d[1]);
  }
#pragma unroll
  for (int off = M::LPG / 2; off > 0; off >>= 1) glast = max(glast, __shfl_xor_sync(kFull, glast, off));  // the group's
  int wmax = glast;
#pragma unroll
  for (int off = 16; off >= M::LPG; off >>= 1) wmax = max(wmax, __shfl_xor_sync(kFull, wmax, off));
  if (wmax == 0) return;

  Walk<M, -1> walk;
  walk.ids = a.ids + job.range.x;
  walk.feat = a.feat;
  walk.sm = &sm;
  walk.n = wmax;
  walk.lane = lane;
  walk.n_items = a.n_items;
  walk.ox = (float)job.ox;
  walk.oy = (float)job.oy;
  walk.bx = (float)bxi;
  walk.by = (float)byi;
  walk.begin();
  const f2x ONE2 = f2_pack(1.f, 1.f);
  // one entry (each group its own, or the same one for all) at place idx of the
  // list: the lane's sums; returns the Gaussian's record
  auto sums = [&](const Entry& en, int idx, float (&v)[10]) -> float* {
    const float4 ea = en.a, eb = en.b, ec = en.c;
    const float dx = __fsub_rn(plx, ea.x);
    const float t0 = __fmul_rn(ea.z, dx);
    f2x TQ[NP], WQ[NP];
    float ar[2 * NP], in[2 * NP];
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      const f2x DY = f2_sub(PLY[p], f2_bcast(ea.y));
      WQ[p] = f2_fma(f2_bcast(ea.w), f2_bcast(dx), DY);
      TQ[p] = f2_mul(WQ[p], f2_bcast(eb.x));
      const f2x Q = f2_fma(f2_bcast(t0), f2_bcast(t0), f2_mul(TQ[p], TQ[p]));
      const f2x ARG = f2_sub(f2_bcast(eb.y), Q);
      ar[2 * p] = ex2_approx(f2_lo(ARG));
      ar[2 * p + 1] = ex2_approx(f2_hi(ARG));
      in[2 * p] = one_if_le_and(f2_lo(Q), eb.w, idx, last[2 * p]);
      in[2 * p + 1] = one_if_le_and(f2_hi(Q), eb.w, idx, last[2 * p + 1]);
    }
    f2x AL[NP], AG[NP];  // alpha, and alpha where it is not clamped: 0 where the pixel takes no part
#pragma unroll
    for (int p = 0; p < NP; ++p) AL[p] = AG[p] = f2_mul(f2_pack(ar[2 * p], ar[2 * p + 1]), f2_pack(in[2 * p], in[2 * p + 1]));
    if (eb.y > rp.log2_clamp) {  // the 0.99 clamp has zero gradient
#pragma unroll
      for (int p = 0; p < NP; ++p) {
        const bool c0 = f2_lo(AL[p]) > rp.alpha_max, c1 = f2_hi(AL[p]) > rp.alpha_max;
        AG[p] = f2_pack(c0 ? 0.f : f2_lo(AL[p]), c1 ? 0.f : f2_hi(AL[p]));
        AL[p] = f2_pack(c0 ? rp.alpha_max : f2_lo(AL[p]), c1 ? rp.alpha_max : f2_hi(AL[p]));
      }
    }
    f2x GA = 0, GT = 0, GW = 0, V6 = 0, V7 = 0, V8 = 0, V9 = 0;  // sums over the lane's pairs
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      const f2x OM = f2_sub(ONE2, AL[p]);  // in [0.01, 1]; 1 where the pixel takes no part: T, U unchanged
      const f2x INV = f2_pack(rcp_approx(f2_lo(OM)), rcp_approx(f2_hi(OM)));
      T[p] = f2_mul(T[p], INV);  // transmittance in front of this Gaussian
      const f2x W = f2_mul(AL[p], T[p]);
      const f2x CD = f2_fma_s(C0[p], ec.x, f2_fma_s(C1[p], ec.y, f2_fma_s(C2[p], ec.z, f2_mul(DD[p], f2_bcast(eb.z)))));
      // d/d alpha_i: colour/depth T_i c_i - (sum behind)/(1 - alpha_i); alpha image + T_final/(1 - alpha_i)
      const f2x GAL = f2_sub(f2_mul(T[p], CD), f2_mul(U[p], INV));
      U[p] = f2_fma(W, CD, U[p]);
      const f2x g = f2_mul(GAL, AG[p]);
      const f2x gt = f2_mul(g, TQ[p]);
      if (p == 0) {
        GA = g;
        GT = gt;
        GW = f2_mul(gt, WQ[p]);
        V6 = f2_mul(W, DD[p]);
        V7 = f2_mul(W, C0[p]);
        V8 = f2_mul(W, C1[p]);
        V9 = f2_mul(W, C2[p]);
      } else {
        GA = f2_add(GA, g);
        GT = f2_add(GT, gt);
        GW = f2_fma(gt, WQ[p], GW);
        V6 = f2_fma(W, DD[p], V6);
        V7 = f2_fma(W, C0[p], V7);
        V8 = f2_fma(W, C1[p], V8);
        V9 = f2_fma(W, C2[p], V9);
      }
    }
    v[5] = f2_lo(GA) + f2_hi(GA);
    v[1] = f2_lo(GT) + f2_hi(GT);
    v[4] = f2_lo(GW) + f2_hi(GW);
    v[6] = f2_lo(V6) + f2_hi(V6);
    v[7] = f2_lo(V7) + f2_hi(V7);
    v[8] = f2_lo(V8) + f2_hi(V8);
    v[9] = f2_lo(V9) + f2_hi(V9);
    v[0] = v[5] * t0;
    v[2] = v[0] * dx;
    v[3] = v[1] * dx;
    return g2d + 12 * (size_t)__float_as_uint(ec.w);
  };
  // the entries `bits` of the chunk at `at` by all groups together, every entry on
  // every block: each Gaussian's sums go over the whole warp and to its record
  // once, not once per block; two at a time
  auto walk_all = [&](unsigned bits, int at) {
    const Entry* e = sm.e + (at & (kRing - 1));
    const int i0 = walk.chunk(at);
    while (bits) {
      const int j = 31 - __clz(bits);
      bits ^= 1u << j;
      float v[10];
      float* rec = sums(e[j], i0 + j, v);
      if (bits) {
        const int k = 31 - __clz(bits);
        bits ^= 1u << k;
        float u[10];
        float* rec_u = sums(e[k], i0 + k, u);
        warp_reduce_add10(v, u, lane, rec, rec_u);
      } else {
        warp_reduce_add10(v, lane, rec);
      }
    }
  };
  if constexpr (PPL == 1) {  // every chunk
    for (; walk.top < walk.end; walk.top += 32) {
      unsigned m;
      bool wide;
      walk.convert(rp, m, wide);
      walk_all(__ballot_sync(kFull, m != 0u), walk.top);
    }
    cp_wait_all();
    return;
  }
  // A chunk taken together, and the entries of another from its first to its last
  // wide one, are held back until the groups are done with what comes before, and
  // then walked by all groups together (the nearest splats of a map of large ones
  // cover the image: 257k additions to one record took 1.30 ms where the pass now
  // takes 0.13).
  unsigned held = 0u, rest = 0u;  // these entries; the group's entries of the chunk after them
  bool all = false;               // the groups have them as their own lists (four pixels per lane; a loop over
                                  // them made the pass 1.3 us slower, 106 -> 107.4)
  for (;;) {
    while (__any_sync(kFull, walk.cur == 0u && walk.off < walk.top)) walk.step();
    const bool can = walk.can_stage() && !held && !all;
    if (can && __any_sync(kFull, walk.cur == 0u)) {  // a group is dry
      unsigned m;
      bool wide;
      unsigned mine = walk.stage(rp, m, wide);
      const int over = walk.chunk(walk.top) + 32 - glast;  // entries behind every pixel of the group
      if (over > 0) mine = over < 32 ? mine & (kFull >> over) : 0u;
      const unsigned whole = __ballot_sync(kFull, kTogether<PPL> ? m == kFull : m != 0u && wide);
      rest = 0u;
      if (whole) {
        const unsigned meet = __ballot_sync(kFull, m != 0u);
        const unsigned w = kTogether<PPL> ? __ballot_sync(kFull, m != 0u && wide) : whole;
        if (kTogether<PPL> && 4 * __popc(whole) >= 3 * __popc(meet)) {
          held = meet;
          mine = 0u;
        } else if (w) {  // (entry 31 comes first)
          const unsigned behind = kFull << (31 - __clz(w)) << 1, front = (1u << (__ffs(w) - 1)) - 1u;
          held = meet & ~behind & ~front;
          rest = mine & front;
          mine &= behind;
        }
      }
      walk.push(mine);
      continue;
    }
    int lim = walk.end;
    if (!held && !all) {
      lim = walk.limit(can);
      if (lim == walk.kEnd) break;
      if (lim == walk.kAgain) continue;
    } else if (!__any_sync(kFull, walk.cur != 0u)) {  // the held entries' turn, or they are done
      if constexpr (kTogether<PPL>) {
        walk_all(held, walk.top - 32);
        held = 0u;
        walk.cur = rest;
      } else {
        walk.cur = all ? rest : held;
        all = !all;
        held = 0u;
      }
      walk.base = walk.off = walk.top - 32;
      continue;
    }
    if (all) {
      do {
        int idx;
        const Entry& en = sm.e[walk.take(idx)];
        float v[10];
        float* rec = sums(en, idx, v);
        warp_reduce_add10(v, lane, rec);
      } while (__any_sync(kFull, walk.cur != 0u));
      continue;
    }
    do {
      int idx;
      const Entry& en = sm.e[walk.take(idx)];
      float v[10];
      float* rec = sums(en, idx, v);
      group_reduce_add10<M::LPG>(v, lane, rec);
    } while (can ? !__any_sync(kFull, walk.cur == 0u) : walk.any_up_to(lim));
  }
  cp_wait_all();
}

// `work` as in raster_fwd_kernel.
template <int TW, int TH, int PPL>
__global__ void __launch_bounds__(kThreads, kBwdCtas) raster_bwd_kernel(const __grid_constant__ RasterArgs a,
                                                                 RasterParams rp,
                                                                 const float* __restrict__ T_final_all,
                                                                 const int32_t* __restrict__ last_all,
                                                                 float* __restrict__ g2d,
                                                                 uint32_t* __restrict__ work) {
  pdl_enter();
  constexpr uint32_t JOBS = 8 / PPL;
  __shared__ __align__(16) WarpSmem s_w[kThreads / 32];
  const int warp = threadIdx.x >> 5;
  init_warp_smem(s_w[warp]);
  const uint32_t n_jobs = JOBS * a.n_tiles;
  uint32_t job;
  while (next_job(work, n_jobs, job)) {
    bwd_job<TW, TH, PPL>(a, rp, job / JOBS, (int)(job % JOBS), s_w[warp], T_final_all, last_all, g2d);
  }
}

// Marks the tiles whose list is cut and holds a pixel that did not stop (one
// CTA of 256 threads per tile) and counts them.
__global__ void __launch_bounds__(256) raster_open_kernel(const __grid_constant__ RasterArgs a,
                                                          const int32_t* __restrict__ last_all,
                                                          const uint8_t* __restrict__ cut,
                                                          uint8_t* __restrict__ level,
                                                          unsigned long long* __restrict__ open) {
  const uint32_t tile = blockIdx.x;
  if (!cut[tile]) return;
  int v = 0;
  for (int k = 1; k < a.views; ++k)
    if (tile >= a.v[k].tile_base) v = k;
  const int lt = (int)(tile - a.v[v].tile_base);
  const int px = lt % a.v[v].tiles_x * a.tile_w + (int)threadIdx.x % a.tile_w;
  const int py = lt / a.v[v].tiles_x * a.tile_h + (int)threadIdx.x / a.tile_w;
  const bool in = px < a.v[v].width && py < a.v[v].height;
  const bool mine = in && (last_all[a.v[v].pix_base + (size_t)py * a.v[v].width + px] & kOpen);
  if (__syncthreads_or(mine) && threadIdx.x == 0) {
    level[tile] += 1;
    atomicAdd(open, 1ull);
  }
}

RasterParams make_params(const RasterArgs& a) {
  RasterParams rp;
  rp.width = rp.height = 0;  // per view, from the view table
  rp.tile_w = a.tile_w;
  rp.tile_h = a.tile_h;
  rp.tiles_x = rp.tiles_y = 0;
  for (int c = 0; c < 3; ++c) rp.bg[c] = a.bg[c];
  rp.alpha_max = a.alpha_max;
  rp.log2_alpha_min = log2f(a.alpha_min);
  rp.qmax_s = 9.f * kHalfLog2e;
  rp.t_eps = a.t_eps;
  rp.log2_clamp = log2f(a.alpha_max) - 1e-5f;
  return rp;
}

}  // namespace

bool raster_shape_supported(int tw, int th) {
  return (tw == 16 && th == 16) || (tw == 8 && th == 32) || (tw == 32 && th == 8);
}

namespace {

// Persistent grid: as many CTAs as fit on the GPU at once (occupancy of the
// kernel x SMs; per_sm caches the occupancy query of one kernel), at most one
// per kThreads / 32 jobs.
template <class K>
int persistent_grid(K kernel, int& per_sm, int n_ctas, int num_sms) {
  if (per_sm == 0) {
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel, kThreads, 0) != cudaSuccess || b < 1) b = 1;
    per_sm = b;
  }
  return std::max(1, std::min(n_ctas, per_sm * std::max(num_sms, 1)));
}

int job_ctas(uint32_t n_tiles, int ppl) {
  return (int)(((int64_t)n_tiles * (8 / ppl) + kThreads / 32 - 1) / (kThreads / 32));
}

template <int TW, int TH, int PPL, bool COUNT, bool LOSS>
void fwd_launch(const RasterArgs& a, const RasterParams& rp, float* T_final, int32_t* last,
                unsigned long long* counters, cudaStream_t s) {
  static int per_sm = 0;
  const int nc = job_ctas(a.n_tiles, PPL);
  auto* k = raster_fwd_kernel<TW, TH, PPL, COUNT, LOSS>;
  launch_pdl(k, a.persistent ? persistent_grid(k, per_sm, nc, a.num_sms) : nc, kThreads, 0, s, a, rp, T_final, last, counters,
             a.work);
}

template <int TW, int TH, bool COUNT, bool LOSS>
void fwd_shape(const RasterArgs& a, const RasterParams& rp, float* T_final, int32_t* last,
               unsigned long long* counters, cudaStream_t s) {
  switch (a.px_per_lane) {
    case 4: fwd_launch<TW, TH, 4, COUNT, LOSS>(a, rp, T_final, last, counters, s); break;
    case 2: fwd_launch<TW, TH, 2, COUNT, LOSS>(a, rp, T_final, last, counters, s); break;
    default: fwd_launch<TW, TH, 1, COUNT, LOSS>(a, rp, T_final, last, counters, s); break;
  }
}

template <bool COUNT, bool LOSS>
void fwd_shapes(const RasterArgs& a, const RasterParams& rp, float* T_final, int32_t* last,
                unsigned long long* counters, cudaStream_t s) {
  if (a.tile_w == 16) fwd_shape<16, 16, COUNT, LOSS>(a, rp, T_final, last, counters, s);
  else if (a.tile_w == 8) fwd_shape<8, 32, COUNT, LOSS>(a, rp, T_final, last, counters, s);
  else fwd_shape<32, 8, COUNT, LOSS>(a, rp, T_final, last, counters, s);
}

template <int TW, int TH, int PPL>
void bwd_launch(const RasterArgs& a, const RasterParams& rp, const float* T_final, const int32_t* last, float* g2d,
                cudaStream_t s) {
  static int per_sm = 0;
  const int nc = job_ctas(a.n_tiles, PPL);
  auto* k = raster_bwd_kernel<TW, TH, PPL>;
  launch_pdl(k, a.persistent ? persistent_grid(k, per_sm, nc, a.num_sms) : nc, kThreads, 0, s, a, rp, T_final, last, g2d,
             a.work);
}

template <int TW, int TH>
void bwd_shape(const RasterArgs& a, const RasterParams& rp, const float* T_final, const int32_t* last, float* g2d,
               cudaStream_t s) {
  switch (a.px_per_lane) {
    case 4: bwd_launch<TW, TH, 4>(a, rp, T_final, last, g2d, s); break;
    case 2: bwd_launch<TW, TH, 2>(a, rp, T_final, last, g2d, s); break;
    default: bwd_launch<TW, TH, 1>(a, rp, T_final, last, g2d, s); break;
  }
}

}  // namespace

// Four pixels per lane share an entry's loads and its list handling, but give
// a tile only two warps.  Below about six tiles per SM the SMs hold too few
// warps to hide a warp's latency, and two pixels per lane (twice the warps,
// each with a shorter walk) are faster; below one tile per SM, one.  Measured,
// forward + backward us at 4 / 2 / 1 pixels per lane: 80 tiles 55 / 48 / 44,
// 300 tiles 55 / 49 / 54, 690 tiles 66 / 62 / 88, 1200 tiles 83 / 87 / 131,
// 1908 tiles 97 / 108 / 176.
int raster_px_per_lane(uint32_t n_tiles, int num_sms, int64_t pairs, int64_t longest) {
  const int64_t sms = std::max(num_sms, 1), warps = sms * kFwdCtas * kThreads / 32;
  int ppl = n_tiles >= 6 * sms ? 4 : n_tiles >= sms ? 2 : 1;
  // A warp walks its list alone: where the longest is several times a warp's
  // share of all (a few tiles whose pixels do not stop), the pass takes as long
  // as that walk, and smaller regions make it shorter.  Lists below 1024 end
  // soon enough.  Not down to one pixel per lane: that has twice the additions
  // to each gradient record, and a larger rounding error for it.  8 views of
  // 234k Gaussians with lists of 334 and one of 15804, forward + backward: 2782
  // us with four pixels per lane, 2237 with two.
  if (ppl == 4 && longest >= 1024 && longest * warps > 8 * pairs) ppl = 2;
  return ppl;
}

void launch_raster_fwd(const RasterArgs& a, float* T_final, int32_t* last, unsigned long long* counters,
                       cudaStream_t s) {
  if (a.n_tiles == 0) return;
  const RasterParams rp = make_params(a);
  if (a.zero_work) cudaMemsetAsync(a.work, 0, sizeof(uint32_t), s);
  const bool loss = a.loss_partials != nullptr;
  if (counters) {
    if (loss) fwd_shapes<true, true>(a, rp, T_final, last, counters, s);
    else fwd_shapes<true, false>(a, rp, T_final, last, counters, s);
  } else {
    if (loss) fwd_shapes<false, true>(a, rp, T_final, last, counters, s);
    else fwd_shapes<false, false>(a, rp, T_final, last, counters, s);
  }
}

void launch_raster_open(const RasterArgs& a, const int32_t* last, const uint8_t* cut, uint8_t* level,
                        unsigned long long* open, cudaStream_t s) {
  if (a.n_tiles) raster_open_kernel<<<a.n_tiles, 256, 0, s>>>(a, last, cut, level, open);
}

void launch_raster_bwd(const RasterArgs& a, const float* T_final, const int32_t* last, float4* g2d, cudaStream_t s) {
  if (a.n_tiles == 0) return;
  const RasterParams rp = make_params(a);
  if (a.zero_work) cudaMemsetAsync(a.work, 0, sizeof(uint32_t), s);
  if (a.tile_w == 16) bwd_shape<16, 16>(a, rp, T_final, last, (float*)g2d, s);
  else if (a.tile_w == 8) bwd_shape<8, 32>(a, rp, T_final, last, (float*)g2d, s);
  else bwd_shape<32, 8>(a, rp, T_final, last, (float*)g2d, s);
}

cudaError_t raster_bind_bounds(uint32_t* word) { return bind_bounds_word(word); }

}  // namespace gs
