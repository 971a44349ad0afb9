// Tile binning: expansion of each visible Gaussian into its (tile, Gaussian) pairs, tile ranges.
//
// The Gaussians arrive sorted by depth (stage one of the two-stage (tile, depth) sort), so the
// pairs are emitted in depth order; a stable sort on the tile id then yields (tile, depth, id)
// order, and each tile's range of the sorted pairs is found by boundary detection.  A pair key
// carries, above the 20-bit tile id, the Gaussian's pixel box clipped to that tile (so that the
// blend can skip pairs by their keys alone).
#include <algorithm>

#include "dev_common.cuh"

namespace v3dg {
namespace {

constexpr int kExpThreads = 256, kExpItems = 4, kExpTile = kExpThreads * kExpItems;
constexpr uint32_t kExpWarps = kExpThreads / 32;
// Boxes of more tiles than this (or wider than a live_row) are left to k_expand_large: one block's
// 1024 Gaussians are then at most 64k pairs.  With the whole list in one kernel, the few blocks that
// held the Gaussians next to the camera (1300 tiles each) took 1.9 ms of a 1080p frame.
constexpr uint32_t kLargeArea = 64;

// Pair key of a Gaussian's box r in tile (tx, ty) with (view, tile) id `id`: above the id, the box
// clipped to the tile, tile-local (rows exact, columns in quads).
__device__ __forceinline__ uint32_t pair_key(uint32_t id, const uint2 r, uint32_t tx, uint32_t ty) {
  const uint32_t x0 = r.x & 0xFFFFu, x1 = r.x >> 16, y0 = r.y & 0xFFFFu, y1 = r.y >> 16;
  const uint32_t bx0 = x0 > 16 * tx ? x0 - 16 * tx : 0u, bx1 = min(x1 - 16 * tx, 15u);
  const uint32_t by0 = y0 > 16 * ty ? y0 - 16 * ty : 0u, by1 = min(y1 - 16 * ty, 15u);
  return id | (by0 << 20) | (by1 << 24) | ((bx0 >> 2) << 28) | ((bx1 >> 2) << 30);
}

// One pass over a slab's depth-sorted Gaussians: each block takes 1024 of them, scans their tile
// counts, finds its first pair position with a bounded look-back and then writes its pairs
// cooperatively: position p of the block's small boxes belongs to the Gaussian j with
// off[j] <= p < off[j + 1], each warp takes one contiguous range of positions and follows the
// owners forward (one binary search per warp and tile), so the work is spread over the whole block
// and the writes are contiguous.  kFilter: only tiles that are still live count and are written.
// (Leaving out the pairs that meet no live 4x4 block of their tile as well cost twice the expansion's
// time, 0.6 -> 1.0 ms on the 1080p crowd, and saved 2% of the tile sort.)
template <bool kFilter>
__global__ void __launch_bounds__(kExpThreads)
k_expand(const uint32_t* __restrict__ slots0, const uint32_t* __restrict__ slots1, const uint2* __restrict__ rect,
         uint32_t cap, uint32_t cap_pairs, int tiles_x, const uint2* __restrict__ list,
         const InstFrame* __restrict__ inst_views, uint32_t tiles_per_view, TileLive live,
         uint32_t* __restrict__ large_slot, uint32_t* __restrict__ large_pos, uint32_t* __restrict__ pk,
         uint32_t* __restrict__ pv, uint32_t* __restrict__ frame, uint32_t* __restrict__ slab,
         uint64_t* __restrict__ status, uint32_t epoch) {
  __shared__ uint32_t s_off[kExpTile + 1];
  __shared__ uint32_t s_out[kExpTile];     // the Gaussian's first pair in the block's output
  __shared__ uint2 s_rect[kExpTile];
  __shared__ uint32_t s_slot[kExpTile];
  __shared__ uint32_t s_view[kExpTile];
  __shared__ uint32_t s_scan[kExpThreads / 32 + 1];
  __shared__ uint32_t s_tile, s_base;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t n = min(slab[kSlabCount], cap);
  const uint32_t ntiles = (n + kExpTile - 1) / kExpTile;
  // an overflowed frame has no pairs; after a wait that gave up the slots may be anything
  if (blockIdx.x >= ntiles || frame[kOverflow] || frame[kTimeout]) return;
  const uint32_t* __restrict__ slots = (sort_passes(slab[kSlabBits]) & 1u) ? slots1 : slots0;
  for (;;) {   // persistent blocks: tiles in the order of an atomic counter
  if (threadIdx.x == 0) s_tile = atomicAdd(slab + kSlabExpandTile, 1u);
  __syncthreads();
  const uint32_t tile = s_tile;
  if (tile >= ntiles) return;
  const uint32_t first = tile * kExpTile;
  // this thread's Gaussians: the pairs of all of them (sum), and of the small ones with their number
  // (packed: at most 64k pairs, 1024 Gaussians)
  uint32_t slot[kExpItems], view[kExpItems], c[kExpItems], sum = 0, dense = 0;
  uint2 r[kExpItems];
  bool small[kExpItems], any_large = false;
#pragma unroll
  for (int i = 0; i < kExpItems; ++i) {
    const uint32_t j = first + threadIdx.x * kExpItems + i;
    c[i] = 0;
    small[i] = true;
    view[i] = 0;
    if (j < n) {
      slot[i] = slots[j];
      r[i] = rect[slot[i]];
      if (inst_views) view[i] = inst_views[list[slot[i] / kSlots].x].view;
      const TileRect t = tile_rect(r[i]);
      small[i] = t.w * t.h <= kLargeArea && t.w <= 32u;
      if (kFilter) {
        const uint32_t* row = live.bits + size_t(view[i] * live.tiles_y + t.y) * live.words;
        for (uint32_t y = 0; y < t.h; ++y, row += live.words)
          for (uint32_t x = 0; x < t.w; x += 32u) c[i] += __popc(live_row(row, t.x + x, min(t.w - x, 32u)));
      } else {
        c[i] = t.w * t.h;
      }
      any_large |= !small[i];
    }
    sum += c[i];
    if (small[i] && c[i]) dense += (c[i] << 11) | 1u;
  }
  uint32_t total, dense_total;
  uint32_t out = block_exclusive_scan<kExpThreads / 32>(sum, s_scan, &total);
  uint32_t ex = block_exclusive_scan<kExpThreads / 32>(dense, s_scan, &dense_total);
  if (threadIdx.x < 32) {   // warp 0: the look-back, 32 tiles per round
    const uint32_t b = chained_exclusive_warp(status, tile, total, epoch, frame + kTimeout);
    if (threadIdx.x == 0) {
      s_base = b;
      if (tile == ntiles - 1) slab[kSlabPairs] = b + total;
    }
  }
  const uint32_t items = dense_total & 2047u, small_pairs = dense_total >> 11;
  if (threadIdx.x == 0) s_off[items] = small_pairs;
#pragma unroll
  for (int i = 0; i < kExpItems; ++i) {
    if (small[i] && c[i]) {
      const uint32_t d = ex & 2047u;
      s_off[d] = ex >> 11;
      s_out[d] = out;
      s_rect[d] = r[i];
      s_slot[d] = slot[i];
      s_view[d] = view[i];
      ex += (c[i] << 11) | 1u;
    }
    out += c[i];
  }
  __syncthreads();
  const uint32_t base = s_base;
  const bool fits = uint64_t(base) + total <= cap_pairs;   // (always: the frame's pairs fit the capacity)
  if (!fits && threadIdx.x == 0) atomicOr(frame + kOverflow, 1u);
  if (any_large && fits) {
    out -= sum;
#pragma unroll
    for (int i = 0; i < kExpItems; ++i) {
      if (!small[i] && c[i]) {
        const uint32_t q = atomicAdd(slab + kSlabLarge, 1u);
        large_slot[q] = slot[i];
        large_pos[q] = base + out;
      }
      out += c[i];
    }
  }
  // Each warp writes one contiguous range of the small boxes' pairs, 32 positions per step.  The owner
  // of position p is the last item j with s_off[j] <= p.  Items start at distinct positions (each
  // has at least one pair), so at most 32 items start within a step: with `ob` the owner
  // of the position before the step, lane i checks item ob + 1 + i, the warp ORs the start
  // offsets that fall in the step into one mask, and a lane's owner is ob plus the starts at or
  // before its position.
  const uint32_t per_warp = ((small_pairs + kExpWarps * 32u - 1u) / (kExpWarps * 32u)) * 32u;
  const uint32_t pw0 = min(uint32_t(warp) * per_warp, small_pairs), pw1 = min(pw0 + per_warp, small_pairs);
  int ob = -1;   // owner of pw0 - 1 (none before position 0)
  if (fits && pw0 > 0) {   // binary search, the same in every lane: s_off[lo] <= pw0 - 1 < s_off[hi]
    uint32_t lo = 0, hi = items;   // (s_off[0] = 0, s_off[items] = small_pairs)
    while (hi - lo > 1) {
      const uint32_t mid = (lo + hi) >> 1;
      if (s_off[mid] <= pw0 - 1u) lo = mid; else hi = mid;
    }
    ob = int(lo);
  }
  for (uint32_t p0 = pw0; fits && p0 < pw1; p0 += 32u) {
    const uint32_t p = p0 + uint32_t(lane);
    const int kk = ob + 1 + lane;
    uint32_t bit = 0;
    if (kk < int(items)) {
      const uint32_t v = s_off[kk] - p0;   // >= 0: item ob + 1 starts after position p0 - 1
      if (v < 32u) bit = 1u << v;
    }
    const uint32_t starts = __reduce_or_sync(0xffffffffu, bit);
    const uint32_t upto = lane == 31 ? 0xffffffffu : ((2u << lane) - 1u);   // positions p0 .. p
    const int owner = ob + __popc(starts & upto);
    ob = __shfl_sync(0xffffffffu, owner, 31);
    if (p >= pw1) continue;
    const uint32_t lo = uint32_t(owner);
    const uint2 b = s_rect[lo];
    const TileRect t = tile_rect(b);
    const uint32_t k = p - s_off[lo];
    uint32_t tx, ty;
    if (kFilter) {   // the k-th live tile of the box
      const uint32_t* row = live.bits + size_t(s_view[lo] * live.tiles_y + t.y) * live.words;
      uint32_t left = k, y = 0, bits = live_row(row, t.x, t.w);
      for (uint32_t in_row = __popc(bits); left >= in_row && y + 1u < t.h; in_row = __popc(bits)) {
        left -= in_row;
        ++y;
        row += live.words;
        bits = live_row(row, t.x, t.w);
      }
      for (; left; --left) bits &= bits - 1u;
      tx = t.x + uint32_t(__ffs(bits) - 1);
      ty = t.y + y;
    } else {
      const uint32_t dy = k / t.w;
      tx = t.x + (k - dy * t.w);
      ty = t.y + dy;
    }
    const uint32_t q = base + s_out[lo] + k;
    pk[q] = pair_key(s_view[lo] * tiles_per_view + ty * uint32_t(tiles_x) + tx, b, tx, ty);
    pv[q] = s_slot[lo];
  }
  __syncthreads();   // the tile's shared data is consumed before the next tile reuses it
  }  // next tile
}

// The Gaussians with large boxes, one warp each: 32 tiles of the box per step, in order.
template <bool kFilter>
__global__ void __launch_bounds__(256)
k_expand_large(const uint32_t* __restrict__ large_slot, const uint32_t* __restrict__ large_pos, uint32_t cap,
               uint32_t cap_pairs, const uint2* __restrict__ rect, int tiles_x, const uint2* __restrict__ list,
               const InstFrame* __restrict__ inst_views, uint32_t tiles_per_view, TileLive live,
               uint32_t* __restrict__ pk, uint32_t* __restrict__ pv, const uint32_t* __restrict__ slab) {
  const uint32_t lane = threadIdx.x & 31u, warps = gridDim.x * blockDim.x / 32u;
  const uint32_t n = min(slab[kSlabLarge], cap);
  for (uint32_t q = (blockIdx.x * blockDim.x + threadIdx.x) / 32u; q < n; q += warps) {
    const uint32_t slot = large_slot[q];
    uint32_t pos = large_pos[q];
    const uint2 b = rect[slot];
    const TileRect t = tile_rect(b);
    const uint32_t view = inst_views ? inst_views[list[slot / kSlots].x].view : 0u;
    const uint32_t area = t.w * t.h;
    for (uint32_t k0 = 0; k0 < area; k0 += 32u) {
      const uint32_t k = k0 + lane;
      const uint32_t dy = k / t.w, tx = t.x + (k - dy * t.w), ty = t.y + dy;
      bool in = k < area;
      uint32_t at = pos + lane;
      if (kFilter) {
        in = in && live_row(live.bits + size_t(view * live.tiles_y + ty) * live.words, tx, 1u);
        const uint32_t m = __ballot_sync(0xffffffffu, in);
        at = pos + __popc(m & lanemask_lt());
        pos += __popc(m);
      } else {
        pos += 32u;
      }
      if (in && at < cap_pairs) {
        pk[at] = pair_key(view * tiles_per_view + ty * uint32_t(tiles_x) + tx, b, tx, ty);
        pv[at] = slot;
      }
    }
  }
}

// Tile ranges by boundary detection: each thread takes four consecutive sorted keys at a time
// (one 16-byte load when the array is 16-byte aligned) and compares each with its neighbours.
__global__ void __launch_bounds__(256)
k_ranges(const uint32_t* __restrict__ tk, uint32_t cap_pairs, const uint32_t* __restrict__ n_pairs,
         uint2* __restrict__ ranges, uint32_t n_tiles) {
  const uint32_t n = min(*n_pairs, cap_pairs);
  const uint32_t groups = (n + 3) / 4;
  const bool aligned = (reinterpret_cast<uintptr_t>(tk) & 15u) == 0;
  for (uint32_t g = blockIdx.x * blockDim.x + threadIdx.x; g < groups; g += gridDim.x * blockDim.x) {
    const uint32_t k0 = 4 * g;
    uint32_t t[6];   // tiles of keys k0 - 1 .. k0 + 4 (0xFFFFFFFF outside [0, n))
    t[0] = k0 > 0 ? tk[k0 - 1] & kPairTileMask : 0xFFFFFFFFu;
    if (aligned && k0 + 4 <= n) {
      const uint4 v = *reinterpret_cast<const uint4*>(tk + k0);
      t[1] = v.x & kPairTileMask;
      t[2] = v.y & kPairTileMask;
      t[3] = v.z & kPairTileMask;
      t[4] = v.w & kPairTileMask;
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) t[1 + i] = k0 + i < n ? tk[k0 + i] & kPairTileMask : 0xFFFFFFFFu;
    }
    t[5] = k0 + 4 < n ? tk[k0 + 4] & kPairTileMask : 0xFFFFFFFFu;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t k = k0 + i, tt = t[1 + i];
      if (k >= n || tt >= n_tiles) continue;
      if (t[i] != tt) ranges[tt].x = k;
      if (t[i + 2] != tt) ranges[tt].y = k + 1;
    }
  }
}

}  // namespace

cudaError_t launch_expand(const uint32_t* slots0, const uint32_t* slots1, const uint2* rect, uint32_t cap_slots,
                          uint32_t cap_pairs, int tiles_x, const uint2* list, const InstFrame* inst_views,
                          uint32_t tiles_per_view, const TileLive& live, bool filter, uint32_t* large_slot,
                          uint32_t* large_pos, uint32_t* pair_keys, uint32_t* pair_vals, uint32_t* frame, int slab,
                          uint64_t* status, uint32_t epoch, int sm_count, cudaStream_t st) {
  // persistent grid: at most the resident blocks (8 of 256 threads per SM), whatever the capacity
  const uint32_t blocks = std::min<uint32_t>((cap_slots + kExpTile - 1) / kExpTile, uint32_t(sm_count) * 8u);
  if (!blocks) return cudaSuccess;
  uint32_t* words = frame + kSlabBase + slab * kSlabWords;
  const auto expand = filter ? k_expand<true> : k_expand<false>;
  expand<<<blocks, kExpThreads, 0, st>>>(slots0, slots1, rect, cap_slots, cap_pairs, tiles_x, list, inst_views,
                                         tiles_per_view, live, large_slot, large_pos, pair_keys, pair_vals, frame, words,
                                         status, epoch);
  const auto large = filter ? k_expand_large<true> : k_expand_large<false>;
  large<<<sm_count * 4, 256, 0, st>>>(large_slot, large_pos, cap_slots, cap_pairs, rect, tiles_x, list, inst_views,
                                      tiles_per_view, live, pair_keys, pair_vals, words);
  return cudaGetLastError();
}

cudaError_t launch_ranges(const uint32_t* tk, uint32_t cap_pairs, const uint32_t* frame, int slab, uint2* ranges,
                          int n_tiles, int sm_count, cudaStream_t st) {
  k_ranges<<<sm_count * 8, 256, 0, st>>>(tk, cap_pairs, frame + kSlabBase + slab * kSlabWords + kSlabPairs, ranges,
                                         uint32_t(n_tiles));
  return cudaGetLastError();
}

}  // namespace v3dg
