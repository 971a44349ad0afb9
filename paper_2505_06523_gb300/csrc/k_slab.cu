// Depth slabs: a frame's visible Gaussians are binned, sorted and blended in up to six slabs, front
// to back, and a slab leaves out what only meets tiles whose pixels have all stopped.
//
// Why: on a composed scene most of what is visible by projection is hidden.  On the 1080p crowd (73M
// visible Gaussians, 176M pairs) the nearest 1/128 of the Gaussians finish a quarter of the tiles,
// and only 34M of the Gaussians behind them meet a tile that is still live; of those behind the
// nearest quarter, 10M of 55M.  Sorting, expanding and sorting again what cannot change a pixel was
// more than half of those stages.  The image does not change: a pixel that has stopped takes no
// further record, and a slab's records come in the same order as in the whole list.
// Measured on a GB300, one slab -> several: depth sort, binning, tile sort and ranges of the 1080p crowd
// 5.2 -> 2.6 ms (its blend 1.3 -> 1.8 ms: each slab waits for its longest tile), of the 5000-instance
// 4K crowd 51 -> 11 ms, of 16 crowd views 50 -> 23.4 ms; one asset filling 1080p (31M pairs of 225k
// Gaussians, all tiles finished after 3% of them) 2.4 -> 0.43 ms.
#include <algorithm>

#include "dev_common.cuh"

namespace v3dg {
namespace {

__global__ void __launch_bounds__(256)
k_frame_init(uint32_t* __restrict__ frame, uint32_t* __restrict__ hist, uint32_t hist_words,
             uint32_t* __restrict__ depth_hist, uint2* __restrict__ ranges, uint32_t n_ranges, TileLive live,
             uint32_t n_tiles, uint32_t n_views) {
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x, step = gridDim.x * blockDim.x;
  for (uint32_t i = t; i < uint32_t(kFrameWords); i += step)
    if (i == kVisible || i == kPairs || i == kPairsEff || i == kConicFp64 || i == kRenderClusters || i == kPairs64 ||
        i == kPairs64 + 1 || i == kKeyMinInv || i == kKeyMax || i > kTileCounters)
      frame[i] = 0;
  for (uint32_t i = t; i < hist_words; i += step) hist[i] = 0;
  for (uint32_t i = t; i < n_ranges; i += step) ranges[i] = make_uint2(0u, 0u);
  if (!live.bits) return;
  for (uint32_t i = t; i < uint32_t(kDepthBins); i += step) depth_hist[i] = 0;
  for (uint32_t i = t; i < n_tiles; i += step) live.blocks[i] = 0xFFFFu;
  const auto row_word = [](uint32_t x, uint32_t n) {   // bits x .. x + 31 of a row of n ones
    return x >= n ? 0u : n - x >= 32u ? 0xFFFFFFFFu : (1u << (n - x)) - 1u;
  };
  for (uint32_t i = t; i < n_views * live.tiles_y * live.words; i += step)
    live.bits[i] = row_word((i % live.words) * 32u, live.tiles_x);
  for (uint32_t i = t; i < n_views * live.groups_y * live.coarse_words; i += step)
    live.coarse[i] = row_word((i % live.coarse_words) * 32u, live.groups_x);
  for (uint32_t i = t; i < n_views * live.groups_y * live.groups_x; i += step) {
    const uint32_t gx = i % live.groups_x, gy = (i / live.groups_x) % live.groups_y;
    live.coarse_tiles[i] = min(8u, live.tiles_x - 8u * gx) * min(8u, live.tiles_y - 8u * gy);
  }
}

// The slabs' limits: at the depths where these thousandths of the frame's pairs lie in front (the first slab
// is kept whole; the last takes what the others have not hidden).  A slab more leaves out a few more pairs
// and costs about 20 launches and a tail of the blend, so larger frames take more of them (see slab_count).
// Whole frames by number of slabs, 3 / 4 / 6: crowd at 1080p (157M pairs) 6.46 / 6.06 / 6.84 ms, 5000 instances at
// 4K (1.9G) 29.8 / 27.1 / 25.5 ms, 16 crowd views (1.3G) 53.6 / 47.8 / 45.2 ms; 2 / 3: crowd of 600 instances (99M)
// 4.34 / 4.72 ms, one asset filling 1080p (31M) 0.87 / 0.95 ms.  Two slabs' limit at 250, 350 and 450: that crowd
// 4.34, 4.48, 4.51 ms; the asset 0.88, 0.87, 0.90 ms, from 3 units (44M) 1.85, 1.64, 1.65 ms: frames of
// large boxes take the later limit.  Limits tried with four: {20, 80, 250}, {30, 120, 350}, {40, 160, 400}, {60, 200, 400}, {70, 250, 450}, {100, 300, 500}: the crowd 7.32,
// 6.68, 6.87, 6.85, 6.32, 6.15 ms.  With six: {30, 90, 200, 340, 520}, {40, 120, 240, 360, 500}, these, {60, 160, 320,
// 500, 700}, {80, 190, 330, 480, 650}, {100, 220, 360, 500, 650}: 5000 instances at 4K 26.0, 24.8, 25.8, 26.2, 27.1,
// 27.0 ms, 16 crowd views 53.0, 53.3, 50.5, 50.6, 50.0, 50.1 ms, five views (869M pairs) 24.0, 24.2, 23.6, 24.1, 24.0,
// 24.4 ms.
__constant__ const uint32_t kLimits2[1] = {250}, kLimits2Large[1] = {350}, kLimits4[3] = {83, 300, 500},
                            kLimits6[5] = {50, 140, 280, 430, 600};

__global__ void __launch_bounds__(256)
k_slab_limits(uint32_t* __restrict__ frame, const uint32_t* __restrict__ depth_hist, int slabs, uint32_t cap_pairs) {
  __shared__ uint32_t s_scan[9], s_edge[kMaxSlabs + 1];
  const unsigned long long total = *reinterpret_cast<const unsigned long long*>(frame + kPairs64);
  const uint32_t kmin = ~frame[kKeyMinInv], kmax = frame[kKeyMax];
  const bool any = frame[kVisible] != 0u;
  if (threadIdx.x <= kMaxSlabs) s_edge[threadIdx.x] = threadIdx.x == 0 ? kmin : any ? kmax + 1u : kmin;
  __syncthreads();
  if (slabs > 1 && total <= 0xFFFFFFFFull) {
    constexpr int kPer = kDepthBins / 256;
    uint32_t v[kPer], sum = 0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      v[i] = depth_hist[threadIdx.x * kPer + i];
      sum += v[i];
    }
    uint32_t all, excl = block_exclusive_scan<8>(sum, s_scan, &all);
    // thousandths of the pairs
    const uint32_t* const limits = slabs == 2 ? (large_boxes(total, frame[kVisible]) ? kLimits2Large : kLimits2) : slabs == 4 ? kLimits4 : kLimits6;
    uint32_t target[kMaxSlabs - 1];
#pragma unroll
    for (int k = 0; k < kMaxSlabs - 1; ++k)
      target[k] = k < slabs - 1 ? max(uint32_t(uint64_t(all) * limits[k] / 1000u), 1u) : 0u;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      for (int k = 0; k < slabs - 1; ++k)
        if (excl < target[k] && excl + v[i] >= target[k])   // one bin crosses each target
          s_edge[k + 1] = min(max(uint32_t(threadIdx.x * kPer + i + 1 + kDepthBase) << kDepthShift, kmin), kmax + 1u);
      excl += v[i];
    }
    __syncthreads();
  }
  if (threadIdx.x < slabs) {
    const uint32_t lo = any ? s_edge[threadIdx.x] : 0u, hi = any ? s_edge[threadIdx.x + 1] : 0u;
    uint32_t* w = frame + kSlabBase + threadIdx.x * kSlabWords;
    w[kSlabLo] = lo;
    w[kSlabHi] = hi;
    w[kSlabBits] = hi > lo + 1u ? 32u - __clz(hi - lo - 1u) : 1u;
  }
  if (threadIdx.x == 0) {
    // a total beyond the capacity (counted in 64 bits, so also one beyond 2^32) overflows the frame
    frame[kPairs] = total > 0xFFFFFFFFull ? 0xFFFFFFFFu : uint32_t(total);
    if (total > cap_pairs) frame[kOverflow] = 1u;
    frame[kPairsEff] = frame[kOverflow] ? 0u : uint32_t(total);
  }
}

// Several slabs: the stable compaction of a slab's slots in three launches without a chain of waits (with
// a look-back, four slabs of the 1080p crowd took 1.5 ms: a thousand tiles in flight wait for one
// another).  (One slab takes none: the depth sort's first pass reads the slots themselves.)  k_mark: a warp takes 32 nodes, drops those whose depth range misses the slab, and writes
// a bit per slot of the others: in the slab and (kFilter) on a live tile; a block's 256 nodes leave
// their count.  k_mark_scan: the counts' prefix sums, by one block.  k_gather: the marked slots.
constexpr int kMarkNodes = 256;   // nodes of a block

template <bool kFilter>
__global__ void __launch_bounds__(256)
k_mark(const uint32_t* __restrict__ keys, const uint2* __restrict__ rect, uint32_t cap_nodes, const uint2* __restrict__ list,
       const InstFrame* __restrict__ inst_views, TileLive live, const float2* __restrict__ depth_range,
       uint2* __restrict__ marks, uint32_t* __restrict__ counts, const uint32_t* __restrict__ frame,
       const uint32_t* __restrict__ slab) {
  __shared__ uint32_t s_warp[8];
  constexpr int kAhead = 4;   // nodes whose keys are loaded together
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const uint32_t n = min(frame[kRenderNodes], cap_nodes);
  const uint32_t n_blocks = (n + kMarkNodes - 1) / kMarkNodes;
  const uint32_t lo = slab[kSlabLo], hi = slab[kSlabHi];
  if (lo >= hi) return;
  for (uint32_t blk = blockIdx.x; blk < n_blocks; blk += gridDim.x) {
    const uint32_t node0 = blk * kMarkNodes + warp * 32u;
    bool cand = false;
    if (node0 + lane < n) {
      const float2 z = depth_range[node0 + lane];   // conservative
      cand = !(z.y < __uint_as_float(lo)) && !(z.x >= __uint_as_float(hi));
    }
    uint32_t todo = __ballot_sync(0xffffffffu, cand);
    uint2 mine = make_uint2(0u, 0u);
    uint32_t count = 0;
    while (todo) {
      uint32_t node[kAhead], key[kAhead][2];
      int m = 0;
#pragma unroll
      for (int a = 0; a < kAhead; ++a) {
        node[a] = node0 + uint32_t(__ffs(todo) - 1);   // (todo == 0: not used)
        if (todo) {
          todo &= todo - 1u;
          m = a + 1;
        }
        key[a][0] = a < m ? keys[size_t(node[a]) * kSlots + lane] : 0xFFFFFFFFu;
        key[a][1] = a < m ? keys[size_t(node[a]) * kSlots + 32 + lane] : 0xFFFFFFFFu;
      }
      // the boxes of the slots in the slab, all on their way before the first is looked at
      uint2 box[kAhead][2];
      bool in[kAhead][2];
#pragma unroll
      for (int a = 0; a < kAhead; ++a)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          in[a][h] = key[a][h] >= lo && key[a][h] < hi;
          if (kFilter) box[a][h] = in[a][h] ? rect[size_t(node[a]) * kSlots + 32 * h + lane] : make_uint2(0u, 0u);
        }
#pragma unroll
      for (int a = 0; a < kAhead; ++a) {
        if (a >= m) break;   // (uniform)
        uint32_t b[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (kFilter && in[a][h]) {
            TileRect r = tile_rect(box[a][h]);
            const uint32_t view = inst_views ? inst_views[list[node[a]].x].view : 0u;
            const uint32_t* row = live.bits + size_t(view * live.tiles_y + r.y) * live.words;
            uint32_t words = live.words;
            if (r.h * ((r.w + 31u) / 32u) > 4u) {   // a large box: the groups of tiles it meets (no more than a superset)
              const uint32_t x1 = (r.x + r.w - 1u) >> 3, y1 = (r.y + r.h - 1u) >> 3;
              r.x >>= 3;
              r.y >>= 3;
              r.w = x1 - r.x + 1u;
              r.h = y1 - r.y + 1u;
              words = live.coarse_words;
              row = live.coarse + size_t(view * live.groups_y + r.y) * words;
            }
            uint32_t any = 0;
            for (uint32_t y = 0; y < r.h && !any; ++y, row += words)
              for (uint32_t x = 0; x < r.w && !any; x += 32u) any = live_row(row, r.x + x, min(r.w - x, 32u));
            in[a][h] = any != 0u;
          }
          b[h] = __ballot_sync(0xffffffffu, in[a][h]);
          count += __popc(b[h]);
        }
        if (lane == node[a] - node0) mine = make_uint2(b[0], b[1]);
      }
    }
    if (node0 + lane < n) marks[node0 + lane] = mine;
    if (lane == 0) s_warp[warp] = count;
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t t = 0;
      for (int w = 0; w < 8; ++w) t += s_warp[w];
      counts[blk] = t;
    }
    __syncthreads();
  }
}

__global__ void __launch_bounds__(1024)
k_mark_scan(uint32_t* __restrict__ counts, uint32_t cap_nodes, const uint32_t* __restrict__ frame,
            uint32_t* __restrict__ slab) {
  __shared__ uint32_t s_scan[33];
  const uint32_t n_blocks = (min(frame[kRenderNodes], cap_nodes) + kMarkNodes - 1) / kMarkNodes;
  if (slab[kSlabLo] >= slab[kSlabHi]) return;   // (the slab keeps its zero count)
  uint32_t base = 0;
  constexpr int kPer = 8;
  for (uint32_t i0 = 0; i0 < n_blocks; i0 += 1024 * kPer) {
    uint32_t v[kPer], sum = 0, total;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const uint32_t i = i0 + threadIdx.x * kPer + k;
      v[k] = i < n_blocks ? counts[i] : 0u;
      sum += v[k];
    }
    uint32_t ex = base + block_exclusive_scan<32>(sum, s_scan, &total);
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const uint32_t i = i0 + threadIdx.x * kPer + k;
      if (i < n_blocks) counts[i] = ex;
      ex += v[k];
    }
    base += total;
  }
  if (threadIdx.x == 0) slab[kSlabCount] = base;
}

__global__ void __launch_bounds__(256)
k_gather(const uint32_t* __restrict__ keys, uint32_t cap_nodes, const uint2* __restrict__ marks,
         const uint32_t* __restrict__ counts, uint32_t* __restrict__ kout, uint32_t* __restrict__ vout,
         const uint32_t* __restrict__ frame, const uint32_t* __restrict__ slab) {
  __shared__ uint32_t s_warp[8];
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const uint32_t n = min(frame[kRenderNodes], cap_nodes);
  const uint32_t n_blocks = (n + kMarkNodes - 1) / kMarkNodes;
  const uint32_t lo = slab[kSlabLo];
  if (lo >= slab[kSlabHi]) return;
  for (uint32_t blk = blockIdx.x; blk < n_blocks; blk += gridDim.x) {
    const uint32_t node0 = blk * kMarkNodes + warp * 32u;
    const uint2 mine = node0 + lane < n ? marks[node0 + lane] : make_uint2(0u, 0u);
    const uint32_t c = __popc(mine.x) + __popc(mine.y);
    uint32_t incl = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= uint32_t(d)) incl += t;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    uint32_t base = counts[blk];
    for (int w = 0; w < int(warp); ++w) base += s_warp[w];
    uint32_t todo = __ballot_sync(0xffffffffu, c != 0u);
    while (todo) {   // four marked nodes at a time, their slots by lanes
      constexpr int kAhead = 4;
      uint32_t key[kAhead][2], m[kAhead][2], first[kAhead], slot[kAhead];
#pragma unroll
      for (int a = 0; a < kAhead; ++a) {
        const int l = todo ? __ffs(todo) - 1 : 0;
        m[a][0] = __shfl_sync(0xffffffffu, mine.x, l);
        m[a][1] = __shfl_sync(0xffffffffu, mine.y, l);
        if (!todo) m[a][0] = m[a][1] = 0u;
        todo &= todo - 1u;
        first[a] = base + __shfl_sync(0xffffffffu, incl - c, l);
        slot[a] = (node0 + uint32_t(l)) * uint32_t(kSlots) + lane;
#pragma unroll
        for (int h = 0; h < 2; ++h) key[a][h] = (m[a][h] >> lane) & 1u ? keys[slot[a] + 32u * h] : 0u;
      }
#pragma unroll
      for (int a = 0; a < kAhead; ++a) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
          if ((m[a][h] >> lane) & 1u) {
            const uint32_t p = first[a] + (h ? __popc(m[a][0]) : 0) + __popc(m[a][h] & lanemask_lt());
            kout[p] = key[a][h] - lo;
            vout[p] = slot[a] + 32u * h;
          }
      }
    }
    __syncthreads();   // s_warp is consumed
  }
}

}  // namespace

cudaError_t launch_frame_init(uint32_t* frame, uint32_t* hist, uint32_t hist_words, uint32_t* depth_hist, uint2* ranges,
                              uint32_t n_ranges, const TileLive& live, uint32_t n_tiles, int n_views, int sm_count,
                              cudaStream_t st) {
  const uint32_t most = std::max(hist_words, n_ranges);
  const uint32_t grid = std::min<uint32_t>((most + 255u) / 256u, uint32_t(sm_count) * 4u);
  k_frame_init<<<grid, 256, 0, st>>>(frame, hist, hist_words, depth_hist, ranges, n_ranges, live, n_tiles,
                                     uint32_t(n_views));
  return cudaGetLastError();
}

cudaError_t launch_slab_limits(uint32_t* frame, const uint32_t* depth_hist, int slabs, uint32_t cap_pairs,
                               cudaStream_t st) {
  k_slab_limits<<<1, 256, 0, st>>>(frame, depth_hist, slabs, cap_pairs);
  return cudaGetLastError();
}

cudaError_t launch_pick_slab(const uint32_t* keys, const uint2* rect, uint32_t cap_nodes, const uint2* list,
                             const InstFrame* inst_views, const TileLive& live, bool filter, const float2* depth_range,
                             uint2* marks, uint32_t* counts, uint32_t* kout, uint32_t* vout, uint32_t* frame, int slab,
                             int sm_count, cudaStream_t st) {
  const uint32_t blocks = (cap_nodes + kMarkNodes - 1) / kMarkNodes;
  if (!blocks) return cudaSuccess;
  uint32_t* words = frame + kSlabBase + slab * kSlabWords;
  const uint32_t grid = std::min<uint32_t>(blocks, uint32_t(sm_count) * 8u);
  const auto mark = filter ? k_mark<true> : k_mark<false>;
  mark<<<grid, 256, 0, st>>>(keys, rect, cap_nodes, list, inst_views, live, depth_range, marks, counts, frame, words);
  k_mark_scan<<<1, 1024, 0, st>>>(counts, cap_nodes, frame, words);
  k_gather<<<grid, 256, 0, st>>>(keys, cap_nodes, marks, counts, kout, vout, frame, words);
  return cudaGetLastError();
}

}  // namespace v3dg
