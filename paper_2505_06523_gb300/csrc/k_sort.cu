// Stable LSD radix sort of (uint32 key, uint32 value) pairs, onesweep style.
//
// One histogram kernel reads the keys once and counts all digit passes (as many passes as 8-bit
// digits need, the key's bits then spread evenly over them: 13 tile bits as 7 + 6); then each
// pass is a single kernel: a block scans the pass's digit counts, then takes the next 4096-key tile (virtual id from an atomic counter),
// ranks its keys per digit within each warp (stable: item-major then lane order within a warp,
// warps in order), publishes its per-digit counts (the sums of the warps' counts), reorders the
// tile by digit in shared memory (so that the global writes come out in runs), and looks back
// across earlier tiles per digit (one thread per digit, 4 status words per round, bounded waits)
// to find its global offsets.
#include <algorithm>
#include <utility>

#include "dev_common.cuh"

namespace v3dg {
namespace {

constexpr int kBins = kSortBins;
constexpr int kLookback = 4;   // status words read per look-back round
constexpr int kWarps = kSortThreads / 32;
constexpr int kSortBlocks = 4;   // resident blocks per SM (64 registers a thread, 52 KB of shared memory)
static_assert(kSortThreads >= kBins, "one thread per digit");

// Digit counts of every pass in one read of the keys (one shared histogram per pass and block).
// A thread counts a run of kHistRun consecutive keys and adds each pass's digit to the shared
// histogram only when it changes (runs of equal digits are common: the high digits of nearby
// keys -- depths of one cluster, tiles of one Gaussian -- coincide), which keeps shared-memory
// atomics on the few hot bins of the high digits from serialising.
constexpr int kHistRun = 16;
constexpr uint32_t kHistShort = 1u << 20;   // fewer keys than this: runs of four, so that more threads take part

// The digits of a sort: pass p covers `width` bits from begin + p * width (the last one what is left
// of them).  On the device, bits_dev replaces the host's bit range.
struct SortDigits {
  int begin, end, passes, width;
};

__host__ __device__ __forceinline__ SortDigits sort_digits(int begin, int end) {
  const int passes = (end - begin + 7) / 8;
  return {begin, end, passes, passes > 0 ? (end - begin + passes - 1) / passes : 8};
}

__device__ __forceinline__ SortDigits sort_digits(SortDigits d, const uint32_t* bits_dev) {
  return bits_dev ? sort_digits(0, int(*bits_dev)) : d;
}

// kOfSlots: of the visible slots' keys (which it also counts).
template <bool kOfSlots>
__global__ void __launch_bounds__(256)
k_hist(const uint32_t* __restrict__ keys, const uint32_t* __restrict__ n_dev, uint32_t cap, SortDigits dg,
       const uint32_t* __restrict__ bits_dev, uint32_t* __restrict__ hist, SortSlots slots) {
  __shared__ uint32_t sh[4][kBins], s_valid;
  const uint32_t n = kOfSlots ? min(slots.frame[kRenderNodes], slots.cap_nodes) * uint32_t(kSlots) : min(*n_dev, cap);
  const uint32_t lo = kOfSlots ? slots.slab[kSlabLo] : 0u;
  uint32_t valid = 0;
  const uint32_t run = n < kHistShort ? 4u : uint32_t(kHistRun);
  if (uint64_t(blockIdx.x) * blockDim.x * run >= n) return;   // no run for this block
  dg = sort_digits(dg, bits_dev);
  const int passes = dg.passes;
  for (int i = threadIdx.x; i < 4 * kBins; i += blockDim.x) sh[i / kBins][i % kBins] = 0;
  if (threadIdx.x == 0) s_valid = 0;
  __syncthreads();
  int sh_[4];
  uint32_t m[4];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    sh_[p] = dg.begin + dg.width * p;
    m[p] = (1u << min(max(dg.end - sh_[p], 0), dg.width)) - 1u;
  }
  const uint32_t runs = (n + run - 1) / run;
  const bool aligned = (reinterpret_cast<uintptr_t>(keys) & 15u) == 0;
  for (uint32_t r = blockIdx.x * blockDim.x + threadIdx.x; r < runs; r += gridDim.x * blockDim.x) {
    const uint32_t i0 = r * run;
    uint32_t cur[4], cnt[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      cur[p] = 0xFFFFFFFFu;
      cnt[p] = 0;
    }
    if (aligned && i0 + run <= n) {   // a full run: 16-byte loads
      const uint4* v = reinterpret_cast<const uint4*>(keys + i0);
#pragma unroll
      for (int q = 0; q < kHistRun / 4; ++q) {
        if (4u * q >= run) break;
        const uint4 k4 = v[q];
        const uint32_t kk[4] = {k4.x, k4.y, k4.z, k4.w};
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          if (kOfSlots && kk[t] == 0xFFFFFFFFu) continue;
          if (kOfSlots) ++valid;
#pragma unroll
          for (int p = 0; p < 4; ++p) {
            if (p >= passes) break;
            const uint32_t d = ((kk[t] - lo) >> sh_[p]) & m[p];
            if (d != cur[p]) {
              if (cnt[p]) atomicAdd(&sh[p][cur[p]], cnt[p]);
              cur[p] = d;
              cnt[p] = 0;
            }
            ++cnt[p];
          }
        }
      }
    } else {
      for (uint32_t i = i0; i < min(i0 + run, n); ++i) {
        const uint32_t k = keys[i];
        if (kOfSlots && k == 0xFFFFFFFFu) continue;
        if (kOfSlots) ++valid;
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          if (p >= passes) break;
          const uint32_t d = ((k - lo) >> sh_[p]) & m[p];
          if (d != cur[p]) {
            if (cnt[p]) atomicAdd(&sh[p][cur[p]], cnt[p]);
            cur[p] = d;
            cnt[p] = 0;
          }
          ++cnt[p];
        }
      }
    }
#pragma unroll
    for (int p = 0; p < 4; ++p)
      if (cnt[p]) atomicAdd(&sh[p][cur[p]], cnt[p]);
  }
  if (kOfSlots) {
    valid = __reduce_add_sync(0xffffffffu, valid);
    if ((threadIdx.x & 31) == 0 && valid) atomicAdd(&s_valid, valid);
  }
  __syncthreads();
  if (kOfSlots && threadIdx.x == 0 && s_valid) atomicAdd(slots.slab + kSlabCount, s_valid);
  for (int i = threadIdx.x; i < passes * kBins; i += blockDim.x) {
    const uint32_t c = sh[i / kBins][i % kBins];
    if (c) atomicAdd(hist + i, c);
  }
}

// The words of a standalone sort: n, tile counters and the gave-up flag, and the digit counts.  One
// launch in place of two memsets and a store (20M pairs, 32 bits: 659 -> 650 us a call; 300k, 13 bits: 72 -> 70).
__global__ void __launch_bounds__(kBins)
k_sort_init(uint32_t* __restrict__ words, uint32_t n, uint32_t* __restrict__ hist) {
  hist[blockIdx.x * kBins + threadIdx.x] = 0;
  if (blockIdx.x == 0 && threadIdx.x < kSortWords) words[threadIdx.x] = threadIdx.x == 0 ? n : 0u;
}

// What bounds a pass (20M pairs, ncu): the shared-memory pipe at 72% (38 wavefronts per 32 keys, most of
// them bank conflicts of the random digits) with 49% of the issue slots, behind it the look-back (9k of
// a tile's 34k cycles).  Pairs and per-digit words are 8 bytes wide so that ranking takes three shared
// accesses a key, not five, and reordering one, not two; full tiles test no bounds.  20M pairs, 32 bits:
// 692 -> 662 us a call, 300k pairs, 13 bits: 84 -> 75 us when they were made.  512 threads of 8 keys at 48 warps per SM: 730 us
// (more warps wait for the same pipe); 8 status words a look-back round: 686 us.
// Shared memory of a tile.
struct SortTile {
  uint2 kv[kSortTile];                // the tile's pairs, reordered by digit
  uint2 digit[kWarps][kBins];         // per warp and digit: the lanes holding it (zero between items), and its
                                      // count so far; after the ranking, its first position in the tile
  uint32_t start[kBins], cnt[kBins];  // each digit's first position in the tile and its count
  uint32_t goff[kBins];               // global destination offset minus start (mod 2^32)
  uint32_t scan[kWarps + 1];
  uint32_t tile;
};

// Ranks of a warp's items: the number of the warp's earlier keys of the same digit (item-major, then
// lane order), 16 bits each.  The lanes that share a digit come from a shared-memory OR of lane bits
// (measured faster than match.any, and than one vote per digit where the warp holds few of them).
// kFull: every item of the tile is a key; else the items with a bit in `live` (one bit each) are.
template <bool kFull>
__device__ __forceinline__ void rank_items(const uint32_t (&key)[kSortItems], uint32_t (&rank)[kSortItems / 2], uint2* mine,
                                           uint32_t live_items, int shift, uint32_t dmask) {
  const uint32_t lane = threadIdx.x & 31u;
#pragma unroll
  for (int i = 0; i < kSortItems; ++i) {
    const uint32_t live = kFull ? 0xffffffffu : __ballot_sync(0xffffffffu, (live_items >> i) & 1u);
    if (i % 2 == 0) rank[i / 2] = 0;
    if (kFull || (live >> lane) & 1u) {
      uint2* const at = mine + ((key[i] >> shift) & dmask);
      atomicOr(&at->x, 1u << lane);
      __syncwarp(live);
      const uint2 v = *at;   // the lanes of this digit, and its earlier keys
      const uint32_t before = __popc(v.x & lanemask_lt());
      __syncwarp(live);
      if (before == 0) *at = make_uint2(0u, v.y + __popc(v.x));   // the digit's first lane
      __syncwarp(live);
      rank[i / 2] |= (v.y + before) << (16 * (i % 2));
    }
  }
}

// Where a pass's keys and values come from: (kin, vin), the key's index as value, or (the first pass over
// a frame's slots) the visible slots' keys with the slot as value.  The last saves a compaction of the
// visible slots before the sort, a launch with a chain of waits and 16 bytes a Gaussian: depth stage of a
// 256x256 view (100k visible) 51 -> 43 us, of 5 instances at 640x360 113 -> 95 us, frames of 30-70M pairs
// 2.94 -> 2.84 and 4.54 -> 4.40 ms.
enum class Source { kPairs, kIndexed, kSlots };

template <Source kFrom>
__global__ void __launch_bounds__(kSortThreads, kSortBlocks)
k_onesweep(const uint32_t* __restrict__ kin, const uint32_t* __restrict__ vin, uint32_t* __restrict__ kout,
           uint32_t* __restrict__ vout, const uint32_t* __restrict__ n_dev, uint32_t cap, SortDigits dg, int pass,
           const uint32_t* __restrict__ bits_dev, const uint32_t* __restrict__ hist, uint64_t* __restrict__ status,
           uint32_t* __restrict__ tile_counter, uint32_t epoch, uint32_t* __restrict__ err,
           SortSlots slots) {
  extern __shared__ __align__(16) unsigned char s_sort[];
  SortTile& S = *reinterpret_cast<SortTile*>(s_sort);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr bool kOfSlots = kFrom == Source::kSlots;
  const uint32_t n = kOfSlots ? min(slots.frame[kRenderNodes], slots.cap_nodes) * uint32_t(kSlots) : min(*n_dev, cap);
  const uint32_t lo = kOfSlots ? slots.slab[kSlabLo] : 0u;
  const uint32_t ntiles = (n + kSortTile - 1) / kSortTile;
  dg = sort_digits(dg, bits_dev);
  if (pass >= dg.passes || blockIdx.x >= ntiles) return;
  const int shift = dg.begin + dg.width * pass;
  const uint32_t dmask = (1u << min(dg.end - shift, dg.width)) - 1u;
  // the first output position of this thread's digit: exclusive scan of the pass's digit counts
  uint32_t all;
  const uint32_t gexcl = block_exclusive_scan<kWarps>(tid < kBins ? hist[tid] : 0u, S.scan, &all);
  // persistent blocks: tiles in the order of an atomic counter, so every tile a look-back waits
  // for is held by a running block
  for (;;) {
    if (tid == 0) S.tile = atomicAdd(tile_counter, 1u);
    __syncthreads();
    const uint32_t tile = S.tile;
    if (tile >= ntiles) return;
    for (int i = tid; i < kWarps * kBins / 2; i += kSortThreads)
      reinterpret_cast<uint4*>(&S.digit[0][0])[i] = make_uint4(0u, 0u, 0u, 0u);
    const uint32_t base = tile * kSortTile + warp * (kSortItems * 32);
    const bool full = !kOfSlots && (tile + 1u) * kSortTile <= n;   // (n is below 2^32 - 4096)
    uint32_t key[kSortItems], val[kSortItems], rank[kSortItems / 2], live = 0;   // (live: unless full, the items that are keys)
#pragma unroll
    for (int i = 0; i < kSortItems; ++i) {
      const uint32_t idx = base + i * 32 + lane;
      const bool ok = full || idx < n;
      key[i] = ok ? kin[idx] : 0xFFFFFFFFu;
      if (!full) live |= uint32_t(kOfSlots ? key[i] != 0xFFFFFFFFu : ok) << i;
      if (kOfSlots) key[i] -= lo;
      val[i] = kFrom != Source::kPairs ? idx : (ok ? vin[idx] : 0u);
    }
    __syncthreads();
    if (full)
      rank_items<true>(key, rank, S.digit[warp], live, shift, dmask);
    else
      rank_items<false>(key, rank, S.digit[warp], live, shift, dmask);
    __syncthreads();
    // per digit (one thread each): the block count and the chain, then every warp's first position
    uint32_t cw[kWarps], cnt = 0;
    if (tid < kBins) {
#pragma unroll
      for (int w = 0; w < kWarps; ++w) {
        cw[w] = S.digit[w][tid].y;
        cnt += cw[w];
      }
    }
    if (tid <= dmask) chain_publish(status + tid, kBins, tile, cnt, epoch);   // as soon as they are known
    uint32_t total;
    const uint32_t start = block_exclusive_scan<kWarps>(cnt, S.scan, &total);
    if (tid < kBins) {
      S.start[tid] = start;
      S.cnt[tid] = cnt;
      uint32_t at = start;
#pragma unroll
      for (int w = 0; w < kWarps; ++w) {
        S.digit[w][tid].y = at;
        at += cw[w];
      }
    }
    __syncthreads();
    // reorder the tile by digit in shared memory (before the look-back, which needs none of the
    // tile's registers and gets the earlier tiles more time to publish)
#pragma unroll
    for (int i = 0; i < kSortItems; ++i) {
      if (full || (live >> i) & 1u) {
        const uint32_t d = (key[i] >> shift) & dmask;
        S.kv[S.digit[warp][d].y + ((rank[i / 2] >> (16 * (i % 2))) & 0xFFFFu)] = make_uint2(key[i], val[i]);
      }
    }
    if (tid <= dmask) {   // (the digit's count and start reloaded: no registers held over the reorder)
      const uint32_t excl = chain_lookback<kLookback>(status + tid, kBins, tile, S.cnt[tid], epoch, err);
      S.goff[tid] = gexcl + excl - S.start[tid];   // wraps; dst = goff + p is exact below 2^32
    }
    __syncthreads();
    if (full) {
#pragma unroll 8
      for (uint32_t i = 0; i < kSortItems; ++i) {
        const uint32_t p = tid + i * kSortThreads;
        const uint2 kv = S.kv[p];
        const uint32_t dst = S.goff[(kv.x >> shift) & dmask] + p;
        kout[dst] = kv.x;
        vout[dst] = kv.y;
      }
    } else {
      const uint32_t valid = total;
      for (uint32_t p = tid; p < valid; p += kSortThreads) {
        const uint2 kv = S.kv[p];
        const uint32_t dst = S.goff[(kv.x >> shift) & dmask] + p;
        kout[dst] = kv.x;
        vout[dst] = kv.y;
      }
    }
    __syncthreads();   // the tile's shared data is consumed before the next tile reuses it
  }  // next tile
}

// Diagnostic of the bounded waits: warp 0 runs the radix-sort passes' look-back (one thread,
// kLookback words per round), warp 1 the warp-wide look-back of the compaction and expansion
// kernels, each as tile 1 of its own two-word chain whose tile 0 publishes the prefix 1000 + warp
// (publish != 0) or never publishes (its word keeps an epoch that is not `epoch`).
__global__ void k_check_wait(uint64_t* __restrict__ status, uint32_t epoch, uint32_t spin_limit, int publish,
                             uint32_t* __restrict__ out) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint64_t* chain = status + 2 * warp;
  if (lane == 0 && publish) chain_publish(chain, 1, 0, 1000u + uint32_t(warp), epoch);
  __syncwarp();
  if (warp == 0) {
    if (lane == 0) out[0] = chain_lookback<kLookback>(chain, 1, 1, 1u, epoch, out + 2, spin_limit);
  } else {
    const uint32_t e = chained_exclusive_warp(chain, 1, 1u, epoch, out + 2, spin_limit);
    if (lane == 0) out[1] = e;
  }
}

}  // namespace

int g_sort_blocks_per_sm = 4;   // resident onesweep blocks per SM (set with the attributes)

cudaError_t sort_set_attributes() {
  const void* fns[] = {(const void*)k_onesweep<Source::kPairs>, (const void*)k_onesweep<Source::kIndexed>,
                       (const void*)k_onesweep<Source::kSlots>};
  for (const void* f : fns) {
    cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sizeof(SortTile)));
    if (e != cudaSuccess) return e;
  }
  int per_sm = 0;
  const cudaError_t e =
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_onesweep<Source::kPairs>, kSortThreads, sizeof(SortTile));
  if (e == cudaSuccess && per_sm > 0) g_sort_blocks_per_sm = per_sm;
  return e;
}

cudaError_t launch_sort_init(uint32_t* words, uint32_t n, uint32_t* hist, cudaStream_t st) {
  k_sort_init<<<kSortPasses, kBins, 0, st>>>(words, n, hist);
  return cudaGetLastError();
}

cudaError_t launch_sort(uint32_t* k0, uint32_t* v0, uint32_t* k1, uint32_t* v1, const uint32_t* n_dev,
                        uint32_t cap, int begin_bit, int end_bit, bool implicit_vals, const SortScratch& sc,
                        uint32_t* err_flag, uint32_t& epoch, int sm_count, cudaStream_t st, bool* result_in_1,
                        int* launches, const uint32_t* bits_dev, const SortSlots* slots) {
  const SortDigits dg = sort_digits(begin_bit, end_bit);
  *result_in_1 = false;
  if (dg.passes <= 0 || cap == 0) return cudaSuccess;
  if (dg.passes > kSortPasses) return cudaErrorInvalidValue;
  const uint32_t max_tiles = (cap + kSortTile - 1) / kSortTile;
  if (max_tiles > sc.max_tiles) return cudaErrorInvalidValue;
  // persistent grid: the resident blocks, whatever the capacity (surplus blocks cost launches)
  const uint32_t grid = std::min<uint32_t>(max_tiles, uint32_t(sm_count) * uint32_t(g_sort_blocks_per_sm));
  cudaError_t e = cudaSuccess;
  const SortSlots from = slots ? *slots : SortSlots{};
  if (slots)
    k_hist<true><<<sm_count * 4, 256, 0, st>>>(from.keys, n_dev, cap, dg, bits_dev, sc.hist, from);
  else
    k_hist<false><<<sm_count * 4, 256, 0, st>>>(k0, n_dev, cap, dg, bits_dev, sc.hist, from);
  ++*launches;
  uint32_t *ki = k0, *vi = v0, *ko = k1, *vo = v1;
  for (int p = 0; p < dg.passes; ++p) {
    epoch = (epoch + 1) & 0x3FFFFFFFu;
    if (epoch == 0) epoch = 1;
    const uint32_t ep = epoch;
    const auto kernel = p > 0           ? k_onesweep<Source::kPairs>
                        : slots         ? k_onesweep<Source::kSlots>
                        : implicit_vals ? k_onesweep<Source::kIndexed>
                                        : k_onesweep<Source::kPairs>;
    kernel<<<grid, kSortThreads, sizeof(SortTile), st>>>(p == 0 && slots ? from.keys : ki, vi, ko, vo, n_dev, cap, dg, p,
                                                         bits_dev, sc.hist + kBins * p, sc.status, sc.tile_counters + p, ep,
                                                         err_flag, from);
    ++*launches;
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    std::swap(ki, ko);
    std::swap(vi, vo);
  }
  *result_in_1 = (dg.passes & 1) != 0;
  return cudaSuccess;
}

cudaError_t launch_check_wait(uint64_t* status, uint32_t epoch, uint32_t spin_limit, int publish, uint32_t* out,
                              cudaStream_t st) {
  k_check_wait<<<1, 64, 0, st>>>(status, epoch, spin_limit, publish, out);
  return cudaGetLastError();
}

}  // namespace v3dg
