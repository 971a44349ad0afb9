// Device helpers shared by the kernels: acquire/release accesses and the bounded chained scan.
#pragma once

#include <cstdint>

#include "v3dg_internal.h"

namespace v3dg {

// A status word carries its flag and its value in one aligned 64-bit word, so a reader that sees
// the flag sees the value with it: relaxed (uncached, single-copy atomic) accesses suffice and no
// fence is needed.
__device__ __forceinline__ uint64_t ld_status(const uint64_t* p) {
  uint64_t v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void st_status(uint64_t* p, uint64_t v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ uint64_t pack_status(uint32_t epoch, uint64_t flag, uint32_t value) {
  return (uint64_t(epoch) << 34) | (flag << 32) | uint64_t(value);
}

// Decoupled look-back.  Tile t owns the status word status[t * stride]; a word whose epoch differs
// from `epoch` counts as not yet written, so the array never needs clearing between launches.
// chain_publish makes the tile's aggregate visible (tile 0 publishes its inclusive prefix);
// chain_lookback then sums the earlier tiles' words back to the first inclusive prefix and
// publishes the tile's own.  Every wait is bounded: after kSpinLimit polls the thread sets *err,
// publishes what it has (so that later tiles do not wait in turn) and returns.
__device__ __forceinline__ void chain_publish(uint64_t* status, uint32_t stride, uint32_t tile, uint32_t agg,
                                              uint32_t epoch) {
  st_status(status + size_t(tile) * stride, pack_status(epoch, tile == 0 ? kFlagPrefix : kFlagAgg, agg));
}

//
// The walk reads kW earlier tiles' words per round with independent loads, so a walk over n
// tiles costs about n / kW memory latencies instead of n: walks are long when tiles reach their
// look-back out of order (a tile passes every earlier one that has only its aggregate).
template <int kW = 1>
__device__ __forceinline__ uint32_t chain_lookback(uint64_t* status, uint32_t stride, uint32_t tile, uint32_t agg,
                                                   uint32_t epoch, uint32_t* err, uint32_t spin_limit = kSpinLimit) {
  if (tile == 0) return 0;
  uint32_t excl = 0;
  int64_t j = int64_t(tile) - 1;
  uint32_t spins = 0;
  while (j >= 0) {
    uint64_t s[kW];
#pragma unroll
    for (int w = 0; w < kW; ++w) s[w] = j - w >= 0 ? ld_status(status + size_t(j - w) * stride) : 0;
    // consume the words in order, up to the first inclusive prefix or the first unwritten word
    int used = 0;
    bool done = false, wait = false;
#pragma unroll
    for (int w = 0; w < kW; ++w) {
      if (done || wait || j - w < 0) continue;
      const uint32_t flag = uint32_t(s[w] >> 32) & 3u;
      if (uint32_t(s[w] >> 34) != epoch || flag == 0) {
        wait = true;
        continue;
      }
      excl += uint32_t(s[w]);
      ++used;
      done = flag == kFlagPrefix;
    }
    if (done) break;
    j -= used;
    if (wait) {
      if (++spins > spin_limit) {
        atomicOr(err, 1u);
        break;
      }
      if (spins > 32) __nanosleep(32);
    }
  }
  st_status(status + size_t(tile) * stride, pack_status(epoch, kFlagPrefix, excl + agg));
  return excl;
}

// The look-back of one chain by a whole warp (all 32 lanes call it, converged): a round reads the
// words of the 128 tiles before j (four independent loads a lane) and consumes them 32 at a time; the
// nearest inclusive prefix or unwritten word ends it.  About a thousand tiles of a persistent grid
// are in flight at once, and a walk passes every one of them that has only its aggregate: with 32
// words a round that took most of the expansion's time.  Returns the exclusive prefix in every lane;
// lane 0 publishes.
__device__ __forceinline__ uint32_t chained_exclusive_warp(uint64_t* status, uint32_t tile, uint32_t agg,
                                                           uint32_t epoch, uint32_t* err,
                                                           uint32_t spin_limit = kSpinLimit) {
  constexpr int kWords = 4;
  const uint32_t lane = threadIdx.x & 31u;
  if (lane == 0) chain_publish(status, 1, tile, agg, epoch);
  if (tile == 0) return 0;
  uint32_t excl = 0, spins = 0;
  int64_t j = int64_t(tile) - 1;
  bool done = false;
  while (!done) {
    uint64_t s[kWords];
#pragma unroll
    for (int w = 0; w < kWords; ++w) {
      const int64_t q = j - 32 * w - int64_t(lane);
      // before tile 0 (never reached: tile 0 publishes an inclusive prefix) reads as a zero prefix
      s[w] = q >= 0 ? ld_status(status + q) : pack_status(epoch, kFlagPrefix, 0);
    }
    bool wait = false;
#pragma unroll
    for (int w = 0; w < kWords; ++w) {
      if (done || wait) continue;   // (uniform)
      const uint32_t flag = uint32_t(s[w] >> 32) & 3u;
      const bool ready = uint32_t(s[w] >> 34) == epoch && flag != 0;
      const uint32_t not_ready = __ballot_sync(0xffffffffu, !ready);
      const uint32_t prefix = __ballot_sync(0xffffffffu, ready && flag == kFlagPrefix);
      const uint32_t first_wait = not_ready ? uint32_t(__ffs(not_ready) - 1) : 32u;
      const uint32_t first_prefix = prefix ? uint32_t(__ffs(prefix) - 1) : 32u;
      done = first_prefix < first_wait;
      wait = !done && first_wait < 32u;
      const uint32_t take = done ? first_prefix + 1 : first_wait;
      excl += __reduce_add_sync(0xffffffffu, lane < take ? uint32_t(s[w]) : 0u);
      j -= take;
    }
    if (wait) {
      if (++spins > spin_limit) {
        if (lane == 0) atomicOr(err, 1u);
        break;
      }
      if (spins > 32) __nanosleep(32);
    }
  }
  if (lane == 0) st_status(status + tile, pack_status(epoch, kFlagPrefix, excl + agg));
  return excl;
}

// Passes that a sort of `bits` key bits takes (the result is in the second buffers when odd).
__device__ __forceinline__ uint32_t sort_passes(uint32_t bits) { return (bits + 7u) / 8u; }

// The tiles of a pixel box (x0 | x1 << 16, y0 | y1 << 16, inclusive pixels).
struct TileRect {
  uint32_t x, y, w, h;
};

__device__ __forceinline__ TileRect tile_rect(const uint2 b) {
  const uint32_t x = (b.x & 0xFFFFu) >> 4, y = (b.y & 0xFFFFu) >> 4;
  return {x, y, ((b.x >> 16) >> 4) - x + 1u, ((b.y >> 16) >> 4) - y + 1u};
}

// Live bits of w <= 32 tiles from column x on; row: the first word of their row in TileLive::bits
// (the spare word after each row makes the second load valid).
__device__ __forceinline__ uint32_t live_row(const uint32_t* __restrict__ row, uint32_t x, uint32_t w) {
  const uint32_t v = __funnelshift_r(row[x >> 5], row[(x >> 5) + 1], x & 31u);
  return w < 32u ? v & ((1u << w) - 1u) : v;
}

__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// Block-wide exclusive scan of one uint32 per thread (blockDim.x == 32 * NW); returns the
// exclusive prefix and writes the block total to *total.  `scratch` holds NW + 1 words.
template <int NW>
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* scratch, uint32_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t incl = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += t;
  }
  if (lane == 31) scratch[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = lane < NW ? scratch[lane] : 0u;
    uint32_t wi = w;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, wi, d);
      if (lane >= d) wi += t;
    }
    if (lane < NW) scratch[lane] = wi - w;
    if (lane == NW - 1) scratch[NW] = wi;
  }
  __syncthreads();
  const uint32_t r = scratch[warp] + incl - v;
  *total = scratch[NW];
  __syncthreads();
  return r;
}

}  // namespace v3dg
