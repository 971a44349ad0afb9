// Per-tile front-to-back alpha blending (Sec. 2.1): C = sum_i c_i a_i prod_{j<i} (1 - a_j).
//
// k_blend (variant 0): the work item is one warp's 8x4 pixels of a 16x16 tile, and no warp ever waits
// for another one.  A warp walks its tile's depth-ordered list of pairs by the keys alone (they
// carry each Gaussian's box within the tile), collects the records whose box meets the bounding
// rectangle of its unfinished pixels, gathers 32 of them at a time (one per lane), stages them in
// two lists, one for each 4x4 half of its pixels, and composites those in order, each half-warp its
// own list: a = min(0.999, 2^(na dx^2 + nb dx dy + nc dy^2 + log2 o)), stopping before
// T (1 - a) < 1e-4.  Key loads, slot loads, record loads and compositing belong to successive
// batches, so the three dependent global latencies overlap with the compositing.
//
// The tiles with the longest lists go first, each sub-tile of them to a whole block (see "long lists").
//
// Why warps and 8x4: the blend is bound by the serial chain of the longest lists (a tile whose pixels
// never all finish walks its whole list: 125k pairs in the 1080p crowd) and, on full frames, by
// issue and shared-memory reads (near asset: 83% issue-active, 74% of the shared-memory pipe).  A block
// per tile with a barrier around each batch (the two-phase kernel before this one) had one block on
// each long list, its warps idle at the barriers.  Blend stage on a GB300, two-phase kernel -> a warp per
// sub-tile -> and long lists by blocks: 96x80 thumbnail 158 -> 37 -> 29 us, 256x256 viewer 266 -> 62 ->
// 51 us, 200 instances at 640x360 655 -> 275 -> 174 us, one asset filling 1080p 1671 -> 346 -> 364 us, the
// same 50 units away 768 -> 230 -> 127 us, crowd at 1080p (four slabs) 2.75 -> 2.03 -> 1.70 ms, 16 crowd
// views 31.9 -> 11.7 -> 12.0 ms (full frames lose a little: five blocks per SM, not six).  (With two
// slabs the near asset takes 353 us, with six the 16 views 12.3 ms; the crowd 1.80 ms on this code.)  The warp kernel
// with 8x8 pixels a warp (two per lane, four lists): 57 us, 510 us, 293 us and 1.74 ms on the thumbnail,
// the 200 instances, the near asset and the crowd; 8x4 with one list: 72, 414, 307 us and 1.41 ms
// against 35, 289, 309 us and 1.29 ms (one slab).
// Each record's mean is stored relative to the pixel origin of its first tile, so dx, dy are
// differences of small numbers.
//
// k_blend_px (variant 1): one block per tile, batches staged by bulk copies (see below).
#include <algorithm>

#include "dev_common.cuh"

namespace v3dg {
namespace {

constexpr int kBlendThreads = 128;   // four warps, independent except on long lists
constexpr int kBlendBlocks = 5;      // resident blocks per SM: 20 warps of at most 96 registers, 37 KB of shared memory each
constexpr uint32_t kLongPairs = 256;   // shortest list that a block blends together
constexpr int kPxThreads = 256;
constexpr int kPxWarps = kPxThreads / 32;
constexpr float kLog2MinAlpha = -7.9943534f;  // log2(1/255)

// log2(alpha) of a staged record at tile-local pixel centre (fx, fy); one definition for both variants
__device__ __forceinline__ float log2_alpha(const float4 g, const float4 c, float fx, float fy) {
  const float dx = fx - g.x, dy = fy - g.y;
  return fmaf(dx, fmaf(g.z, dx, g.w * dy), fmaf(c.x * dy, dy, c.y));
}

// One front-to-back step at a pixel (Sec. 2.1): alpha = min(0.999, 2^l2a), skipped below 1/255 and where
// l2a is not a number (a covariance that overflows), the pixel stops before T (1 - alpha) < 1e-4, else
// C += alpha T c and T *= 1 - alpha.  Variant 1 composites through this function, variant 0 through
// blend_step and blend_alpha: three forms of one rule, with the same roundings in the same order (2^l2a
// has the same bits from exp2f and ex2.approx for l2a >= log2(1/255)), so the images are bit-identical;
// a change goes into all three.  Returns whether the record contributed.
__device__ __forceinline__ bool composite_step(float l2a, float r, float g, float b, float& T, float& cr, float& cg,
                                               float& cb, bool& done) {
  const float a = l2a >= kLog2MinAlpha ? fminf(0.999f, exp2f(l2a)) : 0.f;
  if (a < 1.f / 255.f) return false;
  const float tn = T * (1.f - a);
  if (tn < 1e-4f) {
    done = true;
    return false;
  }
  const float wgt = a * T;
  cr = fmaf(wgt, r, cr);
  cg = fmaf(wgt, g, cg);
  cb = fmaf(wgt, b, cb);
  T = tn;
  return true;
}

// ---------------------------------------------------------------- variant 0: a warp per 8x4 pixels

constexpr int kSubTiles = 8;      // 8x4 pixel blocks of a tile: two across, four down
constexpr int kScanKeys = 8;      // keys per lane and scan step
constexpr int kRing = 512;        // list positions waiting to be gathered: < 32 + 32 * kScanKeys
constexpr uint32_t kNoKey = (15u << 20) | (3u << 28);   // an empty box: meets no rectangle of a sub-tile

constexpr int kAhead = 4;         // records whose alphas are computed ahead of the transmittance chain

// The staged records, one list for each 4x4 half of the sub-tile: the two half-warps composite
// different records at once, so that a small Gaussian occupies 16 lanes and not 32.
struct BlendWarp {
  float4 g[2][32];     // (u, v, na, nb) in the tile's pixel frame
  float4 c[2][32];     // (nc, log2 o, mask of the warp's pixels in the record's box, b)
  float2 rg[2][32];    // (r, g)
  uint32_t ring[kRing];
};

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// One front-to-back step at a pixel, as composite_step, by predicated instructions (a branch per record
// costs more than all of them).  in: not zero where the pixel is unfinished and in the record's box;
// l2a: its log2 alpha; al: min(0.999, 2^l2a).  A record below 1/255 (or not a number) does nothing.
// t carries the transmittance along: past the record that takes it below 1e-4 it stays below, so
// nothing else contributes; T stays as the last contributing record left it.
__device__ __forceinline__ void blend_step(uint32_t in, float l2a, float al, float cr, float cg, float cb, float& t,
                                           float& T, float& r, float& g, float& b) {
  asm("{\n\t.reg .pred p, q;\n\t.reg .f32 om, tn, w;\n\t"
      "setp.ne.u32 p, %5, 0;\n\t"
      "setp.ge.and.f32 p, %6, %11, p;\n\t"
      "setp.ge.and.f32 p, %7, %12, p;\n\t"
      "sub.rn.f32 om, 0f3F800000, %7;\n\t"
      "mul.rn.f32 w, %7, %0;\n\t"
      "mul.rn.f32 tn, %0, om;\n\t"
      "setp.ge.and.f32 q, tn, %13, p;\n\t"
      "@p mov.f32 %0, tn;\n\t"
      "@q mov.f32 %1, tn;\n\t"
      "@q fma.rn.f32 %2, w, %8, %2;\n\t"
      "@q fma.rn.f32 %3, w, %9, %3;\n\t"
      "@q fma.rn.f32 %4, w, %10, %4;\n\t}"
      : "+f"(t), "+f"(T), "+f"(r), "+f"(g), "+f"(b)
      : "r"(in), "f"(l2a), "f"(al), "f"(cr), "f"(cg), "f"(cb), "f"(kLog2MinAlpha), "f"(1.f / 255.f), "f"(1e-4f));
}

// The bounding rectangle of a warp's unfinished pixels, as the constants of key_hits: rows r0..r1
// and column quads c0..c1 of the tile.
struct KeyTest {
  uint32_t lo, hi;
};

// live: the unfinished pixels of the sub-tile, bit 16 (x / 4) + 4 y + x % 4, not zero.
__device__ __forceinline__ KeyTest key_test(uint32_t live, uint32_t sub) {
  const uint32_t any = (live | (live >> 16)) & 0xFFFFu;
  const uint32_t r0 = 4u * (sub >> 1) + (uint32_t(__ffs(any) - 1) >> 2);
  const uint32_t r1 = 4u * (sub >> 1) + (uint32_t(31 - __clz(any)) >> 2);
  const uint32_t c0 = 2u * (sub & 1u) + ((live & 0xFFFFu) ? 0u : 1u);
  const uint32_t c1 = 2u * (sub & 1u) + ((live >> 16) ? 1u : 0u);
  return {((15u - r1) << 20) | ((3u - c1) << 28), ((16u - r0) << 20) | ((4u - c0) << 26)};
}

// Whether the box that a pair key carries (rows y0..y1, column quads q0..q1, see kPairTileMask)
// meets the rectangle.  Four comparisons in two additions: y0 > r1 carries into bit 24 and q0 > c1
// into bit 30 of the first sum, y1 >= r0 into bit 24 and q1 >= c0 into bit 28 of the second.
__device__ __forceinline__ bool key_hits(uint32_t key, KeyTest t) {
  const uint32_t a = (key & 0x30F00000u) + t.lo;
  const uint32_t b = ((key >> 4) & 0x0CF00000u) + t.hi;
  return ((a & 0x41000000u) | (~b & 0x11000000u)) == 0u;
}

// The tile at position i of the classes' regions, one after the other (see k_blend_items; cls_incl:
// in lane c, the tiles of classes 0 .. c).  All lanes call it.
__device__ __forceinline__ uint32_t item_tile(const uint32_t* __restrict__ items, uint32_t n_tiles, uint32_t cls_incl, uint32_t i) {
  const uint32_t cls = __popc(__ballot_sync(0xffffffffu, cls_incl <= i));   // lanes beyond the classes hold 2^32 - 1
  const uint32_t before = __shfl_sync(0xffffffffu, cls_incl, cls ? cls - 1u : 0u);
  return items[size_t(cls) * n_tiles + (i - (cls ? before : 0u))];
}

// In lane c, the tiles of classes 0 .. c.
__device__ __forceinline__ uint32_t item_classes(const uint32_t* __restrict__ class_count) {
  const uint32_t lane = threadIdx.x & 31u;
  uint32_t incl = lane < uint32_t(kItemClasses) ? class_count[lane] : 0u;
#pragma unroll
  for (int d = 1; d < kItemClasses; d <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= uint32_t(d)) incl += t;
  }
  return lane < uint32_t(kItemClasses) ? incl : 0xFFFFFFFFu;
}

// ---- long lists: a block per sub-tile
// What bounds a sub-tile with a long list is its chain: 37k keys of a horizon tile took one warp 0.3 ms,
// a third each for scanning, gathering and compositing, with the chip idle.  So the tiles whose lists
// are at least a warp's share of the slab's pairs go first, each sub-tile to a whole block: three warps
// scan, gather and compute the alphas of every pixel, the fourth only composites.  Hit number
// 96 r + 32 w + j of the list is record j of producer w's batch in round r; in round r the producers make
// that round's batches while the consumer composites the round before, one block barrier per round.
constexpr int kProducers = kBlendThreads / 32 - 1;
constexpr uint32_t kRoundHits = 32 * kProducers;
constexpr int kLongScan = 4;       // keys per producer lane and scan step
// Positions waiting for their slots to be loaded: a scan for one round more starts with less than that
// round's hits missing, all earlier rounds' slots loaded, and ends with at most a step more.
constexpr uint32_t kLongRing = 512;
static_assert(kRoundHits + kRoundHits * kLongScan <= kLongRing, "ring");

struct BlendBlock {
  float4 g[kProducers][2][32];                 // staged records, as in BlendWarp
  float4 c[kProducers][2][32];
  float alpha[2][kProducers][32][32];          // [round parity][producer][record][pixel], 0: does not contribute
  float2 rg[2][kProducers][2][32];             // colours of each half's records
  float blue[2][kProducers][2][32];
  uint32_t n[2][kProducers];                   // records of the longer list, a multiple of 4
  uint32_t ring[kLongRing];
  uint32_t count[kProducers];
  uint32_t live[2], hits[2], ended[2], item;
};

__device__ __forceinline__ void producers_sync() {
  __syncwarp();
  asm volatile("bar.sync 1, %0;" ::"n"(32 * kProducers) : "memory");
}

// blend_step with the alpha ready (0: does nothing).
__device__ __forceinline__ void blend_alpha(float a, const float2 rg, float blue, float& t, float& T, float& r, float& g, float& b) {
  asm("{\n\t.reg .pred q;\n\t.reg .f32 om, w;\n\t"
      "sub.rn.f32 om, 0f3F800000, %5;\n\t"
      "mul.rn.f32 w, %5, %0;\n\t"
      "mul.rn.f32 %0, %0, om;\n\t"
      "setp.gt.f32 q, %5, 0f00000000;\n\t"
      "setp.ge.and.f32 q, %0, %9, q;\n\t"
      "@q mov.f32 %1, %0;\n\t"
      "@q fma.rn.f32 %2, w, %6, %2;\n\t"
      "@q fma.rn.f32 %3, w, %7, %3;\n\t"
      "@q fma.rn.f32 %4, w, %8, %4;\n\t}"
      : "+f"(t), "+f"(T), "+f"(r), "+f"(g), "+f"(b)
      : "f"(a), "f"(rg.x), "f"(rg.y), "f"(blue), "f"(1e-4f));
}

// The mask of a record's box (third float4) within the sub-tile whose first pixel is (ox, oy).
__device__ __forceinline__ uint32_t box_mask(const float4 r2, int ox, int oy) {
  const uint32_t bx = __float_as_uint(r2.z), by = __float_as_uint(r2.w);
  const int x0 = max(int(bx & 0xFFFFu) - ox, 0), x1 = min(int(bx >> 16) - ox, 7);
  const int y0 = max(int(by & 0xFFFFu) - oy, 0), y1 = min(int(by >> 16) - oy, 3);
  if (x0 > x1 || y0 > y1) return 0u;
  const uint32_t cols = (0xFFu >> (7 - x1)) & (0xFFu << x0), rows = (0xFFFFu << (4 * y0)) & (0xFFFFu >> (12 - 4 * y1));
  return (((cols & 15u) * 0x1111u) & rows) | (((((cols >> 4) & 15u) * 0x1111u) & rows) << 16);
}

// One sub-tile by the whole block: list positions [sp, end) of it, `live` pixels.  The consumer warp's
// T, colour and mybit are the pixels' state (bit 0 once stopped), as in k_blend; returns the pixels
// that are left.
template <bool kCount>
__device__ __forceinline__ uint32_t blend_long(BlendBlock& S, uint32_t sp, uint32_t end, uint32_t live, uint32_t sub, int tx,
                                               int ty, float fx, float fy, const uint32_t* __restrict__ tk,
                                               const uint32_t* __restrict__ pv, const float4* __restrict__ rec,
                                               uint32_t cap_slots, float& T, float& cr, float& cg, float& cb,
                                               uint32_t& mybit, uint32_t& n_eval, uint32_t& n_contrib) {
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, half = lane >> 4;
  const int sx = tx * 16 + 8 * int(sub & 1u), sy = ty * 16 + 4 * int(sub >> 1);
  const uint32_t lanebit = 1u << lane;
  const int w = int(warp) - 1;   // producer
  if (threadIdx.x == 0) S.live[1] = live;
  __syncthreads();
  uint32_t tail = 0, key[kLongScan], slot = 0xFFFFFFFFu;
  float4 r0, r1, r2;
  bool valid = false;
  float t = T;
  const auto load_keys = [&] {
#pragma unroll
    for (int k = 0; k < kLongScan; ++k) {
      const uint32_t pos = sp + uint32_t(w) * (32u * kLongScan) + 32u * k + lane;
      key[k] = pos < end ? tk[pos] : kNoKey;
    }
  };
  // more hits until hit number `want` is known (or the list has ended)
  const auto scan = [&](uint32_t want, uint32_t live_now) {
    if (tail >= want || sp >= end) return;
    const KeyTest kt = key_test(live_now, sub);
    do {
      uint32_t b[kLongScan], cnt = 0;
#pragma unroll
      for (int k = 0; k < kLongScan; ++k) {
        b[k] = __ballot_sync(0xffffffffu, key_hits(key[k], kt));
        cnt += __popc(b[k]);
      }
      if (lane == 0) S.count[w] = cnt;
      producers_sync();
      uint32_t at = tail;
#pragma unroll
      for (int p = 0; p < kProducers; ++p) {
        const uint32_t c = S.count[p];
        if (p < w) at += c;
        tail += c;
      }
#pragma unroll
      for (int k = 0; k < kLongScan; ++k) {
        if ((b[k] >> lane) & 1u)
          S.ring[(at + __popc(b[k] & lanemask_lt())) % kLongRing] = sp + uint32_t(w) * (32u * kLongScan) + 32u * k + lane;
        at += __popc(b[k]);
      }
      sp += kRoundHits * kLongScan;
      load_keys();
      producers_sync();   // the counts are read, the ring's new positions visible
    } while (tail < want && sp < end);
  };
  const auto load_slot = [&](uint32_t round) {
    const uint32_t i = round * kRoundHits + 32u * uint32_t(w) + lane;
    slot = i < tail ? pv[S.ring[i % kLongRing]] : 0xFFFFFFFFu;
  };
  const auto load_record = [&] {
    valid = slot < cap_slots;
    if (valid) {
      const float4* r = rec + 3 * size_t(slot);
      r0 = r[0];
      r1 = r[1];
      r2 = r[2];
    }
  };
  if (w >= 0) {
    load_keys();
    scan(kRoundHits, live);
    load_slot(0);
    load_record();
    scan(2u * kRoundHits, live);
    load_slot(1);
  }
  for (uint32_t round = 0;; ++round) {
    const uint32_t par = round & 1u;
    if (w >= 0) {
      const uint32_t live_now = S.live[par ^ 1u];
      scan((round + 3u) * kRoundHits, live_now);
      // stage this round's batch
      const uint32_t m = valid ? box_mask(r2, sx, sy) & live_now : 0u;
      const uint32_t ml = m & 0xFFFFu, mr = m >> 16;
      const uint32_t bl = __ballot_sync(0xffffffffu, ml != 0u), br = __ballot_sync(0xffffffffu, mr != 0u);
      const int nl = __popc(bl), nr = __popc(br), n = (max(nl, nr) + 3) & ~3;
      if (m) {
        const uint32_t org = __float_as_uint(r2.y);
        const float ox = float(16 * (tx - int(org & 0xFFFFu))), oy = float(16 * (ty - int(org >> 16)));
        const float4 g = make_float4(r0.x - ox, r0.y - oy, r0.z, r0.w);
        const float4 c = make_float4(r1.x, r1.y, __uint_as_float(m), 0.f);
        const float2 rg = make_float2(r1.z, r1.w);
        if (ml) {
          const int i = __popc(bl & lanemask_lt());
          S.g[w][0][i] = g;
          S.c[w][0][i] = c;
          S.rg[par][w][0][i] = rg;
          S.blue[par][w][0][i] = r2.x;
        }
        if (mr) {
          const int i = __popc(br & lanemask_lt());
          S.g[w][1][i] = g;
          S.c[w][1][i] = c;
          S.rg[par][w][1][i] = rg;
          S.blue[par][w][1][i] = r2.x;
        }
      }
      if (int(lane) >= nl && int(lane) < n) S.c[w][0][lane].z = 0.f;   // (records without pixels)
      if (int(lane) >= nr && int(lane) < n) S.c[w][1][lane].z = 0.f;
      if (lane == 0) {
        S.n[par][w] = uint32_t(n);
        if (w == 0) {
          S.hits[par] = tail;
          S.ended[par] = sp >= end ? 1u : 0u;
        }
      }
      load_record();
      load_slot(round + 2u);
      __syncwarp();
      for (int i = 0; i < n; i += 4) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float4 c = S.c[w][half][i + q];
          const float l2a = log2_alpha(S.g[w][half][i + q], c, fx, fy);
          const float al = fminf(0.999f, ex2_approx(l2a));
          const bool in = (__float_as_uint(c.z) & lanebit) != 0u;
          if (kCount) n_eval += in ? 1u : 0u;
          S.alpha[par][w][i + q][lane] = in && l2a >= kLog2MinAlpha && al >= 1.f / 255.f ? al : 0.f;
        }
      }
    } else if (round > 0) {
      const uint32_t prev = par ^ 1u;
      for (int p = 0; p < kProducers; ++p) {
        const int n = int(S.n[prev][p]);
        for (int i = 0; i < n; i += 4) {
          float a[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) a[q] = S.alpha[prev][p][i + q][lane];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            if (kCount) n_contrib += a[q] > 0.f && t * (1.f - a[q]) >= 1e-4f ? 1u : 0u;
            blend_alpha(a[q], S.rg[prev][p][half][i + q], S.blue[prev][p][half][i + q], t, T, cr, cg, cb);
          }
        }
      }
      if (t < 1e-4f) mybit = 0u;
      live = __ballot_sync(0xffffffffu, mybit != 0u);
      if (lane == 0) S.live[par] = live;
    } else if (lane == 0) {
      S.live[par] = live;
    }
    __syncthreads();
    // the hits below round * kRoundHits are composited
    if (S.live[par] == 0u || (S.ended[par] && round * kRoundHits >= S.hits[par])) break;
  }
  const uint32_t left = S.live[0] & S.live[1];
  __syncthreads();   // the block's shared words are read
  return left;
}

// kCount: also count the evaluations and contributions into work[0], work[1].
// kSlabbed: one of the frame's depth slabs (the first one covers every tile, later ones those with
// pairs): the pixels' T goes through live.state (negative once the pixel has stopped) and their
// colour through the image, and the 4x4 blocks whose last pixel stops are cleared in live.
template <bool kCount, bool kSlabbed>
__global__ void __launch_bounds__(kBlendThreads, kBlendBlocks)
k_blend(const uint2* __restrict__ ranges, const uint32_t* __restrict__ items, uint32_t n_tiles,
        const uint32_t* __restrict__ class_count, uint32_t* __restrict__ slab, bool first, TileLive live_tiles, const uint32_t* __restrict__ tk,
        const uint32_t* __restrict__ pv, const float4* __restrict__ rec, uint32_t cap_slots, int width, int height,
        int tiles_x, int tiles_per_view, float* __restrict__ rgb, float* __restrict__ t_out,
        unsigned long long* __restrict__ work, uint32_t* __restrict__ frame, uint32_t* __restrict__ sticky) {
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (frame[kOverflow]) atomicOr(sticky, 1u);
    if (frame[kTimeout]) atomicOr(sticky + 1, 1u);
  }
  const uint32_t cls_incl = item_classes(class_count);
  // (a later slab leaves out the tiles without pairs)
  const uint32_t n_items =
      (kSlabbed && !first ? __shfl_sync(0xffffffffu, cls_incl, kItemClasses - 2) : n_tiles) * uint32_t(kSubTiles);
  extern __shared__ __align__(16) unsigned char s_blend[];   // BlendBlock, then BlendWarp x 4
  BlendBlock& B = *reinterpret_cast<BlendBlock*>(s_blend);
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  BlendWarp& S = reinterpret_cast<BlendWarp*>(s_blend)[warp];
  uint32_t n_eval = 0, n_contrib = 0;
  // the classes of long lists: all of them at least a warp's share of the slab's pairs (each key is
  // scanned by eight warps), below which a warp on its own does not hold the frame up, and the block's
  // work beyond the stop of a short chain costs more (half the share: 1001x563 143 -> 170 us; twice:
  // 200 instances 174 -> 256 us), and at least kLongPairs
  const uint32_t share = max(slab[kSlabPairs] / max(gridDim.x * (kBlendThreads / 32u) / kSubTiles, 1u), kLongPairs);
  const int long_classes = min(max(16 - int(32 - __clz(share - 1u)), -1), kItemClasses - 3) + 1;   // class c: 2^(16 - c) pairs or more
  const uint32_t n_long = long_classes ? __shfl_sync(0xffffffffu, cls_incl, long_classes - 1) * uint32_t(kSubTiles) : 0u;
  bool by_block = n_long > 0u;
  for (;;) {
    uint32_t it = 0;
    if (by_block) {
      if (threadIdx.x == 0) B.item = atomicAdd(slab + kSlabBlendLong, 1u);
      __syncthreads();
      it = B.item;
      __syncthreads();
      by_block = it < n_long;
      if (!by_block) continue;
    } else {
      if (lane == 0) it = atomicAdd(slab + kSlabBlendItem, 1u);
      it = __shfl_sync(0xffffffffu, it, 0) + n_long;
      if (it >= n_items) break;
    }
    const int tile = int(item_tile(items, n_tiles, cls_incl, it / kSubTiles));   // (view, tile) id
    const uint32_t sub = it % kSubTiles;
    const int view = tile / tiles_per_view, vt = tile - view * tiles_per_view;
    const int tx = vt % tiles_x, ty = vt / tiles_x;
    const int sx = 8 * int(sub & 1u), sy = 4 * int(sub >> 1);   // the sub-tile's first pixel in the tile
    const int lx = sx + int(4u * (lane >> 4) + (lane & 3u)), ly = sy + int((lane >> 2) & 3u);
    const int px = tx * 16 + lx, py = ty * 16 + ly;
    const float fx = float(lx) + 0.5f, fy = float(ly) + 0.5f;
    const bool inside = px < width && py < height;
    float T = 1.f, cr = 0.f, cg = 0.f, cb = 0.f;
    uint32_t mybit = inside ? 1u << lane : 0u;   // 0 once the pixel has stopped
    const size_t p = (size_t(view) * height + py) * width + px;   // (inside: the pixel's place)
    if (kSlabbed && !first && inside) {
      T = live_tiles.state[p];
      if (T < 0.f) {
        mybit = 0u;
        T = -T;
      }
    }
    uint32_t live = __ballot_sync(0xffffffffu, mybit != 0u);
    if (kSlabbed && !first) {
      if (live == 0u) continue;   // (finished in an earlier slab; the same in all of a block's warps)
      if (inside) {
        cr = rgb[3 * p + 0];
        cg = rgb[3 * p + 1];
        cb = rgb[3 * p + 2];
      }
    }
    const uint2 range = ranges[tile];
    uint32_t sp = range.x;                  // next list position to scan
    const uint32_t end = live ? range.y : range.x;
    if (by_block) {
      if (sp < end)
        live = blend_long<kCount>(B, sp, end, live, sub, tx, ty, fx, fy, tk, pv, rec, cap_slots, T, cr, cg, cb, mybit, n_eval,
                                  n_contrib);
      if (warp != 0u) continue;   // (the consumer has the pixels)
    } else if (sp < end) {
      KeyTest kt = key_test(live, sub);
      uint32_t head = 0, tail = 0;          // the ring's waiting positions
      uint32_t key[kScanKeys];
#pragma unroll
      for (int k = 0; k < kScanKeys; ++k) {
        const uint32_t pos = sp + 32u * k + lane;
        key[k] = pos < end ? tk[pos] : kNoKey;
      }
      // the next at most 32 hits of the list, their slots one per lane; returns their number
      auto next_slots = [&](uint32_t& slot) -> uint32_t {
        while (tail - head < 32u && sp < end) {
#pragma unroll
          for (int k = 0; k < kScanKeys; ++k) {
            const bool hit = key_hits(key[k], kt);
            const uint32_t b = __ballot_sync(0xffffffffu, hit);
            if (hit) S.ring[(tail + __popc(b & lanemask_lt())) % kRing] = sp + 32u * k + lane;
            tail += __popc(b);
          }
          sp += 32u * kScanKeys;
#pragma unroll
          for (int k = 0; k < kScanKeys; ++k) {   // the next step's keys, on their way during the compositing
            const uint32_t pos = sp + 32u * k + lane;
            key[k] = pos < end ? tk[pos] : kNoKey;
          }
        }
        __syncwarp();
        const uint32_t n = min(tail - head, 32u);
        slot = lane < n ? pv[S.ring[(head + lane) % kRing]] : 0xFFFFFFFFu;
        head += n;
        return n;
      };
      float4 r0, r1, r2;
      bool valid = false;
      auto load_record = [&](uint32_t slot) {
        valid = slot < cap_slots;   // (a slot beyond the buffers never occurs in a valid frame)
        if (valid) {
          const float4* r = rec + 3 * size_t(slot);
          r0 = r[0];
          r1 = r[1];
          r2 = r[2];
        }
      };
      uint32_t slot;
      uint32_t n_rec = next_slots(slot);
      load_record(slot);
      uint32_t n_slot = next_slots(slot);
      while (n_rec) {
        // stage the records whose box holds an unfinished pixel of this warp, in order
        const uint32_t m = valid ? box_mask(r2, tx * 16 + sx, ty * 16 + sy) & live : 0u;
        const uint32_t ml = m & 0xFFFFu, mr = m >> 16;   // the left and right 4x4 pixels
        const uint32_t bl = __ballot_sync(0xffffffffu, ml != 0u), br = __ballot_sync(0xffffffffu, mr != 0u);
        const int nl = __popc(bl), nr = __popc(br);
        const int n = (max(nl, nr) + kAhead - 1) / kAhead * kAhead;
        if (m) {
          const uint32_t org = __float_as_uint(r2.y);
          const float ox = float(16 * (tx - int(org & 0xFFFFu))), oy = float(16 * (ty - int(org >> 16)));
          const float4 g = make_float4(r0.x - ox, r0.y - oy, r0.z, r0.w);
          const float4 c = make_float4(r1.x, r1.y, __uint_as_float(m), r2.x);
          const float2 rg = make_float2(r1.z, r1.w);
          if (ml) {
            const int i = __popc(bl & lanemask_lt());
            S.g[0][i] = g;
            S.c[0][i] = c;
            S.rg[0][i] = rg;
          }
          if (mr) {
            const int i = __popc(br & lanemask_lt());
            S.g[1][i] = g;
            S.c[1][i] = c;
            S.rg[1][i] = rg;
          }
        }
        // the shorter list, and both up to a multiple of kAhead, end in records without pixels
        if (int(lane) >= nl && int(lane) < n) S.c[0][lane].z = 0.f;
        if (int(lane) >= nr && int(lane) < n) S.c[1][lane].z = 0.f;
        n_rec = n_slot;
        load_record(slot);
        n_slot = n_rec ? next_slots(slot) : 0u;   // (n_slot == 0: the loop ends after this batch)
        __syncwarp();
        const float4* sg = S.g[lane >> 4];
        const float4* sc = S.c[lane >> 4];
        const float2* srg = S.rg[lane >> 4];
        // kAhead records at a time: their alphas are independent, only t is a chain
        float t = T;
        for (int i = 0; i < n; i += kAhead) {
          float l2a[kAhead], al[kAhead], blue[kAhead];
          uint32_t in[kAhead];
#pragma unroll
          for (int q = 0; q < kAhead; ++q) {
            const float4 c = sc[i + q];
            l2a[q] = log2_alpha(sg[i + q], c, fx, fy);
            al[q] = fminf(0.999f, ex2_approx(l2a[q]));
            in[q] = __float_as_uint(c.z) & mybit;
            blue[q] = c.w;
          }
#pragma unroll
          for (int q = 0; q < kAhead; ++q) {
            if (kCount) {
              n_eval += in[q] ? 1u : 0u;
              n_contrib += in[q] && l2a[q] >= kLog2MinAlpha && al[q] >= 1.f / 255.f && t * (1.f - al[q]) >= 1e-4f ? 1u : 0u;
            }
            const float2 rg = srg[i + q];
            blend_step(in[q], l2a[q], al[q], rg.x, rg.y, blue[q], t, T, cr, cg, cb);
          }
          if (t < 1e-4f) mybit = 0u;   // the pixel has stopped
        }
        live = __ballot_sync(0xffffffffu, mybit != 0u);
        if (live == 0u) break;
        __syncwarp();   // the batch is consumed before the next one is staged
        kt = key_test(live, sub);
      }
      __syncwarp();   // the warp's staged records and ring are free for the next item
    }
    if (inside) {
      rgb[3 * p + 0] = cr;
      rgb[3 * p + 1] = cg;
      rgb[3 * p + 2] = cb;
      if (t_out) t_out[p] = T;
      if (kSlabbed) live_tiles.state[p] = mybit ? T : -T;
    }
    if (kSlabbed && lane == 0 && (!(live & 0xFFFFu) || !(live >> 16))) {
      // 4x4 blocks without an unfinished pixel (again, where an earlier slab finished them)
      const uint32_t left = 1u << (4u * (sub >> 1) + 2u * (sub & 1u));
      const uint32_t gone = (live & 0xFFFFu ? 0u : left) | (live >> 16 ? 0u : left << 1);
      const uint32_t old = atomicAnd(live_tiles.blocks + tile, ~gone);
      if (old != 0u && (old & ~gone) == 0u) {   // the tile's last
        const TileLive& L = live_tiles;
        atomicAnd(L.bits + size_t(view * L.tiles_y + ty) * L.words + (tx >> 5), ~(1u << (tx & 31)));
        const uint32_t gx = uint32_t(tx) >> 3, row = view * L.groups_y + (uint32_t(ty) >> 3);
        if (atomicSub(L.coarse_tiles + size_t(row) * L.groups_x + gx, 1u) == 1u)   // and the group's last
          atomicAnd(L.coarse + size_t(row) * L.coarse_words + (gx >> 5), ~(1u << (gx & 31u)));
      }
    }
  }  // next item
  if (kCount) {
    unsigned long long e = n_eval, cnt = n_contrib;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      e += __shfl_xor_sync(0xffffffffu, e, d);
      cnt += __shfl_xor_sync(0xffffffffu, cnt, d);
    }
    if (lane == 0) {
      atomicAdd(work, e);
      atomicAdd(work + 1, cnt);
    }
  }
}

// True when the box that a pair key carries (see kPairTileMask: rows y0..y1, column quads
// q0..q1) holds a pixel whose bit is set in `live` (one word per row pair: row 2w in bits
// 0..15, row 2w + 1 in 16..31).
__device__ __forceinline__ bool box_live(uint32_t key, const uint32_t* live) {
  const uint32_t y0 = (key >> 20) & 15u, y1 = (key >> 24) & 15u, q0 = (key >> 28) & 3u, q1 = key >> 30;
  const uint32_t cols = (0xFFFFu >> (12u - 4u * q1)) & (0xFFFFu << (4u * q0));
  for (uint32_t y = y0; y <= y1; ++y)
    if ((live[y >> 1] >> ((y & 1u) * 16u)) & cols) return true;
  return false;
}

// The next batch of a work item: the records from list position *sp on whose box (carried by the
// pair key) holds an unfinished pixel, in list order, at most kBatch of them; kScan * 256
// consecutive keys per step.  Writes their slots to s_qslot and, when s_rows is given, the row
// pairs their box spans (bit w: rows 2w, 2w + 1) to s_rows; advances *sp past the last record
// taken and returns the batch size (uniform across the block; called by all threads).
template <int kBatch>
__device__ __forceinline__ uint32_t fill_batch(const uint32_t* __restrict__ tk, const uint32_t* __restrict__ pv,
                                               uint32_t end, uint32_t cap_slots, const uint32_t* s_live,
                                               uint32_t* s_qslot, uint8_t* s_rows, uint32_t* s_cnt,
                                               uint32_t* s_resume, uint32_t* s_total, uint32_t* sp_io) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t sp = *sp_io, q = 0;
  while (q < uint32_t(kBatch) && sp < end) {
    constexpr int kScan = 4;
    uint32_t key[kScan], ball[kScan], hits = 0;
#pragma unroll
    for (int k = 0; k < kScan; ++k) {
      const uint32_t pos = sp + k * kPxThreads + threadIdx.x;
      key[k] = 0;
      if (pos < end) {
        key[k] = tk[pos];
        if (box_live(key[k], s_live)) hits |= 1u << k;
      }
      ball[k] = __ballot_sync(0xffffffffu, (hits >> k) & 1u);
      if (lane == 0) s_cnt[k * kPxWarps + warp] = __popc(ball[k]);
    }
    __syncthreads();
    if (warp == 0) {   // exclusive scan over (step, warp) = list order
      const uint32_t v = s_cnt[lane];
      uint32_t incl = v;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += t;
      }
      s_cnt[lane] = incl - v;
      if (lane == 31) *s_total = incl;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kScan; ++k) {
      if ((hits >> k) & 1u) {
        const uint32_t pos = sp + k * kPxThreads + threadIdx.x;
        const uint32_t idx = q + s_cnt[k * kPxWarps + warp] + __popc(ball[k] & lanemask_lt());
        if (idx < uint32_t(kBatch)) {
          const uint32_t slot = pv[pos];
          s_qslot[idx] = slot;
          if (s_rows) {   // (a slot beyond the buffers never occurs in a valid frame: no warp reads it)
            const uint32_t w0 = ((key[k] >> 20) & 15u) >> 1, w1 = ((key[k] >> 24) & 15u) >> 1;
            s_rows[idx] = slot < cap_slots ? uint8_t((0xFFu >> (7u - w1)) & (0xFFu << w0)) : uint8_t(0);
          }
        } else if (idx == uint32_t(kBatch)) {
          *s_resume = pos;   // the first record left over
        }
      }
    }
    __syncthreads();
    const uint32_t total = *s_total;
    if (q + total > uint32_t(kBatch)) {
      sp = *s_resume;
      q = kBatch;
    } else {
      sp = min(sp + uint32_t(kPxThreads * kScan), end);
      q += total;
    }
    static_assert(kScan * kPxWarps == 32, "one scan lane per (step, warp)");
  }
  *sp_io = sp;
  return q;
}

// ---------------------------------------------------------------- bulk-copy staging
// One non-tensor cp.async.bulk per 48-byte record (16-byte aligned in global and shared memory)
// from this GPU's own memory into the CTA's shared memory, completing on an mbarrier.

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return uint32_t(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

// One poll of the phase with the given parity; the thread may be suspended for up to about 1 us
// (the suspend-time hint) while the phase is incomplete.
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity), "r"(1000u)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Waits for the mbarrier phase of the given parity; false when it has not completed within about
// one second (and at most kSpinLimit polls).
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity) {
  const uint64_t t0 = global_ns();
  for (uint32_t i = 0; i < kSpinLimit; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((i & 63u) == 63u && global_ns() - t0 > 1000000000ull) break;
  }
  return false;
}

__device__ __forceinline__ void bulk_copy_to_shared(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// Resident blocks per SM of the pixel-loop kernel (shared memory: 54 B per record of a batch; at
// six blocks the 40-register limit spills).
constexpr int blend_px_blocks_per_sm(int batch) { return batch == 512 ? 4 : 5; }

// Second blend variant (V3DG_OPT_BLEND_MODE 1): the same batches, staged by bulk copies, then
// composited pixel-parallel with no per-pixel masks.  Warp w owns rows 2w and 2w + 1 of the tile
// (lane = pixel) and walks, in list (= depth) order, only the batch records whose box spans one of
// its rows (known from the pair key at fill time), so a warp never visits a record that cannot
// reach it; each lane evaluates the record where its pixel lies in the record's box and is still
// accumulating, and composites at once (composite_step, the same arithmetic as k_blend, so the image is the same bit for bit).  A warp whose 32 pixels are all done skips the
// rest of the batch.
template <bool kCount, int kBatch>
__global__ void __launch_bounds__(kPxThreads, blend_px_blocks_per_sm(kBatch))
k_blend_px(const uint2* __restrict__ ranges, const uint32_t* __restrict__ items, uint32_t n_items,
           const uint32_t* __restrict__ class_count, uint32_t* __restrict__ tile_counter,
           const uint32_t* __restrict__ tk, const uint32_t* __restrict__ pv,
           const float4* __restrict__ rec, uint32_t cap_slots, int width, int height, int tiles_x, int tiles_per_view,
           float* __restrict__ rgb, float* __restrict__ t_out, unsigned long long* __restrict__ work,
           uint32_t* __restrict__ frame, uint32_t* __restrict__ sticky) {
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (frame[kOverflow]) atomicOr(sticky, 1u);
    if (frame[kTimeout]) atomicOr(sticky + 1, 1u);
  }
  constexpr int kPer = kBatch >= kPxThreads ? kBatch / kPxThreads : 1;
  constexpr int kWords = kBatch / 32;
  static_assert(kBatch % 32 == 0 && kWords <= 32 && (kBatch <= kPxThreads || kBatch % kPxThreads == 0),
                "batch size");
  __shared__ __align__(16) float4 s_rec[3 * kBatch];   // the batch's records, as stored by the projection
  __shared__ uint32_t s_qslot[kBatch];
  __shared__ uint8_t s_rows[kBatch];                   // bit w: the record's box spans rows 2w or 2w + 1
  __shared__ uint32_t s_live[kPxWarps];
  __shared__ uint32_t s_cnt[32];
  __shared__ uint32_t s_next, s_resume, s_total;
  __shared__ __align__(8) uint64_t s_bar;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int lx = threadIdx.x & 15, ly = threadIdx.x >> 4;   // lane = 16 (ly & 1) + lx
  const float fx = float(lx) + 0.5f, fy = float(ly) + 0.5f;
  uint32_t n_eval = 0, n_contrib = 0, phase = 0;
  bool failed = false;
  const uint32_t cls_incl = item_classes(class_count);
  if (threadIdx.x == 0) mbar_init(&s_bar, 1);
  __syncthreads();
  for (;;) {
    if (threadIdx.x == 0) s_next = atomicAdd(tile_counter, 1u);
    __syncthreads();
    const uint32_t next = s_next;
    __syncthreads();
    if (next >= n_items) break;
    const int tile = int(item_tile(items, n_items, cls_incl, next));   // (view, tile) id
    const int view = tile / tiles_per_view, vt = tile - view * tiles_per_view;
    const int tx = vt % tiles_x, ty = vt / tiles_x;
    const int px = tx * 16 + lx, py = ty * 16 + ly;
    const bool inside = px < width && py < height;
    const uint2 range = ranges[tile];
    float T = 1.f, cr = 0.f, cg = 0.f, cb = 0.f;
    bool done = !inside;
    uint32_t sp = range.x;
    for (;;) {
      const uint32_t dword = __ballot_sync(0xffffffffu, done);
      if (lane == 0) s_live[warp] = ~dword;
      __syncthreads();
      uint32_t any_live = 0;
#pragma unroll
      for (int w = 0; w < kPxWarps; ++w) any_live |= s_live[w];
      if (any_live == 0 || sp >= range.y) break;
      const uint32_t q = fill_batch<kBatch>(tk, pv, range.y, cap_slots, s_live, s_qslot, s_rows, s_cnt, &s_resume, &s_total, &sp);
      if (q == 0) break;
      // stage the batch: the previous batch's shared reads ended at the fill's barriers
      if (threadIdx.x == 0) mbar_arrive_expect_tx(&s_bar, q * 48u);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
#pragma unroll
      for (int k = 0; k < kPer; ++k) {
        const uint32_t i = threadIdx.x + k * kPxThreads;
        if (i >= q) continue;
        uint32_t slot = s_qslot[i];
        if (slot >= cap_slots) slot = 0;   // never for a valid frame; no warp reads the record (rows 0)
        bulk_copy_to_shared(&s_rec[3 * i], rec + 3 * size_t(slot), 48u, &s_bar);
      }
      // this warp's records: bit j of word k <=> record 32 k + j spans one of its rows
      uint32_t mine = 0;
#pragma unroll
      for (int k = 0; k < kWords; ++k) {
        __syncwarp();
        const uint32_t j = 32u * k + lane;
        const uint32_t b = __ballot_sync(0xffffffffu, j < q && ((s_rows[j] >> warp) & 1u));
        if (lane == k) mine = b;
      }
      if (!mbar_wait_bounded(&s_bar, phase)) failed = true;
      phase ^= 1u;
      if (__syncthreads_or(failed)) goto out;
      bool wdone = __all_sync(0xffffffffu, done);
      for (int k = 0; k < kWords && !wdone; ++k) {
        uint32_t bits = __shfl_sync(0xffffffffu, mine, k);
        while (bits) {
          const int j = 32 * k + __ffs(bits) - 1;
          bits &= bits - 1;
          const float4 r0 = s_rec[3 * j], r1 = s_rec[3 * j + 1], r2 = s_rec[3 * j + 2];
          const uint32_t bx = __float_as_uint(r2.z), by = __float_as_uint(r2.w);
          if (!done && px >= int(bx & 0xFFFFu) && px <= int(bx >> 16) && py >= int(by & 0xFFFFu) &&
              py <= int(by >> 16)) {
            const uint32_t org = __float_as_uint(r2.y);
            const float ox = float(16 * (tx - int(org & 0xFFFFu))), oy = float(16 * (ty - int(org >> 16)));
            const float l2a = log2_alpha(make_float4(r0.x - ox, r0.y - oy, r0.z, r0.w), r1, fx, fy);
            if (kCount) ++n_eval;
            if (composite_step(l2a, r1.z, r1.w, r2.x, T, cr, cg, cb, done) && kCount) ++n_contrib;
          }
          if (__all_sync(0xffffffffu, done)) {
            wdone = true;
            break;
          }
        }
      }
      __syncthreads();   // the batch's records are consumed before the next batch is staged
    }
    if (inside) {
      const size_t p = (size_t(view) * height + py) * width + px;
      rgb[3 * p + 0] = cr;
      rgb[3 * p + 1] = cg;
      rgb[3 * p + 2] = cb;
      if (t_out) t_out[p] = T;
    }
  }  // next tile
out:
  if (failed) {   // a bounded wait gave up: flag the frame, and let the copies in flight land first
    if (threadIdx.x == 0) {
      atomicOr(frame + kTimeout, 1u);
      atomicOr(sticky + 1, 1u);
    }
    mbar_wait_bounded(&s_bar, phase ^ 1u);
    return;
  }
  if (kCount) {
    unsigned long long e = n_eval, cnt = n_contrib;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      e += __shfl_xor_sync(0xffffffffu, e, d);
      cnt += __shfl_xor_sync(0xffffffffu, cnt, d);
    }
    if (lane == 0) {
      atomicAdd(work, e);
      atomicAdd(work + 1, cnt);
    }
  }
}

// The tiles by the length of their lists, in kItemClasses regions of n_tiles entries (class 0: 2^16
// pairs or more, then an octave each, the last but one: 1 to 7 pairs, the last: none), so that the
// work items that take longest start first.
constexpr int kLastClass = kItemClasses - 1;
__device__ __forceinline__ uint32_t item_class(uint32_t len) {
  return len ? uint32_t(min(max(int(__clz(len)) - 15, 0), kLastClass - 1)) : uint32_t(kLastClass);
}

__global__ void __launch_bounds__(256) k_blend_items(const uint2* __restrict__ ranges, uint32_t n_tiles,
                                                     uint32_t* __restrict__ items, uint32_t* __restrict__ class_count) {
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t mask = __ballot_sync(0xffffffffu, t < n_tiles);
  if (t >= n_tiles) return;
  const uint2 r = ranges[t];
  const uint32_t cls = item_class(r.y - r.x);
  const uint32_t peers = __match_any_sync(mask, cls);
  const int leader = __ffs(peers) - 1;
  uint32_t base = 0;
  if (int(threadIdx.x & 31u) == leader) base = atomicAdd(class_count + cls, __popc(peers));
  base = __shfl_sync(peers, base, leader);
  items[size_t(cls) * n_tiles + base + __popc(peers & lanemask_lt())] = t;
}

}  // namespace

namespace {

template <bool kCount, int kBatch>
void blend_px_launch(int grid, cudaStream_t st, const uint2* ranges, const uint32_t* items, uint32_t n_tiles,
                     const uint32_t* class_count, uint32_t* tile_counter, const uint32_t* tk, const uint32_t* pv,
                     const float4* rec, uint32_t cap_slots, const CamConst& cam, float* rgb, float* t_out, unsigned long long* work,
                     uint32_t* frame, uint32_t* sticky) {
  k_blend_px<kCount, kBatch><<<grid, kPxThreads, 0, st>>>(ranges, items, n_tiles, class_count, tile_counter, tk, pv, rec,
                                                          cap_slots, cam.width, cam.height, cam.tiles_x,
                                                          cam.tiles_x * cam.tiles_y, rgb, t_out, work, frame, sticky);
}

}  // namespace

namespace {
constexpr int kBlendShared = int(std::max(sizeof(BlendBlock), sizeof(BlendWarp) * (kBlendThreads / 32)));
}  // namespace

cudaError_t blend_set_attributes() {
  // several resident blocks per SM, of up to 37 KB shared memory each, want the largest carveout
  const void* fns[] = {(const void*)k_blend<true, false>,   (const void*)k_blend<false, false>,
                       (const void*)k_blend<true, true>,    (const void*)k_blend<false, true>,
                       (const void*)k_blend_px<true, 128>,  (const void*)k_blend_px<false, 128>,
                       (const void*)k_blend_px<true, 256>,  (const void*)k_blend_px<false, 256>,
                       (const void*)k_blend_px<true, 512>,  (const void*)k_blend_px<false, 512>};
  for (const void* f : fns) {
    const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout,
                                               cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_blend(const uint2* ranges, uint32_t* items, uint32_t* class_count, const uint32_t* tk,
                         const uint32_t* pv, const float4* rec, uint32_t cap_slots, const CamConst& cam, float* rgb, float* t_out,
                         unsigned long long* work, uint32_t* frame, uint32_t* sticky, int slab, const TileLive& live,
                         int batch, int mode, int n_views, int sm_count, cudaStream_t st) {
  const int n_tiles = cam.tiles_x * cam.tiles_y * n_views;
  if (n_tiles == 0) return cudaSuccess;
  if (batch != 128 && batch != 256 && batch != 512) return cudaErrorInvalidValue;
  if ((mode != 0 && mode != 1) || (mode == 1 && live.bits)) return cudaErrorInvalidValue;
  uint32_t* words = frame + kSlabBase + slab * kSlabWords;
  k_blend_items<<<(n_tiles + 255) / 256, 256, 0, st>>>(ranges, uint32_t(n_tiles), items, class_count);
  // persistent grids: the resident blocks
  if (mode == 0) {
    const int grid = std::min(kSubTiles * n_tiles, sm_count * kBlendBlocks);
    const auto kernel = live.bits ? (work ? k_blend<true, true> : k_blend<false, true>)
                                  : (work ? k_blend<true, false> : k_blend<false, false>);
    kernel<<<grid, kBlendThreads, kBlendShared, st>>>(ranges, items, uint32_t(n_tiles), class_count, words, slab == 0, live, tk, pv, rec, cap_slots,
                                           cam.width, cam.height, cam.tiles_x, cam.tiles_x * cam.tiles_y, rgb, t_out, work,
                                           frame, sticky);
    return cudaGetLastError();
  }
  const int grid = std::min(n_tiles, sm_count * blend_px_blocks_per_sm(batch));
  const auto launch = batch == 128   ? (work ? blend_px_launch<true, 128> : blend_px_launch<false, 128>)
                      : batch == 256 ? (work ? blend_px_launch<true, 256> : blend_px_launch<false, 256>)
                                     : (work ? blend_px_launch<true, 512> : blend_px_launch<false, 512>);
  launch(grid, st, ranges, items, uint32_t(n_tiles), class_count, words + kSlabBlendItem, tk, pv, rec, cap_slots, cam, rgb, t_out, work,
         frame, sticky);
  return cudaGetLastError();
}

}  // namespace v3dg
