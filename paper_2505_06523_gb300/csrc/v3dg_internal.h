// Internal layouts shared by the host side (v3dg_api.cpp) and the kernels (*.cu).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace v3dg {

constexpr int kTile = 16;              // 16x16 pixel tiles
constexpr int kSlots = 64;             // Gaussian slots per cluster block on the device
constexpr int kMaxShCoeffs = 16;       // degree 3

// Attributes of one asset, one contiguous block per cluster: planes of 64 values (j = 0..63 is
// the Gaussian within the cluster).  First the geometry planes, always float32, then the colour
// planes (opacity, then SH coefficient-major, channel-minor), float32 or -- for assets loaded with
// V3DG_OPT_ATTR_FP16 -- float16.
enum GeoPlane : int { kX = 0, kY, kZ, kLs0, kLs1, kLs2, kQw, kQx, kQy, kQz, kGeoPlanes };
enum ColorPlane : int { kOpacity = 0, kSh0 = 1 };   // SH: kSh0 + 3 * coeff + channel
constexpr int color_planes(int sh_coeffs) { return kSh0 + 3 * sh_coeffs; }
constexpr size_t cluster_block_bytes(int sh_coeffs, bool half) {
  return size_t(kGeoPlanes) * kSlots * 4 + size_t(color_planes(sh_coeffs)) * kSlots * (half ? 2 : 4);
}

// Node flags.
constexpr uint8_t kLeaf = 1, kRoot = 2;

struct AssetDev {
  const float4* own;       // own sphere (cluster group of the node), asset frame
  const float4* par;       // parent's own sphere (root: copy of own, unused)
  const float4* bound;     // sphere around the node's Gaussian means: centre = their mean
  const float* sigma_max;  // max over the node's Gaussians of exp(max log-scale)
  const uint8_t* flags;    // kLeaf | kRoot
  const uint8_t* count;    // Gaussians in the node, 1..64
  const unsigned char* attr;  // n_nodes cluster blocks of `stride` bytes
  uint32_t n_nodes;
  uint32_t stride;         // bytes per cluster block: cluster_block_bytes(sh_coeffs, half_color)
  uint32_t sh_coeffs;      // (degree + 1)^2
  uint32_t half_color;     // 1: opacity and SH stored as float16
  // top-down selection: children of node n are child_list[child_off[n] .. child_off[n + 1]);
  // sub_bound / sub_sigma bound the spheres and sigmas of every node of n's subtree
  const uint32_t* child_off;
  const uint32_t* child_list;
  const float4* sub_bound;
  const float* sub_sigma;
  uint32_t root;
  uint32_t node_base;      // global id of node 0: the node counts of the assets loaded before this one
};

// Per (frame, instance) constants, computed on the host in FP64 (128-byte aligned, 256 B).
struct alignas(16) InstFrame {
  double m64[12];          // M = W [s R | t], row-major 3x4
  float m[12];             // float32 rounding of m64
  float cam_a[3];          // camera centre in the asset frame, R^T (C - t) / s
  float s;                 // uniform scale
  double s64;
  float tau_f;             // area tolerance of this instance's asset
  uint32_t asset;
  uint32_t view;           // the camera (view) this instance frame belongs to
  uint32_t pad[19];
};
static_assert(sizeof(InstFrame) == 256, "InstFrame layout");

// Camera constants passed by value to the kernels.
struct CamConst {
  float fx, fy, cx, cy;
  float near_z;
  float limx, limy;        // Jacobian clamp: 1.3 * (w / 2) / fx
  int width, height;
  int tiles_x, tiles_y;
  double k_foot;           // pi * fx * fy (FP64) for the exact footprint re-test
  float k_foot32;
  float cull_kx, cull_ky;  // conservative pixel half-width factors of the visibility cull
};

// Frame counters (device, uint32 each).
enum Counter : int {
  kCutNodes = 0, kCutGauss, kRenderNodes, kVisible, kPairs, kOverflow, kTimeout,
  kPairsEff = 8,           // pairs of the frame, or 0 when it overflowed
  kTdReached = 9,          // top-down selection: (instance, node) entries it tested
  kConicFp64 = 10,         // Gaussians whose 2D covariance had det < 1e-12 and was inverted in FP64
  kRenderClusters = 11,    // distinct clusters of the render list (projection grouped by cluster)
  kPairs64 = 12,           // [12, 14): the pair total as a 64-bit sum (detects totals beyond 2^32)
  kKeyMinInv = 14,         // ~(lower bound of the visible Gaussians' depth keys); of one slab, the smallest
  kKeyMax = 15,            // upper bound of them; of one slab, the largest
  kTileCounters = 16,      // [16, 32): atomic tile counters: [16] selection, [27, 31) cluster order, [31] projection
  kSlabBase = 32,          // kSlabWords words for each depth slab
};

// A frame is binned, sorted and blended in one or more depth slabs, front to back: slab k holds the
// visible Gaussians with depth keys in [lo, hi).  From the second slab on, Gaussians and pairs that
// only meet tiles whose pixels have all stopped are left out (they cannot change a pixel).
constexpr int kMaxSlabs = 6, kSlabWords = 24, kFrameWords = kSlabBase + kMaxSlabs * kSlabWords;
// A frame whose Gaussians cover many tiles each: a camera close to an asset.
__host__ __device__ inline bool large_boxes(uint64_t pairs, uint64_t visible) { return pairs >= 16u * visible; }
enum SlabWord : int {
  kSlabCount = 0,          // Gaussians picked
  kSlabPairs,              // their pairs
  kSlabDepthTiles,         // tile counters of the kernels (4 words)
  kSlabExpandTile = kSlabDepthTiles + 4,
  kSlabPairTiles,          // 4 words
  kSlabBlendItem = kSlabPairTiles + 4,
  kSlabBlendLong,          // the same of the items that a block blends together
  kSlabLo, kSlabHi,        // depth keys [lo, hi)
  kSlabBits,               // key bits of the slab's depth sort: keys are stored as key - lo
  kSlabLarge,              // Gaussians left to the large-box expansion
};
static_assert(kSlabLarge < kSlabWords, "slab words");
static_assert(kSlabBlendLong == kSlabBlendItem + 1, "the blend's work counters are cleared together");
constexpr int kItemClasses = 16;   // classes of the blend's work items

// Depth histogram of the pairs (weights: tiles covered), for the slabs' limits: 16 bins per octave
// of the float32 depth from 2^-7 up (the first and last bin take what lies beyond).
constexpr int kDepthBins = 2048, kDepthShift = 19, kDepthBase = 1920;

// Which tiles still have an unfinished pixel (several slabs): one bit per tile, rows of `words`
// 32-bit words (one of them spare, zero), row view * tiles_y + ty; and per tile a bit for each of its
// 4x4 pixel blocks (4 row + column) that has one.  NULL bits: a frame of one slab.
struct TileLive {
  uint32_t* bits;
  uint32_t* blocks;
  uint32_t* coarse;        // the same bits of groups of 8x8 tiles, and per group its live tiles
  uint32_t* coarse_tiles;
  float* state;            // per pixel: T, negative once the pixel has stopped
  uint32_t words, coarse_words;
  uint32_t tiles_x, tiles_y, groups_x, groups_y;
};

// Status words of the chained (decoupled look-back) scans: epoch << 34 | flag << 32 | value.
constexpr uint64_t kFlagAgg = 1, kFlagPrefix = 2;
constexpr uint32_t kSpinLimit = 1u << 20;

// Diagnostic of the bounded waits: one look-back as tile 1 of a two-tile chain whose tile 0
// publishes (publish != 0) or never does, with at most spin_limit polls, by one thread and by a
// whole warp.  out[0], out[1]: the prefixes the two look-backs found; out[2]: nonzero if a wait
// gave up.  status: 2 * 2 words.
cudaError_t launch_check_wait(uint64_t* status, uint32_t epoch, uint32_t spin_limit, int publish, uint32_t* out,
                              cudaStream_t st);

// ---------------------------------------------------------------- launch functions (return cudaError)
// Selection (Sec. 3.3-3.4).  mode 0: render list (cut minus the visibility cull) + counters;
// mode 1: the cut itself (parity read-back).  max_nodes: of the assets; items: nodes per thread, as
// select_items gives them; status: a word per 256 * items nodes of every instance.
int select_items(uint64_t instances, uint32_t max_nodes, int sm_count);
cudaError_t launch_select(const InstFrame* inst, int n_inst, const AssetDev* assets, uint32_t max_nodes, int items,
                          const CamConst& cam, int mode, uint2* out, uint32_t cap, uint32_t* frame,
                          uint32_t tile_counter_slot, uint64_t* status, uint32_t epoch, cudaStream_t st);

// Top-down selection (same result as launch_select on trees whose footprints never grow from a
// node to its parent, which the containment of the cluster-group spheres guarantees): level by
// level from each instance's root, a node whose own footprint exceeds tau_F hands its children
// to the next level; the others are selected.  mode 0 also skips every subtree whose bound
// proves the visibility cull of all its nodes.  Marks go to a bitmap of n_inst * wpi words
// (zeroed by the caller), which one ordered compaction turns into the list of launch_select.
// frontier: two buffers of cap_front entries; counts: steps + 1 words (zeroed by the caller).
struct TopDown {
  uint2* frontier[2];
  uint32_t cap_front;
  uint32_t* counts;
  uint32_t* bitmap;
  uint32_t wpi;            // bitmap words per instance: ceil(max nodes / 32)
  int steps;               // largest root level + 1
};
cudaError_t launch_select_topdown(const InstFrame* inst, int n_inst, const AssetDev* assets, const CamConst& cam,
                                  int mode, const TopDown& td, uint2* out, uint32_t cap, uint32_t* frame,
                                  uint32_t tile_counter_slot, uint64_t* status, uint32_t epoch, int sm_count,
                                  cudaStream_t st, int* launches);

// Per render-list entry, its cluster's global id (node_base + node) shifted right by key_shift, the key
// that groups the render list by cluster for the projection.
cudaError_t launch_order_keys(const uint2* render_list, uint32_t cap_nodes, const InstFrame* inst, const AssetDev* assets,
                              const uint32_t* frame, uint32_t* order_keys, int key_shift, int sm_count, cudaStream_t st);

// Records (3 float4 per slot, slot = render index * 64 + j):
//   [0] = (u_rel, v_rel, na, nb), [1] = (nc, log2 o, r, g), [2] = (b, tile origin, x range, y range)
// with (u_rel, v_rel) the 2D mean relative to the pixel origin of the Gaussian's first tile
// (tx0, ty0), log2(alpha) = na dx^2 + nb dx dy + nc dy^2 + log2 o, and the inclusive pixel
// ranges x0 | x1 << 16, y0 | y1 << 16 of the alpha >= 1/255 ellipse's bounding box.
// color_formats: bit 0 set if some loaded asset stores its colour planes in float32, bit 1 if
// some asset stores them in float16 (the kernel is specialised for the formats present).
// order (may be NULL: list order): a permutation of the render-list indices that the warps take
// in turn.  Each entry's outputs stay at its own slots, so the order changes no result; ordered by
// cluster, the instances that draw one cluster read its attributes one after the other, and all
// but the first find them in L2.  sorted_keys (may be NULL): the global cluster id of each
// position of `order`; the distinct ones are counted into frame[kRenderClusters].
// Also adds up frame[kVisible], the pairs (tiles covered) into frame[kPairs64], the smallest and
// largest key, and -- unless depth_hist is NULL -- the depth histogram of the pairs and a conservative
// depth range of every render-list node.
cudaError_t launch_project(const uint2* render_list, uint32_t cap_nodes, const InstFrame* inst,
                           const AssetDev* assets, const CamConst& cam, float4* rec, uint2* rect,
                           uint32_t* keys, uint32_t* frame, const uint32_t* order,
                           const uint32_t* sorted_keys, int color_formats, uint32_t* depth_hist,
                           float2* depth_range, int sm_count, cudaStream_t st);

// Start of a render: the render's counters (the selection's words stay, so that a render list
// overflow still invalidates the frame), the sorts' digit counts, the depth histogram, the tile
// ranges of every slab and the tiles' liveness.
cudaError_t launch_frame_init(uint32_t* frame, uint32_t* hist, uint32_t hist_words, uint32_t* depth_hist, uint2* ranges,
                              uint32_t n_ranges, const TileLive& live, uint32_t n_tiles, int n_views, int sm_count,
                              cudaStream_t st);
// After the projection: the frame's pair count and overflow, and the limits of its `slabs` slabs.
cudaError_t launch_slab_limits(uint32_t* frame, const uint32_t* depth_hist, int slabs, uint32_t cap_pairs,
                               cudaStream_t st);
// The visible Gaussians of one of several slabs, in slot order: (key - lo, slot), keys in [lo, hi) and, with filter, boxes that meet a live tile.
// depth_range: a conservative depth range per render-list node.  marks, counts: scratch of cap_nodes
// and ceil(cap_nodes / 256) entries.
cudaError_t launch_pick_slab(const uint32_t* keys, const uint2* rect, uint32_t cap_nodes, const uint2* list,
                             const InstFrame* inst_views, const TileLive& live, bool filter, const float2* depth_range,
                             uint2* marks, uint32_t* counts, uint32_t* kout, uint32_t* vout, uint32_t* frame, int slab,
                             int sm_count, cudaStream_t st);

// Radix sort of (key, value) pairs, n read from *n_dev (clamped to cap).  Ping-pongs between
// (k0, v0) and (k1, v1); the result lands in (k0, v0) when the pass count is even, else in
// (k1, v1) -- *result_in_1 tells which.  implicit_vals: the values of the first pass are the
// element indices (v0 is not read).  bits_dev (may be NULL): the sort covers key bits
// [0, *bits_dev) instead, in as few passes as 8-bit digits need (the launches beyond return at
// once); the result is in (k1, v1) when that number is odd.
// slots (may be NULL; with bits_dev, no implicit_vals): the first pass reads the slots of a frame's
// render list instead of (k0, v0): the keys of the visible ones less slab[kSlabLo], their slot numbers
// as values; slab[kSlabCount] (n_dev) becomes their number.
struct SortSlots {
  const uint32_t* keys;    // a key per slot, 0xFFFFFFFF: not visible
  const uint32_t* frame;
  uint32_t cap_nodes;
  uint32_t* slab;
};
constexpr int kSortPasses = 4, kSortBins = 256;
struct SortScratch {
  uint32_t* hist;          // kSortPasses * kSortBins digit counts (zero)
  uint64_t* status;        // max_tiles * 256
  uint32_t max_tiles;
  uint32_t* tile_counters; // one per pass (zeroed by the caller's frame memset)
};
constexpr int kSortThreads = 256, kSortItems = 16, kSortTile = kSortThreads * kSortItems;
// Before a standalone sort: words = n, its tile counters ([1..4]) and gave-up flag ([5]); the digit counts.
constexpr int kSortWords = 8;
cudaError_t launch_sort_init(uint32_t* words, uint32_t n, uint32_t* hist, cudaStream_t st);
cudaError_t launch_sort(uint32_t* k0, uint32_t* v0, uint32_t* k1, uint32_t* v1, const uint32_t* n_dev,
                        uint32_t cap, int begin_bit, int end_bit, bool implicit_vals,
                        const SortScratch& sc, uint32_t* err_flag, uint32_t& epoch, int sm_count,
                        cudaStream_t st, bool* result_in_1, int* launches, const uint32_t* bits_dev = nullptr,
                        const SortSlots* slots = nullptr);

// Pair keys: tile id in bits 0..19 (at most 2^20 tiles), then the Gaussian's pixel box clipped
// to the tile, tile-local and inclusive: rows y0 in bits 20..23 and y1 in 24..27, columns rounded
// out to quads of 4, x0 / 4 in bits 28..29 and x1 / 4 in 30..31.
constexpr uint32_t kPairTileMask = 0xFFFFFu;
constexpr int kMaxTiles = 1 << 20;

// Per-device kernel attributes (shared-memory carveouts), set once per context before any launch
// (so that no attribute call happens during a stream capture).
cudaError_t sort_set_attributes();
cudaError_t blend_set_attributes();
cudaError_t project_set_attributes();

// Expansion of a slab's depth-sorted Gaussians into (tile, slot) pairs in depth order (filter: only of
// tiles that are still live); writes the slab's pair count.  slots0 / slots1: the two places where
// the depth sort may have left the slots (see launch_sort, bits_dev).  rect: per slot, the pixel box
// (x0 | x1 << 16, y0 | y1 << 16) of the alpha >= 1/255 ellipse, inclusive.
// Several views: the tile id of a pair is view * tiles_per_view + tile, with the view of the
// Gaussian's instance frame (inst_views[list[slot / 64].x].view; inst_views NULL: one view).
// large_slot, large_pos: cap_slots words each, scratch (the Gaussians with large boxes).
cudaError_t launch_expand(const uint32_t* slots0, const uint32_t* slots1, const uint2* rect, uint32_t cap_slots,
                          uint32_t cap_pairs, int tiles_x, const uint2* list, const InstFrame* inst_views,
                          uint32_t tiles_per_view, const TileLive& live, bool filter, uint32_t* large_slot,
                          uint32_t* large_pos, uint32_t* pair_keys, uint32_t* pair_vals, uint32_t* frame, int slab,
                          uint64_t* status, uint32_t epoch, int sm_count, cudaStream_t st);
// ranges: n_tiles zeroed entries.
cudaError_t launch_ranges(const uint32_t* tile_keys, uint32_t cap_pairs, const uint32_t* frame, int slab,
                          uint2* ranges, int n_tiles, int sm_count, cudaStream_t st);
// work != nullptr: also count (evaluations, contributions) into work[0], work[1].
// sticky[0] |= frame[kOverflow], sticky[1] |= frame[kTimeout] (the flags of every frame since the
// host last cleared them).
// items, class_count: kItemClasses * n_tiles words of scratch and kItemClasses zeroed words (the tiles
// by the length of their lists); the slab's words kSlabBlendItem and kSlabBlendLong are zero.  live.bits != NULL: one of
// several slabs, first to last from 0 -- the pixels' state is kept in live.state and the image
// between them (mode 0 only).
// batch: records that variant 1 stages per batch, 128, 256 or 512.  n_views
// images of cam's size, one after the other in rgb (and t_out); tile ids are (view, tile).
// tk, pair_vals: the sorted pair keys (tile id and in-tile box, see kPairTileMask) and values.
// mode 0: every warp composites 8x4 pixels on its own; mode 1: batches staged by bulk copies and
// composited by warps over row pairs.  The image is the same bit for bit.
cudaError_t launch_blend(const uint2* ranges, uint32_t* items, uint32_t* class_count, const uint32_t* tk,
                         const uint32_t* pair_vals, const float4* rec, uint32_t cap_slots, const CamConst& cam, float* rgb, float* t_out,
                         unsigned long long* work, uint32_t* frame, uint32_t* sticky, int slab, const TileLive& live,
                         int batch, int mode, int n_views, int sm_count, cudaStream_t st);

}  // namespace v3dg
