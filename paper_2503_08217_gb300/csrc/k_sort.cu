// Tile|depth key duplication and the radix sort that orders every tile's
// splats front to back (the rasteriser of Eq. 2), then per-tile ranges.
//
// The sorted order is the one of a stable LSD radix sort on the 64-bit key
// (view-tile id << 32 | FP32 depth bits) over the duplicated pairs in
// projection order (the pairs of the tiles a splat's alpha region reaches,
// see the expansion below). Duplicates of one splat share its depth, so the four
// depth-digit passes run on the splats BEFORE duplication (S keys instead of
// K); the splats are then expanded into (tile, splat) pairs in depth order,
// and the one or two tile-digit passes finish the sort. Every pass is a
// single-pass "onesweep" kernel: persistent CTAs take tiles of kSortTileKeys
// keys (3840 by default) from an atomic counter, rank digits through shared
// memory or with warp ballots (match.any queues on the address-divergence
// unit), get each digit's global offset from a
// precomputed histogram plus a decoupled look-back over tiles, reorder the
// tile in shared memory and write it out coalesced.
#include "s3r_internal.cuh"

namespace s3r {
namespace {

constexpr int kWarps = kSortThreads / 32;
constexpr int kWarpKeys = kSortItems * 32;   // keys per warp per tile
// Predecessor words a digit's look-back reads per round trip (build-time
// define the autotuner varies).
#ifndef S3R_SORT_LOOKBACK
#define S3R_SORT_LOOKBACK 8
#endif
constexpr int kSortLookback = S3R_SORT_LOOKBACK;
static_assert(kSortLookback >= 1 && kSortLookback <= 64, "look-back batch of 1..64 words");

constexpr int kShortBits = 6;   // see k_onesweep

struct PassArgs {
  const uint32_t* keys_in;
  const uint32_t* vals_in;   // null: values are the input positions
  uint32_t* keys_out;
  uint32_t* vals_out;
  const uint32_t* count;     // device count of keys
  int64_t cap;
  int shift;
  const uint32_t* hist;      // [256] global digit histogram of this pass
  uint32_t* ctr;
  unsigned long long* lookback;
  int stage;
};

// Exclusive scan of one value per thread across a 256-thread block.
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t x, uint32_t* s_tmp /*[8]*/,
                                                    uint32_t* total) {
  const uint32_t lane = lane_id();
  const int warp = threadIdx.x >> 5;
  uint32_t incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= (uint32_t)o) incl += y;
  }
  if (lane == 31) s_tmp[warp] = incl;
  __syncthreads();
  uint32_t wbase = 0, tot = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    const uint32_t c = s_tmp[w];
    if (w < warp) wbase += c;
    tot += c;
  }
  __syncthreads();
  if (total) *total = tot;
  return wbase + incl - x;
}

// Keys (and values, or their positions) of one radix tile: warp w reads its
// kWarpKeys consecutive keys as kSortItems coalesced rounds. Slots past the
// end get key 0xffffffff (digit 255) and are never written out.
__device__ __forceinline__ void load_tile(const PassArgs& a, int64_t n, int64_t tile, int warp,
                                          uint32_t lane, uint32_t (&key)[kSortItems],
                                          uint32_t (&val)[kSortItems]) {
  const int64_t first = tile * kSortTileKeys + (int64_t)warp * kWarpKeys + lane;
  // items of this lane below n (one 64-bit compare; the rounds then compare
  // small constants against it), and one base pointer per array
  const int64_t left = n - first;
  const int avail = left <= 0 ? 0 : (left >= (int64_t)kWarpKeys ? kWarpKeys : (int)left);
  const uint32_t* kp = a.keys_in + first;
  const uint32_t* vp = a.vals_in ? a.vals_in + first : nullptr;
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const bool valid = r * 32 < avail;
    key[r] = valid ? __ldcs(kp + r * 32) : 0xffffffffu;
    val[r] = valid ? (vp ? __ldcs(vp + r * 32) : (uint32_t)(first + r * 32)) : 0u;
  }
}

// One LSD pass. Per tile: rank the digits, publish the tile's digit counts for
// the look-back, reorder the tile by digit in shared memory, take the next tile
// and start its loads, then walk the look-back for the global offsets (thread d
// for digit d, eight predecessors per round trip) while those loads are in
// flight, and write the reordered tile out.
//
// The pass is bound by its instructions (177 per 32 keys, most of them on the
// ALU pipe, when digits were ranked with eight ballots a key). kSpread ranks
// through shared memory instead: one OR a key finds the lanes with the same
// digit. That is for digits that spread over many values, since lanes with equal
// digits wait for each other there: the three low digits of the depth and the
// tile digits (23.9M pairs of a seven-camera rig, in a captured step: 0.188 and
// 0.180 -> 0.162 and 0.168 ms a pass; 4.8M splats: 0.046 -> 0.040). The depth's top digit, its exponent, has few values
// and keeps the ballots (0.043 ms, 0.042 either way), and so does a tile digit
// of up to kShortBits bits, which takes a ballot a bit (11.2M pairs, the upper
// six bits of 9,600 tiles: 0.078 ms against 0.090 through shared memory).
//
// Where many keys share a digit, a spread pass takes longer than ballots do: all
// keys alike (a flat wall seen head on, 5M splats) 0.049 ms against 0.045, a tile
// digit of which one value has 0.6 of the keys (12.8M pairs) 0.114 against 0.102.
// A choice by the histogram's largest count inside the kernel mended those passes
// but made every other one 6 to 9 % longer (the rig's tile passes 0.185 -> 0.201
// and 0.192 -> 0.209 ms), so there is none: the passes of such a view together
// took 0.39 to 0.41 ms both ways.

// Place of a digit's word: digits that are multiples of 32, as the low depth digit
// is far from the origin, where depths are coarse, fall into different banks (four
// such values, 5M splats: 0.058 ms in one bank, 0.043 so; ballots 0.045).
__device__ __forceinline__ uint32_t word_of(uint32_t d) { return d ^ (d >> 5); }

template <int kBits, bool kSpread>
__global__ void __launch_bounds__(kSortThreads, S3R_SORT_BLOCKS) k_onesweep(PassArgs a) {
  sequence_begin();
  constexpr uint32_t kMask = (1u << kBits) - 1u;
  // the reorder buffers, which also hold a word per warp and digit while kSpread
  // ranks (more than a tile of fewer than eight keys per thread has)
  constexpr int kBuffer = kSpread && kSortTileKeys < kWarps * kRadix ? kWarps * kRadix : kSortTileKeys;
  __shared__ uint32_t s_keys[kBuffer];
  __shared__ uint32_t s_vals[kBuffer];
  __shared__ uint32_t s_cnt[kWarps][kRadix];   // per-warp digit counts -> exclusive offsets
  __shared__ uint32_t s_gbase[kRadix];         // exclusive scan of the global histogram
  __shared__ uint32_t s_loc[kRadix];           // tile-local start of each digit
  __shared__ uint32_t s_dst[kRadix];           // global start of each digit minus its local start
  __shared__ uint32_t s_tmp[kWarps];
  __shared__ uint32_t s_tile;

  const int64_t n = min((int64_t)*a.count, a.cap);
  const int64_t n_tiles = (n + kSortTileKeys - 1) / kSortTileKeys;
  const uint32_t tag = stage_tag(a.ctr[kCtrEpoch], a.stage);
  const int warp = threadIdx.x >> 5;
  const uint32_t lane = lane_id();
  const uint32_t lt = lanemask_lt();
  const int d_me = threadIdx.x;   // the digit this thread scans / looks back on

  if (threadIdx.x == 0) s_tile = atomicAdd(a.ctr + kCtrTileBase + a.stage, 1u);
  s_gbase[d_me] = block_excl_scan(a.hist[d_me], s_tmp, nullptr);   // synchronises
  int64_t tile = s_tile;
  uint32_t key[kSortItems], val[kSortItems];
  if (tile < n_tiles) load_tile(a, n, tile, warp, lane, key, val);

  while (tile < n_tiles) {
    for (int i = lane; i < kRadix; i += 32) s_cnt[warp][i] = 0;
    __syncwarp();
    uint32_t rank[kSortItems];
    if constexpr (kSpread) {
      // peers with the same digit: each lane sets its bit in the digit's word, two
      // rounds at a time (the reorder buffers hold the words); the first of the
      // peers adds their number to the warp's count
      uint32_t* const words[2] = {s_keys + warp * kRadix, s_vals + warp * kRadix};
      uint32_t before[kSortItems];
      for (int i = lane; i < kRadix; i += 32) words[0][i] = words[1][i] = 0u;
      __syncwarp();
#pragma unroll
      for (int r = 0; r < kSortItems; r += 2) {
#pragma unroll
        for (int q = 0; q < 2 && r + q < kSortItems; ++q)
          atomicOr(words[q] + word_of((key[r + q] >> a.shift) & kMask), 1u << lane);
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 2 && r + q < kSortItems; ++q)
          rank[r + q] = words[q][word_of((key[r + q] >> a.shift) & kMask)];
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 2 && r + q < kSortItems; ++q) {
          const uint32_t d = (key[r + q] >> a.shift) & kMask;
          before[r + q] = 0u;
          if ((rank[r + q] & lt) == 0) {
            words[q][word_of(d)] = 0u;
            before[r + q] = atomicAdd(&s_cnt[warp][d], (uint32_t)__popc(rank[r + q]));
          }
          __syncwarp();
        }
      }
#pragma unroll
      for (int r = 0; r < kSortItems; ++r)
        rank[r] = __shfl_sync(0xffffffffu, before[r], __ffs(rank[r]) - 1) + __popc(rank[r] & lt);
    } else {
#pragma unroll
      for (int r = 0; r < kSortItems; ++r) {
        // peers with the same digit: the AND over the digit's bits of the
        // ballot or its complement
        const uint32_t d = (key[r] >> a.shift) & kMask;
        uint32_t peers = 0xffffffffu;
#pragma unroll
        for (int b = 0; b < kBits; ++b) {
          const bool bit = (d >> b) & 1u;
          const uint32_t bal = __ballot_sync(0xffffffffu, bit);
          peers &= bit ? bal : ~bal;
        }
        const uint32_t before = s_cnt[warp][d];
        rank[r] = before + __popc(peers & lt);
        __syncwarp();
        if ((peers & lt) == 0) s_cnt[warp][d] = before + __popc(peers);
        __syncwarp();
      }
    }
    __syncthreads();

    // per digit: exclusive offsets over warps and the tile's count, published
    // at once for the successors' look-back
    uint32_t tile_cnt = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const uint32_t c = s_cnt[w][d_me];
      s_cnt[w][d_me] = tile_cnt;
      tile_cnt += c;
    }
    lookback_publish(a.lookback + d_me, kRadix, tile, tag, tile == 0 ? 2u : 1u, tile_cnt);
    const uint32_t loc = block_excl_scan(tile_cnt, s_tmp, nullptr);   // synchronises
    s_loc[d_me] = loc;
    __syncthreads();

    // reorder in shared memory by digit (stable)
    const int64_t base = tile * kSortTileKeys + (int64_t)warp * kWarpKeys;
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
      if (base + r * 32 + lane < n) {
        const uint32_t d = (key[r] >> a.shift) & kMask;
        const uint32_t pos = s_loc[d] + s_cnt[warp][d] + rank[r];
        s_keys[pos] = key[r];
        s_vals[pos] = val[r];
      }
    }
    if (threadIdx.x == 0) s_tile = atomicAdd(a.ctr + kCtrTileBase + a.stage, 1u);
    __syncthreads();
    const int64_t next = s_tile;
    // the next tile's loads overlap this tile's look-back and write-out
    if (next < n_tiles) load_tile(a, n, next, warp, lane, key, val);

    uint32_t prefix = 0;
    if (tile > 0) {
      prefix = lookback_walk<kSortLookback>(a.lookback + d_me, kRadix, tile, tag, a.ctr);
      lookback_publish(a.lookback + d_me, kRadix, tile, tag, 2u, prefix + tile_cnt);
    }
    s_dst[d_me] = s_gbase[d_me] + prefix - loc;
    __syncthreads();
    const int tile_n = (int)min((int64_t)kSortTileKeys, n - tile * kSortTileKeys);
    for (int i = threadIdx.x; i < tile_n; i += kSortThreads) {
      const uint32_t k = s_keys[i];
      const uint32_t dst = s_dst[(k >> a.shift) & kMask] + (uint32_t)i;
      __stcs(a.keys_out + dst, k);
      __stcs(a.vals_out + dst, s_vals[i]);
    }
    __syncthreads();   // shared arrays and s_tile are reused
    tile = next;
  }
}

// Expand depth-sorted splats into (view-tile id, splat) pairs, in two kernels
// so that the work is balanced by OUTPUT count: the nearest splats come first
// in depth order and may each cover hundreds of tiles.
//
// A splat is listed in the tiles of its 3-sigma rectangle (the record's rect)
// that its alpha >= 1/255 region reaches: the blend skips every pixel outside
// that region, so the other tiles of the rectangle would only lengthen the
// lists (they are 40-50 % of the rectangle's tiles on the rig workload). With
// the conic q = A dx^2 + 2 B dx dy + C dy^2 the region is the ellipse q <= L,
// L = 2 ln(255 o). A row of tiles is a strip of pixel-centre rows, and the
// ellipse's extent in x within a strip is one interval: its left end
//   x_l(dy) = (-B dy - sqrt(L A - det dy^2)) / A
// is convex in dy with its minimum -sqrt(L C / det) (the ellipse's leftmost
// point) at dy = s = B sqrt(L A / (det (det + B^2))); over a strip it is that
// minimum if s lies in the strip, else the smaller value at the strip's ends.
// The right end is the mirror image (-s, +sqrt(L C / det)). L is raised
// (1.02 L + 0.1), det lowered by a bound on its rounding, the square roots and
// the strip padded, so every interval only grows: a tile is dropped only when
// none of its pixel centres can pass the blend's FP32 test. Splats too
// anisotropic for that guarantee keep their whole rectangle. The square roots
// and reciprocals are the hardware approximations (errors of about 1 ulp, far
// inside the margins), deterministic like the rest of the arithmetic.
//
//  k_splat_tiles: per splat, in depth order (its packed 32-byte record
//                gathered by the sorted id), its tile count (one interval per row of its
//                rectangle) and a 32-byte record for the expansion: the splat
//                id, the tile id of the rectangle's corner, grid and
//                rectangle widths, rectangle height, and its rows: the first
//                kInlineRows in the record, the others 8 bytes each in a row
//                table (columns, and the tiles of the splat before the
//                row, which the expansion files its markers by; offsets from a warp-aggregated bump counter; the warp
//                computes a tall splat's rows together, one per lane), so
//                that the expansion reads most splats' rows without a
//                dependent load. A splat that no longer fits the table
//                stores its region (32 bytes, by splat id) instead, and the
//                expansion recomputes its later rows from it with the same
//                function. Outside the scan below, which would otherwise
//                wait on the few splats with tens of rows.
//  k_dup_scan:   the exclusive scan of the counts (saturating) gives every
//                splat its first output, and every expansion chunk its first
//                splat.
//  k_dup_expand: persistent CTAs take fixed chunks of 256 * kExpItems outputs
//                (3072 at 12: 0.137 ms at the surround rig, 2048 0.150, 1024 0.191,
//                4096 0.148). A lane per splat files each of its rows that falls
//                into the chunk as a marker at the row's first position in
//                shared memory (a row's tile ids are consecutive); then every
//                32 outputs are one coalesced store, each finding its marker
//                with bit operations on the marked positions.
constexpr int kDupThreads = 256;
#ifndef S3R_DUP_EXPAND_ITEMS
#define S3R_DUP_EXPAND_ITEMS 12   // build-time define the autotuner varies
#endif
constexpr int kExpItems = S3R_DUP_EXPAND_ITEMS;       // outputs per thread per chunk
constexpr int kExpChunk = kDupThreads * kExpItems;    // outputs per chunk
static_assert(kExpChunk >= kDupChunkMin, "the chunk map is sized for chunks of kDupChunkMin");
static_assert(kExpChunk % 32 == 0, "a chunk clears whole words of contributor bits");
static_assert(kExpItems <= 14, "not built above 14 outputs per thread (16 took 0.148 ms where 12 took 0.137)");

constexpr float kSpanPad = 0.05f;        // pixels, on the strips and the column bounds

// The alpha >= 1/255 region of a splat in the frame of its rectangle's
// top-left pixel corner. Stored as two float4: (u, v, B, 1/A), (L A, det, ye, xe).
struct Region {
  float u, v, B, inv_A;
  float LA, det;        // det < 0: no usable bound, every tile of a row
  float ye, xe;         // half-extents in y and x; ye < 0: reaches no pixel
  float s;              // dy of the leftmost point (-s: the rightmost)
};

__device__ __forceinline__ void region_store(const Region& g, float4* dst) {
  dst[0] = make_float4(g.u, g.v, g.B, g.inv_A);
  dst[1] = make_float4(g.LA, g.det, g.ye, g.xe);
}

// The stationary point s from the stored fields, so that the scan and the
// expansion derive it identically.
__device__ __forceinline__ void region_finish(Region& g) {
  g.s = (g.det > 0.f && g.ye > 0.f)
            ? __fmul_rn(__fmul_rn(g.B, g.ye), approx_rcp(approx_sqrt(__fmaf_rn(g.B, g.B, g.det))))
            : 0.f;
}

__device__ __forceinline__ Region region_load(const float4 a, const float4 b) {
  Region g;
  g.u = a.x; g.v = a.y; g.B = a.z; g.inv_A = a.w;
  g.LA = b.x; g.det = b.y; g.ye = b.z; g.xe = b.w;
  region_finish(g);
  return g;
}

__device__ __forceinline__ Region region_of(const float2 xy, const float4 co, uint32_t x0,
                                            uint32_t y0) {
  const float A = co.x, B = co.y, C = co.z, o = co.w;
  Region g;
  g.u = __fsub_rn(xy.x, 16.f * (float)x0);
  g.v = __fsub_rn(xy.y, 16.f * (float)y0);
  g.B = B;
  g.inv_A = A > 0.f ? approx_rcp(A) : 0.f;
  g.det = conic_det_lower(A, B, C);
  const float L = __fmaf_rn(2.04f, __logf(__fmul_rn(255.f, o)), 0.1f);   // 1.02 * 2 ln(255 o) + 0.1
  g.LA = __fmul_rn(L, A);
  g.ye = g.xe = 0.f;
  if (g.det > 0.f) {
    if (L > 0.f) {
      g.ye = __fmaf_rn(approx_sqrt(__fmul_rn(g.LA, approx_rcp(g.det))), 1.00001f, kSpanPad);
      g.xe = __fmaf_rn(approx_sqrt(__fmul_rn(__fmul_rn(L, C), approx_rcp(g.det))), 1.00001f, kSpanPad);
    } else {
      g.ye = -1.f;
    }
  }
  region_finish(g);
  return g;
}

// Columns [first, second) (relative to the rectangle, clamped to [0, w)) of
// the tiles in row r of the rectangle that the region reaches.
__device__ __forceinline__ uint2 row_span(const Region& g, uint32_t r, uint32_t w) {
  if (!(g.det > 0.f)) return make_uint2(0u, w);
  const float top = 16.f * (float)r;
  const float lo = fmaxf(__fsub_rn(__fadd_rn(top, 0.5f - kSpanPad), g.v), -g.ye);
  const float hi = fminf(__fsub_rn(__fadd_rn(top, 15.5f + kSpanPad), g.v), g.ye);
  if (!(lo <= hi)) return make_uint2(0u, 0u);
  const float pad = __fmul_rn(4e-6f, g.LA);
  const float rl = approx_sqrt(__fadd_rn(fmaxf(__fmaf_rn(__fmul_rn(-g.det, lo), lo, g.LA), 0.f), pad));
  const float rh = approx_sqrt(__fadd_rn(fmaxf(__fmaf_rn(__fmul_rn(-g.det, hi), hi, g.LA), 0.f), pad));
  const float bl = __fmul_rn(-g.B, lo), bh = __fmul_rn(-g.B, hi);
  float xl = __fmul_rn(fminf(__fsub_rn(bl, rl), __fsub_rn(bh, rh)), g.inv_A);
  float xr = __fmul_rn(fmaxf(__fadd_rn(bl, rl), __fadd_rn(bh, rh)), g.inv_A);
  if (lo <= g.s && g.s <= hi) xl = fminf(xl, -g.xe);
  if (lo <= -g.s && -g.s <= hi) xr = fmaxf(xr, g.xe);
  // tile c holds the pixel centres 16 c + 0.5 .. 16 c + 15.5
  const float ca = ceilf(__fmul_rn(__fsub_rn(__fadd_rn(g.u, xl), 15.5f + kSpanPad), 0.0625f));
  const float cb = floorf(__fmul_rn(__fsub_rn(__fadd_rn(g.u, xr), 0.5f - kSpanPad), 0.0625f)) + 1.f;
  const float fw = (float)w;
  const float a = ca > 0.f ? fminf(ca, fw) : 0.f;           // NaN: 0
  const float b = cb < fw ? fmaxf(cb, 0.f) : fw;            // NaN: w
  return a < b ? make_uint2((uint32_t)a, (uint32_t)b) : make_uint2(0u, 0u);
}

struct DupArgs {
  uint32_t* hist;        // tile-digit histograms of the radix passes that follow
  int tile_passes;
  const uint32_t* sp_cnt;      // [S] tiles each splat reaches, by depth position
  const uint2* row_spans;      // per row of a rectangle: first | end << 16 (columns), and the
                               // splat's tiles before the row
  const float4* sp_region;     // [S][2] region, by splat id, where sp_rowoff is kNoRows
  uint32_t* dup_key;
  uint32_t* dup_val;
  uint32_t* dup_excl;    // [S+1] first output of each sorted splat
  uint4* dup_meta;       // [S][2] records in depth order: (splat, corner tile, gx | w << 16, h),
                         // (first row-table entry or kNoRows, rows 0..2)
  uint32_t* dup_chunk;   // [chunks+1] splat holding each chunk's first output; last: final splat
  int64_t cap_splats, cap_dups;
  uint32_t* ctr;
  unsigned long long* lookback;
  uint32_t* contrib;       // [kBlendBands][contrib_words] the forward's contributor bits, cleared here
  int64_t contrib_words;
};

constexpr int kTilesThreads = 256;
constexpr uint32_t kNoRows = 0xffffffffu;
constexpr int kInlineRows = 3;

struct TilesArgs {
  const uint32_t* sorted;   // depth order -> splat id
  const uint4* tin;         // [S][2] packed splat records (rect and view below: fallback)
  const uint2* rect;
  const uint8_t* view;
  uint32_t* ctr;
  int64_t cap;
  uint32_t* cnt;            // [S] tiles reached, by depth position
  uint4* meta;              // [S][2] expansion records, by depth position
  uint2* row_spans;         // (columns, tiles of the splat before the row)
  int64_t rows_cap;
  float4* region;           // [S][2] by splat id
};

// Four blocks per SM (61 registers): 0.103 ms at the surround rig (4.16M splats),
// three 0.114, five 0.108; without the loads ahead 0.115.
__global__ void __launch_bounds__(kTilesThreads, 4) k_splat_tiles(const __grid_constant__ ViewSet vs,
                                                              TilesArgs a) {
  sequence_begin();
  __shared__ uint32_t s_cnt[kTilesThreads];   // tiles of each lane's rows past the inline ones
  const int64_t n = min((int64_t)a.ctr[kCtrSplats], a.cap);
  const uint32_t lane = lane_id();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t i_first = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  uint32_t sp_next = i_first < n ? a.sorted[i_first] : 0u;
  uint32_t sp_after = i_first + stride < n ? a.sorted[i_first + stride] : 0u;
  uint4 t0_next = make_uint4(0u, 0u, 0u, 0u), t1_next = t0_next;
  if (i_first < n) {
    t0_next = a.tin[2 * (size_t)sp_next];
    t1_next = a.tin[2 * (size_t)sp_next + 1];
  }
  for (int64_t base = blockIdx.x * (int64_t)blockDim.x; base < n; base += stride) {
    const int64_t i = base + threadIdx.x;   // depth position
    const bool live = i < n;
    // the packed inputs: one 32-byte sector per splat, gathered by the sorted id;
    // the next round's are on their way while this one's rows are computed, the
    // ids a round further ahead
    const uint32_t sp = sp_next;
    const uint4 t0 = t0_next, t1 = t1_next;
    sp_next = sp_after;
    if (i + stride < n) {
      t0_next = a.tin[2 * (size_t)sp_next];
      t1_next = a.tin[2 * (size_t)sp_next + 1];
    }
    sp_after = i + 2 * stride < n ? a.sorted[i + 2 * stride] : 0u;
    const float2 sxy = make_float2(__uint_as_float(t0.x), __uint_as_float(t0.y));
    const float4 sco = make_float4(__uint_as_float(t0.z), __uint_as_float(t0.w),
                                   __uint_as_float(t1.x), __uint_as_float(t1.y));
    uint32_t x0 = t1.z & 0xffffu, y0 = t1.z >> 16;
    uint32_t w = t1.w & 0x1fffu, h = (t1.w >> 13) & 0x1fffu;
    uint32_t sview = ((t1.w >> 26) & 0x1fu) | ((t1.w >> 31) ? 0x80u : 0u);   // bit 7: moved
    if (live && t1.w == kTinFallback) {   // a view too large for the packed extent
      const uint2 rc = a.rect[sp];
      x0 = rc.x & 0xffffu;
      y0 = rc.x >> 16;
      w = (rc.y & 0xffffu) - x0;
      h = (rc.y >> 16) - y0;
      sview = a.view[sp];
    }
    // table entries for the rows past the inline ones, one atomic per warp
    const uint32_t need = (live && w != 0 && h > kInlineRows) ? h - kInlineRows : 0u;
    uint32_t incl = need;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= (uint32_t)o) incl += t;
    }
    unsigned long long wbase = 0;
    if (lane == 31 && incl)
      wbase = atomicAdd(reinterpret_cast<unsigned long long*>(a.ctr + kCtrRows),
                        (unsigned long long)incl);
    wbase = __shfl_sync(0xffffffffu, wbase, 31);
    const uint64_t off = wbase + incl - need;
    const bool table = off + need <= (uint64_t)a.rows_cap;
    Region g = {};
    if (live) g = region_of(sxy, sco, x0, y0);
    // each lane: the inline rows of its own splat
    uint32_t cnt = 0;
    uint32_t head[kInlineRows] = {0u, 0u, 0u};
    if (live && w != 0)
#pragma unroll
      for (uint32_t r = 0; r < (uint32_t)kInlineRows; ++r)
        if (r < h) {
          const uint2 c = row_span(g, r, w);
          head[r] = c.x | (c.y << 16);
          cnt += c.y - c.x;
        }
    // the warp: the further rows of its taller splats as one list, a row per
    // lane; row t of the list belongs to the first lane whose running count
    // exceeds t, and the lists of a warp's splats stand together in the table.
    // (A splat at a time, a lane per row, kept 14 lanes of 32 idle.)
    const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
    if (total) {   // warp-uniform
      s_cnt[threadIdx.x] = 0u;
      __syncwarp();
      for (uint32_t t0 = 0; t0 < total; t0 += 32) {
        const uint32_t t = t0 + lane;
        int o = 0;   // owner: lanes below it have incl <= t
#pragma unroll
        for (int step = 16; step > 0; step >>= 1) {
          const uint32_t x = __shfl_sync(0xffffffffu, incl, min(o + step - 1, 31));
          if (x <= t) o += step;
        }
        o = min(o, 31);
        Region gb;
        gb.u = __shfl_sync(0xffffffffu, g.u, o);
        gb.v = __shfl_sync(0xffffffffu, g.v, o);
        gb.B = __shfl_sync(0xffffffffu, g.B, o);
        gb.inv_A = __shfl_sync(0xffffffffu, g.inv_A, o);
        gb.LA = __shfl_sync(0xffffffffu, g.LA, o);
        gb.det = __shfl_sync(0xffffffffu, g.det, o);
        gb.ye = __shfl_sync(0xffffffffu, g.ye, o);
        gb.xe = __shfl_sync(0xffffffffu, g.xe, o);
        gb.s = __shfl_sync(0xffffffffu, g.s, o);
        const uint32_t wb = __shfl_sync(0xffffffffu, w, o);
        const uint32_t before = __shfl_sync(0xffffffffu, incl - need, o);
        const bool tb = __shfl_sync(0xffffffffu, (int)table, o) != 0;
        uint2 c = make_uint2(0u, 0u);
        if (t < total) c = row_span(gb, kInlineRows + (t - before), wb);
        // the splat's tiles before this row: its inline rows', its rows' of
        // earlier rounds, and its rows' of the lanes before in this round
        const uint32_t len = c.y - c.x;
        uint32_t run = len;
#pragma unroll
        for (int st = 1; st < 32; st <<= 1) {
          const uint32_t y = __shfl_up_sync(0xffffffffu, run, st);
          if (lane >= (uint32_t)st) run += y;
        }
        const uint32_t first = before > t0 ? before - t0 : 0u;   // its first lane here
        const uint32_t skip = __shfl_sync(0xffffffffu, run - len, (int)min(first, 31u));
        const uint32_t inline_cnt = __shfl_sync(0xffffffffu, cnt, o);
        uint32_t* far_cnt = &s_cnt[(threadIdx.x & ~31u) + o];
        if (t < total && tb)
          a.row_spans[wbase + t] = make_uint2(c.x | (c.y << 16), inline_cnt + *far_cnt + (run - len - skip));
        __syncwarp();
        if (len) atomicAdd(far_cnt, len);
        __syncwarp();
      }
      cnt += s_cnt[threadIdx.x];
    }
    if (!live) continue;
    const ViewInfo& vi = vs.v[sview & 0x7f];   // bit 7: Eq. 7 moved
    const uint32_t corner = (uint32_t)vi.tile_base + y0 * (uint32_t)vi.gx + x0;
    // a rectangle without columns (an Eq. 7 splat moved out of the frustum)
    // has no rows either for the expansion, which then reads no row table
    a.cnt[i] = cnt;
    a.meta[2 * i] = make_uint4(sp, corner, (uint32_t)vi.gx | (w << 16), w != 0 ? h : 0u);
    a.meta[2 * i + 1] = make_uint4(table ? (uint32_t)off : kNoRows, head[0], head[1], head[2]);
    if (!table) region_store(g, a.region + 2 * sp);
  }
}

// Exclusive saturating scan (sat_add) of one value per thread across a
// 256-thread block; inputs <= kSat.
__device__ __forceinline__ uint32_t block_excl_scan_sat(uint32_t x, uint32_t* s_tmp /*[8]*/,
                                                        uint32_t* total) {
  const uint32_t lane = lane_id();
  const int warp = threadIdx.x >> 5;
  uint32_t incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= (uint32_t)o) incl = sat_add(incl, y);
  }
  uint32_t excl = __shfl_up_sync(0xffffffffu, incl, 1);
  if (lane == 0) excl = 0;
  if (lane == 31) s_tmp[warp] = incl;
  __syncthreads();
  uint32_t wbase = 0, tot = 0;
#pragma unroll
  for (int w = 0; w < kDupThreads / 32; ++w) {
    const uint32_t c = s_tmp[w];
    if (w < warp) wbase = sat_add(wbase, c);
    tot = sat_add(tot, c);
  }
  __syncthreads();
  *total = tot;
  return sat_add(wbase, excl);
}

// Pair offsets saturate at kSat (above every capacity, which is < 2^31), so a
// real pair count of 2^32 or more cannot wrap into a small one: it latches
// the capacity status like any other overflow.
//
// The counts are in depth order already (k_splat_tiles), so this is a plain
// scan: 4096-count tiles, 16 consecutive counts per thread (128-bit loads and
// stores); a CTA scans the tiles of its chunk in the block, gets the chunk's
// offset from the counts all earlier chunks published (chunk_prefix), and
// reads its counts again (from L2) to write the offsets and the expansion
// chunks' first splats.
constexpr int kDupScanItems = 16;
constexpr int kDupScanTile = kDupThreads * kDupScanItems;   // 4096
constexpr int kDupScanChunkTiles = 16;

__global__ void __launch_bounds__(kDupThreads) k_dup_scan(DupArgs a) {
  sequence_begin();
  __shared__ uint32_t s_ex[kDupScanChunkTiles][kDupThreads];   // thread's offset within the chunk
  __shared__ uint32_t s_tmp[kDupThreads / 32];
  __shared__ uint32_t s_chunk;
  const int64_t n = min((int64_t)a.ctr[kCtrSplats], a.cap_splats);
  const int64_t n_tiles = (n + kDupScanTile - 1) / kDupScanTile;
  // one chunk per CTA of the grid where kDupScanChunkTiles tiles allow it (the
  // count is on the device, so every CTA derives the same chunk length)
  const int per = (int)max((int64_t)1, min((int64_t)kDupScanChunkTiles,
                                           (n_tiles + gridDim.x - 1) / (int64_t)gridDim.x));
  const int64_t n_chunks = (n_tiles + per - 1) / per;
  const uint32_t tag = stage_tag(a.ctr[kCtrEpoch], kStageDup);
  auto load = [&](int64_t tile, uint32_t (&c)[kDupScanItems]) {
    const int64_t i0 = tile * kDupScanTile + (int64_t)threadIdx.x * kDupScanItems;
    if (i0 + kDupScanItems <= n) {
      const uint4* p = reinterpret_cast<const uint4*>(a.sp_cnt + i0);
#pragma unroll
      for (int q = 0; q < kDupScanItems / 4; ++q) {
        const uint4 v = p[q];
        c[4 * q] = v.x; c[4 * q + 1] = v.y; c[4 * q + 2] = v.z; c[4 * q + 3] = v.w;
      }
    } else {
#pragma unroll
      for (int k = 0; k < kDupScanItems; ++k) c[k] = i0 + k < n ? a.sp_cnt[i0 + k] : 0u;
    }
#pragma unroll
    for (int k = 0; k < kDupScanItems; ++k) c[k] = min(c[k], kSat);
  };
  for (;;) {
    if (threadIdx.x == 0) s_chunk = atomicAdd(a.ctr + kCtrTileBase + kStageDup, 1u);
    __syncthreads();
    const int64_t chunk = s_chunk;
    if (chunk >= n_chunks) break;
    const int64_t t0 = chunk * per;
    const int nt = (int)min((int64_t)per, n_tiles - t0);
    // 1. per tile: the threads' sums, scanned over the block and carried over
    //    the chunk (the next tile's loads issued first)
    uint32_t c[kDupScanItems];
    load(t0, c);
    uint32_t carry = 0;
    for (int i = 0; i < nt; ++i) {
      uint32_t run = 0;
#pragma unroll
      for (int k = 0; k < kDupScanItems; ++k) run = sat_add(run, c[k]);
      if (i + 1 < nt) load(t0 + i + 1, c);
      uint32_t total;
      const uint32_t ex = block_excl_scan_sat(run, s_tmp, &total);   // synchronises
      s_ex[i][threadIdx.x] = sat_add(carry, ex);
      carry = sat_add(carry, total);
    }
    // 2. the chunk's count, published, and every earlier chunk's count
    if (threadIdx.x == 0) lookback_publish(a.lookback, 1, chunk, tag, 1u, carry);
    const uint32_t prefix =
        chunk_prefix<kDupThreads / 32, true>(a.lookback, chunk, tag, a.ctr, s_tmp);
    if (threadIdx.x == 0 && chunk == n_chunks - 1) {
      const uint32_t all = sat_add(prefix, carry);
      a.ctr[kCtrDups] = all;
      a.dup_excl[n] = all;                          // sentinel
      if ((int64_t)all > a.cap_dups) atomicOr(a.ctr + kCtrStatus, kStatusCapacity);
      // after the last chunk: the last splat (chunks end at an inclusive splat bound)
      const uint64_t tot = min((uint64_t)all, (uint64_t)a.cap_dups);
      a.dup_chunk[(tot + kExpChunk - 1) / kExpChunk] = (uint32_t)(n - 1);
    }
    // 3. every splat's first output, and the expansion chunks starting in it
    load(t0, c);
    for (int i = 0; i < nt; ++i) {
      const int64_t i0 = (t0 + i) * kDupScanTile + (int64_t)threadIdx.x * kDupScanItems;
      uint32_t o[kDupScanItems];
      uint32_t ex = sat_add(prefix, s_ex[i][threadIdx.x]);
#pragma unroll
      for (int k = 0; k < kDupScanItems; ++k) {
        o[k] = ex;
        if (i0 + k < n) {
          // every chunk boundary inside this splat's outputs [ex, ex + c)
          // (below capacity) starts with this splat
          const uint64_t e1 = min((uint64_t)ex + c[k], (uint64_t)a.cap_dups);
          for (uint64_t q = ((uint64_t)ex + kExpChunk - 1) / kExpChunk; q * kExpChunk < e1; ++q)
            a.dup_chunk[q] = (uint32_t)(i0 + k);
        }
        ex = sat_add(ex, c[k]);
      }
      if (i + 1 < nt) load(t0 + i + 1, c);
      if (i0 + kDupScanItems <= n) {
        uint4* p = reinterpret_cast<uint4*>(a.dup_excl + i0);
#pragma unroll
        for (int q = 0; q < kDupScanItems / 4; ++q)
          p[q] = make_uint4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]);
      } else {
#pragma unroll
        for (int k = 0; k < kDupScanItems; ++k)
          if (i0 + k < n) a.dup_excl[i0 + k] = o[k];
      }
    }
    __syncthreads();   // s_chunk / s_ex reuse
  }
}

// A row of one splat's tiles falling into a chunk: `len` pairs from output `o`
// on, their tile ids consecutive from `key`. The part inside the chunk is filed
// as one marker at its first position: the splat, and the tile id less the
// position, so that the pairs of a marker are its value plus their positions.
// The digits above the lowest are counted here, a piece of equal digits at a
// time (pieces end at multiples of 256); the lowest is counted by the pairs.
struct ExpandChunk {
  uint32_t O0, O1;
  uint32_t* key;            // [kExpChunk] tile id less position, at marked positions
  uint32_t* val;            // [kExpChunk] splat
  uint32_t* mark;           // [kExpChunk / 32] bits
  uint32_t (*hist)[kRadix];
  int passes;
};
__device__ __forceinline__ void file_row(const ExpandChunk& c, uint32_t splat, uint32_t o, uint32_t len,
                                         uint32_t key) {
  const uint32_t lo = max(o, c.O0), hi = min(o + len, c.O1);
  if (lo >= hi) return;
  const uint32_t pos = lo - c.O0;
  uint32_t k = key + (lo - o);
  c.key[pos] = k - pos;
  c.val[pos] = splat;
  atomicOr(c.mark + (pos >> 5), 1u << (pos & 31u));
  if (c.passes < 2) return;
  for (uint32_t left = hi - lo; left > 0;) {
    const uint32_t n = min(left, kRadix - (k & (kRadix - 1)));
    for (int p = 1; p < c.passes; ++p) atomicAdd(&c.hist[p][(k >> (8 * p)) & 0xffu], n);
    k += n;
    left -= n;
  }
}

// Five blocks per SM (48 registers): 0.137 ms at the surround rig, with four 0.155.
__global__ void __launch_bounds__(kDupThreads, 5) k_dup_expand(DupArgs a) {
  sequence_begin();
  __shared__ uint32_t s_key[kExpChunk];
  __shared__ uint32_t s_val[kExpChunk];
  __shared__ uint32_t s_mark[kExpChunk / 32];
  __shared__ uint32_t s_chunk;
  __shared__ uint32_t s_hist[4][kRadix];
  constexpr int kWordsPerWarp = kExpChunk / 32 / (kDupThreads / 32);
  for (int i = threadIdx.x; i < 4 * kRadix; i += kDupThreads) (&s_hist[0][0])[i] = 0;
  const int64_t total = min((int64_t)a.ctr[kCtrDups], a.cap_dups);
  const int64_t n_chunks = (total + kExpChunk - 1) / kExpChunk;
  const uint32_t lane = lane_id();
  const int warp = threadIdx.x >> 5;
  for (;;) {
    if (threadIdx.x == 0) s_chunk = atomicAdd(a.ctr + kCtrTileBase + kStageExpand, 1u);
    for (int i = threadIdx.x; i < kExpChunk / 32; i += kDupThreads) s_mark[i] = 0u;
    __syncthreads();
    const int64_t chunk = s_chunk;
    if (chunk >= n_chunks) break;
    ExpandChunk c;
    c.O0 = (uint32_t)(chunk * kExpChunk);
    c.O1 = (uint32_t)min((int64_t)c.O0 + kExpChunk, total);   // exclusive
    c.key = s_key;
    c.val = s_val;
    c.mark = s_mark;
    c.hist = s_hist;
    c.passes = a.tile_passes;
    // 1. the chunk's splats, from the one holding its first output to (at most)
    //    the one holding the next chunk's first output (the scan's map), a lane
    //    each: the inline rows by their lane, the further rows of the taller
    //    ones by the warp, a row per lane
    const uint32_t q0 = a.dup_chunk[chunk], q1 = a.dup_chunk[chunk + 1];
    for (uint32_t qb = q0 + warp * 32; qb <= q1; qb += kDupThreads) {
      const uint32_t q = qb + lane;
      uint32_t o = c.O1, o0 = c.O1, corner = 0, gx = 0, w = 0, h = 0, off = 0, sp = 0;
      uint4 d = make_uint4(0u, 0u, 0u, 0u), e = d;
      if (q <= q1) {
        d = a.dup_meta[2 * (size_t)q];
        e = a.dup_meta[2 * (size_t)q + 1];
        o0 = o = a.dup_excl[q];
      }
      // The last chunk's map ends at the last splat, and splats without a pair (too
      // faint to reach a tile) may follow the last one that has some: past the
      // chunk's outputs nothing is left to file. (A view of 82,000 pairs with 960,000
      // faint splats behind them took 2.3 ms here without this.)
      if (chunk == n_chunks - 1 && __shfl_sync(0xffffffffu, o0, 0) >= c.O1) break;
      if (q <= q1) {
        sp = d.x;
        corner = d.y;
        gx = d.z & 0xffffu;
        w = d.z >> 16;
        h = d.w;
        off = e.x;
        const uint32_t head[kInlineRows] = {e.y, e.z, e.w};
#pragma unroll
        for (uint32_t r = 0; r < (uint32_t)kInlineRows; ++r)
          if (r < h) {
            const uint32_t first = head[r] & 0xffffu, len = (head[r] >> 16) - first;
            file_row(c, sp, o, len, corner + r * gx + first);
            o += len;
          }
      }
      // the further rows in the table, as one list (see k_splat_tiles)
      const bool tall = h > (uint32_t)kInlineRows && o < c.O1;
      const uint32_t need = tall && off != kNoRows ? h - kInlineRows : 0u;
      uint32_t incl = need;
#pragma unroll
      for (int st = 1; st < 32; st <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, st);
        if (lane >= (uint32_t)st) incl += y;
      }
      const uint32_t rows = __shfl_sync(0xffffffffu, incl, 31);
      for (uint32_t t0 = 0; t0 < rows; t0 += 32) {
        const uint32_t t = t0 + lane;
        int b = 0;   // owner: lanes below it have incl <= t
#pragma unroll
        for (int st = 16; st > 0; st >>= 1) {
          const uint32_t x = __shfl_sync(0xffffffffu, incl, min(b + st - 1, 31));
          if (x <= t) b += st;
        }
        b = min(b, 31);
        const uint32_t r = t - __shfl_sync(0xffffffffu, incl - need, b);   // past the inline ones
        const uint32_t fb = __shfl_sync(0xffffffffu, off, b), gb = __shfl_sync(0xffffffffu, gx, b);
        const uint32_t cb = __shfl_sync(0xffffffffu, corner, b), sb = __shfl_sync(0xffffffffu, sp, b);
        const uint32_t ob = __shfl_sync(0xffffffffu, o0, b);
        if (t < rows) {
          const uint2 row = a.row_spans[fb + r];
          const uint32_t first = row.x & 0xffffu;
          file_row(c, sb, ob + row.y, (row.x >> 16) - first, cb + (r + kInlineRows) * gb + first);
        }
      }
      // and those the table had no room for: from the stored region, through the
      // function that counted them, a splat at a time
      uint32_t loose = __ballot_sync(0xffffffffu, tall && off == kNoRows);
      while (loose) {
        const int b = __ffs(loose) - 1;
        loose &= loose - 1;
        const uint32_t hb = __shfl_sync(0xffffffffu, h, b), gb = __shfl_sync(0xffffffffu, gx, b);
        const uint32_t cb = __shfl_sync(0xffffffffu, corner, b), sb = __shfl_sync(0xffffffffu, sp, b);
        const uint32_t wb = __shfl_sync(0xffffffffu, w, b);
        uint32_t ob = __shfl_sync(0xffffffffu, o, b);
        const Region g = region_load(a.sp_region[2 * (size_t)sb], a.sp_region[2 * (size_t)sb + 1]);
        for (uint32_t r0 = kInlineRows; r0 < hb && ob < c.O1; r0 += 32) {
          const uint32_t r = r0 + lane;
          const uint2 row = r < hb ? row_span(g, r, wb) : make_uint2(0u, 0u);
          const uint32_t len = row.y - row.x;
          uint32_t run = len;
#pragma unroll
          for (int st = 1; st < 32; st <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, run, st);
            if (lane >= (uint32_t)st) run += y;
          }
          file_row(c, sb, ob + run - len, len, cb + r * gb + row.x);
          ob += __shfl_sync(0xffffffffu, run, 31);
        }
      }
    }
    __syncthreads();
    // 2. the pairs, 32 positions at a time: a pair belongs to the last marker at
    //    or before its position (the chunk's first position has one)
    const uint32_t n_here = c.O1 - c.O0;
    uint32_t word = (uint32_t)(warp * kWordsPerWarp);
    uint32_t carry = 0;   // last marked position before the word
    for (uint32_t x = word; x > 0;) {
      const uint32_t bits = s_mark[--x];
      if (bits) {
        carry = x * 32u + 31u - __clz(bits);
        break;
      }
    }
#pragma unroll
    for (int i = 0; i < kWordsPerWarp; ++i, ++word) {
      const uint32_t bits = s_mark[word], pos = word * 32u + lane;
      const uint32_t at_or_before = bits & (0xffffffffu >> (31u - lane));
      const uint32_t m = at_or_before ? word * 32u + 31u - __clz(at_or_before) : carry;
      if (pos < n_here) {
        const uint32_t key = s_key[m] + pos;
        __stcs(a.dup_key + c.O0 + pos, key);
        __stcs(a.dup_val + c.O0 + pos, s_val[m]);
        atomicAdd(&s_hist[0][key & 0xffu], 1u);
      }
      if (bits) carry = word * 32u + 31u - __clz(bits);
    }
    // the contributor bits of the chunk's pair positions, for the forward: as
    // many words as there are pairs, where clearing them for the whole pair
    // capacity in the tile-range launch (a few CTAs on small images) took most
    // of that launch
    for (int b = 0; b < kBlendBands; ++b)
      for (uint32_t i = threadIdx.x; i < (n_here + 31u) / 32u; i += kDupThreads)
        a.contrib[b * a.contrib_words + c.O0 / 32u + i] = 0u;
    __syncthreads();   // the markers are rewritten by the next chunk
  }
  __syncthreads();
  for (int i = threadIdx.x; i < a.tile_passes * kRadix; i += kDupThreads) {
    const uint32_t c = (&s_hist[0][0])[i];
    if (c) atomicAdd(a.hist + i, c);
  }
}

// Tile ranges and the blend queue's classes, one thread per tile: the
// tile's first pair is the lower bound of its id in the sorted pair keys
// (a search), its end the next tile's first pair (the neighbouring lane's
// search). Every tile's [start, end) is written ([0, 0) for a tile without
// pairs), and the tile is filed under class clz(end - start) (32 for the
// empty ones): a shared count per class, one global atomic per class and
// block for the block's slots, then the ids. The launch is bound by the latency
// of the search's dependent loads, so a step probes seven keys at once and
// keeps an eighth: 9 steps over 28 million pairs where halving takes 25.
constexpr int kRangeThreads = 256;

// First position whose key is not below v, among n sorted keys.
__device__ __forceinline__ uint32_t lower_bound_u32(const uint32_t* keys, uint32_t n,
                                                    uint32_t v) {
  uint32_t lo = 0, len = n;   // the answer is in [lo, lo + len]
  while (len >= 8) {
    const uint32_t s = len >> 3;
    uint32_t below = 0;       // of the seven probes at the eighths' last keys
#pragma unroll
    for (uint32_t i = 1; i < 8; ++i) below += keys[lo + i * s - 1] < v ? 1u : 0u;
    lo += below * s;
    len = below == 7 ? len - 7 * s : s - 1;
  }
  uint32_t below = 0;
#pragma unroll
  for (uint32_t i = 0; i < 7; ++i) below += (i < len && keys[lo + i] < v) ? 1u : 0u;
  return lo + below;
}

__global__ void __launch_bounds__(kRangeThreads) k_tile_ranges(
    const uint32_t* keys, const uint32_t* ctr, int64_t cap, int tiles, uint2* ranges,
    uint32_t* class_cnt, uint32_t* class_list) {
  sequence_begin();
  __shared__ uint32_t s_cnt[kTileClasses], s_base[kTileClasses];
  const uint32_t K = (uint32_t)min((int64_t)ctr[kCtrDups], cap);
  const uint32_t lane = lane_id();
  for (int base = blockIdx.x * kRangeThreads; base < tiles; base += gridDim.x * kRangeThreads) {
    if (threadIdx.x < kTileClasses) s_cnt[threadIdx.x] = 0u;
    __syncthreads();
    const int t = base + (int)threadIdx.x;
    const bool live = t < tiles;
    const uint32_t start = live ? lower_bound_u32(keys, K, (uint32_t)t) : K;
    uint32_t end = __shfl_down_sync(0xffffffffu, start, 1);
    if (live && (lane == 31 || t + 1 >= tiles)) end = lower_bound_u32(keys, K, (uint32_t)t + 1u);
    int cls = 0;
    uint32_t slot = 0;
    if (live) {
      const uint32_t len = end - start;
      ranges[t] = len ? make_uint2(start, end) : make_uint2(0u, 0u);
      cls = len ? __clz(len) : 32;
      slot = atomicAdd(&s_cnt[cls], 1u);
    }
    __syncthreads();
    if (threadIdx.x < kTileClasses && s_cnt[threadIdx.x])
      s_base[threadIdx.x] = atomicAdd(class_cnt + threadIdx.x, s_cnt[threadIdx.x]);
    __syncthreads();
    if (live) class_list[(size_t)cls * tiles + s_base[cls] + slot] = (uint32_t)t;
    __syncthreads();
  }
}

int per_sm_for(const void* fn, int threads) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, 0) != cudaSuccess ||
      per_sm < 1)
    per_sm = 1;
  return per_sm;
}

}  // namespace

cudaError_t launch_sort(s3r_workspace* ws, cudaStream_t st) {
  cudaError_t e;
  // occupancy is queried once (outside any graph capture: the first call)
  static thread_local int sweep_per_sm = 0, dup_per_sm = 0, exp_per_sm = 0;
  if (!sweep_per_sm)
    sweep_per_sm = min(per_sm_for((const void*)k_onesweep<kRadixBits, true>, kSortThreads),
                       min(per_sm_for((const void*)k_onesweep<kRadixBits, false>, kSortThreads),
                           per_sm_for((const void*)k_onesweep<kShortBits, false>, kSortThreads)));
  if (!dup_per_sm) dup_per_sm = per_sm_for((const void*)k_dup_scan, kDupThreads);
  if (!exp_per_sm) exp_per_sm = per_sm_for((const void*)k_dup_expand, kDupThreads);
  const int g_sweep = ws->num_sms * sweep_per_sm;
  // depth digits on the splats: 4 passes, result back in buffer 0
  for (int p = 0; p < 4; ++p) {
    PassArgs a;
    a.keys_in = ws->depth_key[p & 1];
    a.vals_in = p == 0 ? nullptr : ws->depth_val[p & 1];
    a.keys_out = ws->depth_key[(p + 1) & 1];
    a.vals_out = ws->depth_val[(p + 1) & 1];
    a.count = ws->ctr + kCtrSplats;
    a.cap = ws->cap.max_splats;
    a.shift = 8 * p;
    a.hist = ws->hist + (kHistDepth + p) * kRadix;
    a.ctr = ws->ctr;
    a.lookback = ws->lookback;
    a.stage = kStageDepth0 + p;
    KernelTimer timer(ws, kKDepth0 + p, st);
    e = launch_in_sequence(ws, p < 3 ? k_onesweep<kRadixBits, true> : k_onesweep<kRadixBits, false>, g_sweep,
                           kSortThreads, 0, st, a);
    if (e != cudaSuccess) return e;
  }
  ws->depth_final = 0;
  // expand into (tile, splat) pairs in depth order
  DupArgs d;
  d.sp_cnt = ws->sp_tiles;
  d.row_spans = ws->row_spans;
  d.sp_region = reinterpret_cast<const float4*>(ws->sp_region);
  d.dup_key = ws->dup_key[0];
  d.dup_val = ws->dup_val[0];
  d.dup_excl = ws->dup_excl;
  d.dup_meta = reinterpret_cast<uint4*>(ws->dup_meta);
  d.dup_chunk = ws->dup_chunk;
  d.cap_splats = ws->cap.max_splats;
  d.cap_dups = ws->cap.max_duplicates;
  d.ctr = ws->ctr;
  d.lookback = ws->lookback;
  d.hist = ws->hist + kHistTile * kRadix;
  d.tile_passes = ws->tile_passes;
  d.contrib = ws->contrib;
  d.contrib_words = ws->contrib_words;
  {
    static thread_local int tiles_per_sm = 0;
    if (!tiles_per_sm) tiles_per_sm = per_sm_for((const void*)k_splat_tiles, kTilesThreads);
    KernelTimer timer(ws, kKSplatTiles, st);
    TilesArgs t;
    t.rect = ws->sp_rect;
    t.view = ws->sp_view;
    t.ctr = ws->ctr;
    t.cap = ws->cap.max_splats;
    t.sorted = ws->depth_val[0];
    t.tin = reinterpret_cast<const uint4*>(ws->sp_tin);
    t.cnt = ws->sp_tiles;
    t.meta = reinterpret_cast<uint4*>(ws->dup_meta);
    t.row_spans = ws->row_spans;
    t.rows_cap = ws->rows_cap;
    t.region = reinterpret_cast<float4*>(ws->sp_region);
    e = launch_in_sequence(ws, k_splat_tiles, (int64_t)ws->num_sms * tiles_per_sm, kTilesThreads, 0, st,
                           ws->views, t);
  }
  if (e != cudaSuccess) return e;
  {
    KernelTimer timer(ws, kKDuplicate, st);
    e = launch_in_sequence(ws, k_dup_scan, scan_ctas((int64_t)ws->num_sms * dup_per_sm), kDupThreads, 0,
                           st, d);
  }
  if (e != cudaSuccess) return e;
  {
    KernelTimer timer(ws, kKExpand, st);
    e = launch_in_sequence(ws, k_dup_expand, (int64_t)ws->num_sms * exp_per_sm, kDupThreads, 0, st, d);
  }
  if (e != cudaSuccess) return e;
  // tile digits on the pairs
  for (int p = 0; p < ws->tile_passes; ++p) {
    PassArgs a;
    a.keys_in = ws->dup_key[p & 1];
    a.vals_in = ws->dup_val[p & 1];
    a.keys_out = ws->dup_key[(p + 1) & 1];
    a.vals_out = ws->dup_val[(p + 1) & 1];
    a.count = ws->ctr + kCtrDups;
    a.cap = ws->cap.max_duplicates;
    a.shift = 8 * p;
    a.hist = ws->hist + (kHistTile + p) * kRadix;
    a.ctr = ws->ctr;
    a.lookback = ws->lookback;
    a.stage = kStageTile0 + p;
    KernelTimer timer(ws, kKTile0 + p, st);
    // tile ids are below total_tiles, so the last digit may have few bits (see k_onesweep)
    const bool few = ((ws->views.total_tiles - 1) >> (8 * p)) < (1 << kShortBits);
    e = launch_in_sequence(ws, few ? k_onesweep<kShortBits, false> : k_onesweep<kRadixBits, true>, g_sweep,
                           kSortThreads, 0, st, a);
    if (e != cudaSuccess) return e;
  }
  ws->dup_final = ws->tile_passes & 1;
  // every tile's range and class (the blend queue)
  {
    const int tiles = ws->views.total_tiles;
    int64_t grid = (tiles + kRangeThreads - 1) / kRangeThreads;
    if (grid > (int64_t)ws->num_sms * 8) grid = (int64_t)ws->num_sms * 8;
    if (grid < 1) grid = 1;
    KernelTimer timer(ws, kKTileRanges, st);
    e = launch_in_sequence(ws, k_tile_ranges, grid, kRangeThreads, 0, st, ws->dup_key[ws->dup_final],
                           ws->ctr, ws->cap.max_duplicates, tiles, ws->ranges, ws->tile_class_cnt,
                           ws->tile_class_list);
  }
  return e;
}

}  // namespace s3r
