// Front-to-back alpha blending of every 16x16 tile (Eq. 2) and its exact
// adjoint.
//
// Forward: one CTA of two warps per tile, each warp a 16x8 band, four pixels
// per lane, the two of a column evaluated as one packed f32x2 pair (on small
// images four warps, each a 16x4 band, two pixels per lane). The
// tile's front-to-back splat list is consumed in batches (64 by default) staged in
// shared memory (uv, base-2 conic, opacity, rgb as duplicated pairs, and the
// box where the splat can reach alpha >= 1/255); per 32 splats a warp ballots which of
// them can reach alpha >= 1/255 somewhere in its band (box, then the exact
// ellipse-rectangle test) and evaluates only those. alpha = min(0.99, o G) is
// skipped below 1/255, and a pixel stops before its transmittance would fall
// under 1e-4; a warp stops when all its pixels have stopped. The final
// transmittance and the position of the last blended splat are stored per
// pixel, and the splats blended into at least one pixel of a band are
// recorded as bits for the backward.
//
// Backward: the same tiles and bands walked back to front, starting at each
// warp's last blended splat and visiting only the recorded splats. The
// transmittance before each splat is recovered from the stored final value as
// T <- T / (1 - alpha), so no per-pixel lists are kept; a lane's two pixels
// of a column again form one packed pair. Per splat the nine
// adjoints (uv, conic, opacity, rgb) are summed over the warp through shared
// memory, then over the CTA (one shared atomic per two splats and warp),
// and flushed to global memory with one vector atomic per four floats.
#include <type_traits>

#include "s3r_internal.cuh"

namespace s3r {
namespace {

// Launch shapes. Each is a build-time define, so that the autotuner
// (autotune.py beside this package's build script) can build and time
// alternatives; the values here are its choice at the surround-rig workload.
#ifndef S3R_BLEND_FWD_BATCH
#define S3R_BLEND_FWD_BATCH 64    // splats staged per batch (forward)
#endif
#ifndef S3R_BLEND_FWD_BLOCKS
#define S3R_BLEND_FWD_BLOCKS 18   // resident forward blocks per SM (register budget)
#endif
#ifndef S3R_BLEND_BWD_BATCH
#define S3R_BLEND_BWD_BATCH 64    // splats staged per batch (backward)
#endif
#ifndef S3R_BLEND_BWD_BLOCKS
#define S3R_BLEND_BWD_BLOCKS 14   // resident backward blocks per SM (register budget)
#endif

constexpr int kBatchBwd = S3R_BLEND_BWD_BATCH;
constexpr float kAlphaMax = 0.99f;
constexpr float kAlphaMin = 1.0f / 255.0f;
constexpr float kTStop = 1e-4f;

// Persistent tile queue: a launch of (SMs x resident blocks) CTAs takes
// positions from an atomic cursor. Tiles come longest lists first
// (k_tile_ranges files every tile under class clz(length), class 0 the
// longest, 32 the empty tiles). Chunks of memory-bound zeroing are spread
// evenly between the tiles (position i is a chunk when floor((i+1) C / P)
// > floor(i C / P), C chunks among P positions), so that their stores run
// while other CTAs of the SM blend (where the forward has a CTA for every tile they
// follow the tiles instead): the forward clears the per-splat adjoints
// the backward sums into, the backward in overwrite mode clears the caller's
// gradient arrays. The last CTA to leave resets the cursor for the next launch.
struct TileQueue {
  uint32_t* cursor;
  uint32_t* exits;
};

// Overwrite mode of the backward: the arrays of 1-4 floats per Gaussian are
// zeroed in full (the projection backward, which runs next, writes the kept
// rows), the SH rows only of the Gaussians that no view kept.
constexpr int kZeroChunk = 2048;   // Gaussians (or splats) per chunk (64 words of the kept bitmap)
struct GradZero {
  const uint32_t* kept_bits;
  int64_t n;                       // 0: nothing to zero (accumulate mode)
  s3r_grads g;
  int sh_floats;                   // 3 (K + 1)^2
};

// Which of a call's forward launches works: always, where the longest list decides
// the time, or where the work of all lists does (see long_list_decides).
enum Pick { kPickAlways = 0, kPickLongList, kPickEvenLists };

struct BlendArgs {
  const uint2* ranges;
  const uint32_t* class_cnt;    // [kTileClasses] tiles per class
  const uint32_t* class_list;   // [kTileClasses][tiles] tile ids per class
  int tiles;
  TileQueue fwd_queue, bwd_queue;
  GradZero zero;          // backward only
  const uint32_t* sorted_splats;
  const uint4* sp_tin;     // [S][2] packed splat record: (u, v, conic a, b), (conic c, opacity, ..)
  const float4* sp_rgb_d;
  const float* bg;
  const float* dL;        // backward only
  float* out;             // forward only
  float* final_T;
  uint32_t* n_contrib;
  float* sp_grad;         // [S*12]: zeroed by the forward (chunks in its queue), summed by the backward
  const uint32_t* ctr;
  int64_t cap_splats, cap_dups;
  int pick;               // forward only: which of two launches of a call works (see launch_fwd)
  unsigned long long* pairs;     // counting mode: list pairs the forward walked
  unsigned long long* eval_fwd;  // counting mode: pairs the forward evaluated
  unsigned long long* eval_bwd;  // counting mode: pairs the backward evaluated
  uint32_t* contrib;          // [kBlendBands][contrib_words]: pair blended into >= 1 pixel of the band
  int64_t contrib_words;
};

// Set the bits of `bits` (positions gp .. gp+31 of the sorted pairs) in a
// bit array; the window may straddle two words (shared with a neighbour tile).
__device__ __forceinline__ void or_bits(uint32_t* arr, uint32_t gp, uint32_t bits) {
  const uint32_t w = gp >> 5, sh = gp & 31u;
  atomicOr(arr + w, bits << sh);
  if (sh) atomicOr(arr + w + 1, bits >> (32u - sh));
}
__device__ __forceinline__ uint32_t get_bits(const uint32_t* arr, uint32_t gp) {
  const uint32_t w = gp >> 5, sh = gp & 31u;
  return __funnelshift_r(arr[w], arr[w + 1], sh);
}

// Class starts of the queue (exclusive scan of the class counts) and the
// number of zeroing chunks, once per CTA; thread 0 takes the CTA's first
// queue position.
__device__ __forceinline__ void queue_init(const BlendArgs& a, const TileQueue& q, uint32_t* s_cstart,
                                           uint32_t n_chunks, uint32_t& pending) {
  if (threadIdx.x == 0) {
    uint32_t run = 0;
    for (int c = 0; c < kTileClasses; ++c) {
      s_cstart[c] = run;
      run += a.class_cnt[c];
    }
    s_cstart[kTileClasses] = run;
    s_cstart[kTileClasses + 1] = n_chunks;
    pending = atomicAdd(q.cursor, 1u);
  }
  __syncthreads();
}

// The CTA's next work item (block-uniform): a tile id (>= 0), a zeroing
// chunk c as -2 - c, or -1 when the queue is empty. Thread 0 holds the
// position taken one item ahead, so that the atomic's round trip overlaps
// the current item's work.
__device__ __forceinline__ int queue_next(const BlendArgs& a, const TileQueue& q,
                                          const uint32_t* s_cstart, int* s_tile, uint32_t& pending) {
  if (threadIdx.x == 0) {
    const uint32_t i = pending;
    const uint64_t T = s_cstart[kTileClasses], C = s_cstart[kTileClasses + 1];
    const uint64_t P = T + C;
    int t = -1;
    if (i < P) {
      pending = atomicAdd(q.cursor, 1u);
      const uint64_t cb = C ? (uint64_t)i * C / P : 0u;              // chunks before position i
      const uint64_t cb1 = C ? ((uint64_t)i + 1u) * C / P : 0u;
      if (cb1 > cb) {
        t = -2 - (int)cb;
      } else {
        const uint32_t ti = (uint32_t)(i - cb);                          // tiles before position i
        int c = 0;
        while (ti >= s_cstart[c + 1]) ++c;
        t = (int)a.class_list[(size_t)c * a.tiles + (ti - s_cstart[c])];
      }
    }
    *s_tile = t;
  }
  __syncthreads();
  return *s_tile;
}

// Every CTA has taken its last item: the last one to leave resets the cursor.
__device__ __forceinline__ void queue_exit(const TileQueue& q) {
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(q.exits, 1u) == gridDim.x - 1) {
      *q.cursor = 0u;
      *q.exits = 0u;
      __threadfence();
    }
  }
}

// The forward's form of the same queue: the CTA's first warp finds the class
// starts with one load per lane (not 33 dependent ones) and a position's class
// with one compare per lane. A CTA's first position is its own number, the cursor
// counts those after the grid: an SM's CTAs start together, and where they drew
// their first positions from the cursor, the longest lists met on one SM. Where
// the launch has a CTA for every tile it is direct: CTA i takes tile i, then the
// zeroing chunks grid - 1 - i, + grid, ..., so that the chunks go to the CTAs
// without a tile or with the shortest ones first and the cursor stays untouched. (Chunks spread among the tiles, as the
// cursor hands them out, held the last tiles back until others had ended: 1,196
// tiles of a view of 381,000 splats 86 us, 57 us without any zeroing.)
struct QueueState {
  uint32_t pending;   // warp 0: the position taken, one item ahead; direct: the
                      // tile, from gridDim.x on that plus the next chunk
  bool direct;
};
// Whether the forward's time is that of the tile with the longest list, from the
// first class that has tiles: that list at least three times the mean, and so few
// pairs that the SMs do not wait for issue slots (launch_fwd has the times).
constexpr uint32_t kFewPairs = 300000, kLongList = 3;
__device__ __forceinline__ bool long_list_decides(const BlendArgs& a, uint32_t first_class) {
  const uint32_t pairs = (uint32_t)min((int64_t)a.ctr[kCtrDups], a.cap_dups);
  const uint32_t longest = 0x80000000u >> first_class;   // and less than twice that
  return pairs <= kFewPairs && (uint64_t)longest * (uint32_t)a.tiles >= (uint64_t)kLongList * pairs;
}

// False: this launch is not the one that works.
__device__ __forceinline__ bool fwd_queue_init(const BlendArgs& a, uint32_t* s_cstart, int* s_works,
                                               uint32_t n_chunks, QueueState& st) {
  static_assert(kTileClasses == 33, "a lane per class, and one more");
  st.pending = blockIdx.x;
  st.direct = (uint32_t)a.tiles <= gridDim.x;
  if (threadIdx.x < 32) {
    const uint32_t lane = threadIdx.x;
    const uint32_t c = a.class_cnt[lane], c_last = a.class_cnt[kTileClasses - 1];
    uint32_t incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= (uint32_t)o) incl += y;
    }
    s_cstart[lane] = incl - c;
    if (lane == 31) {
      s_cstart[kTileClasses - 1] = incl;
      s_cstart[kTileClasses] = incl + c_last;
      s_cstart[kTileClasses + 1] = n_chunks;
    }
    if (a.pick != kPickAlways) {
      const uint32_t listed = __ballot_sync(0xffffffffu, c > 0u);
      const bool decides = listed && long_list_decides(a, (uint32_t)__ffs(listed) - 1u);
      if (lane == 0) *s_works = decides == (a.pick == kPickLongList);
    }
  }
  __syncthreads();
  return a.pick == kPickAlways || *s_works;
}

__device__ __forceinline__ int fwd_queue_next(const BlendArgs& a, const uint32_t* s_cstart,
                                              int* s_tile, QueueState& st) {
  if (threadIdx.x < 32) {
    uint32_t i = __shfl_sync(0xffffffffu, st.pending, 0);
    const uint32_t T = s_cstart[kTileClasses], C = s_cstart[kTileClasses + 1];
    int t = -1;
    uint32_t ti = 0xffffffffu;   // the tile's place in the queue, if the item is one
    if (st.direct) {
      if (i < gridDim.x) {
        if (i < T) ti = i;
        i = 2u * gridDim.x - 1u - i;   // the first chunk, which is the item where there is no tile
        st.pending = i;
      }
      if (ti == 0xffffffffu && i - gridDim.x < C) {
        t = -2 - (int)(i - gridDim.x);
        st.pending = i + gridDim.x;
      }
    } else if (i < (uint64_t)T + C) {
      if (threadIdx.x == 0) st.pending = gridDim.x + atomicAdd(a.fwd_queue.cursor, 1u);
      const uint64_t P = (uint64_t)T + C;
      const uint64_t cb = C ? (uint64_t)i * C / P : 0u;              // chunks before position i
      const uint64_t cb1 = C ? ((uint64_t)i + 1u) * C / P : 0u;
      if (cb1 > cb)
        t = -2 - (int)cb;
      else
        ti = (uint32_t)(i - cb);                                       // tiles before position i
    }
    if (ti != 0xffffffffu) {
      // class starts ascend: the class is the number of later starts at or below ti
      const int c = __popc(__ballot_sync(0xffffffffu, ti >= s_cstart[threadIdx.x + 1]));
      t = (int)a.class_list[(size_t)c * a.tiles + (ti - s_cstart[c])];
    }
    if (threadIdx.x == 0) *s_tile = t;
  }
  __syncthreads();
  return *s_tile;
}

__device__ __forceinline__ void fwd_queue_exit(const BlendArgs& a, const QueueState& st) {
  if (threadIdx.x == 0 && !st.direct) {
    __threadfence();
    if (atomicAdd(a.fwd_queue.exits, 1u) == gridDim.x - 1) {
      *a.fwd_queue.cursor = 0u;
      *a.fwd_queue.exits = 0u;
      __threadfence();
    }
  }
}

__device__ __forceinline__ void zero_span(float* p, int64_t lo, int64_t hi) {
  if (!p) return;
  for (int64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) p[i] = 0.f;
}

template <int SHF>
__device__ __forceinline__ void zero_sh_unkept(const GradZero& z, int64_t w0, int64_t w1) {
  const uint32_t lane = threadIdx.x & 31u;
  const int nwarps = (int)(blockDim.x >> 5);
  for (int64_t w = w0 + (threadIdx.x >> 5); w < w1; w += nwarps) {
    const int64_t g0 = w * 32;
    const int cnt = (int)min((int64_t)32, z.n - g0);
    const uint32_t live = cnt == 32 ? 0xffffffffu : ((1u << cnt) - 1u);
    const uint32_t zero = ~z.kept_bits[w] & live;
    if (!zero) continue;
    if constexpr (SHF % 4 == 0) {
      constexpr int W4 = SHF / 4;
      float4* p = reinterpret_cast<float4*>(z.g.sh) + g0 * W4;
      for (int i = (int)lane; i < W4 * cnt; i += 32)
        if ((zero >> (i / W4)) & 1u) p[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    } else {
      float* p = z.g.sh + g0 * SHF;
      for (int i = (int)lane; i < SHF * cnt; i += 32)
        if ((zero >> (i / SHF)) & 1u) p[i] = 0.f;
    }
  }
}

// Zeroing chunk c of the forward: the per-splat adjoints (12 floats per
// splat) of splats [c kZeroChunk, (c + 1) kZeroChunk).
__device__ __forceinline__ uint32_t splat_grad_chunks(const BlendArgs& a) {
  const int64_t n = min((int64_t)a.ctr[kCtrSplats], a.cap_splats);
  return (uint32_t)((n + kZeroChunk - 1) / kZeroChunk);
}
__device__ void splat_grad_zero_chunk(const BlendArgs& a, int64_t c) {
  const int64_t n = min((int64_t)a.ctr[kCtrSplats], a.cap_splats);
  float4* g = reinterpret_cast<float4*>(a.sp_grad);
  const int64_t lo = 3 * c * kZeroChunk, hi = 3 * min(n, (c + 1) * kZeroChunk);
  for (int64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) g[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// Zeroing chunk c of the backward: Gaussians [c kZeroChunk, (c + 1) kZeroChunk).
__device__ __forceinline__ uint32_t grad_chunks(const GradZero& z) {
  return (uint32_t)((z.n + kZeroChunk - 1) / kZeroChunk);
}
__device__ void grad_zero_chunk(const GradZero& z, int64_t c) {
  const int64_t g0 = c * kZeroChunk, g1 = min(z.n, g0 + kZeroChunk);
  zero_span(z.g.means, 3 * g0, 3 * g1);
  zero_span(z.g.log_scales, 3 * g0, 3 * g1);
  zero_span(z.g.quats, 4 * g0, 4 * g1);
  zero_span(z.g.opacity_logits, g0, g1);
  if (z.g.sh) {
    const int64_t w0 = g0 / 32, w1 = (g1 + 31) / 32;
    switch (z.sh_floats) {
      case 3: zero_sh_unkept<3>(z, w0, w1); break;
      case 12: zero_sh_unkept<12>(z, w0, w1); break;
      case 27: zero_sh_unkept<27>(z, w0, w1); break;
      default: zero_sh_unkept<48>(z, w0, w1); break;
    }
  }
}

__device__ __forceinline__ int view_of_tile(const ViewSet& vs, int tile) {
  int v = 0;
  while (v + 1 < vs.n_views && vs.v[v + 1].tile_base <= tile) ++v;
  return v;
}

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.69314718055994531f;

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Shared-memory form of a splat for the blend: the conic is pre-scaled so that
// the exponent is evaluated directly in base 2:
//   a = (u, v, A2, B2), b = (C2, opacity, r, g), c = b-channel, with
//   A2 = -A/2 log2(e), B2 = -B log2(e), C2 = -C/2 log2(e)
// so that power * log2(e) = dx (A2 dx + B2 dy) + C2 dy^2 and G = 2^that.
__device__ __forceinline__ void stage_splat(const float2 xy, const float4 co, const float4 rgb,
                                            float4& a, float4& b, float& c) {
  a = make_float4(xy.x, xy.y, -0.5f * kLog2e * co.x, -kLog2e * co.y);
  b = make_float4(-0.5f * kLog2e * co.z, co.w, rgb.x, rgb.y);
  c = rgb.z;
}

// Exponent (base 2) and alpha of a staged splat at pixel centre (fx, fy), as
// both blend kernels evaluate them (in packed pairs, with these operations in
// this order, so that both take the same FP32 decisions):
//   dx = u - fx, dy = v - fy, p = fma(dx, fma(A2, dx, B2 dy), (C2 dy) dy),
//   G = 2^p (ex2.approx), raw = o G, alpha = min(0.99, raw);
// the pixel takes the splat iff p <= 0 and alpha >= 1/255.

// Bounding box of the region where a staged splat can reach alpha >= 1/255:
// the ellipse d^T Q d <= 2 ln(255 o) (Q the conic), grown by a small relative
// and absolute margin so that FP32 rounding of the exact test can never fall
// outside it. Empty (xmin = +inf) when o < 1/255; unbounded for a splat too
// anisotropic for that guarantee (the per-pixel test then decides alone).
__device__ __forceinline__ float4 alpha_box(const float2 xy, const float4 co) {
  const float o = co.w;
  if (!(o * 255.f > 1.f)) return make_float4(INFINITY, -INFINITY, INFINITY, -INFINITY);
  const float det = conic_det_lower(co.x, co.y, co.z);
  if (det < 0.f) {
    const float sum = co.x + co.y + co.z;
    return make_float4(sum != sum ? sum : -INFINITY, INFINITY, -INFINITY, INFINITY);
  }
  const float L2 = 2.f * __logf(255.f * o);
  const float ex = sqrtf(fmaxf(L2 * co.z / det, 0.f)) * 1.002f + 0.02f;
  const float ey = sqrtf(fmaxf(L2 * co.x / det, 0.f)) * 1.002f + 0.02f;
  return make_float4(xy.x - ex, xy.x + ex, xy.y - ey, xy.y + ey);
}

// The blend kernels run kBandWarps warps per tile; warp r covers the band of
// 16 / kBandWarps rows starting at row r * 16 / kBandWarps, and lane (x, y) =
// (l & 7, l >> 3) owns the pixels (x + 8c, y + 4k) of that band, c = 0, 1.
// The forward's footprint test and contributor bits are per band, and the
// backward walks a band's bits. Neighbouring 8x8 blocks share almost all their
// contributors (a 16x8 band's set is 3 % larger than an 8x8 block's at the rig
// workload), while the per-splat work of a warp (the footprint ballot, the
// loop and the loads; in the backward the nine-value warp sum, its dominant
// cost) is shared by 2 * (4 / kBandWarps) pixels per lane.
constexpr int kBandWarps = kBlendBands;
constexpr int kBandThreads = 32 * kBandWarps;
constexpr int kBandRows = 4 / kBandWarps;       // pixel rows per lane and column
constexpr int kBandPix = 2 * kBandRows;         // pixels per lane
static_assert(S3R_BLEND_FWD_BATCH % 32 == 0 && S3R_BLEND_FWD_BATCH <= 256 &&
                  S3R_BLEND_BWD_BATCH % 32 == 0 && S3R_BLEND_BWD_BATCH <= 256,
              "batches are whole 32-splat ballots and stay within static shared memory");
static_assert(S3R_BLEND_FWD_BLOCKS >= 1 && S3R_BLEND_FWD_BLOCKS * kBandThreads <= 2048 &&
                  S3R_BLEND_BWD_BLOCKS >= 1 && S3R_BLEND_BWD_BLOCKS * kBandThreads <= 2048,
              "an SM holds at most 2048 threads");

struct Band {
  int X0, Y0;              // pixel (0, 0) of this lane
  float bx0, bx1, by0, by1;   // pixel-centre extent of the warp's band
};
template <int kWarpsT>
__device__ __forceinline__ Band band_pixels(const ViewInfo& vi, int lt, int warp, uint32_t lane) {
  Band b;
  const int bx = (lt % vi.gx) * kTile, by = (lt / vi.gx) * kTile + warp * (kTile / kWarpsT);
  b.X0 = bx + (int)(lane & 7u);
  b.Y0 = by + (int)(lane >> 3);
  b.bx0 = bx + 0.5f;
  b.bx1 = bx + 15.5f;
  b.by0 = by + 0.5f;
  b.by1 = by + (kTile / kWarpsT) - 0.5f;
  return b;
}

// Whether a staged splat can reach alpha >= 1/255 at some pixel centre of the
// band. The base-2 exponent p = dx (A2 dx + B2 dy) + C2 dy^2 (dx = u - px,
// dy = v - py) is concave, so its maximum over the band's pixel-centre
// rectangle is 0 if the centre lies inside and otherwise lies on an edge, at
// the clamped stationary point of that edge (dy = -B2 X / (2 C2) on the edge
// dx = X, dx = -B2 Y / (2 A2) on dy = Y). The splat passes if that maximum
// reaches log2(1 / (255 o)) less a margin far above FP32 rounding, so that no
// splat the per-pixel test would keep is dropped. Most splats are small and
// anisotropic, and their bounding box touches many bands that the ellipse
// itself misses.
__device__ __forceinline__ bool ellipse_reaches(const float4 a, const float4 b, const Band& t) {
  // the staged conic is (A, B, C) scaled by -log2(e) (A2 = -A/2, B2 = -B, C2 = -C/2)
  if (conic_det_lower(-a.z, -0.5f * a.w, -b.x) < 0.f) return true;
  const float dx0 = a.x - t.bx1, dx1 = a.x - t.bx0;
  const float dy0 = a.y - t.by1, dy1 = a.y - t.by0;
  const bool inside = (dx0 <= 0.f) & (dx1 >= 0.f) & (dy0 <= 0.f) & (dy1 >= 0.f);
  const float A2 = a.z, B2 = a.w, C2 = b.x;
  const float kx = -0.5f * B2 * rcp_approx(C2), ky = -0.5f * B2 * rcp_approx(A2);
  float best = -INFINITY;
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const float X = s ? dx1 : dx0;
    const float dy = fminf(fmaxf(kx * X, dy0), dy1);
    best = fmaxf(best, fmaf(X, fmaf(A2, X, B2 * dy), C2 * dy * dy));
    const float Y = s ? dy1 : dy0;
    const float dx = fminf(fmaxf(ky * Y, dx0), dx1);
    best = fmaxf(best, fmaf(dx, fmaf(A2, dx, B2 * Y), C2 * Y * Y));
  }
  const float thr = -__log2f(255.f * b.y);
  return inside | (best >= thr - (0.05f + 1e-3f * fabsf(thr)));
}

__device__ __forceinline__ bool box_misses(const float4 b, const Band& t) {
  return b.x > t.bx1 || b.y < t.bx0 || b.z > t.by1 || b.w < t.by0;
}

// kCount: also count the (pixel, splat) pairs walked (list positions up to
// each pixel's stop) and evaluated (footprint test passed, pixel not stopped).
//
// A lane's two pixels of a column (rows y and y + 4) are evaluated as one
// packed pair: the splat's values are staged in shared memory as duplicated
// pairs (A2 A2 B2 B2 | C2 C2 o o | r r g g | b b v v | u u), so every operand
// of the packed arithmetic comes straight from a 64-bit shared load. The
// arithmetic is the exponent and alpha of stage_splat's comment, in that
// order, so the backward's recomputation takes the same decisions.
constexpr int kBatchFwd = S3R_BLEND_FWD_BATCH;
// The forward's decision for one pixel as one predicate chain (three compares,
// three selects; written as compiler booleans the same decisions took about
// twice the integer-pipe instructions, and that pipe is the forward's busiest).
// `floor_` is the least alpha the pixel still takes: 1/255 until it stops, then
// infinity. The splat is taken where p <= 0, alpha >= floor_ and the
// transmittance nT it would leave is not under 1e-4; where only the last fails
// the pixel stops. It took 6.5 % off the kernel's instructions. Returns the
// applied alpha and moves the last position.
__device__ __forceinline__ float blend_alpha(float p, float al, float nT, int pos, float& floor_,
                                             int& last) {
  float ab;
  asm("{\n\t.reg .pred q, s, b;\n\t"
      "setp.leu.f32 q, %3, 0f00000000;\n\t"
      "setp.geu.and.f32 q, %4, %1, q;\n\t"
      "setp.lt.and.f32 s|b, %5, %7, q;\n\t"
      "selp.f32 %0, %4, 0f00000000, b;\n\t"
      "selp.b32 %2, %6, %2, b;\n\t"
      "selp.f32 %1, 0f7F800000, %1, s;\n\t}"
      : "=&f"(ab), "+f"(floor_), "+r"(last)
      : "f"(p), "f"(al), "f"(nT), "r"(pos), "f"(kTStop));
  return ab;
}

// One splat of the forward's walk over a lane's pixels, kPairs packed pairs:
// two columns of two rows each with two warps per tile, one row of two columns
// with four (FX and FY hold the pairs' pixel centres accordingly). kClamp: the
// splat's opacity exceeds 0.99, so alpha = o G may reach the 0.99 cap; for o <= 0.99 it cannot (G = 2^p <= 1 where p <= 0, up
// to the last ulp of ex2.approx at p = 0), and the clamp is left out. The
// backward takes the same branch per splat, and the FP64 o G of the exact
// definition never reaches the cap for those splats either.
//
// fwd_eval: the exponents and alphas, which depend on the splat and the pixel
// alone. `cap`: the alpha cap, or NaN where the splat cannot reach it.
// fwd_apply: the decisions and the compositing, in the splats' order.
template <int kPairs>
struct SplatEval {
  float p[2 * kPairs], al[2 * kPairs];
};
template <bool kClamp, int kPairs>
__device__ __forceinline__ void fwd_eval(const float4 q0, const float4 q1, const float4 q3, const float2 qu,
                                         float cap, const f2 FY, const f2 (&FX)[kPairs],
                                         SplatEval<kPairs>& e) {
  const f2 A2 = pk(q0.x, q0.y), B2 = pk(q0.z, q0.w), C2c = pk(q1.x, q1.y), O2 = pk(q1.z, q1.w);
  const f2 V2 = pk(q3.z, q3.w), U2 = pk(qu.x, qu.y);
  // the rows' dy and the dy terms of the exponent, shared by the pairs
  const f2 dy = sub2(V2, FY);
  const f2 bdy = mul2(B2, dy);
  const f2 cdy = mul2(mul2(C2c, dy), dy);
#pragma unroll
  for (int c = 0; c < kPairs; ++c) {
    const f2 dx = sub2(U2, FX[c]);
    const f2 pw = fma2(dx, fma2(A2, dx, bdy), cdy);
    upk(pw, e.p[2 * c], e.p[2 * c + 1]);
    float raw[2];
    upk(mul2(O2, pk(ex2_approx(e.p[2 * c]), ex2_approx(e.p[2 * c + 1]))), raw[0], raw[1]);
#pragma unroll
    for (int r = 0; r < 2; ++r) e.al[2 * c + r] = kClamp ? fminf(cap, raw[r]) : raw[r];
  }
}
template <bool kCount, int kPairs>
__device__ __forceinline__ void fwd_apply(const SplatEval<kPairs>& e, const float4 q2, const float4 q3,
                                          const f2 ONE, int pos, f2 (&T2)[kPairs],
                                          f2 (&C2)[kPairs][3], int (&last)[2 * kPairs],
                                          int (&endp)[2 * kPairs], float (&floor_)[2 * kPairs],
                                          uint32_t& n_eval, bool& any_blend) {
  // a blended pixel takes alpha >= 1/255 > 0, a skipped one 0: the splat was
  // blended somewhere in the lane's pixels iff the applied alphas sum above 0
  f2 ab_sum;
  const f2 R2 = pk(q2.x, q2.y), G2 = pk(q2.z, q2.w), Bl2 = pk(q3.x, q3.y);
#pragma unroll
  for (int c = 0; c < kPairs; ++c) {
    float ab[2], nT[2];
    upk(mul2(T2[c], sub2(ONE, pk(e.al[2 * c], e.al[2 * c + 1]))), nT[0], nT[1]);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int k = 2 * c + r;
      const bool was_done = floor_[k] > 1.f;
      if constexpr (kCount) n_eval += was_done ? 0u : 1u;
      // one select: T (1 - 0) = T exactly where the splat is not blended
      ab[r] = blend_alpha(e.p[k], e.al[k], nT[r], pos, floor_[k], last[k]);
      if constexpr (kCount) endp[k] = !was_done && floor_[k] > 1.f ? pos : endp[k];
    }
    const f2 AB = pk(ab[0], ab[1]);
    ab_sum = c == 0 ? AB : add2(ab_sum, AB);
    const f2 w = mul2(AB, T2[c]);
    C2[c][0] = fma2(R2, w, C2[c][0]);
    C2[c][1] = fma2(G2, w, C2[c][1]);
    C2[c][2] = fma2(Bl2, w, C2[c][2]);
    T2[c] = mul2(T2[c], sub2(ONE, AB));
  }
  float s0, s1;
  upk(ab_sum, s0, s1);
  any_blend = s0 + s1 > 0.f;
}

// A splat without a conic (an entry NaN: a Gaussian so long that its 2D covariance
// overflows) has alpha NaN, and makes NaN of the pixels that walk it. The decisions
// let NaN pass, as those of a splat that a pixel takes, so a pixel that has stopped
// is given alpha 0 here.
template <int kPairs>
__device__ __forceinline__ void guard_stopped(SplatEval<kPairs>& e, const float (&floor_)[2 * kPairs]) {
#pragma unroll
  for (int k = 0; k < 2 * kPairs; ++k) e.al[k] = floor_[k] > 1.f ? 0.f : e.al[k];
}

template <int kPix>
__device__ __forceinline__ bool all_stopped(const float (&floor_)[kPix]) {
  float least = floor_[0];
#pragma unroll
  for (int k = 1; k < kPix; ++k) least = fminf(least, floor_[k]);
  return least > 1.f;
}

// S3R_BLEND_FWD_BLOCKS: 18 blocks per SM (56 registers). At the surround rig
// (27.7M pairs, 1.07G evaluated) 18 blocks took 1.043 ms, 20 (48 registers)
// 1.084 ms and 16 (64 registers) 1.148 ms: the kernel needs the warps, and a
// few registers more than 48 end the spills.
//
// kWarpsT: warps per tile. Two (16x8 bands, four pixels per lane) share a
// splat's loads and loop between the most pixels. On a small image the time is
// that of the longest list walked by one pair of warps, and four (16x4 bands, two
// pixels per lane) walk it faster: see launch_fwd for the line and its times. The
// contributor bits stay those of the backward's 16x8 bands, two warps adding
// to each.
template <bool kCount, int kWarpsT>
__global__ void __launch_bounds__(32 * kWarpsT, S3R_BLEND_FWD_BLOCKS * kBandWarps / kWarpsT) k_blend_fwd(
    const __grid_constant__ ViewSet vs, BlendArgs a) {
  sequence_begin();
  static_assert(kWarpsT == 2 || kWarpsT == 4, "bands of 16x8 or 16x4 pixels");
  constexpr int kPairs = 4 / kWarpsT, kPix = 2 * kPairs, kThreadsT = 32 * kWarpsT;
  constexpr int kAhead = 2;   // splats evaluated together by four warps (1: 0.184 ms, 2: 0.149, 3 and 4: 0.162)
  constexpr int kStage = (kBatchFwd + kThreadsT - 1) / kThreadsT;   // splats a thread stages per batch
  __shared__ float4 s_p0[kBatchFwd];   // A2 A2 B2 B2
  __shared__ float4 s_p1[kBatchFwd];   // C2 C2 o o
  __shared__ float4 s_p2[kBatchFwd];   // r r g g
  __shared__ float4 s_p3[kBatchFwd];   // b b v v
  __shared__ float2 s_u[kBatchFwd];    // u u
  __shared__ float4 s_box[kBatchFwd];
  __shared__ uint32_t s_cstart[kTileClasses + 2];
  __shared__ int s_tile, s_works;
  QueueState queue;
  if (!fwd_queue_init(a, s_cstart, &s_works, splat_grad_chunks(a), queue)) return;
  for (;;) {
    const int tile = fwd_queue_next(a, s_cstart, &s_tile, queue);
    if (tile == -1) break;
    if (tile < -1) {
      splat_grad_zero_chunk(a, -2 - (int64_t)tile);
      __syncthreads();   // s_tile is rewritten by the next queue_next
      continue;
    }
    const int v = view_of_tile(vs, tile);
    const ViewInfo& vi = vs.v[v];
    const int lt = tile - vi.tile_base;
    const int warp = threadIdx.x >> 5;
    const uint32_t lane = lane_id();
    const Band P = band_pixels<kWarpsT>(vi, lt, warp, lane);
    // pixel k = 2 c + r of the lane: column c, row r of two warps' bands, else
    // column r of the one row
    int px[kPix], py[kPix];
#pragma unroll
    for (int k = 0; k < kPix; ++k) {
      px[k] = P.X0 + 8 * (kPairs == 2 ? k >> 1 : k);
      py[k] = P.Y0 + (kPairs == 2 ? 4 * (k & 1) : 0);
    }
    const uint2 range = a.ranges[tile];
    const int n = (int)(range.y - range.x);
    const f2 FY = pk((float)py[0] + 0.5f, (float)py[1] + 0.5f);
    f2 FX[kPairs];
    const f2 ONE = pk(1.f, 1.f);

    // per pair; scalar per-pixel state
    f2 T2[kPairs], C2[kPairs][3];
    int last[kPix], endp[kPix];
    float floor_[kPix];   // least alpha taken; infinity once the pixel has stopped
    uint32_t n_eval = 0;
  #pragma unroll
    for (int c = 0; c < kPairs; ++c) {
      FX[c] = pk((float)px[2 * c] + 0.5f, (float)px[2 * c + 1] + 0.5f);
      T2[c] = ONE;
      C2[c][0] = C2[c][1] = C2[c][2] = pk(0.f, 0.f);
    }
  #pragma unroll
    for (int k = 0; k < kPix; ++k) {
      const bool inside = px[k] < vi.width && py[k] < vi.height;
      last[k] = 0;
      floor_[k] = inside ? kAlphaMin : INFINITY;
      endp[k] = inside ? n : 0;      // positions walked
    }
    uint32_t* wbits = a.contrib + (warp * kBandWarps / kWarpsT) * a.contrib_words;
    uint32_t ahead[kStage];   // the next batch's splat ids, loaded one batch ahead
#pragma unroll
    for (int q = 0; q < kStage; ++q) {
      const int i = (int)threadIdx.x + q * kThreadsT;
      ahead[q] = i < kBatchFwd && i < n ? a.sorted_splats[range.x + i] : 0u;
    }
    for (int b0 = 0; b0 < n; b0 += kBatchFwd) {
      // whether every pixel has stopped: tested once per chunk and batch, not per splat
      if (__syncthreads_and(all_stopped(floor_))) break;
#pragma unroll
      for (int q = 0; q < kStage; ++q) {
        const int i = (int)threadIdx.x + q * kThreadsT;
        if (i >= kBatchFwd || b0 + i >= n) continue;
        const uint32_t s = ahead[q];
        const uint4 t0 = a.sp_tin[2 * (size_t)s], t1 = a.sp_tin[2 * (size_t)s + 1];
        const float2 xy = make_float2(__uint_as_float(t0.x), __uint_as_float(t0.y));
        const float4 co = make_float4(__uint_as_float(t0.z), __uint_as_float(t0.w),
                                      __uint_as_float(t1.x), __uint_as_float(t1.y));
        const float4 rgb = a.sp_rgb_d[s];
        float4 sa, sb;
        float sc;
        stage_splat(xy, co, rgb, sa, sb, sc);
        s_p0[i] = make_float4(sa.z, sa.z, sa.w, sa.w);
        s_p1[i] = make_float4(sb.x, sb.x, sb.y, sb.y);
        s_p2[i] = make_float4(sb.z, sb.z, sb.w, sb.w);
        s_p3[i] = make_float4(sc, sc, sa.y, sa.y);
        s_u[i] = make_float2(sa.x, sa.x);
        s_box[i] = alpha_box(xy, co);
        if (b0 + kBatchFwd + i < n) ahead[q] = a.sorted_splats[range.x + b0 + kBatchFwd + i];
      }
      __syncthreads();
      const int m = min(kBatchFwd, n - b0);
      for (int c0 = 0; c0 < m; c0 += 32) {
        if (__all_sync(0xffffffffu, all_stopped(floor_))) break;
        // which of the next 32 splats can reach alpha >= 1/255 in this warp's band
        const int jl = c0 + (int)lane;
        bool reach = false, no_conic = false;
        if (jl < m) {
          const float4 p0 = s_p0[jl], p1 = s_p1[jl], p3 = s_p3[jl];
          const float4 ea = make_float4(s_u[jl].x, p3.z, p0.x, p0.z);
          const float4 eb = make_float4(p1.x, p1.z, 0.f, 0.f);
          const float4 box = s_box[jl];
          reach = !box_misses(box, P) && ellipse_reaches(ea, eb, P);
          no_conic = box.x != box.x;
        }
        uint32_t todo = __ballot_sync(0xffffffffu, reach);
        uint32_t blended = 0;     // splats of this chunk blended into some pixel of the band
        // the chunk's walk; kGuard where it has a splat without a conic (see guard_stopped)
        auto walk = [&](auto guard) {
          constexpr bool kGuard = decltype(guard)::value;
          if constexpr (kWarpsT == 2) {
            while (todo) {
              const int j = c0 + __ffs(todo) - 1;
              todo &= todo - 1;
              const float4 q0 = s_p0[j], q1 = s_p1[j], q2 = s_p2[j], q3 = s_p3[j];
              const float2 qu = s_u[j];
              bool any_blend = false;
              SplatEval<kPairs> e;
              // warp-uniform: every lane walks the same splat
              if (q1.z > kAlphaMax) {
                fwd_eval<true, kPairs>(q0, q1, q3, qu, kAlphaMax, FY, FX, e);
                fwd_apply<kCount, kPairs>(e, q2, q3, ONE, b0 + j + 1, T2, C2, last, endp, floor_, n_eval,
                                          any_blend);
              } else {
                fwd_eval<false, kPairs>(q0, q1, q3, qu, 0.f, FY, FX, e);
                if constexpr (kGuard) guard_stopped<kPairs>(e, floor_);
                fwd_apply<kCount, kPairs>(e, q2, q3, ONE, b0 + j + 1, T2, C2, last, endp, floor_, n_eval,
                                          any_blend);
              }
              if (__any_sync(0xffffffffu, any_blend)) blended |= 1u << (j - c0);
            }
          } else {
            // kAhead splats at a time: their exponents and alphas are independent
            // and overlap, only the compositing is a chain
            while (todo) {
              int js[kAhead];
              SplatEval<kPairs> e[kAhead];
              int m_here = 0;
#pragma unroll
              for (int u = 0; u < kAhead; ++u) {
                js[u] = c0 + (todo ? __ffs(todo) - 1 : 0);
                m_here += todo ? 1 : 0;
                todo &= todo - 1;
              }
#pragma unroll
              for (int u = 0; u < kAhead; ++u) {
                const int j = js[u];
                const float4 q1 = s_p1[j];
                // where there is no cap, NaN: the minimum is then the alpha, NaN included
                fwd_eval<true, kPairs>(s_p0[j], q1, s_p3[j], s_u[j], q1.z > kAlphaMax ? kAlphaMax : NAN, FY, FX,
                                       e[u]);
              }
#pragma unroll
              for (int u = 0; u < kAhead; ++u) {
                if (u >= m_here) break;
                const int j = js[u];
                bool any_blend = false;
                if constexpr (kGuard) guard_stopped<kPairs>(e[u], floor_);
                fwd_apply<kCount, kPairs>(e[u], s_p2[j], s_p3[j], ONE, b0 + j + 1, T2, C2, last, endp, floor_,
                                          n_eval, any_blend);
                if (__any_sync(0xffffffffu, any_blend)) blended |= 1u << (j - c0);
              }
            }
          }
        };
        if (__ballot_sync(0xffffffffu, no_conic))
          walk(std::true_type{});
        else
          walk(std::false_type{});
        if (lane == 0 && blended) or_bits(wbits, range.x + b0 + c0, blended);
      }
    }
    if constexpr (kCount) {
      // work accounting, one 64-bit atomic per warp and counter
      unsigned long long walked = 0;
  #pragma unroll
      for (int k = 0; k < kPix; ++k) walked += (unsigned long long)endp[k];
      unsigned long long evald = n_eval;
  #pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        walked += __shfl_xor_sync(0xffffffffu, walked, o);
        evald += __shfl_xor_sync(0xffffffffu, evald, o);
      }
      if (lane == 0 && walked) atomicAdd(a.pairs, walked);
      if (lane == 0 && evald) atomicAdd(a.eval_fwd, evald);
    }
    const int64_t plane = (int64_t)vi.width * vi.height;
  #pragma unroll
    for (int c = 0; c < kPairs; ++c) {
      float T[2], Cr[2], Cg[2], Cb[2];
      upk(T2[c], T[0], T[1]);
      upk(C2[c][0], Cr[0], Cr[1]);
      upk(C2[c][1], Cg[0], Cg[1]);
      upk(C2[c][2], Cb[0], Cb[1]);
  #pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int k = 2 * c + r;
        if (px[k] < vi.width && py[k] < vi.height) {
          const int64_t pix = (int64_t)py[k] * vi.width + px[k];
          float* o = a.out + 3 * (int64_t)vi.pix_base + pix;
          o[0] = fmaf(T[r], a.bg[0], Cr[r]);
          o[plane] = fmaf(T[r], a.bg[1], Cg[r]);
          o[2 * plane] = fmaf(T[r], a.bg[2], Cb[r]);
          a.final_T[vi.pix_base + pix] = T[r];
          a.n_contrib[vi.pix_base + pix] = (uint32_t)last[k];
        }
      }
    }
    __syncthreads();   // shared staging is reused by the next tile
  }
  fwd_queue_exit(a, queue);
}

// a ? x : y as one selp. Written out because the compiler turned the
// lane-dependent selects of the warp sum below into divergent branches around
// the shuffles (57 branch instructions per splat in the backward), which made
// the sum several times dearer than its 14 shuffles.
__device__ __forceinline__ float select_f(bool a, float x, float y) {
  float r;
  asm("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\tselp.f32 %0, %1, %2, p;\n\t}"
      : "=f"(r)
      : "f"(x), "f"(y), "r"((int)a));
  return r;
}

// The backward's decision for one pixel as one predicate chain: G is kept where
// the forward blended the splat (position before the pixel's last contributor,
// p <= 0, alpha >= 1/255) and becomes 0 elsewhere.
__device__ __forceinline__ void keep_taken(float p, float al, float& G, int pos, int last) {
  asm("{\n\t.reg .pred q;\n\t"
      "setp.lt.s32 q, %3, %4;\n\t"
      "setp.leu.and.f32 q, %2, 0f00000000, q;\n\t"
      "setp.geu.and.f32 q, %1, %5, q;\n\t"
      "selp.f32 %0, %0, 0f00000000, q;\n\t}"
      : "+f"(G)
      : "f"(al), "f"(p), "r"(pos), "r"(last), "f"(kAlphaMin));
}

__device__ __forceinline__ void red_shared(float* addr, float v) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(addr);
  asm volatile("red.shared.add.f32 [%0], %1;" ::"r"(sa), "f"(v) : "memory");
}

__device__ __forceinline__ void red_v4(float* p, float x, float y, float z, float w) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(x), "f"(y), "f"(z),
               "f"(w)
               : "memory");
}

// Per-pixel state of the reverse walk: the recovered transmittance in front
// of the current splat, and the colour already composited behind it, dotted
// with dL/dC and in absolute terms,
//   Bd = T_final (bg . d) + sum over blended splats k behind of (c_k . d) alpha_k T_k,
// so that dL/dalpha_i = T_i (c_i . d) - Bd / (1 - alpha_i) (Eq. 2 differentiated).
struct BwdPixel {
  float T, Bd, d0, d1, d2;
  int last;
};

// One splat's contribution to the adjoints at one pixel (reverse order), with
// act = the forward blended it there: T <- T / (1 - alpha) where act;
// cd = c . d; dL/dalpha = T cd - Bd / (1 - alpha); w = act ? alpha T : 0;
// Bd += cd w; dL/dopacity = (act and raw <= 0.99 ? G : 0) dL/dalpha (alpha =
// 0.99 is constant); dpow = o dL/dopacity is dL/d(power). The per-splat sums
// are kept in moment form over the warp's pixels,
//   g0 = sum dpow dx, g1 = sum dpow dy, g2 = sum dpow dx^2, g3 = sum dpow dx dy,
//   g4 = sum dpow dy^2, g5 = sum dL/dopacity, g6..8 = sum w dL/dC,
// (a column's pixels share dx, so g0..g3 take its sums of dpow and dpow dy)
// and turned into the adjoints of (u, v, conic) once per splat at the flush.

__device__ __forceinline__ void bwd_init(BwdPixel& q, const BlendArgs& a, const ViewInfo& vi,
                                         int px, int py, bool inside) {
  q.T = 1.f; q.d0 = q.d1 = q.d2 = 0.f; q.last = 0;
  if (inside) {
    const int64_t plane = (int64_t)vi.width * vi.height;
    const int64_t pix = (int64_t)py * vi.width + px;
    const float* g = a.dL + 3 * (int64_t)vi.pix_base + pix;
    q.d0 = g[0];
    q.d1 = g[plane];
    q.d2 = g[2 * plane];
    q.T = a.final_T[vi.pix_base + pix];
    q.last = (int)a.n_contrib[vi.pix_base + pix];
  }
  q.Bd = q.T * (a.bg[0] * q.d0 + a.bg[1] * q.d1 + a.bg[2] * q.d2);
}

// One splat of the backward's walk (see above) over a lane's two packed
// pixel pairs: updates T and Bd, returns the lane's shares of the nine sums in
// g. kClamp as for fwd_eval, per splat.
//
// A pixel that does not take the splat gets G = 0, hence alpha 0: 1 / (1 - 0) is
// exactly 1, so T, the weight and every sum are left unchanged by the same
// arithmetic, with one select per pixel. A thin splat's moments cancel in the
// chain to its covariance, which magnifies their last bits by the splat's
// aspect ratio, so the sums' order of additions is kept fixed (here and in
// sum_rows).
template <bool kCount, bool kClamp>
__device__ __forceinline__ void bwd_splat(const float4 q0, const float4 q1, const float4 q2,
                                          const float4 q3, const float2 qu, const f2 FY,
                                          const f2 (&FX)[2], const f2 ONE, int pos,
                                          const int (&last)[kBandPix], f2 (&T2)[2], f2 (&Bd2)[2],
                                          const f2 (&Q0)[2], const f2 (&Q1)[2], const f2 (&Q2)[2],
                                          uint32_t& n_eval, float (&g)[9]) {
  constexpr int kRows = kBandRows;
  const f2 A2 = pk(q0.x, q0.y), B2 = pk(q0.z, q0.w), C2c = pk(q1.x, q1.y), O2 = pk(q1.z, q1.w);
  const f2 R2 = pk(q2.x, q2.y), G2 = pk(q2.z, q2.w), Bl2 = pk(q3.x, q3.y), V2 = pk(q3.z, q3.w);
  const f2 U2 = pk(qu.x, qu.y);
  const f2 dy = sub2(V2, FY);
  const f2 bdy = mul2(B2, dy);
  const f2 cdy = mul2(mul2(C2c, dy), dy);
  f2 gdy, gop, w0, w1, w2;
  float D[2], E[2], dx[2], dyv[2], x, y;
  upk(dy, dyv[0], dyv[1]);
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const f2 dx2 = sub2(U2, FX[c]);
    const f2 pw = fma2(dx2, fma2(A2, dx2, bdy), cdy);
    float p[2], G[2], raw[2], inv[2];
    upk(pw, p[0], p[1]);
    G[0] = ex2_approx(p[0]);
    G[1] = ex2_approx(p[1]);
    upk(mul2(O2, pk(G[0], G[1])), raw[0], raw[1]);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int k = c * kRows + r;
      if constexpr (kCount) n_eval += pos < last[k] ? 1u : 0u;
      keep_taken(p[r], kClamp ? fminf(kAlphaMax, raw[r]) : raw[r], G[r], pos, last[k]);
    }
    f2 AL = mul2(O2, pk(G[0], G[1]));
    if constexpr (kClamp) {
      // alpha = 0.99 is constant in the splat's parameters
      upk(AL, x, y);
      AL = pk(fminf(kAlphaMax, x), fminf(kAlphaMax, y));
      G[0] = select_f(x > kAlphaMax, 0.f, G[0]);
      G[1] = select_f(y > kAlphaMax, 0.f, G[1]);
    }
    upk(sub2(ONE, AL), inv[0], inv[1]);
    inv[0] = rcp_approx(inv[0]);
    inv[1] = rcp_approx(inv[1]);
    // T before this splat; Bd the colour behind it
    T2[c] = mul2(T2[c], pk(inv[0], inv[1]));
    const f2 cd = fma2(R2, Q0[c], fma2(G2, Q1[c], mul2(Bl2, Q2[c])));
    const f2 dal = fma2(T2[c], cd, mul2(Bd2[c], pk(-inv[0], -inv[1])));   // dL/dalpha
    const f2 w = mul2(AL, T2[c]);
    Bd2[c] = fma2(cd, w, Bd2[c]);
    const f2 gd = mul2(pk(G[0], G[1]), dal);
    const f2 dpow = mul2(O2, gd);                       // dL/d(power), natural units
    const f2 pdy = mul2(dpow, dy);
    gdy = c == 0 ? mul2(pdy, dy) : fma2(pdy, dy, gdy);
    gop = c == 0 ? gd : add2(gop, gd);
    w0 = c == 0 ? mul2(w, Q0[c]) : fma2(w, Q0[c], w0);
    w1 = c == 0 ? mul2(w, Q1[c]) : fma2(w, Q1[c], w1);
    w2 = c == 0 ? mul2(w, Q2[c]) : fma2(w, Q2[c], w2);
    // the column's sums of dpow and dpow * dy (dx is shared by its rows)
    float dp0, dp1;
    upk(dpow, dp0, dp1);
    upk(pdy, x, y);
    D[c] = dp0 + dp1;
    E[c] = fmaf(dp1, dyv[1], x);
    upk(dx2, dx[c], x);
  }
  const float t0 = dx[0] * D[0], t1 = dx[1] * D[1];
  g[0] = t0 + t1;
  g[1] = E[0] + E[1];
  g[2] = fmaf(t1, dx[1], t0 * dx[0]);
  g[3] = fmaf(dx[1], E[1], dx[0] * E[0]);
  upk(gdy, x, y);
  g[4] = x + y;
  upk(gop, x, y);
  g[5] = x + y;
  upk(w0, x, y);
  g[6] = x + y;
  upk(w1, x, y);
  g[7] = x + y;
  upk(w2, x, y);
  g[8] = x + y;
}

// Warp sums of the nine values of two splats through shared memory. Each lane
// stores its nine shares of a splat as one column of nine rows of 32 (pitch
// 36 words: the stores and the row reads below are both free of bank
// conflicts). Once two splats are stored, lane l sums half (16 floats, four
// 128-bit loads, packed adds) of row (l / 2) of the sixteen rows of values
// 0..7, and 16 lanes per splat share the row of value 8. That is 18 stores, 6
// loads and about 14 additions and shuffles per two splats, where a butterfly
// with transposition took 14 shuffles, 14 selects and 14 additions per splat
// (plus its latency of five dependent shuffles). The columns stand in the order
// (even lanes, odd lanes), so that the halves' sums pair lanes 16, 8, 4, 2
// and 1 apart, in that order, as the butterfly does: the totals have its bits.
// At 14 CTAs per SM (72 registers) one 1080p view's backward went from 0.330 to
// 0.321 ms and a 1001 x 563 view's from 0.083 to 0.081 ms; the surround rig
// (1.05G evaluated pairs) stayed at 1.79 ms, where a packed FMA costs the
// issue slots of two scalar ones and the shuffles had hidden behind them. 16
// CTAs (64 registers) took 0.332 and 1.785 ms, 12 (80) 0.328 and 1.850 ms.
constexpr int kSumPitch = 36;
constexpr int kSumSlot = 9 * kSumPitch;           // words per splat
constexpr int kSumWords = 2 * kSumSlot;           // words per warp

__device__ __forceinline__ void sum_store(float* col, const float (&g)[9]) {
#pragma unroll
  for (int v = 0; v < 9; ++v) col[v * kSumPitch] = g[v];
}

// `half_row` and `ninth` are this lane's read positions. On return, even lanes
// hold the total of value (l / 2) % 8 of splat l / 16 in `tot`, and every lane
// the total of value 8 of splat l / 16 in `tot9`.
__device__ __forceinline__ void sum_rows(const float* half_row, const float* ninth, float& tot,
                                         float& tot9) {
  const float4* h = reinterpret_cast<const float4*>(half_row);
  const float4 a = h[0], b = h[1], c = h[2], d = h[3];
  const f2 lo = add2(add2(pk(a.x, a.y), pk(c.x, c.y)), add2(pk(b.x, b.y), pk(d.x, d.y)));
  const f2 hi = add2(add2(pk(a.z, a.w), pk(c.z, c.w)), add2(pk(b.z, b.w), pk(d.z, d.w)));
  float x, y;
  upk(add2(lo, hi), x, y);
  tot = x + y;
  tot += __shfl_xor_sync(0xffffffffu, tot, 1);
  tot9 = ninth[0] + ninth[8];
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) tot9 += __shfl_xor_sync(0xffffffffu, tot9, o);
}

// The reverse walk evaluates a lane's two pixels of a column (rows y and
// y + 4) as one packed pair, like the forward: the splat is staged as
// duplicated pairs, the per-pixel state (T, Bd, dL/dC) is held as pairs per
// column, and the recomputation, the recovery of T and dL/dalpha are the
// scalar expressions in the same order. Only the order in which a lane adds
// up its four pixels' shares of the nine sums differs from a scalar walk.
template <bool kCount>
__global__ void __launch_bounds__(kBandThreads, S3R_BLEND_BWD_BLOCKS) k_blend_bwd(
    const __grid_constant__ ViewSet vs, BlendArgs a) {
  sequence_begin();
  static_assert(kBandRows == 2, "the packed backward pairs the two rows of a lane's column");
  constexpr int kT = kBandThreads;
  constexpr int kRows = kBandRows;
  constexpr int kPix = kBandPix;
  __shared__ float4 s_p0[kBatchBwd];   // A2 A2 B2 B2
  __shared__ float4 s_p1[kBatchBwd];   // C2 C2 o o
  __shared__ float4 s_p2[kBatchBwd];   // r r g g
  __shared__ float4 s_p3[kBatchBwd];   // b b v v
  __shared__ float2 s_u[kBatchBwd];    // u u
  __shared__ uint32_t s_id[kBatchBwd];
  __shared__ float s_g[kBatchBwd][9];
  __shared__ float s_sink[kBandThreads];   // target of the lanes with no sum to add
  __shared__ __align__(16) float s_sum[kBandWarps][kSumWords];
  __shared__ int s_max;
  __shared__ uint32_t s_cstart[kTileClasses + 2];
  __shared__ int s_tile;
  uint32_t pending = 0;
  queue_init(a, a.bwd_queue, s_cstart, grad_chunks(a.zero), pending);
  for (;;) {
    const int tile = queue_next(a, a.bwd_queue, s_cstart, &s_tile, pending);
    if (tile == -1) break;
    if (tile < -1) {
      grad_zero_chunk(a.zero, -2 - (int64_t)tile);
      __syncthreads();   // s_tile is rewritten by the next queue_next
      continue;
    }
    const int v = view_of_tile(vs, tile);
    const ViewInfo& vi = vs.v[v];
    const int lt = tile - vi.tile_base;
    const int warp = threadIdx.x >> 5;
    const uint32_t lane = lane_id();
    const int X0 = (lt % vi.gx) * kTile + (int)(lane & 7u);
    const int Y0 = (lt / vi.gx) * kTile + warp * (kTile / kBandWarps) + (int)(lane >> 3);
    const uint2 range = a.ranges[tile];

    float fx[2], fy[kRows];
  #pragma unroll
    for (int c = 0; c < 2; ++c) fx[c] = (float)(X0 + 8 * c) + 0.5f;
  #pragma unroll
    for (int r = 0; r < kRows; ++r) fy[r] = (float)(Y0 + 4 * r) + 0.5f;
    const f2 FY = pk(fy[0], fy[1]);
    const f2 FX[2] = {pk(fx[0], fx[0]), pk(fx[1], fx[1])};
    const f2 ONE = pk(1.f, 1.f);
    // per column c: (row 0, row 1) pairs of T, Bd and dL/dC; scalar last contributor
    f2 T2[2], Bd2[2], Q0[2], Q1[2], Q2[2];
    int last[kPix];
    int wlast = 0;
  #pragma unroll
    for (int c = 0; c < 2; ++c) {
      BwdPixel qq[kRows];
  #pragma unroll
      for (int r = 0; r < kRows; ++r) {
        const int px = X0 + 8 * c, py = Y0 + 4 * r;
        bwd_init(qq[r], a, vi, px, py, px < vi.width && py < vi.height);
        last[c * kRows + r] = qq[r].last;
        wlast = max(wlast, qq[r].last);
      }
      T2[c] = pk(qq[0].T, qq[1].T);
      Bd2[c] = pk(qq[0].Bd, qq[1].Bd);
      Q0[c] = pk(qq[0].d0, qq[1].d0);
      Q1[c] = pk(qq[0].d1, qq[1].d1);
      Q2[c] = pk(qq[0].d2, qq[1].d2);
    }
    if (threadIdx.x == 0) s_max = 0;
    __syncthreads();
  #pragma unroll
    for (int o = 16; o > 0; o >>= 1) wlast = max(wlast, __shfl_xor_sync(0xffffffffu, wlast, o));
    if (lane == 0 && wlast) atomicMax(&s_max, wlast);
    __syncthreads();
    const int n = s_max;
    uint32_t n_eval = 0;   // counting mode: pairs inside their pixel's walk
    // the lane's column, half row and ninth-row positions of the warp's sums
    float* sum_col = s_sum[warp] + (lane & 1u) * 16u + (lane >> 1);
    const float* sum_half = s_sum[warp] + (lane >> 4) * kSumSlot + ((lane >> 1) & 7u) * kSumPitch +
                            (lane & 1u) * 16u;
    const float* sum_ninth = s_sum[warp] + (lane >> 4) * kSumSlot + 8 * kSumPitch + (lane & 1u) * 16u +
                             ((lane & 15u) >> 1);
    const int sum_value = (lane & 1u) ? 8 : (int)((lane >> 1) & 7u);
    const bool sum_owner = (lane & 1u) == 0 || (lane & 15u) == 1u;
    // the forward recorded its contributors per band, with the same bands
    const uint32_t* wbits = a.contrib + warp * a.contrib_words;

    for (int hi = n; hi > 0; hi -= kBatchBwd) {
      const int lo = max(0, hi - kBatchBwd);
      const int m = hi - lo;
      __syncthreads();
      for (int i = threadIdx.x; i < m; i += kT) {
        const uint32_t s = a.sorted_splats[range.x + lo + i];
        s_id[i] = s;
        const uint4 t0 = a.sp_tin[2 * (size_t)s], t1 = a.sp_tin[2 * (size_t)s + 1];
        const float2 xy = make_float2(__uint_as_float(t0.x), __uint_as_float(t0.y));
        const float4 co = make_float4(__uint_as_float(t0.z), __uint_as_float(t0.w),
                                      __uint_as_float(t1.x), __uint_as_float(t1.y));
        float4 sa, sb;
        float sc;
        stage_splat(xy, co, a.sp_rgb_d[s], sa, sb, sc);
        s_p0[i] = make_float4(sa.z, sa.z, sa.w, sa.w);
        s_p1[i] = make_float4(sb.x, sb.x, sb.y, sb.y);
        s_p2[i] = make_float4(sb.z, sb.z, sb.w, sb.w);
        s_p3[i] = make_float4(sc, sc, sa.y, sa.y);
        s_u[i] = make_float2(sa.x, sa.x);
      }
      for (int i = threadIdx.x; i < kBatchBwd * 9; i += kT) (&s_g[0][0])[i] = 0.f;
      __syncthreads();
      // this warp's splats end at its own last contributor; walk them back to
      // front, 32 at a time, visiting only the splats the forward blended into
      // at least one pixel of the band (recorded bits)
      for (int c1 = min(m, wlast - lo) - 1; c1 >= 0; c1 -= 32) {
        const int c0 = max(0, c1 - 31);
        uint32_t todo = get_bits(wbits, range.x + lo + c0);
        const int span = c1 - c0 + 1;
        if (span < 32) todo &= (1u << span) - 1u;
        // as a ballot result the mask is warp-uniform to the compiler as well
        todo = __ballot_sync(0xffffffffu, (todo >> lane) & 1u);
        int jA = 0;
        bool second = false;   // the slot of the next splat
        while (todo) {
          const int bit = 31 - __clz(todo);
          todo &= ~(1u << bit);
          const int j = c0 + bit;
          const float4 q0 = s_p0[j], q1 = s_p1[j], q2 = s_p2[j], q3 = s_p3[j];
          const float2 qu = s_u[j];
          const int pos = lo + j;
          float g[9];
          // warp-uniform: every lane walks the same splat
          if (q1.z > kAlphaMax)
            bwd_splat<kCount, true>(q0, q1, q2, q3, qu, FY, FX, ONE, pos, last, T2, Bd2, Q0, Q1, Q2,
                                    n_eval, g);
          else
            bwd_splat<kCount, false>(q0, q1, q2, q3, qu, FY, FX, ONE, pos, last, T2, Bd2, Q0, Q1, Q2,
                                     n_eval, g);
          sum_store(sum_col + (second ? kSumSlot : 0), g);
          if (!second) jA = j;
          if (second || todo == 0) {
            __syncwarp();
            float tot, tot9;
            sum_rows(sum_half, sum_ninth, tot, tot9);
            // one shared atomic per warp and two splats: even lanes add value
            // (l / 2) % 8, lanes 1 and 17 the ninth, the rest (and the second
            // splat's lanes where there is none) to their own sink word
            const bool high = lane >= 16u;
            float* dst = s_g[high ? j : jA] + sum_value;
            const bool own = sum_owner && (second || !high);
            dst = own ? dst : &s_sink[threadIdx.x];
            red_shared(dst, select_f((lane & 1u) == 0, tot, tot9));
            __syncwarp();   // the rows are rewritten
          }
          second = !second;
        }
      }
      __syncthreads();
      for (int i = threadIdx.x; i < m; i += kT) {
        const float* sg = s_g[i];
        bool any = false;
  #pragma unroll
        for (int r = 0; r < 9; ++r) any |= sg[r] != 0.f;
        if (any) {
          float* dst = a.sp_grad + 12 * (size_t)s_id[i];
          // moments -> adjoints: power*log2(e) = dx (A2 dx + B2 dy) + C2 dy^2 with
          // dx = u - px, so d/du = ln 2 (2 A2 g0 + B2 g1), d/dv = ln 2 (B2 g0 + 2 C2 g1)
          const float A2 = s_p0[i].x, B2 = s_p0[i].z, C2 = s_p1[i].x;
          const float gu = kLn2 * fmaf(2.f * A2, sg[0], B2 * sg[1]);
          const float gv = kLn2 * fmaf(B2, sg[0], 2.f * C2 * sg[1]);
          red_v4(dst, gu, gv, -0.5f * sg[2], -sg[3]);
          red_v4(dst + 4, -0.5f * sg[4], sg[5], sg[6], sg[7]);
          atomicAdd(dst + 8, sg[8]);
        }
      }
    }
    if constexpr (kCount) {
      unsigned long long evald = n_eval;
  #pragma unroll
      for (int o = 16; o > 0; o >>= 1) evald += __shfl_xor_sync(0xffffffffu, evald, o);
      if (lane == 0 && evald) atomicAdd(a.eval_bwd, evald);
    }
    __syncthreads();   // shared staging is reused by the next tile
  }
  queue_exit(a.bwd_queue);
}

// Zero the per-splat adjoints of the splats written by the last projection.
__global__ void k_zero_grads(float4* g, const uint32_t* ctr, int64_t cap) {
  sequence_begin();
  const int64_t n = 3 * min((int64_t)ctr[kCtrSplats], cap);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    g[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}

}  // namespace

static BlendArgs make_args(s3r_workspace* ws) {
  BlendArgs a;
  a.ranges = ws->ranges;
  a.class_cnt = ws->tile_class_cnt;
  a.class_list = ws->tile_class_list;
  a.tiles = ws->views.total_tiles;
  a.fwd_queue = TileQueue{ws->ctr + kCtrBlendFwdCursor, ws->ctr + kCtrBlendFwdExits};
  a.ctr = ws->ctr;
  a.cap_splats = ws->cap.max_splats;
  a.cap_dups = ws->cap.max_duplicates;
  a.pick = kPickAlways;
  a.bwd_queue = TileQueue{ws->ctr + kCtrBlendBwdCursor, ws->ctr + kCtrBlendBwdExits};
  a.zero = GradZero{nullptr, 0, {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr}, 0};
  a.sorted_splats = ws->dup_val[ws->dup_final];
  a.sp_tin = reinterpret_cast<const uint4*>(ws->sp_tin);
  a.sp_rgb_d = ws->sp_rgb_d;
  a.final_T = ws->final_T;
  a.n_contrib = ws->n_contrib;
  a.sp_grad = ws->sp_grad;
  a.pairs = reinterpret_cast<unsigned long long*>(ws->ctr + kCtrPairs);
  a.eval_fwd = reinterpret_cast<unsigned long long*>(ws->ctr + kCtrEvalFwd);
  a.eval_bwd = reinterpret_cast<unsigned long long*>(ws->ctr + kCtrEvalBwd);
  a.contrib = ws->contrib;
  a.contrib_words = ws->contrib_words;
  a.bg = nullptr;
  a.dL = nullptr;
  a.out = nullptr;
  return a;
}

// Resident CTAs per SM of a blend instantiation, queried once per thread.
template <typename K>
int blend_blocks_per_sm(K kernel, int threads, int* cache) {
  if (*cache == 0) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0) != cudaSuccess ||
        per_sm < 1)
      per_sm = 1;
    *cache = per_sm;
  }
  return *cache;
}

// CTAs of a forward launch: as many as are resident at once.
template <bool kCount, int kWarpsT>
int fwd_grid(const s3r_workspace* ws) {
  static thread_local int per_sm = 0;
  return ws->num_sms * blend_blocks_per_sm(k_blend_fwd<kCount, kWarpsT>, 32 * kWarpsT, &per_sm);
}

// Four warps per tile where every tile has a resident CTA of them (1,368 tiles on
// 152 SMs): they walk the longest list faster. With up to twice as many tiles it is
// in the lists, which only the device knows, whether one of them or the work of all
// decides: both forms are launched, and the one that is not to work returns at once
// (about 2 us). With more tiles still, two warps. Times of the kernel with two and
// with four warps, us (corridors; by tiles, then with the pairs and the longest list
// over the mean):
//   Gaussians        240        920      1,296      1,674      2,405      2,800
//   300,000     125 / 80    80 / 59    74 / 61    74 / 84   80 / 117   88 / 119
//   1M           94 / 61    68 / 53    68 / 57    70 / 84   76 / 108   90 / 113
//   4M           74 / 49    55 / 53    59 / 59    63 / 96   76 / 104  100 / 113
//   1,500 to 2,700 tiles
//     109,000 pairs, 56: 205 / 139     173,000, 44: 295 / 170    152,000, 18: 72 / 53
//     205,000 pairs, 2:   55 / 86      450,000, 3:   80 / 125    380,000, 4:  60 / 90
//     667,000 pairs, 16:  80 / 123     842,000, 43:  84 / 94     327,000, 8: 102 / 80
// Of 67 such images drawn at random the rule takes the slower form in 8, by 4 to 43 us;
// all with two warps took 7 % longer together, all with four 17 %.
//
// Only the smallest of these launches overlap their predecessor's end: placed then, a
// grid that is resident at once ends up unevenly over the SMs, and the longest lists
// share some. Whole forward, us, overlapped and not: 22,000 Gaussians, 320 x 192 165
// and 167, 960 x 540 155 and 157; 150,000 at 320 x 192 172 and 176, 640 x 360 168 and
// 162, 960 x 540 212 and 193; 300,000 at 960 x 540 241 and 209, three views of 576 x
// 324 295 and 245; 1M at 640 x 360 244 and 225, at 1080p (more tiles than CTAs) equal.
constexpr int64_t kOverlapBlendGaussians = 50000;
constexpr int kOverlapBlendTiles = 2;   // per SM
template <bool kCount>
cudaError_t launch_fwd(s3r_workspace* ws, BlendArgs& a, cudaStream_t st) {
  const int g4 = fwd_grid<kCount, 4>(ws), g2 = fwd_grid<kCount, 2>(ws);
  const int tiles = ws->views.total_tiles;
  const bool by_lists = tiles > g4 && tiles <= g2;
  const bool overlap = ws->overlap && (ws->n <= kOverlapBlendGaussians || tiles <= kOverlapBlendTiles * ws->num_sms);
  if (tiles > g4) {
    a.pick = by_lists ? kPickEvenLists : kPickAlways;
    const cudaError_t e = launch_overlapping(overlap, k_blend_fwd<kCount, 2>, g2, 64, 0, st, ws->views, a);
    if (e != cudaSuccess || !by_lists) return e;
  }
  a.pick = by_lists ? kPickLongList : kPickAlways;
  return launch_overlapping(overlap && !by_lists, k_blend_fwd<kCount, 4>, g4, 128, 0, st, ws->views, a);
}

cudaError_t launch_render_fwd(s3r_workspace* ws, const float* bg, float* out, cudaStream_t st) {
  BlendArgs a = make_args(ws);
  a.bg = bg;
  a.out = out;
  if (ws->views.total_tiles == 0) return cudaSuccess;
  cudaError_t e;
  if (ws->counting) {
    // pairs walked and evaluated (two adjacent 64-bit counters)
    if ((e = cudaMemsetAsync(a.pairs, 0, 2 * sizeof(unsigned long long), st)) != cudaSuccess) return e;
  }
  // the contributor bits were cleared by the sort's pair expansion
  KernelTimer timer(ws, kKBlendFwd, st);
  e = ws->counting ? launch_fwd<true>(ws, a, st) : launch_fwd<false>(ws, a, st);
  ws->sp_grad_clean = 1;
  return e;
}

cudaError_t launch_render_bwd(s3r_workspace* ws, const float* bg, const float* dL,
                              const s3r_grads* grads, cudaStream_t st) {
  BlendArgs a = make_args(ws);
  a.bg = bg;
  a.dL = dL;
  // the splat adjoints start at zero: cleared by the forward (chunks in its queue), or here
  // when a backward has used them since
  if (!ws->sp_grad_clean) {
    KernelTimer timer(ws, kKZeroGrads, st);
    const cudaError_t e0 =
        launch_in_sequence(ws, k_zero_grads, (int64_t)ws->num_sms * 4, 256, 0, st,
                           reinterpret_cast<float4*>(ws->sp_grad), ws->ctr, ws->cap.max_splats);
    if (e0 != cudaSuccess) return e0;
  }
  ws->sp_grad_clean = 0;
  if (ws->grad_mode == S3R_GRAD_OVERWRITE && ws->n > 0 &&
      (grads->means || grads->log_scales || grads->quats || grads->opacity_logits || grads->sh)) {
    a.zero.kept_bits = ws->kept_bits;
    a.zero.n = ws->n;
    a.zero.g = *grads;
    a.zero.sh_floats = 3 * (ws->sh_degree + 1) * (ws->sh_degree + 1);
  }
  cudaError_t e;
  if (ws->counting && (e = cudaMemsetAsync(a.eval_bwd, 0, sizeof(unsigned long long), st)) != cudaSuccess)
    return e;
  static thread_local int per_sm[2] = {0, 0};
  KernelTimer timer(ws, kKBlendBwd, st);
  if (ws->counting)
    return launch_in_sequence(
        ws, k_blend_bwd<true>,
        (int64_t)ws->num_sms * blend_blocks_per_sm(k_blend_bwd<true>, kBandThreads, &per_sm[1]),
        kBandThreads, 0, st, ws->views, a);
  return launch_in_sequence(
      ws, k_blend_bwd<false>,
      (int64_t)ws->num_sms * blend_blocks_per_sm(k_blend_bwd<false>, kBandThreads, &per_sm[0]),
      kBandThreads, 0, st, ws->views, a);
}

}  // namespace s3r
