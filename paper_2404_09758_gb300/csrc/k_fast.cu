// Batched estimator, fast path: tiles that keep at most kLightBin live triangles after pruning,
// and the pruning pass itself.
//
// Once per call and (view, tile), k_bin_prune: the bin's triangles are set up unperturbed; a
// triangle stays live if some pixel of the tile may see it under SOME perturbation of the call
// (each edge function pushed out by the triangle's margin: the support of the box every snapped
// perturbed vertex stays in) and it is not surely behind a triangle that surely covers the pixel
// (farther than the largest vertex move from each of its edges, so every perturbed version still
// covers it, and depth intervals apart).  Live triangles are compacted to the front of the bin;
// each pixel's candidates among them (at most CMAX; more: test them all) are stored, so that a
// pair tests a handful of triangles, not the bin.
//
// Work item = (view, 16x16 tile, run of antithetic pairs), one CTA.  Its pairs run in groups of up to
// GMAX (as many as the set-ups and sums fit in shared memory), with barriers only between a group's
// steps (Eq. 8 for each pair's sign vector s, Algorithms 1-2):
//   S   every live triangle is set up on both sides (theta + s eps, theta - s eps) for every pair of
//       the group, in shared memory, from the projected perturbed vertices of the vertex pass
//       (k_vertex.cu), with its 9 coordinate signs; the item's texel window (below) gets the
//       group's sign bits;
//   then the warps take units, an 8 x 4 pixel block of one pair each, from a shared counter; per side
//   R   each pixel finds its visible triangle among its candidates (smallest packed depth|id key);
//   U   computes its UV and bilinear footprint;
//   G   samples its perturbed texels (values and signs from the window; outside it from memory) and
//       shades them; then forms f+ - f- and credits it: the visible triangle (all three vertices at
//       once, or single corners where the sides disagree) and the union of the texel footprints;
//   F   the group's sums are folded with its pairs' signs and issue one global atomic per corner or
//       texel channel.  The counts of texels follow once per item.
//
// Texel window: the bounding box of the first pair's footprints, two texels wider, whose texel values sit
// in shared memory and whose slots take the credits.  A footprint's four texels get the same
// f+ - f-, so a pixel makes ONE addition, to the footprint's cell; a texel's sum is that of the four
// cells around it (fold).  Only texels of side - outside side +'s footprint are credited one by
// one.  Footprints outside the window (cut where it would not fit, or absent) get hashed cells.
//
// Bound by instruction issue: no contraction, under 0.1 B of DRAM per pixel and pair.  One barrier pair
// per group instead of two barriers and a fold per pair, the window instead of global loads and a
// sign-plane look-up per texel, one sum per footprint instead of four, lit frames once per triangle
// and side instead of per pixel, and 32 (lit: 16) warps per SM instead of 16 (8) took the kernel from
// 10.5 to 6.2 ms (unlit, 8,192 triangles, 512^2, 8 views x 64 pairs), 35.8 to 11.9 ms (Lambert, 32,768
// triangles, 1024^2, 8 x 16), 28.8 to 11.2 ms (GGX, 1 M triangles, 2048^2, 4 x 4).
// Measured and not kept: lanes strided over the tile instead of blocks (fewer atomic conflicts, +7 %),
// 8 or 12 warps per CTA (+8 to +30 %), two lit CTAs of 8 warps per SM (+10 %).
#include <cuda_runtime.h>

#define SGE_FILE_ID 4  // range-check sites of this file (checked build)
#include "sge_device.cuh"

namespace sge {

namespace {

constexpr int NB = kLightBin;
constexpr int CMAX = 16 * kCandWords;  // candidates kept per pixel (a pixel with more tests every live triangle)
constexpr int GMAX = 8;   // pairs of one group: set up together, one barrier before and after their pixels

// Sum of v over the run of consecutive lanes (in lane order) that share key k, for the run's
// last lane; every lane of the warp calls it.  Returns whether the lane ends its run and sets n
// to the run's length.
__device__ __forceinline__ bool run_sum(int k, float& v, int& n) {
  const int lane = threadIdx.x & 31;
  const int kp = __shfl_up_sync(0xffffffffu, k, 1);
  const int kn = __shfl_down_sync(0xffffffffu, k, 1);
  const unsigned heads = __ballot_sync(0xffffffffu, lane == 0 || kp != k);
  const int start = 31 - __clz(heads & (0xffffffffu >> (31 - lane)));
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const float o = __shfl_up_sync(0xffffffffu, v, d);
    if (lane - d >= start) v += o;
  }
  n = lane - start + 1;
  return lane == 31 || kn != k;
}

// A bin triangle's unperturbed edge functions for the pruning pass, with its margin; 64 bytes.
// small (over the tile, offsets 0..15 * 256, every test value fits 32 bits: |a|, |b| < 2^16, |e0| < 2^29,
// margin < 2^10): es[k] = E_k - reach_k - 1 and em[k] = E_k + margin (|a_k| + |b_k|) at the tile's
// first pixel centre, so that a pixel is surely / maybe inside where all three are >= 0 there.
struct __align__(16) TriS {
  union {
    long long e0[3];  // (not small) oriented edge functions at the tile's first pixel centre
    struct {
      int es[3], em[3];
    };
  };
  int a[3], b[3];  // oriented edge steps per fixed-point unit in x and y
  int tri;         // triangle id; -2: not drawable unperturbed, so always a candidate
  int margin;      // perturbation margin, fixed-point units
  int small;
  int pad;
};

// How far (edge-function units) a pixel must lie inside an edge with steps a, b to stay inside under every
// perturbation: each vertex moves at most margin per axis, so at most sqrt(2) margin (+ slack).
__device__ __forceinline__ long long sure_reach(int a, int b, int margin) {
  const float fa = (float)a, fb = (float)b;
  return (long long)ceilf(1.41422f * (float)margin * sqrtf(fa * fa + fb * fb) * 1.0001f + 2.0f);
}

// ---------------------------------------------------------------- bin pruning
// Unperturbed set-up of a bin triangle from its record (k_bin.cu) with its perturbation margin; a triangle
// not drawable unperturbed (zero area, a vertex behind the near limit) gets tri = -2: a perturbed version
// may still be drawable, so it is a candidate everywhere.  span: the pixels that may pass surely_covers
// (inside the triangle) and maybe_covers (inside its edges pushed out by the margin terms); a triangle
// those tests always fail / pass: none / all.
__device__ __forceinline__ void stage_unperturbed(const int4& r0, const int4& r1, int tri, int rx, int ry, TriS& d,
                                                  uint32_t (&span)[2]) {
  const bool ok = r1.w != 0;
  const PVert v[3] = {PVert{r0.x, r0.y, 0.f, 0.f, ok}, PVert{r0.z, r0.w, 0.f, 0.f, ok}, PVert{r1.x, r1.y, 0.f, 0.f, ok}};
  SideTri t;
  set_up_side(t, v, rx, ry);
  const bool drawable = !(t.e.x == -1 && t.e.z == 0 && t.e.w == 0);
  d.tri = drawable ? tri : -2;
  d.margin = r1.z;
  const bool can = drawable && d.margin != 0x7FFFFFFF;
  span[0] = 0u;
  span[1] = 0xFFFFFFFFu;
  d.small = 0;
  if (!can) return;
  span[1] = box_span(v, rx, ry, d.margin);
  long long e[3];
  if (!(t.e.w & kBig)) {
    e[0] = t.e.x, e[1] = t.e.y, e[2] = t.e.z - t.e.x - t.e.y;
    d.a[0] = t.ab.x, d.a[1] = t.ab.y, d.a[2] = -t.ab.x - t.ab.y;
    d.b[0] = t.ab.z, d.b[1] = t.ab.w, d.b[2] = -t.ab.z - t.ab.w;
    d.small = d.margin < (1 << 10);
  } else {
    Tri g;
    setup_tri(v[0], v[1], v[2], rx, ry, g);
#pragma unroll
    for (int k = 0; k < 3; ++k) e[k] = g.e0[k], d.a[k] = g.a[k], d.b[k] = g.b[k];
  }
  // a pixel inside all three edges by their reach has E_0 + E_1 + E_2 = area above the reaches' sum:
  // triangles no wider than the perturbation moves them surely cover nothing
  long long reach[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) reach[k] = sure_reach(d.a[k], d.b[k], d.margin);
  if (e[0] + e[1] + e[2] > reach[0] + reach[1] + reach[2]) span[0] = box_span(v, rx, ry, 0);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    if (d.small) {
      // (reach and the margin terms stay below 2^28 here, so both fit)
      d.es[k] = (int)(e[k] - reach[k] - 1);
      d.em[k] = (int)e[k] + d.margin * (abs(d.a[k]) + abs(d.b[k]));
    }
  }
  if (!d.small) {
#pragma unroll
    for (int k = 0; k < 3; ++k) d.e0[k] = e[k];
  }
}

// Not small: does every perturbed version of t cover pixel (dx, dy)?  (t drawable, its margin bounded.)
__device__ __forceinline__ bool surely_covers(const TriS& t, int dx, int dy) {
  bool sure = true;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const long long e = t.e0[k] + (long long)t.a[k] * (dx * 256) + (long long)t.b[k] * (dy * 256);
    sure = sure && e > sure_reach(t.a[k], t.b[k], t.margin);
  }
  return sure;
}

// Not small: may some perturbed version of t cover pixel (dx, dy)?  (t drawable, its margin bounded.)
__device__ __forceinline__ bool maybe_covers(const TriS& t, int dx, int dy) {
  bool maybe = true;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const long long e = t.e0[k] + (long long)t.a[k] * (dx * 256) + (long long)t.b[k] * (dy * 256);
    maybe = maybe && (e + (long long)t.margin * (long long)(abs(t.a[k]) + abs(t.b[k])) >= 0);
  }
  return maybe;
}

struct PruneSmem {
  TriS t[NB];
  float2 zr[NB];
  uint32_t id[NB];
  uint32_t key[NB];      // ordered bits of the smallest depths, by bin position
  uint32_t span[NB][2];  // the pixels of the sure-cover and the maybe-visible tests
  uint32_t zsure[TILE_PX];         // ordered bits of the nearest far end of a surely covering triangle
  uint32_t mask[NB / 32][TILE_PX]; // each pixel's candidates among the staged triangles
  uint8_t live[NB];
  uint8_t remap[NB];     // compacted position of each live entry of a single-chunk bin
  int wsum[TILE_PX / 32];
};

// Exclusive prefix of flag over the CTA (256 threads); returns this thread's position and
// the total in *total.
__device__ __forceinline__ int block_prefix(int flag, int* wsum, int* total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const unsigned b = __ballot_sync(0xffffffffu, flag);
  const int in_warp = __popc(b & ((1u << lane) - 1u));
  __syncthreads();
  if (lane == 0) wsum[wid] = __popc(b);
  __syncthreads();
  int before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < TILE_PX / 32; ++w) {
    before += w < wid ? wsum[w] : 0;
    all += wsum[w];
  }
  *total = all;
  return before + in_warp;
}

// The staged triangles j < cnt go into the pixels they reach, inside columns <= cmax and rows <= rmax.
// kMark = 0: the nearest far end of a triangle that surely covers each pixel; 1: the candidates that may be
// visible, not wholly behind that (a triangle whose perturbed versions are not bounded is one everywhere).
// kStep threads take the rows of one triangle's box in turn; a warp's lanes meet again after each triangle (left
// to themselves they ran its loops one after another: 2.0 G instead of 1.3 G warp instructions at 1 M triangles).
template <int kMark, int kStep>
__device__ __forceinline__ void for_rows(PruneSmem& sm, int cnt, int cmax, int rmax) {
  for (int u0 = threadIdx.x & ~31; u0 < cnt * kStep; u0 += TILE_PX) {
    const int u = u0 + (threadIdx.x & 31), j = u / kStep;
    const uint32_t s = u < cnt * kStep ? sm.span[j][kMark] : 0u;
    // (columns and rows are both empty or both not)
    const int r0 = __ffs((int)(s >> 16)) - 1 + u % kStep, r1 = min(15 - __clz((int)s), rmax);
    if (s && r0 <= r1) {
      const int c0 = __ffs((int)s) - 1, c1 = min(31 - __clz((int)(s & 0xFFFFu)), cmax);
      const TriS& t = sm.t[j];
      const float z = kMark ? sm.zr[j].x : sm.zr[j].y;
      const uint32_t bit = 1u << (j & 31);
      uint32_t* mask = sm.mask[j >> 5];
      if (t.small) {
        const uint32_t zb = kMark || z == z ? ordered_bits(z) : 0xFFFFFFFFu;
        const int* e = kMark ? t.em : t.es;
        const int a0 = t.a[0] * 256, a1 = t.a[1] * 256, a2 = t.a[2] * 256, b0 = t.b[0] * 256, b1 = t.b[1] * 256, b2 = t.b[2] * 256;
        bool live = false;
        for (int row = r0; row <= r1; row += kStep) {
          int e0 = e[0] + a0 * c0 + b0 * row, e1 = e[1] + a1 * c0 + b1 * row, e2 = e[2] + a2 * c0 + b2 * row;
          for (int p = row * TILE + c0; p <= row * TILE + c1; ++p, e0 += a0, e1 += a1, e2 += a2) {
            if (min(min(e0, e1), e2) < 0) continue;
            if (!kMark) {
              atomicMin(&sm.zsure[p], zb);
            } else if (zb <= sm.zsure[p]) {
              live = true;
              atomicOr(mask + p, bit);
            }
          }
        }
        if (live) sm.live[j] = 1;
      } else {
        const bool all = t.tri == -2 || t.margin == 0x7FFFFFFF;
        for (int row = r0; row <= r1; row += kStep)
          for (int c = c0; c <= c1; ++c) {
            const int p = row * TILE + c;
            if (!kMark) {
              if (z == z && surely_covers(t, c, row)) atomicMin(&sm.zsure[p], ordered_bits(z));
            } else if (all || (maybe_covers(t, c, row) && ordered_bits(z) <= sm.zsure[p])) {
              sm.live[j] = 1;
              atomicOr(mask + p, bit);
            }
          }
      }
    }
    __syncwarp();
  }
}

// Per (view slot, tile): drop from the bin every triangle that no perturbation of the call can
// make visible at any pixel of the tile (outside all margin-widened pixel tests, or behind a
// triangle that surely covers the pixel), compact the rest to the front of the bin's range,
// record their number in tile_live and list the tile as a light item (<= light_bin live
// triangles) or a heavy one, and store each pixel's candidate triangles of a light one in cand/ncand
// (up to CMAX live indices).  The pruned triangles never change any render of the call in this tile.
//
// A light tile's live triangles are in ascending order of their smallest depth under any
// perturbation (ordered bits, a total order with NaN; ties by bin position), so each pixel's list
// is: the estimator stops at the first candidate wholly behind the nearest covering one found.
// Bound by instruction issue.  The bin is ranked once per tile (a comparison per pair of triangles)
// instead of every pixel sorting its list; the triangles go by rows into the pixels of their boxes instead of
// every pixel testing every triangle, a pixel's candidates are the bits of a mask, which come out in
// rank order, and the projected vertices come from the binning.  Before any of this / now: 29.4 / 21.1 us (2,048
// triangles, 256^2, one view), 260 / 135 us (8,192 triangles, 512^2, 8 views), 9,955 / 1,965 us (1 M
// triangles, 2048^2, 4 views).
template <int kStep>
__device__ __forceinline__ void prune_tile(const SceneDev& S, const Workspace& ws, int n_views, int slot, int tile,
                                           int light_bin, PruneSmem& sm) {
  const int tid = threadIdx.x;
  const int ntl = n_tiles(S), n_all = n_views * ntl;
  if (*bin_total(ws) > (unsigned long long)ws.bin_capacity) return;  // overflow: the bins were not stored
  const uint32_t beg = ws.tile_off[slot * ntl + tile];
  const int nb = (int)ws.tile_count[slot * ntl + tile];
  if (nb == 0) return;
  const int tx = tile % S.tiles_x, ty = tile / S.tiles_x;
  const int cmax = min(TILE, S.W - tx * TILE) - 1, rmax = min(TILE, S.H - ty * TILE) - 1;
  const int rx = 256 * (tx * TILE) + 128, ry = 256 * (ty * TILE) + 128;
  const long long tix = (long long)slot * ntl + tile;
  sm.zsure[tid] = ordered_bits(3.4e38f);
  // a chunk of the bin set up; ranked: in ascending order of the smallest depths
  auto stage = [&](int c0, int cnt, bool ranked) {
    int tri = 0, at = tid;
    float2 zr = make_float2(0.f, 0.f);
    int4 r0, r1;
    if (tid < cnt) {
      tri = (int)bin_at(S, ws, beg + c0 + tid);
      const long long i = (long long)slot * S.nt + tri;
      zr = ws.tri_z[i];
      r0 = ws.tri_rec[2 * i];
      r1 = ws.tri_rec[2 * i + 1];
      sm.key[tid] = ordered_bits(zr.x);
    }
#pragma unroll
    for (int w = 0; w < NB / 32; ++w) sm.mask[w][tid] = 0u;
    __syncthreads();
    if (tid < cnt) {
      if (ranked) {
        // ties by bin position: entries of the warps before count when equal too, of the warps behind not
        const uint32_t k = sm.key[tid];
        const int w0 = tid & ~31, w1 = min(w0 + 32, cnt);
        at = 0;
#pragma unroll 8
        for (int j = 0; j < w0; ++j) at += sm.key[j] <= k ? 1 : 0;
#pragma unroll 8
        for (int j = w0; j < w1; ++j) at += sm.key[j] < k || (sm.key[j] == k && j < tid) ? 1 : 0;
#pragma unroll 8
        for (int j = w1; j < cnt; ++j) at += sm.key[j] < k ? 1 : 0;
      }
      sm.id[at] = (uint32_t)tri;
      sm.zr[at] = zr;
      sm.live[at] = 0;
      stage_unperturbed(r0, r1, tri, rx, ry, sm.t[at], sm.span[at]);
    }
    __syncthreads();
  };
  // mark the staged triangles some pixel may see, and each pixel's
  auto mark = [&](int cnt) {
    for_rows<1, kStep>(sm, cnt, cmax, rmax);
    __syncthreads();
  };
  const bool single = nb <= NB;
  // pass 1: nearest far end of the triangles that surely cover each pixel
  for (int c0 = 0; c0 < nb; c0 += NB) {
    const int cnt = min(NB, nb - c0);
    __syncthreads();
    stage(c0, cnt, single);
    for_rows<0, kStep>(sm, cnt, cmax, rmax);
  }
  // pass 2: mark and compact the triangles some pixel may see (a single chunk is still staged)
  int n_live = 0;
  for (int c0 = 0; c0 < nb; c0 += NB) {
    const int cnt = min(NB, nb - c0);
    __syncthreads();
    if (!single) stage(c0, cnt, false);
    mark(cnt);
    const int f = tid < cnt ? sm.live[tid] : 0;
    int total;
    const int pos = block_prefix(f, sm.wsum, &total);
    // positions only move towards the front, past entries this CTA has already read
    if (f) {
      if (CHK(S, (long long)beg + n_live + pos, S.chk.bins)) ws.bins[beg + n_live + pos] = sm.id[tid];
      if (single) sm.remap[tid] = (uint8_t)pos;
    }
    n_live += total;
  }
  if (tid == 0) {
    ws.tile_live[tix] = (uint32_t)n_live;
    const uint32_t it = ((uint32_t)slot << 24) | (uint32_t)tile;
    if (n_live <= min(light_bin, kBigBin)) ws.items[atomicAdd(ws.counters + 0, 1u)] = it;
    else if (n_live <= light_bin) ws.tile_cur[atomicAdd(ws.counters + 6, 1u)] = it;
    else ws.items[n_all - 1 - (int)atomicAdd(ws.counters + 4, 1u)] = it;
  }
  if (n_live > light_bin) return;  // (the dense estimator takes no lists)
  if (!single && n_live > 0) {
    // pass 3 (bins of more than one chunk): the live triangles are one chunk, ranked by depth here and
    // stored back in that order, and each pixel's candidates are found among them
    __syncthreads();
    stage(0, n_live, true);
    if (tid < n_live) {
      sm.remap[tid] = (uint8_t)tid;
      if (CHK(S, (long long)beg + tid, S.chk.bins)) ws.bins[beg + tid] = sm.id[tid];
    }
    mark(n_live);
  } else {
    __syncthreads();
  }
  // this pixel's list: the live indices of its mask's bits, in rank order, the first CMAX of them
  static_assert(CMAX == 16 * kCandWords, "sixteen indices to an int4 word");
  int n = 0;
  uint32_t word[4] = {0u, 0u, 0u, 0u};
  int4* out = ws.cand + tix * kCandWords * TILE_PX + tid;
#pragma unroll 1
  for (int w = 0; w < NB / 32 && w * 32 < nb; ++w)
    for (uint32_t m = sm.mask[w][tid]; m; m &= m - 1) {
      if (n < CMAX) {
        const uint32_t bits = (uint32_t)sm.remap[w * 32 + __ffs((int)m) - 1] << (8 * (n & 3));
        const int i = (n >> 2) & 3;
#pragma unroll
        for (int x = 0; x < 4; ++x) word[x] |= x == i ? bits : 0u;
        if ((n & 15) == 15) {
          out[(n >> 4) * TILE_PX] = make_int4((int)word[0], (int)word[1], (int)word[2], (int)word[3]);
          word[0] = word[1] = word[2] = word[3] = 0u;
        }
      }
      ++n;
    }
  if (n < CMAX && (n & 15)) out[(n >> 4) * TILE_PX] = make_int4((int)word[0], (int)word[1], (int)word[2], (int)word[3]);
  ws.ncand[tix * TILE_PX + tid] = (uint8_t)min(n, 255);
}

template <int kStep, int kCtas>
__global__ void __launch_bounds__(TILE_PX, kCtas) k_bin_prune(SceneDev S, Workspace ws, ViewList vl) {
  __shared__ PruneSmem sm;
  prune_tile<kStep>(S, ws, vl.n, blockIdx.y, blockIdx.x, ws.light_bin, sm);
}

// Batched form: every (tile, view slot, asset) of a batched call in one launch; each CTA reads
// its asset's scene and workspace from the asset's launch descriptor in device memory.
template <int kStep, int kCtas>
__global__ void __launch_bounds__(TILE_PX, kCtas) k_bin_prune_batch(const BatchArgs P) {
  __shared__ PruneSmem sm;
  const BatchAsset& A = P.as[blockIdx.z];
  const int slot = blockIdx.y;
  if (slot >= A.n_views) return;
  const AssetDesc& D = *A.desc;
  if ((int)blockIdx.x >= D.S.tiles_x * D.S.tiles_y) return;
  prune_tile<kStep>(D.S, D.ws, A.n_views, slot, blockIdx.x, P.light_bin, sm);
}

// ---------------------------------------------------------------- the estimator
// Sizes of one model's kernel.  GR: the read textures share one size, so every pixel's bilinear
// footprint is the same texels in all of them, and one window slot carries all their channels.
template <int SH, bool GR = false>
struct Model {
  static constexpr int NREAD = SH == SHADE_UNLIT ? 1 : (SH == SHADE_LAMBERT ? 2 : 4);
  // footprints (and texel windows) per side: one for a group, one per texture otherwise
  static constexpr int NFOOT = GR ? 1 : NREAD;
  static constexpr bool LIT = SH != SHADE_UNLIT;
  static constexpr int WARPS = 16;     // warps of a CTA
  static constexpr int CTAS = LIT ? 1 : 2;        // resident CTAs per SM
  static constexpr int THREADS = 32 * WARPS;
  static constexpr int SLOTS = LIT ? 2 * NB : NB; // (pair, live triangle) set-ups staged per side
  static constexpr int WCAP = LIT ? 1024 : 768;   // texel slots of all windows together
  static constexpr int ACAP = LIT ? 8192 : 7168;  // (pair, cell or texel) sums
  static constexpr int NV = GR ? 2 : 1;           // float4s of texel values per slot
  static constexpr int SPP = GR ? 4 * NREAD : 4;  // sign bits per slot and pair
  static constexpr int GPW = 32 / SPP;            // pairs per sign word
  static constexpr int NW = GMAX / GPW;           // sign words per slot
  // the sign words use the float4s' free components (unlit and ungrouped textures: w of the first;
  // grouped Lambert: z, w of the second); grouped GGX has none free
  static constexpr bool SIGNS_APART = GR && SH == SHADE_GGX;
};
constexpr int kHashNoWindow = 512, kHashWindow = 128;  // hashed footprints of an item without / with a window
constexpr int kHashProbe = 8;
constexpr int kDenseTri = NB * 11 / 4;

template <int SH, bool GR>
struct FastSmem {
  using M = Model<SH, GR>;
  SideTri side[2][M::SLOTS];      // slot g nb + j: triangle j of the group's pair g
  float4 th[M::NV][M::WCAP];      // unperturbed texel values the shading reads (zero: absent channels)
  int4 cand[TILE_PX];             // each pixel's candidates (8-bit live indices), by block and lane
  uint32_t ts[M::SIGNS_APART ? M::NW : 1][M::SIGNS_APART ? M::WCAP : 1];  // the group's sign bits
  uint32_t tcnt[M::WCAP];         // item counts: low half the slot's cell, high half the texel alone
  float tA[M::ACAP];              // the group's sums, per pair: window cells, hashed cells, window texels
  uint32_t hkey[kHashNoWindow];   // hashed footprints (credit codes) and their item counts
  uint32_t hcnt[kHashNoWindow];
  float frame[M::LIT ? 2 : 1][M::LIT ? M::SLOTS : 1][6];  // lit: the set-up's face normal and u tangent
  float tgt[3][TILE_PX];          // target colours, by block and lane
  union {
    struct {
      float uv[NB][6];
      int vid[NB][3];
      int btri[NB];               // triangle id of each live entry
      uint32_t zminb[NB];         // ordered bits of its smallest depth under any perturbation of the call
    };
    int4 dense[kDenseTri];        // (dense_items) vertices and id of the first live triangles
  };
  uint32_t sgn9[2][M::SLOTS];     // bit 3k+c: coordinate c of corner k has s = -1 (by group parity)
  float A_tri[M::SLOTS];          // f+ - f- of the pixels that see the triangle (side +, else side -)
  uint32_t n_tri[M::SLOTS];
  float A_cor[M::SLOTS][3];       // and of the pixels that add single corners of it
  uint32_t n_cor[M::SLOTS];       // their counts, 10 bits per corner (at most 256 pixels)
  int4 win[M::NFOOT];             // texel windows: first column (before wrapping), first row, width, height
  int wbase[M::NFOOT + 1];        // first slot of each window; the total
  double loss[SGE_MAX_VIEWS_PER_CALL];  // this CTA's image error per view slot, added to the global one at the end
  float red[M::WARPS];
  uint32_t item, unit;            // work counters: the kernel's item, the group's next (block, pair)
  uint32_t act[TILE_PX / 32], nact;  // blocks of the tile with a candidate at some pixel
  uint8_t ncand[TILE_PX];
};

static_assert(2 * (sizeof(FastSmem<SHADE_UNLIT, false>) + 1024) <= 228 * 1024, "two unlit CTAs must fit an SM");
static_assert(sizeof(FastSmem<SHADE_GGX, true>) + sizeof(BatchSmem) <= 227 * 1024, "lit");
static_assert(sizeof(FastSmem<SHADE_GGX, false>) + sizeof(BatchSmem) <= 227 * 1024, "lit");

// The perturbed positions of live triangle j's corners (sign bits sg; side - already inverted).
__device__ __forceinline__ void corner_positions(const SceneDev& S, const int* vid, uint32_t sg, float3 p[3]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float* src = S.pos + 3ll * vid[k];
    float q[3];
#pragma unroll
    for (int c = 0; c < 3; ++c)
      q[c] = __fadd_rn(__ldg(src + c), ((sg >> (3 * k + c)) & 1) ? -S.eps_pos : S.eps_pos);
    p[k] = f3(q[0], q[1], q[2]);
  }
}

// Sign-flip mask of bit b of a word whose wanted bit sits `up` places below bit 31.
__device__ __forceinline__ float signed_eps(uint32_t word, int up, float eps) {
  return __uint_as_float(((word << up) & 0x80000000u) ^ __float_as_uint(eps));
}

// Channels of a read texture the shading uses (albedo, normal: 3; roughness, metallic: 1).
__device__ __forceinline__ constexpr int used_channels(int r) { return r < 2 ? 3 : 1; }

// Texel id of window slot t.
__device__ __forceinline__ int window_texel(const int4& win, int t, int w) {
  const int row = t / win.z;
  return (win.y + row) * w + wrap_i(win.x + t - row * win.z, w);
}

// Credit code of a pixel's side in footprint r: the window cell (the slot of the footprint's first
// texel), or with kOut a footprint code (Quad) and r above it.  In the hash a code without kOut is one texel.
constexpr uint32_t kOut = 1u << 31, EMPTY = 0xFFFFFFFFu;
constexpr int kFootShift = 29;

// Sign bits of texel t's channels (bit c: s = -1) in one texture's sign plane of an estimate.
__device__ __forceinline__ uint32_t plane_nibble(const SceneDev& S, const uint32_t* planes, int off, int t) {
  const long long w = (long long)off + (t >> 3);
  if (!CHK(S, w, S.chk.sign_words)) return 0u;
  return (__ldg(planes + w) >> (4 * (t & 7))) & 0xFu;
}

// Hashed slot of an outside code (inserted if new), or -1: no room near its place.
__device__ __forceinline__ int hash_slot(uint32_t* hkey, uint32_t code, int size) {
  uint32_t h = code ^ (code >> 16);
  h *= 0x7feb352du;
  h ^= h >> 15;
#pragma unroll 1
  for (int p = 0; p < kHashProbe; ++p, ++h) {
    const int slot = (int)(h & (uint32_t)(size - 1));
    uint32_t k = *(volatile uint32_t*)&hkey[slot];
    if (k == EMPTY) {
      k = atomicCAS(&hkey[slot], EMPTY, code);
      if (k == EMPTY) return slot;
    }
    if (k == code) return slot;
  }
  return -1;
}

// The sign bits of window slot s for pair g of the group, from bit 28 - SPP (g mod GPW) + ... on:
// the word that holds them.
template <int SH, bool GR>
__device__ __forceinline__ uint32_t sign_word_of(const FastSmem<SH, GR>& sm, int s, int g) {
  using M = Model<SH, GR>;
  if constexpr (M::SIGNS_APART) return sm.ts[g / M::GPW][s];
  else if constexpr (!GR) return __float_as_uint(sm.th[0][s].w);
  else return __float_as_uint(g < M::GPW ? sm.th[1][s].z : sm.th[1][s].w);
}

// After a group's pixels: fold its sums with its pairs' signs into the global sums.  A pixel credits the
// 2 x 2 texels of a footprint with one sum in the footprint's cell, so a texel's sum is that of the
// four cells around it plus what was credited to it alone.  (The cells are cleared by clear_cells.)
template <int SH, bool GR>
__device__ __forceinline__ void fold(const SceneDev& S, const Workspace& ws, const EstimateArgs& a,
                                     FastSmem<SH, GR>& sm, int nb, int G, int par, int nh, const uint32_t* planes) {
  using M = Model<SH, GR>;
  constexpr int NC = GR ? 4 * M::NREAD : 4;
  const int n_all = sm.wbase[M::NFOOT], stride = 2 * n_all + nh;
  for (int r = 0; r < M::NFOOT; ++r) {
    const int base = sm.wbase[r], n = sm.wbase[r + 1] - base;
    const int4 win = sm.win[r];
    for (int t = threadIdx.x; t < n; t += M::THREADS) {
      float acc[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c) acc[c] = 0.0f;
      bool any = false;
      float* cell = sm.tA + base + t;
      for (int g = 0; g < G; ++g, cell += stride) {
        // (no footprint starts in a window's last column: left of a row's first texel lies a zero)
        float A = cell[0] + cell[n_all + nh];
        if (t > 0) A += cell[-1];
        if (t >= win.z) A += cell[-win.z];
        if (t > win.z) A += cell[-win.z - 1];
        if (A == 0.0f) continue;
        any = true;
        const uint32_t sb = sign_word_of<SH, GR>(sm, base + t, g) >> (M::SPP * (g % M::GPW));
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[c] += ((sb >> c) & 1) ? -A : A;
      }
      if (!any) continue;
      const int texel = window_texel(win, t, S.rtex[r].w);
#pragma unroll
      for (int q = 0; q < (GR ? M::NREAD : 1); ++q) {
        const TexDev& T = S.rtex[GR ? q : r];
        const long long p = T.offset + (long long)texel * T.c;
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (c < T.c && CHK(S, p + c, S.chk.params)) atomicAdd(a.grad + p + c, acc[4 * q + c]);
      }
    }
  }
  // hashed footprints: their texels, whose sign words are fetched together (one after another a window-less item's fold took
  // 8 us on average, and 15 us in the fullest tile of a 256^2 call; soup of 10,240 triangles, one pair 150 -> 143 us)
  for (int h = threadIdx.x; h < nh; h += M::THREADS) {
    const uint32_t code = sm.hkey[h];
    if (code == EMPTY) continue;
    const int r = GR ? 0 : (int)((code >> kFootShift) & 3u);
    const int tw = S.rtex[r].w;
    const Quad Q(code, tw);
    const int nq = S.foot_nearest || (!M::LIT && !(code & kOut)) ? 1 : 4;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (q >= nq || Q.repeats(q)) continue;
      const int texel = Q.texel(q, tw);
#pragma unroll 1
      for (int k = 0; k < (GR ? M::NREAD : 1); ++k) {
        const TexDev& T = S.rtex[GR ? k : r];
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        for (int g = 0; g < G; ++g) {
          const float A = sm.tA[g * stride + n_all + h];
          if (A == 0.0f) continue;
          const uint32_t sb = plane_nibble(S, planes + g * ws.sgn_words, ws.sgn_off[T.index], texel);
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[c] += ((sb >> c) & 1) ? -A : A;
        }
        const long long p = T.offset + (long long)texel * T.c;
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (c < T.c && CHK(S, p + c, S.chk.params)) atomicAdd(a.grad + p + c, acc[c]);
      }
    }
  }
  const int j = threadIdx.x;
  if (j < nb) {
    float acc[9] = {};
    uint32_t cnt[3] = {};
    for (int g = 0; g < G; ++g) {
      const int s = g * nb + j;
      const uint32_t nt = sm.n_tri[s], nc = sm.n_cor[s];
      if ((nt | nc) == 0u) continue;
      const float at = sm.A_tri[s];
      const uint32_t sg = sm.sgn9[par][s];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float v = at + sm.A_cor[s][k];
        cnt[k] += nt + ((nc >> (10 * k)) & 1023u);
#pragma unroll
        for (int c = 0; c < 3; ++c) acc[3 * k + c] += ((sg >> (3 * k + c)) & 1) ? -v : v;
        sm.A_cor[s][k] = 0.0f;
      }
      sm.A_tri[s] = 0.0f;
      sm.n_tri[s] = 0u;
      sm.n_cor[s] = 0u;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      if (!cnt[k]) continue;
      const long long p = 3ll * sm.vid[j][k];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        if (!CHK(S, p + c, S.chk.params)) continue;
        atomicAdd(a.grad + p + c, acc[3 * k + c]);
        atomicAdd(a.counts + p + c, cnt[k]);
      }
    }
  }
}

// The sums of G pairs back to zero (after every thread has folded).
template <int SH, bool GR>
__device__ __forceinline__ void clear_sums(FastSmem<SH, GR>& sm, int G, int nh) {
  using M = Model<SH, GR>;
  const int n = G * (2 * sm.wbase[M::NFOOT] + nh);
  for (int i = threadIdx.x; i < n; i += M::THREADS) sm.tA[i] = 0.0f;
}

// The item's texel counts into the global counts (its counters are cleared after a barrier).
template <int SH, bool GR>
__device__ __forceinline__ void flush_counts(const SceneDev& S, const EstimateArgs& a, FastSmem<SH, GR>& sm, int nh) {
  using M = Model<SH, GR>;
  for (int r = 0; r < M::NFOOT; ++r) {
    const int base = sm.wbase[r], n = sm.wbase[r + 1] - base;
    const int4 win = sm.win[r];
    for (int t = threadIdx.x; t < n; t += M::THREADS) {
      const uint32_t* cnt = sm.tcnt + base + t;
      uint32_t c = (cnt[0] >> 16) + (cnt[0] & 0xFFFFu);
      if (t > 0) c += cnt[-1] & 0xFFFFu;
      if (t >= win.z) c += cnt[-win.z] & 0xFFFFu;
      if (t > win.z) c += cnt[-win.z - 1] & 0xFFFFu;
      if (c == 0u) continue;
      const int texel = window_texel(win, t, S.rtex[r].w);
#pragma unroll
      for (int q = 0; q < (GR ? M::NREAD : 1); ++q) {
        const TexDev& T = S.rtex[GR ? q : r];
        const long long p = T.offset + (long long)texel * T.c;
        for (int k = 0; k < T.c; ++k)
          if (CHK(S, p + k, S.chk.params)) atomicAdd(a.counts + p + k, c);
      }
    }
  }
  for (int h = threadIdx.x; h < nh; h += M::THREADS) {
    const uint32_t code = sm.hkey[h], c = sm.hcnt[h];
    if (code == EMPTY) continue;
    sm.hkey[h] = EMPTY;
    sm.hcnt[h] = 0u;
    const int r = GR ? 0 : (int)((code >> kFootShift) & 3u);
    const int tw = S.rtex[r].w;
    const Quad Q(code, tw);
    const int nq = S.foot_nearest || (!M::LIT && !(code & kOut)) ? 1 : 4;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (q >= nq || Q.repeats(q)) continue;
      const int texel = Q.texel(q, tw);
#pragma unroll 1
      for (int k = 0; k < (GR ? M::NREAD : 1); ++k) {
        const TexDev& T = S.rtex[GR ? k : r];
        const long long p = T.offset + (long long)texel * T.c;
        for (int i = 0; i < T.c; ++i)
          if (CHK(S, p + i, S.chk.params)) atomicAdd(a.counts + p + i, c);
      }
    }
  }
}

// The windows' sign bits of the group's G pairs (planes: the first one's).
template <int SH, bool GR>
__device__ __forceinline__ void load_signs(const SceneDev& S, const Workspace& ws, FastSmem<SH, GR>& sm,
                                           const uint32_t* planes, int G) {
  using M = Model<SH, GR>;
  constexpr int NG = GR ? M::NREAD : 1;
  for (int r = 0; r < M::NFOOT; ++r) {
    const int base = sm.wbase[r], n = sm.wbase[r + 1] - base;
    const int4 win = sm.win[r];
    for (int t = threadIdx.x; t < n; t += M::THREADS) {
      const int texel = window_texel(win, t, S.rtex[r].w), sh = 4 * (texel & 7);
      uint32_t word[M::NW];
#pragma unroll
      for (int w = 0; w < M::NW; ++w) word[w] = 0u;
#pragma unroll
      for (int q = 0; q < NG; ++q) {
        const TexDev& T = S.rtex[GR ? q : r];
        const long long wi = (long long)ws.sgn_off[T.index] + (texel >> 3);
        if (!CHK(S, wi, S.chk.sign_words)) continue;
        const uint32_t* p = planes + wi;
#pragma unroll
        for (int g = 0; g < GMAX; ++g) {
          uint32_t nib = 0;
          if (g < G) nib = (__ldg(p) >> sh) & 0xFu;
          if (T.c == 1) nib *= 7u;  // the shading reads the one channel as all three
          word[g / M::GPW] |= nib << (M::SPP * (g % M::GPW) + 4 * q);
          p += ws.sgn_words;
        }
      }
      if constexpr (M::SIGNS_APART) {
#pragma unroll
        for (int w = 0; w < M::NW; ++w) sm.ts[w][base + t] = word[w];
      } else if constexpr (!GR) {
        sm.th[0][base + t].w = __uint_as_float(word[0]);
      } else {
        sm.th[1][base + t].z = __uint_as_float(word[0]);
        sm.th[1][base + t].w = __uint_as_float(word[1]);
      }
    }
  }
}

// The windows of an item from the bounds (columns, rows) of its first pair's footprints in
// sm.win = (min column, min row, max column, max row): two texels of margin (a perturbation moves a
// footprint by a fraction of a texel), cut around the middle where it does not fit.  One thread.
template <int SH, bool GR>
__device__ __forceinline__ void make_windows(const SceneDev& S, FastSmem<SH, GR>& sm) {
  using M = Model<SH, GR>;
  int base = 0;
  for (int r = 0; r < M::NFOOT; ++r) {
    const TexDev& T = S.rtex[r];
    constexpr int cap = M::WCAP / M::NFOOT;
    const int4 b = sm.win[r];  // (min > max where no pixel has a footprint)
    int x0 = b.x - 2, y0 = max(b.y - 2, 0);
    // no texel twice (at most the texture's width): one slot per texel
    int w = b.z < b.x ? 0 : min(min(b.z - b.x, 1 << 28) + 6, T.w), h = b.z < b.x ? 0 : min(b.w + 3, T.h - 1) - y0 + 1;
    if (w >= 2 && h >= 2 && (long long)w * h > cap) {
      if (w >= h) {
        const int keep = cap / h;
        x0 += (w - keep) / 2;
        w = keep;
      } else {
        const int keep = cap / w;
        y0 += (h - keep) / 2;
        h = keep;
      }
    }
    if (w < 2 || h < 2) w = h = 0;
    sm.win[r] = make_int4(x0, y0, w, h);
    sm.wbase[r] = base;
    base += w * h;
  }
  sm.wbase[M::NFOOT] = base;
}

// The windows' unperturbed texel values.
template <int SH, bool GR>
__device__ __forceinline__ void load_window(const SceneDev& S, FastSmem<SH, GR>& sm) {
  using M = Model<SH, GR>;
  constexpr int NG = GR ? M::NREAD : 1;
#pragma unroll 1
  for (int r = 0; r < M::NFOOT; ++r) {
    const int base = sm.wbase[r], n = sm.wbase[r + 1] - base;
    const int4 win = sm.win[r];
    for (int t = threadIdx.x; t < n; t += M::THREADS) {
      const int texel = window_texel(win, t, S.rtex[r].w);
      float tv[8] = {};
#pragma unroll
      for (int k = 0; k < NG; ++k) {
        const TexDev& T = S.rtex[GR ? k : r];
        const float* src = T.ptr + (long long)texel * T.c;
#pragma unroll
        for (int c = 0; c < (GR ? used_channels(k) : 3); ++c)
          if (c < T.c || T.c == 1) tv[(GR ? (k < 2 ? 3 * k : 4 + k) : 0) + c] = __ldg(src + (T.c == 1 ? 0 : c));
      }
      sm.th[0][base + t] = make_float4(tv[0], tv[1], tv[2], tv[3]);
      if constexpr (GR) sm.th[1][base + t] = make_float4(tv[4], tv[5], tv[6], tv[7]);
    }
  }
}

// A pixel's footprints (in: it sees a triangle, at UV (u0, v0)) into the windows' bounds; whole warps.
template <int SH, bool GR>
__device__ __forceinline__ void add_bounds(const SceneDev& S, FastSmem<SH, GR>& sm, bool seen, float u0, float v0) {
#pragma unroll
  for (int r = 0; r < Model<SH, GR>::NFOOT; ++r) {
    const Foot f = footprint(u0, v0, S.rtex[r].w, S.rtex[r].h);
    const bool in = seen && abs(f.ix) < (1 << 28);
    const int x0 = __reduce_min_sync(0xffffffffu, in ? f.ix : 0x3FFFFFFF);
    const int x1 = __reduce_max_sync(0xffffffffu, in ? f.ix : -0x3FFFFFFF);
    const int y0 = __reduce_min_sync(0xffffffffu, in ? f.y0 : 0x3FFFFFFF);
    const int y1 = __reduce_max_sync(0xffffffffu, in ? f.y0 : -0x3FFFFFFF);
    if ((threadIdx.x & 31) == 0 && x0 <= x1) {
      atomicMin(&sm.win[r].x, x0);
      atomicMin(&sm.win[r].y, y0);
      atomicMax(&sm.win[r].z, x1);
      atomicMax(&sm.win[r].w, y1);
    }
  }
}

// One side of a pixel at UV (u0, v0), pair g of the group (planes: the group's first pair's): the perturbed
// texels sampled (values and signs from the window, else from memory) into val, the channels of each
// read texture the shading uses, and the side's credit codes into cr.
template <int SH, bool GR>
__device__ __forceinline__ void sample_side(const SceneDev& S, const Workspace& ws, const FastSmem<SH, GR>& sm,
                                            const uint32_t* planes, int g, int sd, float u0, float v0, int n_win,
                                            uint32_t (&cr)[Model<SH, GR>::NFOOT], float (&val)[Model<SH, GR>::NREAD][3]) {
  using M = Model<SH, GR>;
  constexpr int NREAD = M::NREAD, NFOOT = M::NFOOT, NG = GR ? NREAD : 1;
#pragma unroll
  for (int r = 0; r < NFOOT; ++r) {
    const TexDev& T = S.rtex[r];
    const int4 win = sm.win[r];
    const float x = __fsub_rn(__fmul_rn(u0, (float)T.w), 0.5f), y = __fsub_rn(__fmul_rn(v0, (float)T.h), 0.5f);
    const float xf = floorf(x), yf = floorf(y);
    const float fx = __fsub_rn(x, xf), fy = __fsub_rn(y, yf);
    const float wq[4] = {(1.0f - fx) * (1.0f - fy), fx * (1.0f - fy), (1.0f - fx) * fy, fx * fy};
    const int wx = (int)xf - win.x, wy = (int)yf - win.y;
#pragma unroll
    for (int q = 0; q < NG; ++q) val[GR ? q : r][0] = val[GR ? q : r][1] = val[GR ? q : r][2] = 0.0f;
    // (a column or row far from the window never passes, wrapped or not; no window: 0 < -1 fails)
    bool inside = (uint32_t)wx < (uint32_t)max(win.z - 1, 0) && (uint32_t)wy < (uint32_t)max(win.w - 1, 0);
    int nq = 0;  // nearest footprint: which of the four texels it is
    if (S.foot_nearest && inside) {
      const int nx = (int)floorf(__fmul_rn(u0, (float)T.w)) - (int)xf;
      const int ny = (int)floorf(__fmul_rn(v0, (float)T.h)) - (int)yf;
      inside = (uint32_t)nx < 2u && (uint32_t)ny < 2u;
      nq = nx + ny * win.z;
    }
    if (inside) {
      const int s00 = (NFOOT == 1 ? 0 : sm.wbase[r]) + wy * win.z + wx;
      cr[r] = (uint32_t)(s00 + nq);
      if (!CHK(S, s00 + win.z + 1, n_win)) continue;
      const int up = 28 - M::SPP * (g % M::GPW);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int sq = s00 + (q & 1) + (q & 2 ? win.z : 0);
        const float4 t0 = sm.th[0][sq];
        if constexpr (!GR) {
          const uint32_t sb = __float_as_uint(t0.w);
          const float e = sd ? -T.eps : T.eps;
          const float tv[3] = {t0.x, t0.y, t0.z};
#pragma unroll
          for (int c = 0; c < (M::LIT && r >= 2 ? 1 : 3); ++c)
            val[r][c] += wq[q] * __fadd_rn(tv[c], (c < T.c || T.c == 1) ? signed_eps(sb, up + 3 - c, e) : 0.0f);
        } else {
          const float4 t1 = sm.th[M::NV - 1][sq];
          const float tv[8] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w};
          uint32_t sb;
          if constexpr (M::SIGNS_APART) sb = sm.ts[g / M::GPW][sq];
          else sb = __float_as_uint(g < M::GPW ? t1.z : t1.w);
#pragma unroll
          for (int k = 0; k < NREAD; ++k) {
            const TexDev& U = S.rtex[k];
            const float e = sd ? -U.eps : U.eps;
#pragma unroll
            for (int c = 0; c < used_channels(k); ++c)
              val[k][c] += wq[q] * __fadd_rn(tv[(k < 2 ? 3 * k : 4 + k) + c],
                                             (c < U.c || U.c == 1) ? signed_eps(sb, up + 3 - c - 4 * k, e) : 0.0f);
          }
        }
      }
    } else {
      const Foot f = footprint(u0, v0, T.w, T.h);
      const uint32_t code = kOut | ((uint32_t)(GR ? 0 : r) << kFootShift) | (f.y1 == f.y0 ? kOneRow : 0u) |
                          (uint32_t)(f.y0 * T.w + f.x0);
      cr[r] = S.foot_nearest ? kOut | ((uint32_t)(GR ? 0 : r) << kFootShift) | kOneRow |
                                    (uint32_t)nearest_texel(u0, v0, T.w, T.h)
                              : code;
      int texel[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        texel[q] = (q & 2 ? f.y1 : f.y0) * T.w + (q & 1 ? f.x1 : f.x0);
        if (!CHK(S, texel[q], (long long)T.w * T.h)) texel[q] = 0;
      }
      // (a texture at a time, its four texels' loads in flight together)
#pragma unroll
      for (int k = 0; k < NG; ++k) {
        const TexDev& U = S.rtex[GR ? k : r];
        uint32_t sb[4];
        float tv[4][3];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          sb[q] = plane_nibble(S, planes + g * ws.sgn_words, ws.sgn_off[U.index], texel[q]);
          const float* src = U.ptr + (long long)texel[q] * U.c;
#pragma unroll
          for (int c = 0; c < 3; ++c) tv[q][c] = c < U.c ? __ldg(src + c) : 0.0f;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (sd) sb[q] = ~sb[q];
#pragma unroll
          for (int c = 0; c < 3; ++c)
            if (c < U.c) val[GR ? k : r][c] += wq[q] * __fadd_rn(tv[q][c], ((sb[q] >> c) & 1) ? -U.eps : U.eps);
        }
      }
#pragma unroll
      for (int k = 0; k < NG; ++k)
        if (S.rtex[GR ? k : r].c == 1) val[GR ? k : r][1] = val[GR ? k : r][2] = val[GR ? k : r][0];
    }
  }
}

// The colour of a sampled pixel: fr the triangle's frame (lit), vid its vertices, sg its 9 coordinate
// signs on this side, pw the pixel's perspective-correct weights (GGX).
template <int SH, bool GR>
__device__ __forceinline__ float3 shade_side(const SceneDev& S, int view, const float (&val)[Model<SH, GR>::NREAD][3],
                                             const float* fr, const int* vid, uint32_t sg, const PerspW& pw) {
  if constexpr (SH == SHADE_UNLIT) {
    return f3(val[0][0], val[0][1], val[0][2]);
  } else {
    float3 P = f3(0.f, 0.f, 0.f);
    float rough = 0.5f, metal = 0.0f;
    if constexpr (SH == SHADE_GGX) {
      float3 p[3];
      corner_positions(S, vid, sg, p);
      const float b[3] = {pw.q[0] / pw.qs, pw.q[1] / pw.qs, pw.q[2] / pw.qs};
      P = f3(b[0] * p[0].x + b[1] * p[1].x + b[2] * p[2].x, b[0] * p[0].y + b[1] * p[1].y + b[2] * p[2].y,
             b[0] * p[0].z + b[1] * p[1].z + b[2] * p[2].z);
      rough = val[2][0];
      metal = val[3][0];
    }
    return shade_lit<SH>(S, view, val[0], val[1], rough, metal, f3(fr[0], fr[1], fr[2]), f3(fr[3], fr[4], fr[5]), P);
  }
}

// Credit f+ - f- of a pixel of pair g to the texels of the union of both sides' footprints of every read
// texture (of the group); inA, inB: the sides that see a triangle (at least one).
template <int SH, bool GR>
__device__ __forceinline__ void credit_texels(const SceneDev& S, const Workspace& ws, const EstimateArgs& a,
                                              FastSmem<SH, GR>& sm, const uint32_t* planes, int g, int stride, int n_win,
                                              int nh, float df, bool inA, bool inB,
                                              const uint32_t (&crA)[Model<SH, GR>::NFOOT],
                                              const uint32_t (&crB)[Model<SH, GR>::NFOOT]) {
  using M = Model<SH, GR>;
  constexpr int NFOOT = M::NFOOT, NG = GR ? M::NREAD : 1;
  float* sums = sm.tA + g * stride;
#pragma unroll
  for (int r = 0; r < NFOOT; ++r) {
    const TexDev& T = S.rtex[r];
    const uint32_t A = inA ? crA[r] : crB[r], B = inB ? crB[r] : crA[r];
    // one texel by its id, straight to the global sums
    auto credit_id = [&](int id) {
#pragma unroll 1
      for (int k = 0; k < NG; ++k) {
        const TexDev& U = S.rtex[GR ? k : r];
        const uint32_t sb = plane_nibble(S, planes + g * ws.sgn_words, ws.sgn_off[U.index], id);
        const long long base = U.offset + (long long)id * U.c;
        for (int c = 0; c < U.c; ++c) {
          if (!CHK(S, base + c, S.chk.params)) continue;
          atomicAdd(a.grad + base + c, ((sb >> c) & 1) ? -df : df);
          atomicAdd(a.counts + base + c, 1u);
        }
      }
    };
    // a footprint's texels by one sum in its cell (nearest: the one texel)
    auto credit_cell = [&](uint32_t c) {
      if (!(c & kOut)) {
        if (!CHK(S, c, n_win)) return;
        atomicAdd(sums + c + (S.foot_nearest ? n_win + nh : 0), df);
        atomicAdd(sm.tcnt + c, S.foot_nearest ? 1u << 16 : 1u);
        return;
      }
      const int h = hash_slot(sm.hkey, c, nh);
      if (h >= 0) {
        atomicAdd(sums + n_win + h, df);
        atomicAdd(sm.hcnt + h, 1u);
        return;
      }
      const Quad Q(c, T.w);
#pragma unroll 1
      for (int q = 0; q < (S.foot_nearest ? 1 : 4); ++q)
        if (!Q.repeats(q)) credit_id(Q.texel(q, T.w));
    };
    credit_cell(A);
    if (B == A) continue;
    if (S.foot_nearest) {
      // one texel each: a window slot and an outside id may be the same texel
      bool dup = false;
      if ((A ^ B) & kOut) {
        const uint32_t in = (A & kOut) ? B : A, out = (A & kOut) ? A : B;
        dup = window_texel(sm.win[r], (int)in - (NFOOT == 1 ? 0 : sm.wbase[r]), T.w) == (int)(out & 0x0FFFFFFFu);
      }
      if (!dup) credit_cell(B);
      continue;
    }
    if (!((A | B) & kOut)) {
      // side -'s texels outside side +'s footprint
      const uint32_t ww = (uint32_t)sm.win[r].z;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint32_t s = B + (q & 1) + (q & 2 ? ww : 0u), d = s - A;
        if (d <= 1u || d - ww <= 1u || !CHK(S, s, n_win)) continue;
        atomicAdd(sums + n_win + nh + s, df);
        atomicAdd(sm.tcnt + s, 1u << 16);
      }
      continue;
    }
    // some side outside the window: by texel id
    auto as_id = [&](uint32_t c) {
      if (c & kOut) return c;
      return kOut | (uint32_t)window_texel(sm.win[r], (int)c - (NFOOT == 1 ? 0 : sm.wbase[r]), T.w);
    };
    const Quad QA(as_id(A), T.w), QB(as_id(B), T.w);
    uint32_t mine = 0, all = 0;  // side -'s texels (its footprint's own repeats left out), those not in side +'s
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (QB.repeats(q)) continue;
      all |= 1u << q;
      if (!QA.holds(QB, q)) mine |= 1u << q;
    }
    if (mine == all) {
      credit_cell(B);
    } else {
      // One texel each, straight to the global sums; unlit, of footprints of one row through the hash: a flat triangle's colour is a texel
      // of such a texture, footprints at its centre differ by rounding, and one that covers the image would send every pixel's
      // to the same place (64 of them, 512^2, 8 pairs: 1.60 -> 0.92 ms).  Of other footprints few pixels share a texel, and hashed it costs
      // more to find, fold and count than it saves (3 views of 413 x 311, Lambert, 5 pairs: 356 us, 413 us with all hashed).
#pragma unroll 1
      for (; mine; mine &= mine - 1) {
        const int id = QB.texel(__ffs((int)mine) - 1, T.w);
        const int h = !M::LIT && (B & kOneRow) ? hash_slot(sm.hkey, (uint32_t)id, nh) : -1;
        if (h >= 0) {
          atomicAdd(sums + n_win + h, df);
          atomicAdd(sm.hcnt + h, 1u);
        } else {
          credit_id(id);
        }
      }
    }
  }
}

// An empty start of a CTA's loop over items (every item, and the end of each asset's, leaves it empty again).
template <int SH, bool GR>
__device__ __forceinline__ void reset_smem(FastSmem<SH, GR>& sm) {
  using M = Model<SH, GR>;
  for (int s = threadIdx.x; s < M::ACAP; s += M::THREADS) sm.tA[s] = 0.0f;
  for (int s = threadIdx.x; s < M::WCAP; s += M::THREADS) sm.tcnt[s] = 0u;
  for (int s = threadIdx.x; s < kHashNoWindow; s += M::THREADS) sm.hkey[s] = EMPTY, sm.hcnt[s] = 0u;
  for (int s = threadIdx.x; s < M::SLOTS; s += M::THREADS) {
    sm.A_tri[s] = sm.A_cor[s][0] = sm.A_cor[s][1] = sm.A_cor[s][2] = 0.0f;
    sm.n_tri[s] = sm.n_cor[s] = 0u;
  }
  for (int s = threadIdx.x; s < SGE_MAX_VIEWS_PER_CALL; s += M::THREADS) sm.loss[s] = 0.0;
  if (threadIdx.x == 0) sm.nact = 0u;
  if (threadIdx.x < M::NFOOT) sm.win[threadIdx.x] = make_int4(0x3FFFFFFF, 0x3FFFFFFF, -0x3FFFFFFF, -0x3FFFFFFF);
  if (threadIdx.x <= M::NFOOT) sm.wbase[threadIdx.x] = 0;
}

// The end of an item: its loss to the CTA's sum of the view slot, its counters back to empty, the next item.
template <int SH, bool GR>
__device__ __forceinline__ void end_item(const EstimateArgs& a, FastSmem<SH, GR>& sm, int slot, float loss_acc,
                                         uint32_t next) {
  using M = Model<SH, GR>;
  const int tid = threadIdx.x;
  if (a.loss) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) loss_acc += __shfl_xor_sync(0xffffffffu, loss_acc, o);
    if ((tid & 31) == 0) sm.red[tid >> 5] = loss_acc;
  }
  __syncthreads();
  for (int s = tid; s < sm.wbase[M::NFOOT]; s += M::THREADS) sm.tcnt[s] = 0u;
  if (tid == 0) {
    if (a.loss) {
      double sum = 0.0;
      for (int i = 0; i < M::WARPS; ++i) sum += sm.red[i];
      sm.loss[slot] += sum;
    }
    sm.item = next;
    sm.nact = 0u;
  }
  __syncthreads();
  if (tid < M::NFOOT) sm.win[tid] = make_int4(0x3FFFFFFF, 0x3FFFFFFF, -0x3FFFFFFF, -0x3FFFFFFF);
  if (tid <= M::NFOOT) sm.wbase[tid] = 0;
}

template <int SH, bool GR>
__device__ __forceinline__ void add_losses(const EstimateArgs& a, FastSmem<SH, GR>& sm, int n_slots) {
  // one addition per CTA and view, however many items the call is cut into: their rounding stays below that
  // of the pixels' own sums
  if (a.loss)
    for (int s = threadIdx.x; s < n_slots; s += Model<SH, GR>::THREADS)
      if (sm.loss[s] != 0.0) {
        atomicAdd(a.loss + s, (float)(sm.loss[s] / (double)a.pairs));
        sm.loss[s] = 0.0;
      }
}

// Pairs per item: `lo` doubled up to `hi` while every CTA still gets at least 16 items (a longer run
// amortises the item's staging and texel windows, a shorter one balances the CTAs).
__device__ __forceinline__ int run_of(const EstimateArgs& a, int n_items, int lo, int hi) {
  int run = lo;
  while (2 * run <= hi && (long long)n_items * (a.pair_count / (2 * run)) >= 16ll * gridDim.x) run *= 2;
  return run;
}

// Every light work item of one scene's call, taken one at a time from the scene's work
// counter until none is left.  clean: sm is as reset_smem leaves it.  alone: no other
// scene shares the launch.  own_first: a CTA's first item is its own index, without a round trip to
// the counter (a launch's first asset, which every CTA starts at the same time).
template <int SH, bool GR>
__device__ __forceinline__ void fast_items(const SceneDev& S, const Workspace& ws, const ViewList& vl,
                                           const EstimateArgs& a, FastSmem<SH, GR>& sm, bool own_first, bool& clean,
                                           bool alone) {
  using M = Model<SH, GR>;
  constexpr int NREAD = M::NREAD, NFOOT = M::NFOOT;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // a warp's pixels: an 8 x 4 block, odd rows right to left, so that runs of lanes follow the surface
  const int lx = (lane & 8) ? 7 - (lane & 7) : (lane & 7), ly = lane >> 3;
  const int ntl = n_tiles(S);
  // Tiles with more than kBigBin live triangles go first and, unless there are many, in runs a quarter as
  // long: an item of such a tile costs up to ten times the average one, and as the last one taken it
  // would leave the other CTAs idle (4 views x 16 pairs at 501 x 397: CTAs busy 0.55 of 1.06 ms without
  // this, the kernel 0.63 ms with it; 8 views x 64 pairs at 512^2: 7.2 -> 5.9 ms with the longer runs).
  const int n_small = (int)ws.counters[0], n_big = (int)ws.counters[6];
  // No run is of one pair where the call has more: its units would be half as many as the CTA's warps, and
  // a window would be found, filled and read for it alone (8,192 triangles, 512^2, 8 views x 64 pairs, pairs_per_item = 1: 21.3 ms
  // in runs of one pair, 12.1 ms of two; a batch of 8 uneven assets 22.1 and 16.7 ms).
  const int ppi = a.pairs_per_item > 0 ? max(2, a.pairs_per_item) : kRun;
  const int run = a.pairs_per_item > 0 ? ppi : run_of(a, n_small, ppi, 4 * kRun), run_big = run_of(a, n_big, max(2, ppi / 4), ppi);
  const int chunks = (a.pair_count + run - 1) / run, chunks_big = (a.pair_count + run_big - 1) / run_big;
  const long long work_big = (long long)n_big * chunks_big, n_work = work_big + (long long)n_small * chunks;
  if (!clean) reset_smem<SH, GR>(sm);
  clean = true;
  const uint32_t first_of = own_first ? gridDim.x : 0u;
  if (tid == 0) sm.item = own_first ? blockIdx.x : atomicAdd(ws.counters + 1, 1u);
  __syncthreads();

  for (long long w = sm.item; w < n_work; w = sm.item) {
    const bool big = w < work_big;
    const int nch = big ? chunks_big : chunks, at = (int)((big ? w : w - work_big) / nch);
    const int chunk = (int)((big ? w : w - work_big) - (long long)at * nch), len = big ? run_big : run;
    const uint32_t it = big ? ws.tile_cur[at] : ws.items[at];
    const int slot = it >> 24, tile = it & 0xFFFFFF;
    uint32_t next = 0;
    if (tid == 0) next = first_of + atomicAdd(ws.counters + 1, 1u);  // (in flight while this item is staged)
    if (!CHK(S, slot, vl.n) || !CHK(S, tile, ntl)) {  // (checked build; uniform over the CTA)
      __syncthreads();
      if (tid == 0) sm.item = next;
      __syncthreads();
      continue;
    }
    const int view = vl.id[slot];
    const int tx = tile % S.tiles_x, ty = tile / S.tiles_x;
    const int rx = 256 * (tx * TILE) + 128, ry = 256 * (ty * TILE) + 128;
    const uint32_t bin_beg = ws.tile_off[slot * ntl + tile];
    const int nb = (int)ws.tile_live[slot * ntl + tile];
    const int p0 = a.pair_begin + chunk * len;
    const int p1 = min(a.pair_begin + a.pair_count, p0 + len);
    float loss_acc = 0.0f;

    // ---- per item: the bin's live triangles (pruned and compacted by k_bin_prune) and their smallest
    //      depths; the pixels' targets and candidates (in order of that depth), block by block
    for (int j = tid; j < nb; j += M::THREADS) {
      const int tri = (int)bin_at(S, ws, bin_beg + j);
      sm.btri[j] = tri;
      sm.zminb[j] = ordered_bits(ws.tri_z[(long long)slot * S.nt + tri].x);
#pragma unroll
      for (int k = 0; k < 3; ++k) sm.vid[j][k] = vert_of(S, tri, k);
      load_uvs(S, tri, sm.uv[j]);
    }
    for (int b = warp; b < TILE_PX / 32; b += M::WARPS) {
      const int dx = (b & 1) * 8 + lx, dy = (b >> 1) * 4 + ly, px = tx * TILE + dx, py = ty * TILE + dy;
      const bool valid = px < S.W && py < S.H;
      const long long tix = (long long)slot * ntl + tile;
      const int n = valid ? ws.ncand[tix * TILE_PX + dy * TILE + dx] : 0;
      float3 t = f3(0.f, 0.f, 0.f);
      if (valid) {
        const float* tp = S.targets + (((long long)view * S.H + py) * S.W + px) * 3;
        t = f3(__ldg(tp), __ldg(tp + 1), __ldg(tp + 2));
      }
      if (__any_sync(0xffffffffu, n > 0)) {
        sm.cand[b * 32 + lane] = ws.cand[tix * kCandWords * TILE_PX + dy * TILE + dx];
        sm.ncand[b * 32 + lane] = (uint8_t)n;
        sm.tgt[0][b * 32 + lane] = t.x;
        sm.tgt[1][b * 32 + lane] = t.y;
        sm.tgt[2][b * 32 + lane] = t.z;
        if (lane == 0) sm.act[atomicAdd(&sm.nact, 1u)] = (uint32_t)b;
      } else if (valid) {
        // a block no triangle can reach: the background on both sides of every pair
        const float3 bg = f3(S.bg[0], S.bg[1], S.bg[2]);
        float fp, fm;
        loss_diff(bg, bg, t, fp, fm);
        loss_acc += 0.5f * (fp + fm) * (float)(p1 - p0);
      }
    }
    __syncthreads();
    const int nact = (int)sm.nact;
    // pairs of a group: as many as the set-ups, the sign words and (below) the sums hold
    int Gcap = min(GMAX, M::SLOTS / max(nb, 1)), par = 0, G = 0, nh = 0;
    // unlit calls of one or two pairs and few items take no window: finding its bounds costs half a pair and lengthens each
    // CTA's chain, and the footprints all go through hashed cells (one 256^2 estimate: the kernel 37.0 -> 29.5 us; lit items
    // lose, 11.2 -> 20.1 ms).  With many items the pixels' own work counts, which a window makes less (whole calls,
    // 8,192 triangles, one pair a view, without / with: 512^2 1 view 145 / 147 us, 640^2 4 views 419 / 408 us, 1024^2 4 views
    // 963 / 905 us; two pairs: 512^2 1 view 202 / 200 us, 8 views 608 / 562 us; the line lies where the two meet), and so it does beside other assets
    // (!alone: batches of 4 assets of 8,192 triangles, 512^2, 2 views, one pair 907 / 782 us, two 1,096 / 887 us)
    const bool windowed = M::LIT || a.pair_count > 2 || !alone || n_work * a.pair_count > 6ll * gridDim.x;
    if (!windowed) {
      nh = kHashNoWindow;
      Gcap = min(Gcap, M::ACAP / nh);
    }
    bool first = true;
    const uint32_t* planes0 =
        ws.tsign + ((long long)slot * ws.max_pairs + (p0 - a.pair_begin)) * ws.sgn_words;  // the item's first pair's

    for (int pg = p0; pg < p1 && nact > 0; pg += G) {
      const uint32_t* planes = planes0 + (long long)(pg - p0) * ws.sgn_words;
      // ---- F: fold the previous group's sums with its signs
      if (!first) {
        fold<SH, GR>(S, ws, a, sm, nb, G, par ^ 1, nh, planes - (long long)G * ws.sgn_words);
        __syncthreads();
        clear_sums(sm, G, nh);
      }
      G = min(Gcap, p1 - pg);
      // ---- S: this group's triangles set up on both sides from the projected perturbed vertices
      for (int t2 = tid; t2 < 2 * G * nb; t2 += M::THREADS) {
        const int sd = t2 & 1, s = t2 >> 1, g = s / nb, j = s - g * nb;
        const long long vb = ((long long)slot * ws.max_pairs + (pg - a.pair_begin) + g) * S.nv;
        PVert v[3];
        uint32_t sg = 0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const long long o = vb + sm.vid[j][k];
          const int4 q = __ldg(ws.pverts + 2 * o + sd);
          v[k].X = q.x;
          v[k].Y = q.y;
          v[k].z = __int_as_float(q.z);
          v[k].iw = __int_as_float(q.w);
          v[k].ok = q.x != kNotDrawn;
          if (M::LIT || sd == 0) sg |= ((uint32_t)__ldg(ws.vbits + o) & 7u) << (3 * k);
        }
        if (sd == 0) sm.sgn9[par][s] = sg;
        set_up_side(sm.side[sd][s], v, rx, ry);
        if (M::LIT) {
          float3 p[3];
          corner_positions(S, sm.vid[j], sd ? sg ^ 0x1FFu : sg, p);
          tri_frame(p, sm.uv[j], sm.frame[sd][s]);
        }
      }
      if (!first && windowed) load_signs<SH, GR>(S, ws, sm, planes, G);
      if (tid == 0) sm.unit = 0u;
      __syncthreads();

      // ---- the group's units, a block of 32 pixels of one pair each, taken by the warps as they come
      //      free; in the item's first group side + of the first pair comes first, up to its
      //      footprints, whose bounds give the item's texel windows
      bool bounds = first && windowed;
      int g = 0, i = 0, u = 0;  // the warp's unit u = g nact + i: pair g of the group, block act[i]
      for (;;) {
        if (!bounds) {
          int next = 0;
          if (lane == 0) next = (int)atomicAdd(&sm.unit, 1u);
          next = __shfl_sync(0xffffffffu, next, 0);
          i += next - u;
          u = next;
          for (; i >= nact; i -= nact) ++g;
          if (g >= G) break;
        } else {
          i = warp < nact ? warp : 0;
        }
        const int n_win = sm.wbase[NFOOT], stride = 2 * n_win + nh;
        const int blk = (int)sm.act[i];
        const int dx = (blk & 1) * 8 + lx, dy = (blk >> 1) * 4 + ly, X = dx * 256, Y = dy * 256;
        const int px = tx * TILE + dx, py = ty * TILE + dy;
        const bool valid = px < S.W && py < S.H;
        const int4* cands = ws.cand + ((long long)slot * ntl + tile) * kCandWords * TILE_PX + dy * TILE + dx;
        int ncand = sm.ncand[blk * 32 + lane];
        if (bounds && (warp >= nact || ncand > CMAX)) ncand = 0;
        const int sbase = g * nb;
        int jA, jB = -1;                    // visible triangles: side +, side - (after the loop)
        float3 cA, cB = f3(0.f, 0.f, 0.f);  // colours
        uint32_t crA[NFOOT], crB[NFOOT];    // credit codes
#pragma unroll
        for (int r = 0; r < NFOOT; ++r) crB[r] = 0;
        // one copy of the code serves both sides (the second pass moves the first's results on)
#pragma unroll 1
        for (int sd = 0; sd < 2; ++sd) {
          jA = jB;
          cA = cB;
#pragma unroll
          for (int r = 0; r < NFOOT; ++r) crA[r] = crB[r];
          jB = -1;
          cB = f3(S.bg[0], S.bg[1], S.bg[2]);
          // -- R: the visible triangle among the candidates, nearest first (one wholly behind the
          //    best so far ends the search)
          uint32_t bz = 0xFFFFFFFFu;
          float l[3] = {0.f, 0.f, 0.f};
          const SideTri* sides = sm.side[sd] + sbase;
          auto test = [&](int j) {
            float q[3];
            float4 z;
            if (!cover_lambdas(sides[j], X, Y, q, z)) return;
            const float zz[3] = {z.x, z.y, z.z};
            const uint32_t zb = ordered_bits(interp_depth(q, zz));
            if (zb < bz || (zb == bz && (jB < 0 || sm.btri[j] < sm.btri[jB]))) {
              bz = zb;
              jB = j;
              l[0] = q[0], l[1] = q[1], l[2] = q[2];
            }
          };
          if (ncand > CMAX) {
            for (int j = 0; j < nb; ++j) test(j);
          } else {
            int4 list = sm.cand[blk * 32 + lane];
            for (int q = 0; q < ncand; ++q) {
              const int j = list.x & 0xFF;
              list.x = (int)((uint32_t)list.x >> 8);
              if ((q & 3) == 3) {
                if (q == 15) list = __ldg(cands + TILE_PX);  // the list's second half (few pixels have one)
                else list.x = list.y, list.y = list.z, list.z = list.w;
              }
              if (!CHK(S, j, nb)) continue;
              if (sm.zminb[j] > bz) break;
              test(j);
            }
          }
          // -- U: the UV buffer value and footprints
          float u0 = 0.f, v0 = 0.f;
          PerspW pw;
          if (jB >= 0) {
            const float4 iw4 = sides[jB].iw;
            const float iw[3] = {iw4.x, iw4.y, iw4.z};
            pw = persp(l, iw);
            const float* uvt = sm.uv[jB];
            u0 = persp_interp(pw, uvt[0], uvt[2], uvt[4]);
            v0 = persp_interp(pw, uvt[1], uvt[3], uvt[5]);
          }
          if (bounds) {
            add_bounds<SH, GR>(S, sm, jB >= 0, u0, v0);
            break;
          }
          if (jB < 0) continue;
          // -- G: sample the perturbed texels and shade
          float val[NREAD][3];
          sample_side<SH, GR>(S, ws, sm, planes, g, sd, u0, v0, n_win, crB, val);
          cB = shade_side<SH, GR>(S, view, val, sm.frame[M::LIT ? sd : 0][M::LIT ? sbase + jB : 0], sm.vid[jB],
                                  sm.sgn9[par][sbase + jB] ^ (sd ? 0x1FFu : 0u), pw);
        }
        if (bounds) {
          bounds = false;
          i = 0;
          __syncthreads();
          if (tid == 0) make_windows(S, sm);
          __syncthreads();
          load_window<SH, GR>(S, sm);
          const int n = sm.wbase[NFOOT];
          nh = n > 0 ? kHashWindow : kHashNoWindow;
          Gcap = min(Gcap, M::ACAP / (2 * n + nh));
          G = min(G, Gcap);
          load_signs<SH, GR>(S, ws, sm, planes, G);
          __syncthreads();
          continue;
        }

        // -- f+ - f- and its credits
        float df = 0.0f;
        if (valid) {
          const float3 tgt = f3(sm.tgt[0][blk * 32 + lane], sm.tgt[1][blk * 32 + lane], sm.tgt[2][blk * 32 + lane]);
          float fp, fm;
          df = loss_diff(cA, cB, tgt, fp, fm);  // 0 where both sides show the background
          loss_acc += 0.5f * (fp + fm);
          if (a.delta_f) a.delta_f[(((long long)slot * a.pairs + pg + g) * S.H + py) * S.W + px] = df;
        }
        // vertices: the visible triangle of side + (else side -), summed over each run of lanes that
        // share it, one shared atomic per run
        {
          const int kt = jA >= 0 ? jA : jB;
          float v = df;
          int n;
          if (run_sum(kt, v, n) && kt >= 0) {
            atomicAdd(&sm.A_tri[sbase + kt], v);
            atomicAdd(&sm.n_tri[sbase + kt], (uint32_t)n);
          }
        }
        if (jA >= 0 && jB >= 0 && jB != jA) {
          // side -'s corners that side +'s triangle does not share
          uint32_t add = 0;
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            const int v = sm.vid[jB][k];
            if (v != sm.vid[jA][0] && v != sm.vid[jA][1] && v != sm.vid[jA][2]) {
              atomicAdd(&sm.A_cor[sbase + jB][k], df);
              add |= 1u << (10 * k);
            }
          }
          if (add) atomicAdd(&sm.n_cor[sbase + jB], add);
        }
        if (jA >= 0 || jB >= 0)
          credit_texels<SH, GR>(S, ws, a, sm, planes, g, stride, n_win, nh, df, jA >= 0, jB >= 0, crA, crB);
      }
      __syncthreads();
      first = false;
      par ^= 1;
    }
    // ---- the last group's fold, the texel counts, the item's loss; then everything back to empty
    if (nact > 0) {
      fold<SH, GR>(S, ws, a, sm, nb, G, par ^ 1, nh, planes0 + (long long)((p1 - G) - p0) * ws.sgn_words);
      __syncthreads();
      flush_counts<SH, GR>(S, a, sm, nh);
      clear_sums(sm, G, nh);
    }
    end_item<SH, GR>(a, sm, slot, loss_acc, next);
  }
  add_losses<SH, GR>(a, sm, vl.n);
}

// Every heavy work item of one scene's call: tiles with more live triangles than the fast path's set-ups
// hold (dense meshes, poles, silhouettes seen edge-on).  The same steps with another split:
// the triangles are many and small (a pixel may have a hundred candidates), so R goes by triangle: each
// is set up and tested at the pixel centres of its box, and the nearest key wins by an atomic minimum; then
// a warp keeps one block of the tile and one of P pairs, and each pixel sets its visible triangles up
// again by itself (one is seen by a pixel or two, so there is nothing to share) and shades.  Vertex
// credits go to the global sums directly, texel credits through the windows and cells as in the fast path.
// Bound by instruction issue (R is 70 % of it).  Against the general kernel it replaces, which set every
// live triangle up in shared memory per pair, tested up to all of them at each pixel and hashed vertices and
// texels: 24.6 -> 7.6 ms (GGX, 1 M triangles, 6,175 dense tiles x 4 pairs), 4.82 -> 1.73 ms (a batch of 8 unlit
// assets), 1.32 -> 0.26 ms (Lambert, 41 tiles x 16 pairs).
template <int SH, bool GR>
__device__ __forceinline__ void dense_items(const SceneDev& S, const Workspace& ws, const ViewList& vl,
                                            const EstimateArgs& a, FastSmem<SH, GR>& sm, bool own_first, bool& clean) {
  using M = Model<SH, GR>;
  constexpr int NREAD = M::NREAD, NFOOT = M::NFOOT, BLOCKS = TILE_PX / 32;
  constexpr int P = M::WARPS / BLOCKS;  // pairs at a time
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, stream = warp / BLOCKS, blk = warp % BLOCKS;
  const int dx = (blk & 1) * 8 + (lane & 7), dy = (blk >> 1) * 4 + (lane >> 3), X = dx * 256, Y = dy * 256;
  // the visible triangle's (depth bits << 32 | id) per pair, side and pixel, in the fast path's set-ups' place
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(&sm.side[0][0]);
  static_assert(sizeof(sm.side) >= 2 * P * TILE_PX * sizeof(unsigned long long), "keys");
  const int ntl = n_tiles(S), n_heavy = (int)ws.counters[4];
  // (the P pairs at a time need P pairs an item: one, a quarter of pairs_per_item = 1..7, leaves half the warps
  // without a pair.  100 K triangles at 256^2, 2 views x 8 pairs, pairs_per_item = 4: 857 us with one, 754 us with two)
  const int ppi = a.pairs_per_item > 0 ? a.pairs_per_item : kRun;
  const int run = run_of(a, n_heavy, max(P, ppi / 4), max(P, ppi));
  const int chunks = (a.pair_count + run - 1) / run;
  const long long n_work = (long long)n_heavy * chunks;
  if (n_work == 0 || (own_first && blockIdx.x >= n_work)) return;  // (uniform over the CTA)
  if (!clean) reset_smem<SH, GR>(sm);
  clean = true;
  const uint32_t first_of = own_first ? gridDim.x : 0u;
  if (tid == 0) sm.item = own_first ? blockIdx.x : atomicAdd(ws.counters + 5, 1u);
  __syncthreads();

  for (long long w = sm.item; w < n_work; w = sm.item) {
    const int at = (int)(w / chunks), chunk = (int)(w - (long long)at * chunks);
    const uint32_t it = ws.items[vl.n * ntl - 1 - at];
    const int slot = it >> 24, tile = it & 0xFFFFFF;
    uint32_t next = 0;
    if (tid == 0) next = first_of + atomicAdd(ws.counters + 5, 1u);
    if (!CHK(S, slot, vl.n) || !CHK(S, tile, ntl)) {  // (checked build; uniform over the CTA)
      __syncthreads();
      if (tid == 0) sm.item = next;
      __syncthreads();
      continue;
    }
    const int view = vl.id[slot];
    const int tx = tile % S.tiles_x, ty = tile / S.tiles_x;
    const int rx = 256 * (tx * TILE) + 128, ry = 256 * (ty * TILE) + 128;
    const uint32_t bin_beg = ws.tile_off[slot * ntl + tile];
    const int nb = (int)ws.tile_live[slot * ntl + tile];  // pruned and compacted by k_bin_prune
    const int p0 = a.pair_begin + chunk * run, p1 = min(a.pair_begin + a.pair_count, p0 + run);
    const int px = tx * TILE + dx, py = ty * TILE + dy;
    const bool valid = px < S.W && py < S.H;
    // ---- per item: the first live triangles' vertices and this pixel's target
    for (int j = tid; j < min(nb, kDenseTri); j += M::THREADS) {
      const int tri = (int)bin_at(S, ws, bin_beg + j);
      sm.dense[j] = make_int4(vert_of(S, tri, 0), vert_of(S, tri, 1), vert_of(S, tri, 2), tri);
    }
    // live triangle j: its vertices and id
    auto triangle = [&](int j) {
      if (j < kDenseTri) return sm.dense[j];
      const int tri = (int)bin_at(S, ws, bin_beg + j);
      return make_int4(vert_of(S, tri, 0), vert_of(S, tri, 1), vert_of(S, tri, 2), tri);
    };
    // its projected vertices for one side of a pair (vb: the pair's first vertex record)
    auto vertices = [&](const int4& t, long long vb, int sd, PVert (&v)[3]) {
      const int id[3] = {t.x, t.y, t.z};
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int4 q = __ldg(ws.pverts + 2 * (vb + id[k]) + sd);
        v[k].X = q.x;
        v[k].Y = q.y;
        v[k].z = __int_as_float(q.z);
        v[k].iw = __int_as_float(q.w);
        v[k].ok = q.x != kNotDrawn;
      }
    };
    float3 tgt = f3(0.f, 0.f, 0.f);
    if (valid) {
      const float* tp = S.targets + (((long long)view * S.H + py) * S.W + px) * 3;
      tgt = f3(__ldg(tp), __ldg(tp + 1), __ldg(tp + 2));
    }
    float loss_acc = 0.0f;
    int Gcap = GMAX, G = 0, nh = 0;
    const bool windowed = M::LIT || a.pair_count > 2;  // as in fast_items
    if (!windowed) {
      nh = kHashNoWindow;
      Gcap = min(Gcap, M::ACAP / nh);
    }
    bool first = true;
    const uint32_t* planes0 = ws.tsign + ((long long)slot * ws.max_pairs + (p0 - a.pair_begin)) * ws.sgn_words;

    for (int pg = p0; pg < p1; pg += G) {
      const uint32_t* planes = planes0 + (long long)(pg - p0) * ws.sgn_words;
      if (!first) {
        fold<SH, GR>(S, ws, a, sm, 0, G, 0, nh, planes - (long long)G * ws.sgn_words);
        __syncthreads();
        clear_sums(sm, G, nh);
      }
      G = min(Gcap, p1 - pg);
      if (!first && windowed) load_signs<SH, GR>(S, ws, sm, planes, G);
      bool bounds = first && windowed;
      for (int s0 = 0; s0 < G; s0 += P) {
        const int g = s0 + stream;  // this warp's pair of the group, if there is one
        const long long vb0 = ((long long)slot * ws.max_pairs + (pg - a.pair_begin) + s0) * S.nv;
        // ---- R: every live triangle into the pixels of its box, both sides of the step's pairs
        __syncthreads();  // the previous step's keys (or the item's set-up) are done with
        for (int i = tid; i < 2 * P * TILE_PX; i += M::THREADS) keys[i] = ~0ull;
        __syncthreads();
        for (int st = 0; st < P && s0 + st < G; ++st) {
          // (the next triangle's vertices are in flight while one is rasterized)
          const long long vb1 = vb0 + (long long)st * S.nv;
          int4 t, q[3];
          auto fetch = [&](int t2) {
            t = triangle(t2 >> 1);
            const int4* p = ws.pverts + 2 * vb1 + (t2 & 1);
            q[0] = __ldg(p + 2ll * t.x);
            q[1] = __ldg(p + 2ll * t.y);
            q[2] = __ldg(p + 2ll * t.z);
          };
          if (tid < 2 * nb) fetch(tid);
          for (int t2 = tid; t2 - lane < 2 * nb; t2 += M::THREADS) {
            const int4 v0 = q[0], v1 = q[1], v2 = q[2];
            const int id = t.w;
            if (t2 + M::THREADS < 2 * nb) fetch(t2 + M::THREADS);
            int c0, c1, r0, r1;
            if (t2 < 2 * nb && tri_box(v0, v1, v2, rx, ry, c0, c1, r0, r1))
              raster_tri(v0, v1, v2, id, rx, ry, c0, c1, r0, r1, keys + (st * 2 + (t2 & 1)) * TILE_PX);
            __syncwarp();  // (lanes left to themselves stay apart after one's box: 9.6 instead of 7.6 ms)
          }
        }
        __syncthreads();
        int tri[2] = {-1, -1};
        if (valid && g < G) {
#pragma unroll
          for (int sd = 0; sd < 2; ++sd) {
            const unsigned long long k = keys[(stream * 2 + sd) * TILE_PX + dy * TILE + dx];
            if (k != ~0ull) tri[sd] = (int)(uint32_t)k;
          }
        }
        // ---- U, G: both sides' winners, set up, sampled and shaded by their pixel
        const long long vb = vb0 + (long long)stream * S.nv;
        int n_win = sm.wbase[NFOOT];
        int vidA[3], vidB[3] = {-1, -1, -1};  // the visible triangles' vertices and signs: side +, side -
        uint32_t sgA = 0, sgB = 0;
        float3 cA, cB = f3(0.f, 0.f, 0.f);
        uint32_t crA[NFOOT], crB[NFOOT];
#pragma unroll
        for (int r = 0; r < NFOOT; ++r) crB[r] = 0;
#pragma unroll 1
        for (int sd = 0; sd < 2; ++sd) {
          const int vis = sd == 0 ? tri[0] : tri[1];
          cA = cB;
          sgA = sgB;
#pragma unroll
          for (int k = 0; k < 3; ++k) vidA[k] = vidB[k];
#pragma unroll
          for (int r = 0; r < NFOOT; ++r) crA[r] = crB[r];
          vidB[0] = vidB[1] = vidB[2] = -1;
          cB = f3(S.bg[0], S.bg[1], S.bg[2]);
          float u0 = 0.f, v0 = 0.f;
          PerspW pw;
          float uvt[6];
          if (vis >= 0) {
            const int4 t = make_int4(vert_of(S, vis, 0), vert_of(S, vis, 1), vert_of(S, vis, 2), vis);
            vidB[0] = t.x, vidB[1] = t.y, vidB[2] = t.z;
            PVert v[3];
            vertices(t, vb, sd, v);
            sgB = 0;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
              sgB |= ((uint32_t)__ldg(ws.vbits + vb + vidB[k]) & 7u) << (3 * k);
            }
            load_uvs(S, t.w, uvt);
            SideTri d;
            set_up_side(d, v, rx, ry);
            float l[3] = {0.f, 0.f, 0.f};
            float4 z;
            cover_lambdas(d, X, Y, l, z);
            const float iw[3] = {v[0].iw, v[1].iw, v[2].iw};
            pw = persp(l, iw);
            u0 = persp_interp(pw, uvt[0], uvt[2], uvt[4]);
            v0 = persp_interp(pw, uvt[1], uvt[3], uvt[5]);
          }
          if (bounds) {
            // the item's first pairs: their side + footprints bound the windows
            bounds = false;
            add_bounds<SH, GR>(S, sm, vis >= 0, u0, v0);
            __syncthreads();
            if (tid == 0) make_windows(S, sm);
            __syncthreads();
            load_window<SH, GR>(S, sm);
            n_win = sm.wbase[NFOOT];
            nh = n_win > 0 ? kHashWindow : kHashNoWindow;
            Gcap = min(Gcap, M::ACAP / (2 * n_win + nh));
            G = min(G, Gcap);
            load_signs<SH, GR>(S, ws, sm, planes, G);
            __syncthreads();
          }
          if (vis < 0) continue;
          float val[NREAD][3];
          sample_side<SH, GR>(S, ws, sm, planes, g, sd, u0, v0, n_win, crB, val);
          const uint32_t sg = sgB ^ (sd ? 0x1FFu : 0u);
          float fr[6];
          if constexpr (M::LIT) {
            float3 p[3];
            corner_positions(S, vidB, sg, p);
            tri_frame(p, uvt, fr);
          }
          cB = shade_side<SH, GR>(S, view, val, fr, vidB, sg, pw);
        }
        // ---- f+ - f- and its credits
        if (g >= G) continue;
        const int stride = 2 * n_win + nh;
        float df = 0.0f;
        if (valid) {
          float fp, fm;
          df = loss_diff(cA, cB, tgt, fp, fm);
          loss_acc += 0.5f * (fp + fm);
          if (a.delta_f) a.delta_f[(((long long)slot * a.pairs + pg + g) * S.H + py) * S.W + px] = df;
        }
        const bool inA = vidA[0] >= 0, inB = vidB[0] >= 0;
        if (!inA && !inB) continue;
#pragma unroll 1
        for (int i = 0; i < 6; ++i) {
          const int k = i % 3;
          const int v = i < 3 ? (k == 0 ? vidA[0] : (k == 1 ? vidA[1] : vidA[2])) : (k == 0 ? vidB[0] : (k == 1 ? vidB[1] : vidB[2]));
          if (v < 0 || (i >= 3 && inA && (v == vidA[0] || v == vidA[1] || v == vidA[2]))) continue;
          const uint32_t sb = (i < 3 ? sgA : sgB) >> (3 * k);
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const long long p = 3ll * v + c;
            if (!CHK(S, p, S.chk.params)) continue;
            atomicAdd(a.grad + p, ((sb >> c) & 1) ? -df : df);
            atomicAdd(a.counts + p, 1u);
          }
        }
        credit_texels<SH, GR>(S, ws, a, sm, planes, g, stride, n_win, nh, df, inA, inB, crA, crB);
      }
      __syncthreads();
      first = false;
    }
    fold<SH, GR>(S, ws, a, sm, 0, G, 0, nh, planes0 + (long long)((p1 - G) - p0) * ws.sgn_words);
    __syncthreads();
    flush_counts<SH, GR>(S, a, sm, nh);
    clear_sums(sm, G, nh);
    end_item<SH, GR>(a, sm, slot, loss_acc, next);
  }
  add_losses<SH, GR>(a, sm, vl.n);
}

template <int SH, bool GR>
__global__ void __launch_bounds__(Model<SH, GR>::THREADS, Model<SH, GR>::CTAS)
    k_estimate_fast(SceneDev S, Workspace ws, ViewList vl, EstimateArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  bool clean = false;
  fast_items<SH, GR>(S, ws, vl, a, *reinterpret_cast<FastSmem<SH, GR>*>(smem_raw), true, clean, true);
}

template <int SH, bool GR>
__global__ void __launch_bounds__(Model<SH, GR>::THREADS, 1)
    k_estimate_dense(SceneDev S, Workspace ws, ViewList vl, EstimateArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  bool clean = false;
  dense_items<SH, GR>(S, ws, vl, a, *reinterpret_cast<FastSmem<SH, GR>*>(smem_raw), true, clean);
}

// The batched kernel keeps its asset after FastSmem, 16-byte aligned.  (Batched calls use the
// per-texture windows: their assets need not share texture sizes.)
template <int SH>
__host__ __device__ constexpr size_t fast_batch_off() {
  return (sizeof(FastSmem<SH, false>) + 15) & ~(size_t)15;
}

// Batched form: the assets of P in order, each until its light items run out.
template <int SH>
__global__ void __launch_bounds__(Model<SH>::THREADS, Model<SH>::CTAS) k_estimate_fast_batch(const BatchArgs P) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  auto& sm = *reinterpret_cast<FastSmem<SH, false>*>(smem_raw);
  BatchSmem& b = *reinterpret_cast<BatchSmem*>(smem_raw + fast_batch_off<SH>());
  bool clean = false;
  for (int ai = 0; ai < P.n; ++ai) {
    __syncthreads();
    load_asset(P, ai, b);
    __syncthreads();
    fast_items<SH, false>(b.d.S, b.d.ws, b.vl, b.a, sm, ai == 0, clean, P.n == 1);
  }
}

// and each until its heavy items run out.
template <int SH>
__global__ void __launch_bounds__(Model<SH>::THREADS, 1) k_estimate_dense_batch(const BatchArgs P) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  auto& sm = *reinterpret_cast<FastSmem<SH, false>*>(smem_raw);
  BatchSmem& b = *reinterpret_cast<BatchSmem*>(smem_raw + fast_batch_off<SH>());
  bool clean = false;
  for (int ai = 0; ai < P.n; ++ai) {
    __syncthreads();
    load_asset(P, ai, b);
    __syncthreads();
    dense_items<SH, false>(b.d.S, b.d.ws, b.vl, b.a, sm, ai == 0, clean);
  }
}

template <int SH, bool GR>
size_t fast_smem() {
  return sizeof(FastSmem<SH, GR>);
}

template <int SH>
size_t fast_batch_smem() {
  return fast_batch_off<SH>() + sizeof(BatchSmem);
}

template <int SH>
cudaError_t launch_fast_batch_t(const BatchArgs& P, int grid, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(k_estimate_fast_batch<SH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)fast_batch_smem<SH>());
  if (e != cudaSuccess) return e;
  k_estimate_fast_batch<SH><<<grid, Model<SH>::THREADS, fast_batch_smem<SH>(), st>>>(P);
  return cudaGetLastError();
}

template <int SH>
cudaError_t launch_dense_batch_t(const BatchArgs& P, int grid, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(k_estimate_dense_batch<SH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)fast_batch_smem<SH>());
  if (e != cudaSuccess) return e;
  k_estimate_dense_batch<SH><<<grid, Model<SH>::THREADS, fast_batch_smem<SH>(), st>>>(P);
  return cudaGetLastError();
}

template <int SH, bool GR>
cudaError_t launch_dense_t(const SceneDev& S, const Workspace& ws, const ViewList& vl, const EstimateArgs& a, int grid,
                           cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(k_estimate_dense<SH, GR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)fast_smem<SH, GR>());
  if (e != cudaSuccess) return e;
  k_estimate_dense<SH, GR><<<grid, Model<SH, GR>::THREADS, fast_smem<SH, GR>(), st>>>(S, ws, vl, a);
  return cudaGetLastError();
}

template <int SH>
int fast_batch_blocks_per_sm_t() {
  int n = 0;
  cudaFuncSetAttribute(k_estimate_fast_batch<SH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)fast_batch_smem<SH>());
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_estimate_fast_batch<SH>, Model<SH>::THREADS, fast_batch_smem<SH>());
  return n > 0 ? n : 1;
}

template <int SH, bool GR>
cudaError_t launch_fast_t(const SceneDev& S, const Workspace& ws, const ViewList& vl, const EstimateArgs& a,
                          int grid, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(k_estimate_fast<SH, GR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)fast_smem<SH, GR>());
  if (e != cudaSuccess) return e;
  k_estimate_fast<SH, GR><<<grid, Model<SH, GR>::THREADS, fast_smem<SH, GR>(), st>>>(S, ws, vl, a);
  return cudaGetLastError();
}

template <int SH, bool GR>
int fast_blocks_per_sm_t() {
  int n = 0;
  cudaFuncSetAttribute(k_estimate_fast<SH, GR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)fast_smem<SH, GR>());
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_estimate_fast<SH, GR>, Model<SH, GR>::THREADS, fast_smem<SH, GR>());
  return n > 0 ? n : 1;
}

}  // namespace

cudaError_t launch_fast(const SceneDev& S, const Workspace& ws, const ViewList& vl, const EstimateArgs& a, int grid,
                        cudaStream_t st) {
  if (S.shading == SHADE_UNLIT) return launch_fast_t<SHADE_UNLIT, false>(S, ws, vl, a, grid, st);
  if (S.shading == SHADE_LAMBERT)
    return S.grouped ? launch_fast_t<SHADE_LAMBERT, true>(S, ws, vl, a, grid, st)
                     : launch_fast_t<SHADE_LAMBERT, false>(S, ws, vl, a, grid, st);
  return S.grouped ? launch_fast_t<SHADE_GGX, true>(S, ws, vl, a, grid, st)
                   : launch_fast_t<SHADE_GGX, false>(S, ws, vl, a, grid, st);
}

cudaError_t launch_dense(const SceneDev& S, const Workspace& ws, const ViewList& vl, const EstimateArgs& a, int grid,
                         cudaStream_t st) {
  if (S.shading == SHADE_UNLIT) return launch_dense_t<SHADE_UNLIT, false>(S, ws, vl, a, grid, st);
  if (S.shading == SHADE_LAMBERT)
    return S.grouped ? launch_dense_t<SHADE_LAMBERT, true>(S, ws, vl, a, grid, st)
                     : launch_dense_t<SHADE_LAMBERT, false>(S, ws, vl, a, grid, st);
  return S.grouped ? launch_dense_t<SHADE_GGX, true>(S, ws, vl, a, grid, st)
                   : launch_dense_t<SHADE_GGX, false>(S, ws, vl, a, grid, st);
}

// Grids of up to two CTAs per SM run at once and take as long as their fullest tile: a row per thread and
// registers without spills.  Larger grids are bound by issue: 7 resident CTAs in 32 registers, whose barriers
// hide behind one another, and 4 threads to a triangle, so small boxes leave few lanes idle (8,192 triangles,
// 512^2, 8 views / 1 M triangles, 2048^2, 4 views: 7 CTAs 135 us / 1.96 ms, 5 CTAs 169 us / 2.29 ms; 8 threads
// to a triangle 127 us / 2.16 ms; one wave of 256 tiles: 21.1 us with 16 threads, 24.1 us with 4).
// Up to one wave of those the fullest tile still counts: a row per thread (soup of 10,240 triangles, 512^2, one view:
// 55.6 us before all this, 39.1 us; 47.0 us with 4 threads to a triangle).
constexpr int kPruneOneWave = 2 * 152, kPruneSevenWave = 7 * 152;

cudaError_t launch_prune(const SceneDev& S, const Workspace& ws, const ViewList& vl, cudaStream_t st) {
  const dim3 grid(n_tiles(S), vl.n);
  if ((long long)grid.x * grid.y <= kPruneOneWave)
    k_bin_prune<16, 2><<<grid, TILE_PX, 0, st>>>(S, ws, vl);
  else if ((long long)grid.x * grid.y <= kPruneSevenWave)
    k_bin_prune<16, 7><<<grid, TILE_PX, 0, st>>>(S, ws, vl);
  else
    k_bin_prune<4, 7><<<grid, TILE_PX, 0, st>>>(S, ws, vl);
  return cudaGetLastError();
}

cudaError_t launch_prune_batch(const BatchArgs& P, int max_tiles, int max_views, cudaStream_t st) {
  const dim3 grid(max_tiles, max_views, P.n);
  const long long ctas = (long long)grid.x * grid.y * grid.z;
  if (ctas <= kPruneOneWave)
    k_bin_prune_batch<16, 2><<<grid, TILE_PX, 0, st>>>(P);
  else if (ctas <= kPruneSevenWave)
    k_bin_prune_batch<16, 7><<<grid, TILE_PX, 0, st>>>(P);
  else
    k_bin_prune_batch<4, 7><<<grid, TILE_PX, 0, st>>>(P);
  return cudaGetLastError();
}

cudaError_t launch_fast_batch(const BatchArgs& P, int shading, int grid, cudaStream_t st) {
  if (shading == SHADE_UNLIT) return launch_fast_batch_t<SHADE_UNLIT>(P, grid, st);
  if (shading == SHADE_LAMBERT) return launch_fast_batch_t<SHADE_LAMBERT>(P, grid, st);
  return launch_fast_batch_t<SHADE_GGX>(P, grid, st);
}

cudaError_t launch_dense_batch(const BatchArgs& P, int shading, int grid, cudaStream_t st) {
  if (shading == SHADE_UNLIT) return launch_dense_batch_t<SHADE_UNLIT>(P, grid, st);
  if (shading == SHADE_LAMBERT) return launch_dense_batch_t<SHADE_LAMBERT>(P, grid, st);
  return launch_dense_batch_t<SHADE_GGX>(P, grid, st);
}

int fast_batch_blocks_per_sm(int shading) {
  if (shading == SHADE_UNLIT) return fast_batch_blocks_per_sm_t<SHADE_UNLIT>();
  if (shading == SHADE_LAMBERT) return fast_batch_blocks_per_sm_t<SHADE_LAMBERT>();
  return fast_batch_blocks_per_sm_t<SHADE_GGX>();
}

int fast_blocks_per_sm(int shading, int grouped) {
  if (shading == SHADE_UNLIT) return fast_blocks_per_sm_t<SHADE_UNLIT, false>();
  if (shading == SHADE_LAMBERT)
    return grouped ? fast_blocks_per_sm_t<SHADE_LAMBERT, true>() : fast_blocks_per_sm_t<SHADE_LAMBERT, false>();
  return grouped ? fast_blocks_per_sm_t<SHADE_GGX, true>() : fast_blocks_per_sm_t<SHADE_GGX, false>();
}

}  // namespace sge
