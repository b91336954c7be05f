// Transparent geometry (Section 4.4): the raster pass keeps a deep ID buffer (each pixel's
// SGE_MAX_LAYERS nearest fragments, ascending (depth bits, triangle id) keys), the shading
// composites the listed RGBA fragments front to back over the background, and G walks the list,
// crediting every listed fragment's vertices and albedo footprint as the opaque case credits
// its one visible triangle.
//
// One CTA per (16 x 16 tile, estimate).  The tile's binned triangles are set up for both sides
// in shared memory a chunk at a time; each pixel keeps both sides' lists in registers (with each
// entry's chunk slot, so that a bin of one chunk is not set up again to shade), then shades,
// forms f+ - f- and credits the union of its fragments' parameters.  When the bin fits one chunk
// the vertex credits are summed per staged triangle in shared memory and reach the global
// sums once per corner at the end of the CTA; texel credits (and every credit of a larger bin) go
// to global atomics per pixel.  Bins come from the conservative binning without pruning: a
// fragment behind another is still listed.
//
// Bound by instruction issue.  The set-up uses every thread and 32-bit edge functions, warps visit only the
// triangles whose box reaches their 8 x 4 block, a triangle whose corners are all new credits them with
// one sum, and the union over the two lists compares footprints by the difference of their first
// texels' ids and triangles by a 32-bit signature instead of searching lists of keys in local memory.
// 9.3 -> 5.3 ms per call (6,144 triangles, 512^2, 8 views x 16 pairs); 3 CTAs per SM instead of 4 take 5.9 ms,
// 5 no less, with 0.8 GB of spilled registers reaching DRAM.
#include <cuda_runtime.h>

#define SGE_FILE_ID 2  // range-check sites of this file (checked build)
#include "sge_device.cuh"

namespace sge {

namespace {

constexpr int K = SGE_MAX_LAYERS;
constexpr int DCHUNK = 128;              // binned triangles staged per pass
constexpr int kDeepEstimates = 16384;    // estimates (grid rows) of one launch

template <int NS>
struct DeepSmem {
  SideTri t[NS][DCHUNK];
  uint32_t span[DCHUNK][2];  // box_span of each staged side-triangle: the pixels it may cover
  int tri[DCHUNK];
  float uv[DCHUNK][6];
  // estimator (two sides) with a bin of one chunk: each staged triangle's welded vertices, and the
  // sums of f+ - f- and the counts of the pixels that credit them through this triangle
  static constexpr int NV = NS == 2 ? DCHUNK : 1;
  int vid[NV][3];
  uint32_t sig[NV];  // bit v mod 32 of each vertex v: triangles without a common bit share no vertex
  float A_tri[NV];   // credited through all three corners at once
  uint32_t n_tri[NV];
  float A_cor[NV][3];  // and through single corners (counts: 10 bits each, at most 256 pixels)
  uint32_t n_cor[NV];
  float m[16];
  float red[TILE_PX / 32];
};

// Insert key k (staged at shared-memory slot q) into the ascending list L (slots P); the
// largest key falls off the end.
__device__ __forceinline__ void deep_insert(unsigned long long (&L)[K], int (&P)[K], unsigned long long k, int q) {
#pragma unroll
  for (int j = 0; j < K; ++j) {
    const bool lt = k < L[j];
    const unsigned long long lo = lt ? k : L[j];
    const int qlo = lt ? q : P[j];
    k = lt ? L[j] : k;
    q = lt ? P[j] : q;
    L[j] = lo;
    P[j] = qlo;
  }
}

// Deep lists of one pixel of the tile for NS sides (sides[s] = +1, -1 or 0), with each entry's
// slot in the staged chunk.  Returns the number of binned triangles it rasterized; when that is at
// most DCHUNK the whole bin fit one chunk, and sm.t[s][P[s][j]] (and sm.vid[P[s][j]]) still hold
// entry j's set-up when the raster is done.
// pv: the estimate's projected vertices from the vertex pass ([nv][2]: sides +, -), for the two
// sides of an estimate; NULL: each triangle is projected from the scene with key and sides[].
template <int NS>
__device__ __forceinline__ int deep_raster(const SceneDev& S, const Workspace& ws, DeepSmem<NS>& sm, int slot,
                                            int tile, uint64_t key, const int (&sides)[NS],
                                            unsigned long long (&L)[NS][K], int (&P)[NS][K], int rx, int ry,
                                            int dx, int dy, const int4* pv = nullptr) {
  const int ntl = n_tiles(S);
  const uint32_t block = (0xFFu << (dx & 8)) | (0xF0000u << (dy & 12));  // the warp's 8 x 4 pixels
  const uint32_t beg = ws.tile_off[slot * ntl + tile];
  int nb = (int)ws.tile_count[slot * ntl + tile];
  // after a bin overflow (reported in the status word) the tile's list was not stored
  if ((long long)beg + nb > ws.bin_capacity) nb = 0;
#pragma unroll
  for (int s = 0; s < NS; ++s)
#pragma unroll
    for (int j = 0; j < K; ++j) L[s][j] = ~0ull, P[s][j] = 0;
  for (int c0 = 0; c0 < nb; c0 += DCHUNK) {
    const int cnt = min(DCHUNK, nb - c0);
    __syncthreads();
    for (int t2 = threadIdx.x; t2 < NS * cnt; t2 += TILE_PX) {
      // (two sides: neighbouring threads, whose projected vertices lie next to each other)
      const int s = NS == 2 ? t2 & 1 : 0, j = NS == 2 ? t2 >> 1 : t2;
      const int tri = (int)bin_at(S, ws, beg + c0 + j);
      uint32_t sig = 0u;
      PVert v[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int vi = vert_of(S, tri, k);
        if (pv) {
          const int4 q = __ldg(pv + 2 * vi + s);
          v[k].X = q.x;
          v[k].Y = q.y;
          v[k].z = __int_as_float(q.z);
          v[k].iw = __int_as_float(q.w);
          v[k].ok = q.x != kNotDrawn;
        } else {
          const float3 p = perturbed_pos(S, vi, key, s == 0 ? sides[0] : sides[NS - 1]);
          v[k] = project(sm.m, p.x, p.y, p.z, S.W, S.H, S.near_w);
        }
        if constexpr (NS == 2) {
          if (s == 0) {
            sm.vid[j][k] = vi;
            sm.A_cor[j][k] = 0.0f;
            sig |= 1u << (vi & 31);
          }
        }
      }
      if (s == 0) {
        if constexpr (NS == 2) {
          sm.sig[j] = sig;
          sm.A_tri[j] = 0.0f;
          sm.n_tri[j] = sm.n_cor[j] = 0u;
        }
        sm.tri[j] = tri;
        load_uvs(S, tri, sm.uv[j]);
      }
      set_up_side<true>(sm.t[s][j], v, rx, ry);
      // a covered pixel centre lies in the triangle's vertex box
      sm.span[j][s] = v[0].ok && v[1].ok && v[2].ok ? box_span(v, rx, ry, 0) : 0u;
    }
    __syncthreads();
#pragma unroll 1
    for (int s = 0; s < NS; ++s) {
      // (one copy of the insertion for both sides: the lists change places)
      unsigned long long (&M)[K] = L[0];
      int (&Q)[K] = P[0];
      for_spans(sm.span, s, cnt, block, dx, dy, [&](int j) {
        float l[3];
        float4 z;
        if (!cover_lambdas<true>(sm.t[s][j], dx * 256, dy * 256, l, z)) return;
        const float zz[3] = {z.x, z.y, z.z};
        deep_insert(M, Q, ((unsigned long long)ordered_bits(interp_depth(l, zz)) << 32) | (uint32_t)sm.tri[j], j);
      });
      if constexpr (NS == 2) {
#pragma unroll
        for (int k = 0; k < K; ++k) {
          const unsigned long long x = L[0][k];
          L[0][k] = L[1][k], L[1][k] = x;
          const int y = P[0][k];
          P[0][k] = P[1][k], P[1][k] = y;
        }
      }
    }
  }
  return nb;
}

// Front-to-back composite of one side's list at one pixel: T = 1; per listed fragment
// C += T a rgb, T *= 1 - a with a = clamp(alpha, 0, 1); C += T background.  on_fragment(tri,
// foot, j, q) is called for each listed fragment with its triangle, albedo footprint, layer and
// chunk slot.
// staged: the side's set-ups in shared memory (slots P) when the bin fit one chunk, else NULL
// (each fragment is set up again; the same arithmetic gives the same set-up).
// ps: the estimate's precomputed signs (vertex bits, texel planes), or NULL to hash with key.
template <typename F>
__device__ __forceinline__ float3 deep_composite(const SceneDev& S, const float* m, uint64_t key, int side,
                                                 const unsigned long long (&L)[K], const int (&P)[K],
                                                 const SideTri* staged, const float (*uvs)[6], int rx, int ry, int dx, int dy,
                                                 F&& on_fragment, const PairSigns* ps = nullptr,
                                                 const int4* pv = nullptr) {
  const TexDev& A = S.rtex[0];  // the RGBA albedo, the one texture this model reads
  float c0 = 0.0f, c1 = 0.0f, c2 = 0.0f, T = 1.0f;
  // not unrolled: one copy of the fragment's set-up, sampling and credit code per side keeps the
  // kernel's code within the instruction cache (the lists are read from local memory instead)
#pragma unroll 1
  for (int j = 0; j < K; ++j) {
    if (L[j] == ~0ull) break;  // (ascending: nothing follows)
    const int tri = (int)(L[j] & 0xFFFFFFFFu);
    float l[3] = {0.f, 0.f, 0.f}, iw[3], uv[6];
    float4 z;
    if (staged) {
      const SideTri& t = staged[P[j]];
      cover_lambdas<true>(t, dx * 256, dy * 256, l, z);
      iw[0] = t.iw.x, iw[1] = t.iw.y, iw[2] = t.iw.z;
#pragma unroll
      for (int k = 0; k < 6; ++k) uv[k] = uvs[P[j]][k];
    } else {
      PVert v[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int vi = vert_of(S, tri, k);
        if (pv) {
          const int4 q = __ldg(pv + 2 * vi + (side < 0 ? 1 : 0));
          v[k].X = q.x;
          v[k].Y = q.y;
          v[k].z = __int_as_float(q.z);
          v[k].iw = __int_as_float(q.w);
          v[k].ok = q.x != kNotDrawn;
        } else {
          const float3 p = perturbed_pos(S, vi, key, side);
          v[k] = project(m, p.x, p.y, p.z, S.W, S.H, S.near_w);
        }
        iw[k] = v[k].iw;
      }
      SideTri own;
      set_up_side<true>(own, v, rx, ry);
      cover_lambdas<true>(own, dx * 256, dy * 256, l, z);
      load_uvs(S, tri, uv);
    }
    const PerspW pw = persp(l, iw);
    const float u = persp_interp(pw, uv[0], uv[2], uv[4]), v = persp_interp(pw, uv[1], uv[3], uv[5]);
    Foot f = footprint(u, v, A.w, A.h);
    if (S.foot_nearest) f.nearest = nearest_texel(u, v, A.w, A.h);
    float a[4];
    // an RGBA albedo in a 16-byte aligned array: one vector load per texel
    if (ps && A.c == 4 && ((reinterpret_cast<uintptr_t>(A.ptr) & 15) == 0)) {
      const float w4[4] = {(1.0f - f.fx) * (1.0f - f.fy), f.fx * (1.0f - f.fy), (1.0f - f.fx) * f.fy, f.fx * f.fy};
      const int tx[4] = {f.x0, f.x1, f.x0, f.x1};
      const int ty[4] = {f.y0, f.y0, f.y1, f.y1};
#pragma unroll
      for (int c = 0; c < 4; ++c) a[c] = 0.0f;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const long long tt = (long long)ty[q] * A.w + tx[q];
        const float4 v4 = __ldg(reinterpret_cast<const float4*>(A.ptr + tt * 4));
        uint32_t sb = texel_signs(*ps, A.index, tt);
        if (side < 0) sb = ~sb;
        a[0] += w4[q] * __fadd_rn(v4.x, (sb & 1) ? -A.eps : A.eps);
        a[1] += w4[q] * __fadd_rn(v4.y, (sb & 2) ? -A.eps : A.eps);
        a[2] += w4[q] * __fadd_rn(v4.z, (sb & 4) ? -A.eps : A.eps);
        a[3] += w4[q] * __fadd_rn(v4.w, (sb & 8) ? -A.eps : A.eps);
      }
    } else if (ps) {
      sample_tex_ps(A, f, *ps, side, a);
    } else {
      sample_tex(A, f, key, side, a);
    }
    const float al = fminf(fmaxf(a[3], 0.0f), 1.0f);
    const float w = T * al;
    c0 += w * a[0];
    c1 += w * a[1];
    c2 += w * a[2];
    T *= 1.0f - al;
    on_fragment(tri, f, j, P[j]);
  }
  return f3(c0 + T * S.bg[0], c1 + T * S.bg[1], c2 + T * S.bg[2]);
}

// Sum of v over the CTA, added to *out by thread 0.
__device__ __forceinline__ void cta_add(float v, float* red, float* out) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    float sum = 0.0f;
    for (int i = 0; i < TILE_PX / 32; ++i) sum += red[i];
    if (sum != 0.0f) atomicAdd(out, sum);
  }
}

// One estimate per grid row: blockIdx.y = slot * pair_count + (pair - pair_begin).
__global__ void __launch_bounds__(TILE_PX, 4) k_estimate_deep(SceneDev S, Workspace ws, ViewList vl, EstimateArgs a,
                                                           int row0) {
  __shared__ DeepSmem<2> sm;
  const int tile = blockIdx.x;
  const int row = row0 + (int)blockIdx.y;
  const int slot = row / a.pair_count, pair = a.pair_begin + row % a.pair_count;
  const int view = vl.id[slot];
  const uint64_t key = pair_key(a.seed, iter_of(a), (uint32_t)view, (uint32_t)pair);
  const int tx = tile % S.tiles_x, ty = tile / S.tiles_x;
  // warps own 8 x 4 blocks
  const int dx = ((threadIdx.x >> 5) & 1) * 8 + (threadIdx.x & 7), dy = (threadIdx.x >> 6) * 4 + ((threadIdx.x >> 3) & 3);
  const int px = tx * TILE + dx, py = ty * TILE + dy;
  const int rx = 256 * (tx * TILE) + 128, ry = 256 * (ty * TILE) + 128;
  if (threadIdx.x < 16) sm.m[threadIdx.x] = S.mvp[16 * view + threadIdx.x];
  __syncthreads();
  unsigned long long L[2][K];
  int P[2][K];
  const int sides[2] = {1, -1};
  // the estimate's projected vertices and signs, from the vertex pass and the texel sign planes
  const int pb = pair - a.pair_begin;
  const int4* pv = ws.pverts + 2 * (((long long)slot * ws.max_pairs + pb) * S.nv);
  const PairSigns ps = pair_signs(S, ws, slot, pb);
  const int nb = deep_raster<2>(S, ws, sm, slot, tile, key, sides, L, P, rx, ry, dx, dy, pv);
  const bool resident = nb <= DCHUNK;
  float lv = 0.0f;
  if (px < S.W && py < S.H) {
    const long long npx = (long long)S.W * S.H, p = (long long)py * S.W + px;
    // every listed fragment of both sides, gathered while compositing: its triangle (chunk slot where the
    // bin is one chunk, else id) and its footprint's code (nearest footprint: the texel)
    const TexDev& A = S.rtex[0];
    uint32_t code[2 * K];
    int who[2 * K], n = 0;
    bool odd = false;  // some footprint wraps, is clamped to a row or is one texel wide
    auto fragment = [&](int tri, const Foot& f, int, int q) {
      if (S.foot_nearest) {
        code[n] = (uint32_t)f.nearest;
      } else {
        code[n] = (uint32_t)(f.y0 * A.w + f.x0) | (f.y1 == f.y0 ? kOneRow : 0u);
        odd = odd || f.y1 == f.y0 || f.x1 != f.x0 + 1;
      }
      who[n++] = resident ? q : tri;
    };
    const float3 cp = deep_composite(S, sm.m, key, 1, L[0], P[0], resident ? sm.t[0] : nullptr, sm.uv, rx, ry, dx, dy,
                                     fragment, &ps, pv);
    const float3 cm = deep_composite(S, sm.m, key, -1, L[1], P[1], resident ? sm.t[1] : nullptr, sm.uv, rx, ry, dx, dy,
                                     fragment, &ps, pv);
    const float* tp = S.targets + ((long long)view * npx + p) * 3;
    float fp, fm;
    const float df = loss_diff(cp, cm, f3(__ldg(tp), __ldg(tp + 1), __ldg(tp + 2)), fp, fm);
    lv = 0.5f * (fp + fm);
    if (a.delta_f) a.delta_f[((long long)slot * a.pairs + pair) * npx + p] = df;
    // vertices of the distinct listed triangles, each vertex once
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
      const int q = who[i];
      uint32_t mask = 7u;
#pragma unroll 1
      for (int j = 0; j < i && mask; ++j) {
        const int o = who[j];
        if (o == q) mask = 0u;
        else if (!resident || (sm.sig[q] & sm.sig[o])) {
#pragma unroll
          for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int kk = 0; kk < 3; ++kk)
              if ((resident ? sm.vid[q][k] : vert_of(S, q, k)) == (resident ? sm.vid[o][kk] : vert_of(S, o, kk)))
                mask &= ~(1u << k);
        }
      }
      if (resident) {
        if (mask == 7u) {
          atomicAdd(&sm.A_tri[q], df);
          atomicAdd(&sm.n_tri[q], 1u);
        } else if (mask) {
          uint32_t add = 0u;
#pragma unroll
          for (int k = 0; k < 3; ++k)
            if ((mask >> k) & 1u) {
              atomicAdd(&sm.A_cor[q][k], df);
              add |= 1u << (10 * k);
            }
          atomicAdd(&sm.n_cor[q], add);
        }
        continue;
      }
      for (; mask; mask &= mask - 1) {
        const int v = vert_of(S, q, __ffs((int)mask) - 1);
        if (CHK(S, v, ws.n_kcount)) atomicAdd(ws.kcount + v, 1u);
        const uint32_t sb = vertex_signs(ps, v);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const long long p = 3ll * v + c;
          if (CHK(S, p, S.chk.params)) atomicAdd(a.grad + p, ((sb >> c) & 1) ? -df : df);
        }
      }
    }
    // texels of the distinct footprints, each texel once: one count per key (k_expand_counts gives it to
    // every channel after the call), a signed sum per channel (RGBA texels of an 8-byte aligned gradient:
    // two vector reductions)
    const bool pairs4 = A.c == 4 && ((reinterpret_cast<uintptr_t>(a.grad + A.offset) & 7) == 0);
    auto credit_texel = [&](int id) {
      const long long kc = ws.kc_off[A.index] + id;
      if (CHK(S, kc, ws.n_kcount)) atomicAdd(ws.kcount + kc, 1u);
      const long long base = A.offset + (long long)id * A.c;
      const uint32_t sb = texel_signs(ps, A.index, id);
      if (pairs4) {
        if (!CHK(S, base + 3, S.chk.params)) return;
        atomicAdd(reinterpret_cast<float2*>(a.grad + base), make_float2((sb & 1) ? -df : df, (sb & 2) ? -df : df));
        atomicAdd(reinterpret_cast<float2*>(a.grad + base + 2), make_float2((sb & 4) ? -df : df, (sb & 8) ? -df : df));
        return;
      }
      for (int c = 0; c < A.c; ++c)
        if (CHK(S, base + c, S.chk.params)) atomicAdd(a.grad + base + c, ((sb >> c) & 1) ? -df : df);
    };
    const uint32_t w = (uint32_t)A.w;
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
      uint32_t mask = S.foot_nearest ? 1u : 15u;
      if (!odd || S.foot_nearest) {
        // ids c, c + 1, c + w, c + w + 1: membership in an earlier footprint by id differences
#pragma unroll 1
        for (int j = 0; j < i && mask; ++j) {
          const uint32_t d = code[i] - code[j];
          if (d == 0u) mask = 0u;
          else if (!S.foot_nearest && d + w + 1u <= 2u * w + 2u) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const uint32_t s = d + (q & 1) + (q & 2 ? w : 0u);
              if (s <= 1u || s - w <= 1u) mask &= ~(1u << q);
            }
          }
        }
        for (; mask; mask &= mask - 1) {
          const int q = __ffs((int)mask) - 1;
          credit_texel((int)(code[i] + (q & 1) + (q & 2 ? w : 0u)));
        }
        continue;
      }
      const Quad Q(code[i], A.w);
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (Q.repeats(q)) mask &= ~(1u << q);
#pragma unroll 1
      for (int j = 0; j < i && mask; ++j) {
        const Quad E(code[j], A.w);
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (E.holds(Q, q)) mask &= ~(1u << q);
      }
      for (; mask; mask &= mask - 1) credit_texel(Q.texel(__ffs((int)mask) - 1, A.w));
    }
  }
  if (resident) {
    // every staged corner credited by some pixel: one count and one signed sum per channel
    __syncthreads();
    const int t = threadIdx.x;
    if (t < nb) {
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const uint32_t n = sm.n_tri[t] + ((sm.n_cor[t] >> (10 * k)) & 1023u);
        if (!n) continue;
        const int v = sm.vid[t][k];
        if (CHK(S, v, ws.n_kcount)) atomicAdd(ws.kcount + v, n);
        const float A = sm.A_tri[t] + sm.A_cor[t][k];
        if (A == 0.0f) continue;
        const uint32_t sb = vertex_signs(ps, v);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const long long q = 3ll * v + c;
          if (CHK(S, q, S.chk.params)) atomicAdd(a.grad + q, ((sb >> c) & 1) ? -A : A);
        }
      }
    }
  }
  if (a.loss) cta_add(lv / (float)a.pairs, sm.red, a.loss + slot);
}

// One render's deep lists and composite (side -1, 0 or +1); with loss, the image error of the
// render against the view's target is added to loss[slot].
__global__ void __launch_bounds__(TILE_PX) k_render_deep(SceneDev S, Workspace ws, int slot, int view, uint64_t key,
                                                         int side, unsigned long long* deep, float* rgb, float* loss) {
  __shared__ DeepSmem<1> sm;
  const int tile = blockIdx.x;
  const int tx = tile % S.tiles_x, ty = tile / S.tiles_x;
  // warps own 8 x 4 blocks
  const int dx = ((threadIdx.x >> 5) & 1) * 8 + (threadIdx.x & 7), dy = (threadIdx.x >> 6) * 4 + ((threadIdx.x >> 3) & 3);
  const int px = tx * TILE + dx, py = ty * TILE + dy;
  const int rx = 256 * (tx * TILE) + 128, ry = 256 * (ty * TILE) + 128;
  if (threadIdx.x < 16) sm.m[threadIdx.x] = S.mvp[16 * view + threadIdx.x];
  __syncthreads();
  unsigned long long L[1][K];
  int P[1][K];
  const int sides[1] = {side};
  const bool resident = deep_raster<1>(S, ws, sm, slot, tile, key, sides, L, P, rx, ry, dx, dy) <= DCHUNK;
  float f = 0.0f;
  if (px < S.W && py < S.H) {
    const long long npx = (long long)S.W * S.H, p = (long long)py * S.W + px;
    if (deep) {
#pragma unroll
      for (int j = 0; j < K; ++j) deep[j * npx + p] = L[0][j];
    }
    if (rgb || loss) {
      const float3 c = deep_composite(S, sm.m, key, side, L[0], P[0], resident ? sm.t[0] : nullptr, sm.uv, rx, ry, dx, dy,
                                      [](int, const Foot&, int, int) {});
      if (rgb) rgb[3 * p] = c.x, rgb[3 * p + 1] = c.y, rgb[3 * p + 2] = c.z;
      if (loss) {
        const float* tp = S.targets + ((long long)view * npx + p) * 3;
        const float d0 = c.x - __ldg(tp), d1 = c.y - __ldg(tp + 1), d2 = c.z - __ldg(tp + 2);
        f = d0 * d0 + d1 * d1 + d2 * d2;
      }
    }
  }
  if (loss) cta_add(f, sm.red, loss + slot);
}

}  // namespace

cudaError_t launch_deep_estimate(const SceneDev& S, const Workspace& ws, const ViewList& vl, const EstimateArgs& a,
                                 cudaStream_t st) {
  const int rows = vl.n * a.pair_count;
  for (int r0 = 0; r0 < rows; r0 += kDeepEstimates) {
    const int nr = rows - r0 < kDeepEstimates ? rows - r0 : kDeepEstimates;
    k_estimate_deep<<<dim3(n_tiles(S), nr), TILE_PX, 0, st>>>(S, ws, vl, a, r0);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Every key's contributions of the call into the counts of its channels (each parameter belongs to
// one key: plain adds), and the key counts back to zero.
__global__ void k_expand_counts(SceneDev S, Workspace ws, uint32_t* counts) {
  const long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= ws.n_kcount) return;
  const uint32_t n = ws.kcount[j];
  if (n == 0) return;
  ws.kcount[j] = 0u;
  long long base = 3 * j;
  int nch = 3;
  if (j >= S.nv) {
    for (int k = 0; k < S.ntex; ++k)
      if (ws.kc_off[k] >= 0 && j >= ws.kc_off[k] && j < ws.kc_off[k] + (long long)S.tex[k].w * S.tex[k].h) {
        base = S.tex[k].offset + (j - ws.kc_off[k]) * S.tex[k].c;
        nch = S.tex[k].c;
      }
  }
  for (int c = 0; c < nch; ++c)
    if (CHK(S, base + c, S.chk.params)) counts[base + c] += n;
}

cudaError_t launch_expand_counts(const SceneDev& S, const Workspace& ws, uint32_t* counts, cudaStream_t st) {
  if (ws.n_kcount == 0) return cudaSuccess;
  k_expand_counts<<<(unsigned)((ws.n_kcount + 255) / 256), 256, 0, st>>>(S, ws, counts);
  return cudaGetLastError();
}

cudaError_t launch_render_deep(const SceneDev& S, const Workspace& ws, int slot, int view, uint64_t key, int side,
                               unsigned long long* deep, float* rgb, float* loss, cudaStream_t st) {
  k_render_deep<<<n_tiles(S), TILE_PX, 0, st>>>(S, ws, slot, view, key, side, deep, rgb, loss);
  return cudaGetLastError();
}

}  // namespace sge
