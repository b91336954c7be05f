// Staged kernels: one render of R with its ID and UV buffers (Section 4.4), and
// the plain one-estimate-at-a-time path (Section 5's loop of P, R and G, with G
// as in Algorithm 2: per-pixel loss difference and a global AtomicAdd per
// contributing parameter).
#include <cuda_runtime.h>

#define SGE_FILE_ID 5  // range-check sites of this file (checked build)
#include "sge_device.cuh"

namespace sge {

namespace {

constexpr int RCHUNK = TILE_PX;  // binned triangles staged per pass, one per thread
// Pixels of the largest box that one lane walks alone in a bin of more than one chunk.
constexpr int kLaneBox = 32;

template <int NS>
struct RSmem {
  SideTri t[NS][RCHUNK];
  unsigned long long keys[NS][TILE_PX];
  uint32_t span[RCHUNK][2];  // pixels each staged triangle may cover, per side
  int tri[RCHUNK];
  // (one side) each staged triangle's UVs and frame, where the kernel shades
  float uv[NS == 1 ? RCHUNK : 1][6], fr[NS == 1 ? RCHUNK : 1][6];
  float m[16];
};

// What one side of a pixel sees: the nearest (depth bits << 32 | id), ~0 where nothing, and the barycentric
// weights and 1 / w of that triangle there.
struct Hit {
  unsigned long long key;
  float l[3], iw[3];
  int slot;  // its place in the staged chunk, or -1
};

// No pixel's interpolated depth of the triangle is below this: interp_depth's weights are not negative and sum to 1
// within 5 u (three conversions, products by one rounded reciprocal), its five operations add 3 u max |z|, and 32 u are
// taken.  Where a depth is not finite there is no bound.
__device__ __forceinline__ float depth_floor(const PVert (&v)[3]) {
  const float lo = fminf(v[0].z, fminf(v[1].z, v[2].z));
  const float far = fmaxf(fabsf(v[0].z), fmaxf(fabsf(v[1].z), fabsf(v[2].z)));
  const float d = lo - (2e-6f * far + 1e-37f);
  return d > -3.4e38f && d < 3.4e38f ? d : -INFINITY;
}

// This thread's pixel of the tile: 8 x 4 blocks per warp.
__device__ __forceinline__ int pixel_dx() { return ((threadIdx.x >> 5) & 1) * 8 + (threadIdx.x & 7); }
__device__ __forceinline__ int pixel_dy() { return (threadIdx.x >> 6) * 4 + ((threadIdx.x >> 3) & 3); }

// Visible triangle of every pixel of a tile for NS sides.  A bin of one chunk is set up in shared memory
// and each pixel tests the triangles whose box holds it (warps skip those that miss their block); of a larger
// one the triangles of small boxes (dense meshes) go into the pixels of their boxes, a triangle per lane, and only
// the others are set up and tested as before (by lane alone, a render of 100 K triangles grown over a 512^2
// image walks up to 256 pixels in a lane: 9.96 ms an iteration of 8 pairs, this 4.4 ms, testing all of them 6.3 ms), unless the
// triangle lies behind what the pixel has already (8 pairs of 2,048 triangles of half a 512^2 image: 17.4 -> 6.9 ms; most of such a
// test is the depth, three conversions from 64 bits).  Bound by instruction issue;
// 64-bit tests of every binned triangle at every pixel, and a second set-up per pixel, took 190 us for a view
// of 32,768 triangles at 1024^2 (Lambert) where this takes 84 us.
template <int NS>
__device__ __forceinline__ void raster_tile(const SceneDev& S, const Workspace& ws, RSmem<NS>& sm, int slot, int tile,
                                            uint64_t key, const int (&sides)[NS], Hit (&hit)[NS], int rx, int ry,
                                            bool surfaces = false) {
  const int ntl = n_tiles(S), tid = threadIdx.x, dx = pixel_dx(), dy = pixel_dy();
  const uint32_t block = (0xFFu << (dx & 8)) | (0xF0000u << (dy & 12));
  const uint32_t beg = ws.tile_off[slot * ntl + tile];
  int nb = (int)ws.tile_count[slot * ntl + tile];
  // after a bin overflow (reported in the status word) the tile's list was not stored
  if ((long long)beg + nb > ws.bin_capacity) nb = 0;
#pragma unroll
  for (int s = 0; s < NS; ++s) hit[s].key = ~0ull, hit[s].slot = -1;
  if (nb == 0) return;
  auto project_side = [&](int tri, int s, PVert (&v)[3]) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float3 q = perturbed_pos(S, vert_of(S, tri, k), key, sides[s]);
      v[k] = project(sm.m, q.x, q.y, q.z, S.W, S.H, S.near_w);
    }
  };
  if (nb <= RCHUNK) {
    if (tid < nb) {
      const int tri = (int)bin_at(S, ws, beg + tid);
      sm.tri[tid] = tri;
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        PVert v[3];
        project_side(tri, s, v);
        set_up_side(sm.t[s][tid], v, rx, ry);
        sm.span[tid][s] = v[0].ok && v[1].ok && v[2].ok ? box_span(v, rx, ry, 0) : 0u;
      }
      if constexpr (NS == 1)
        if (surfaces) load_surface(S, tri, key, sides[0], sm.uv[tid], sm.fr[tid]);
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      int& best = hit[s].slot;
      for_spans(sm.span, s, nb, block, dx, dy, [&](int j) {
        float l[3];
        float4 z;
        if (!cover_lambdas(sm.t[s][j], dx * 256, dy * 256, l, z)) return;
        const float zz[3] = {z.x, z.y, z.z};
        const unsigned long long k = ((unsigned long long)ordered_bits(interp_depth(l, zz)) << 32) | (uint32_t)sm.tri[j];
        if (k >= hit[s].key) return;
        hit[s].key = k;
        hit[s].l[0] = l[0], hit[s].l[1] = l[1], hit[s].l[2] = l[2];
        best = j;
      });
      if (best >= 0) {
        const float4 iw = sm.t[s][best].iw;
        hit[s].iw[0] = iw.x, hit[s].iw[1] = iw.y, hit[s].iw[2] = iw.z;
      }
    }
    return;
  }
#pragma unroll
  for (int s = 0; s < NS; ++s) sm.keys[s][tid] = ~0ull;
  for (int c0 = 0; c0 < nb; c0 += RCHUNK) {
    const int cnt = min(RCHUNK, nb - c0);
    bool staged = false;
    __syncthreads();  // the keys are empty, the last chunk's set-ups are done with
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      uint32_t span = 0u;
      if (tid < cnt) {
        const int tri = (int)bin_at(S, ws, beg + c0 + tid);
        PVert v[3];
        project_side(tri, s, v);
        int4 q[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) q[k] = make_int4(v[k].ok ? v[k].X : kNotDrawn, v[k].Y, __float_as_int(v[k].z), 0);
        int xa, xb, ya, yb;
        if (tri_box(q[0], q[1], q[2], rx, ry, xa, xb, ya, yb)) {
          if ((xb - xa + 1) * (yb - ya + 1) <= kLaneBox) {
            raster_tri(q[0], q[1], q[2], tri, rx, ry, xa, xb, ya, yb, sm.keys[s]);
          } else {
            set_up_side(sm.t[s][tid], v, rx, ry);
            sm.t[s][tid].iw.x = __uint_as_float(ordered_bits(depth_floor(v)));  // (1 / w is formed again below)
            span = box_span(v, rx, ry, 0);
            sm.tri[tid] = tri;
            staged = true;
          }
        }
      }
      sm.span[tid][s] = span;
      __syncwarp();
    }
    if (!__syncthreads_or(staged)) continue;
#pragma unroll
    for (int s = 0; s < NS; ++s)
      for_spans(sm.span, s, cnt, block, dx, dy, [&](int j) {
        if (__float_as_uint(sm.t[s][j].iw.x) > (uint32_t)(hit[s].key >> 32)) return;
        float l[3];
        float4 z;
        if (!cover_lambdas(sm.t[s][j], dx * 256, dy * 256, l, z)) return;
        const float zz[3] = {z.x, z.y, z.z};
        const unsigned long long k = ((unsigned long long)ordered_bits(interp_depth(l, zz)) << 32) | (uint32_t)sm.tri[j];
        hit[s].key = min(hit[s].key, k);
      });
  }
  __syncthreads();
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    hit[s].key = min(hit[s].key, sm.keys[s][dy * TILE + dx]);
    if (hit[s].key == ~0ull) continue;
    PVert v[3];
    project_side((int)(uint32_t)hit[s].key, s, v);
    SideTri d;
    set_up_side(d, v, rx, ry);
    float4 z;
    cover_lambdas(d, dx * 256, dy * 256, hit[s].l, z);
#pragma unroll
    for (int k = 0; k < 3; ++k) hit[s].iw[k] = v[k].iw;
  }
}

// Shade what a pixel sees; the triangle's UVs and frame come from the staged chunk where it is one.
__device__ __forceinline__ void surface_hit(const SceneDev& S, int view, const RSmem<1>& sm, const Hit& hit, uint64_t key,
                                            int side, Surf& sf) {
  const int tri = (int)(uint32_t)hit.key;
  if (hit.slot >= 0) {
    surface(S, view, tri, hit.l, hit.iw, sm.uv[hit.slot], sm.fr[hit.slot], key, side, sf);
    return;
  }
  float uv[6], fr[6];
  load_surface(S, tri, key, side, uv, fr);
  surface(S, view, tri, hit.l, hit.iw, uv, fr, key, side, sf);
}

__global__ void __launch_bounds__(TILE_PX, 4) k_render(SceneDev S, Workspace ws, int slot, int view, uint64_t key,
                                                    int side, unsigned long long* keys, float2* uv, float* rgb) {
  __shared__ RSmem<1> sm;
  const int tile = blockIdx.x;
  const int tx = tile % S.tiles_x, ty = tile / S.tiles_x;
  const int px = tx * TILE + pixel_dx(), py = ty * TILE + pixel_dy();
  if (threadIdx.x < 16) sm.m[threadIdx.x] = S.mvp[16 * view + threadIdx.x];
  __syncthreads();
  Hit hit[1];
  const int sides[1] = {side};
  raster_tile<1>(S, ws, sm, slot, tile, key, sides, hit, 256 * (tx * TILE) + 128, 256 * (ty * TILE) + 128, rgb != nullptr || uv != nullptr);
  if (px >= S.W || py >= S.H) return;
  const long long p = (long long)py * S.W + px;
  if (keys) keys[p] = hit[0].key;
  if (hit[0].key == ~0ull) {
    if (uv) uv[p] = make_float2(0.f, 0.f);
    if (rgb) rgb[3 * p] = S.bg[0], rgb[3 * p + 1] = S.bg[1], rgb[3 * p + 2] = S.bg[2];
    return;
  }
  if (!uv && !rgb) return;
  Surf sf;
  surface_hit(S, view, sm, hit[0], key, side, sf);
  if (uv) uv[p] = make_float2(sf.u, sf.v);
  if (rgb) rgb[3 * p] = sf.rgb.x, rgb[3 * p + 1] = sf.rgb.y, rgb[3 * p + 2] = sf.rgb.z;
}

// Unperturbed render of one view reduced to its image error f = sum_p || I_p(theta) - I_p ||^2
// (Table 1): the forward value of the autograd form.  Adds the view's sum to loss[slot].
__global__ void __launch_bounds__(TILE_PX, 4) k_render_loss(SceneDev S, Workspace ws, int slot, int view, float* loss) {
  __shared__ RSmem<1> sm;
  __shared__ float red[TILE_PX / 32];
  const int tile = blockIdx.x;
  const int tx = tile % S.tiles_x, ty = tile / S.tiles_x;
  const int px = tx * TILE + pixel_dx(), py = ty * TILE + pixel_dy();
  if (threadIdx.x < 16) sm.m[threadIdx.x] = S.mvp[16 * view + threadIdx.x];
  __syncthreads();
  Hit hit[1];
  const int sides[1] = {0};
  raster_tile<1>(S, ws, sm, slot, tile, 0, sides, hit, 256 * (tx * TILE) + 128, 256 * (ty * TILE) + 128, true);
  float f = 0.0f;
  if (px < S.W && py < S.H) {
    float3 c = f3(S.bg[0], S.bg[1], S.bg[2]);
    if (hit[0].key != ~0ull) {
      Surf sf;
      surface_hit(S, view, sm, hit[0], 0, 0, sf);
      c = sf.rgb;
    }
    const float* tp = S.targets + (((long long)view * S.H + py) * S.W + px) * 3;
    const float d0 = c.x - __ldg(tp), d1 = c.y - __ldg(tp + 1), d2 = c.z - __ldg(tp + 2);
    f = d0 * d0 + d1 * d1 + d2 * d2;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = f;
  __syncthreads();
  if (threadIdx.x == 0) {
    float sum = 0.0f;
    for (int i = 0; i < TILE_PX / 32; ++i) sum += red[i];
    atomicAdd(loss + slot, sum);
  }
}

// Plain path, step R: both sides' depth|ID and UV buffers of one estimate.
__global__ void __launch_bounds__(TILE_PX, 3) k_raster_pair(SceneDev S, Workspace ws, int slot, int view, uint64_t key) {
  __shared__ RSmem<2> sm;
  const int tile = blockIdx.x;
  const int tx = tile % S.tiles_x, ty = tile / S.tiles_x;
  const int px = tx * TILE + pixel_dx(), py = ty * TILE + pixel_dy();
  if (threadIdx.x < 16) sm.m[threadIdx.x] = S.mvp[16 * view + threadIdx.x];
  __syncthreads();
  Hit hit[2];
  const int sides[2] = {1, -1};
  raster_tile<2>(S, ws, sm, slot, tile, key, sides, hit, 256 * (tx * TILE) + 128, 256 * (ty * TILE) + 128);
  if (px >= S.W || py >= S.H) return;
  const long long npx = (long long)S.W * S.H, p = (long long)py * S.W + px;
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    ws.keys[s * npx + p] = hit[s].key;
    float2 uvv = make_float2(0.f, 0.f);
    if (hit[s].key != ~0ull) {
      const int tri = (int)(uint32_t)hit[s].key;
      PerspW pw = persp(hit[s].l, hit[s].iw);
      int t0 = uv_of(S, tri, 0), t1 = uv_of(S, tri, 1), t2 = uv_of(S, tri, 2);
      uvv.x = persp_interp(pw, __ldg(S.uvs + 2 * t0), __ldg(S.uvs + 2 * t1), __ldg(S.uvs + 2 * t2));
      uvv.y = persp_interp(pw, __ldg(S.uvs + 2 * t0 + 1), __ldg(S.uvs + 2 * t1 + 1), __ldg(S.uvs + 2 * t2 + 1));
    }
    ws.uvbuf[s * npx + p] = uvv;
  }
}

// Plain path, step G part 1: shade both sides from the buffers, f+ - f- per pixel.
__global__ void k_shade_delta(SceneDev S, Workspace ws, int view, uint64_t key, float* loss, float loss_scale,
                              int slot) {
  const long long npx = (long long)S.W * S.H;
  const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  float lv = 0.0f;
  if (p < npx) {
    const int px = (int)(p % S.W), py = (int)(p / S.W);
    const int tx = px / TILE, ty = py / TILE;
    const long long rx = 256ll * (tx * TILE) + 128, ry = 256ll * (ty * TILE) + 128;
    const float* m = S.mvp + 16 * view;
    float3 col[2];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      col[s] = f3(S.bg[0], S.bg[1], S.bg[2]);
      unsigned long long k = ws.keys[s * npx + p];
      if (k == ~0ull) continue;
      const int tri = (int)(k & 0xFFFFFFFFu), side = s == 0 ? 1 : -1;
      Tri t;
      setup_from_scene(S, m, tri, key, side, rx, ry, t);
      long long e[3];
      cover(t, px - tx * TILE, py - ty * TILE, e);
      float l[3];
      lambdas(e, t.inv_area, l);
      float uv[6], fr[6];
      load_surface(S, tri, key, side, uv, fr);
      Surf sf;
      surface(S, view, tri, l, t.iw, uv, fr, key, side, sf);
      col[s] = sf.rgb;
    }
    const float* tp = S.targets + ((long long)view * npx + p) * 3;
    float fp, fm;
    ws.dfbuf[p] = loss_diff(col[0], col[1], f3(__ldg(tp), __ldg(tp + 1), __ldg(tp + 2)), fp, fm);
    lv = 0.5f * (fp + fm);
  }
  if (loss) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) lv += __shfl_xor_sync(0xffffffffu, lv, o);
    if ((threadIdx.x & 31) == 0 && lv != 0.0f) atomicAdd(loss + slot, lv * loss_scale);
  }
}

// Plain path, step G part 2: AtomicAdd of (f+ - f-) s_i into every contributing parameter.
__global__ void k_scatter(SceneDev S, Workspace ws, uint64_t key, float* grad, uint32_t* counts) {
  const long long npx = (long long)S.W * S.H;
  const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= npx) return;
  int tris[2];
  Foot foot[2][MAX_READ];
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    unsigned long long k = ws.keys[s * npx + p];
    tris[s] = k == ~0ull ? -1 : (int)(k & 0xFFFFFFFFu);
    if (tris[s] < 0) continue;
    float2 uv = ws.uvbuf[s * npx + p];
#pragma unroll
    for (int r = 0; r < MAX_READ; ++r)
      if (r < S.nread) {
        const TexDev& T = S.tex[S.read_k[r]];
        foot[s][r] = footprint(uv.x, uv.y, T.w, T.h);
        if (S.foot_nearest) foot[s][r].nearest = nearest_texel(uv.x, uv.y, T.w, T.h);
      }
  }
  const float df = ws.dfbuf[p];
  for_each_contrib(S, tris, foot, [&](uint32_t ck) {
    long long base;
    int nch;
    key_params(S, ck, base, nch);
    const uint32_t sb = sign_bits(key, (uint64_t)base, nch);
    for (int c = 0; c < nch; ++c) {
      if (!CHK(S, base + c, S.chk.params)) continue;
      atomicAdd(grad + base + c, ((sb >> c) & 1) ? -df : df);
      atomicAdd(counts + base + c, 1u);
    }
  });
}

// Full-image estimator (Eq. 4), step G: the estimate's whole-image loss difference
// sum_p (f+_p - f-_p), from the staged per-pixel differences, added to *out.
__global__ void __launch_bounds__(256) k_reduce_image(const float* df, long long npx, float* out) {
  __shared__ float red[8];
  float v = 0.0f;
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < npx; p += (long long)gridDim.x * blockDim.x)
    v += df[p];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    float sum = 0.0f;
    for (int i = 0; i < 8; ++i) sum += red[i];
    atomicAdd(out, sum);
  }
}

__global__ void k_validate(SceneDev S, uint32_t* status) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 3ll * S.nt) return;
  const int pv = S.pidx[i], uv = S.uvidx[i];
  bool bad = pv < 0 || pv >= S.nv || uv < 0 || uv >= S.nuv;
  if (bad) atomicCAS(status, 0u, (uint32_t)SGE_ERR_BAD_INDEX);
}

}  // namespace

cudaError_t launch_render(const SceneDev& S, const Workspace& ws, int slot, int view, uint64_t key, int side,
                          unsigned long long* keys, float2* uv, float* rgb, cudaStream_t st) {
  k_render<<<n_tiles(S), TILE_PX, 0, st>>>(S, ws, slot, view, key, side, keys, uv, rgb);
  return cudaGetLastError();
}

cudaError_t launch_render_loss(const SceneDev& S, const Workspace& ws, int slot, int view, float* loss,
                               cudaStream_t st) {
  k_render_loss<<<n_tiles(S), TILE_PX, 0, st>>>(S, ws, slot, view, loss);
  return cudaGetLastError();
}

cudaError_t launch_plain_pair(const SceneDev& S, const Workspace& ws, int slot, int view, uint64_t key,
                              const EstimateArgs& a, float loss_scale, cudaStream_t st) {
  const long long npx = (long long)S.W * S.H;
  const int blocks = (int)((npx + 255) / 256);
  k_raster_pair<<<n_tiles(S), TILE_PX, 0, st>>>(S, ws, slot, view, key);
  k_shade_delta<<<blocks, 256, 0, st>>>(S, ws, view, key, a.loss, loss_scale, slot);
  k_scatter<<<blocks, 256, 0, st>>>(S, ws, key, a.grad, a.counts);
  return cudaGetLastError();
}

cudaError_t launch_image_delta(const SceneDev& S, const Workspace& ws, int slot, int view, uint64_t key, float* out,
                               cudaStream_t st) {
  const long long npx = (long long)S.W * S.H;
  const int blocks = (int)((npx + 255) / 256);
  k_raster_pair<<<n_tiles(S), TILE_PX, 0, st>>>(S, ws, slot, view, key);
  k_shade_delta<<<blocks, 256, 0, st>>>(S, ws, view, key, nullptr, 0.0f, slot);
  k_reduce_image<<<blocks < 1024 ? blocks : 1024, 256, 0, st>>>(ws.dfbuf, npx, out);
  return cudaGetLastError();
}

cudaError_t launch_validate(const SceneDev& S, uint32_t* status, cudaStream_t st) {
  const long long n = 3ll * S.nt;
  k_validate<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(S, status);
  return cudaGetLastError();
}

}  // namespace sge
