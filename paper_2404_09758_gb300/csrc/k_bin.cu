// Tile binning shared by every pair and both sides of an estimate.
//
// The paper's rasterizer R (Section 4.3) renders theta + s eps and theta - s eps
// for every estimate.  All those scenes differ from theta by at most eps_pos per
// vertex coordinate, so one binning per view and call serves every render of
// that view: each triangle is binned into the tiles its screen bounding box can
// reach under any such perturbation (interval bounds of the projection plus a
// one-pixel margin).  A render then tests, per tile, only the triangles in the
// tile's bin, with the exact perturbed vertices.
#include <cuda_runtime.h>

#define SGE_FILE_ID 1  // range-check sites of this file (checked build)
#include "sge_device.cuh"

namespace sge {

namespace {

// Interval of one clip coordinate row of M over the box p +- eps (per coordinate).
__device__ __forceinline__ float clip_interval(const float* m, float x, float y, float z, float eps, float& lo,
                                               float& hi) {
  float c = m[0] * x + m[1] * y + m[2] * z + m[3];
  float r = eps * (fabsf(m[0]) + fabsf(m[1]) + fabsf(m[2]));
  r = r * 1.0001f + 1e-6f * (fabsf(c) + fabsf(m[3]) + 1.0f);
  lo = c - r;
  hi = c + r;
  return c;
}

__global__ void k_bin_rect_count(SceneDev S, Workspace ws, ViewList vl) {
  __shared__ float m[16];
  int slot = blockIdx.y;
  int view = vl.id[slot];
  // the call's counters: items and their work counters, bin entries (the status word stays)
  if (blockIdx.x == 0 && slot == 0 && threadIdx.x < 7 && threadIdx.x != 3) ws.counters[threadIdx.x] = 0u;
  if (blockIdx.x == 0 && slot == 0 && threadIdx.x == 7) *bin_total(ws) = 0ull;
  if (threadIdx.x < 16) m[threadIdx.x] = S.mvp[16 * view + threadIdx.x];
  __syncthreads();
  int tri = blockIdx.x * blockDim.x + threadIdx.x;
  if (tri >= S.nt) return;
  int vi[3] = {vert_of(S, tri, 0), vert_of(S, tri, 1), vert_of(S, tri, 2)};
  int4 rect = make_int4(1, 1, 0, 0);  // empty
  bool skip = vi[0] == vi[1] || vi[1] == vi[2] || vi[0] == vi[2];  // welded duplicates: zero area always
  // a triangle with an index out of range is never binned, so no render reads through it
  for (int k = 0; k < 3; ++k) {
    const int ti = uv_of(S, tri, k);
    if (ti < 0 || ti >= S.nuv) skip = true;
  }
  float sx0 = 3.4e38f, sx1 = -3.4e38f, sy0 = 3.4e38f, sy1 = -3.4e38f;
  float disp = 0.0f;  // widest screen interval of a vertex under the perturbation, pixels
  float zlo = 3.4e38f, zhi = -3.4e38f;  // depth interval of the triangle under the perturbation
  bool full = false;
  for (int k = 0; k < 3 && !skip; ++k) {
    if (vi[k] < 0 || vi[k] >= S.nv) { skip = true; break; }
    const float* p = S.pos + 3ll * vi[k];
    float x = p[0], y = p[1], z = p[2];
    float xl, xh, yl, yh, zl, zh, wl, wh;
    const float cx = clip_interval(m + 0, x, y, z, S.eps_pos, xl, xh);
    const float cy = clip_interval(m + 4, x, y, z, S.eps_pos, yl, yh);
    clip_interval(m + 8, x, y, z, S.eps_pos, zl, zh);
    const float cw = clip_interval(m + 12, x, y, z, S.eps_pos, wl, wh);
    if (wh <= S.near_w) { skip = true; break; }  // always behind the near limit: triangle never drawn
    if (wl <= S.near_w) {
      // may or may not be drawn: bin everywhere, at any depth (a bound without this vertex would rank the triangle
      // behind ones it hides, and the search for the nearest would end before it)
      full = true;
      zlo = -3.4e38f;
      zhi = 3.4e38f;
      continue;
    }
    float nx0 = fminf(fminf(xl / wl, xl / wh), fminf(xh / wl, xh / wh));
    float nx1 = fmaxf(fmaxf(xl / wl, xl / wh), fmaxf(xh / wl, xh / wh));
    float ny0 = fminf(fminf(yl / wl, yl / wh), fminf(yh / wl, yh / wh));
    float ny1 = fmaxf(fmaxf(yl / wl, yl / wh), fmaxf(yh / wl, yh / wh));
    zlo = fminf(zlo, fminf(fminf(zl / wl, zl / wh), fminf(zh / wl, zh / wh)));
    zhi = fmaxf(zhi, fmaxf(fmaxf(zl / wl, zl / wh), fmaxf(zh / wl, zh / wh)));
    const float vx0 = (nx0 * 0.5f + 0.5f) * S.W, vx1 = (nx1 * 0.5f + 0.5f) * S.W;
    const float vy0 = (0.5f - ny1 * 0.5f) * S.H, vy1 = (0.5f - ny0 * 0.5f) * S.H;
    sx0 = fminf(sx0, vx0);
    sx1 = fmaxf(sx1, vx1);
    sy0 = fminf(sy0, vy0);
    sy1 = fmaxf(sy1, vy1);
    // farthest any perturbed screen position lies from the unperturbed one
    const float ux = (cx / cw * 0.5f + 0.5f) * S.W, uy = (0.5f - cy / cw * 0.5f) * S.H;
    disp = fmaxf(disp, fmaxf(fmaxf(vx1 - ux, ux - vx0), fmaxf(vy1 - uy, uy - vy0)));
    // near the guard band the drop rule may flip under the perturbation
    if (!(fmaxf(fabsf(vx0), fabsf(vx1)) < 30000.0f && fmaxf(fabsf(vy0), fabsf(vy1)) < 30000.0f)) full = true;
  }
  // Margin (fixed-point units) that bounds, per axis, how far any snapped perturbed
  // vertex can be from the snapped unperturbed one: the farthest interval end, one
  // unit for the two snaps and slack for float rounding; "full" = unbounded.
  int margin = 0x7FFFFFFF;
  if (!full && !skip && disp < 1.0e4f) margin = (int)ceilf(disp * 256.0f * 1.002f) + 4;
  if (ws.tri_rec && !skip) {
    PVert v[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float* p = S.pos + 3ll * vi[k];
      v[k] = project(m, p[0], p[1], p[2], S.W, S.H, S.near_w);
    }
    int4* rec = ws.tri_rec + 2 * ((long long)slot * S.nt + tri);
    rec[0] = make_int4(v[0].X, v[0].Y, v[1].X, v[1].Y);
    rec[1] = make_int4(v[2].X, v[2].Y, margin, v[0].ok && v[1].ok && v[2].ok ? 1 : 0);
  }
  // interpolated depth of a covered pixel lies between the vertex depths; slack for float rounding
  ws.tri_z[(long long)slot * S.nt + tri] =
      make_float2(zlo - (1e-6f + 1e-5f * fabsf(zlo)), zhi + (1e-6f + 1e-5f * fabsf(zhi)));
  if (!skip) {
    int px0, px1, py0, py1;
    if (full) {
      px0 = 0; py0 = 0; px1 = S.W - 1; py1 = S.H - 1;
    } else {
      // pixel centres px + 0.5 inside [sx0, sx1], one pixel of margin each way
      px0 = (int)fmaxf(floorf(sx0) - 1.0f, 0.0f);
      py0 = (int)fmaxf(floorf(sy0) - 1.0f, 0.0f);
      px1 = (int)fminf(floorf(sx1) + 1.0f, (float)(S.W - 1));
      py1 = (int)fminf(floorf(sy1) + 1.0f, (float)(S.H - 1));
    }
    if (px0 <= px1 && py0 <= py1) rect = make_int4(px0 / TILE, py0 / TILE, px1 / TILE, py1 / TILE);
  }
  ws.tri_rect[(long long)slot * S.nt + tri] = rect;
  int nt = n_tiles(S);
  for (int ty = rect.y; ty <= rect.w; ++ty)
    for (int tx = rect.x; tx <= rect.z; ++tx)
      atomicAdd(ws.tile_count + (long long)slot * nt + ty * S.tiles_x + tx, 1u);
}

// Each (slot, tile)'s place in the bins: a CTA's 1,024 counts are scanned and the CTA takes its range
// from the running total, in whatever order the CTAs come; then the fill cursors.  Nothing
// needs the tiles in order, and one CTA scanning every count of a call serially took 12.5 us for
// 8,192 counts and 160 us for 65,536 (both 3 us here).
__global__ void __launch_bounds__(1024) k_bin_place(Workspace ws, int n, int n_triangles) {
  __shared__ unsigned long long wsum[32], base;
  const int i = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t c = i < n ? ws.tile_count[i] : 0u;
  unsigned long long x = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[wid] = x;
  __syncthreads();
  if (wid == 0) {
    unsigned long long w = wsum[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    wsum[lane] = w;
    if (lane == 31) {
      base = atomicAdd(bin_total(ws), w);
      if (base + w > (unsigned long long)ws.bin_capacity) atomicCAS(ws.counters + 3, 0u, (uint32_t)SGE_ERR_BIN_OVERFLOW);
    }
  }
  __syncthreads();
  if (i >= n) return;
  const uint32_t off = bin_start(base + (wid ? wsum[wid - 1] : 0ull) + x - c, c, ws.bin_capacity);
  ws.tile_off[i] = off;
  ws.tile_cur[i] = bin_cursor(off, n_triangles);
}

__global__ void k_bin_fill(SceneDev S, Workspace ws) {
  int slot = blockIdx.y;
  int tri = blockIdx.x * blockDim.x + threadIdx.x;
  if (tri >= S.nt) return;
  int4 rect = ws.tri_rect[(long long)slot * S.nt + tri];
  int nt = n_tiles(S);
  auto fill = [&](auto stores) {
    for (int ty = rect.y; ty <= rect.w; ++ty)
      for (int tx = rect.x; tx <= rect.z; ++tx) {
        const long long t = (long long)slot * nt + ty * S.tiles_x + tx;
        const uint32_t pos = atomicAdd(ws.tile_cur + t, 1u);
        if (stores(pos, t) && CHK(S, pos, S.chk.bins)) ws.bins[pos] = (uint32_t)tri;
      }
  };
  // (apart, so that the usual loop reads nothing: a large triangle's is a chain of atomics)
  if (cursors_above(ws.bin_capacity, S.nt))
    fill([&](uint32_t pos, long long) { return (long long)pos < ws.bin_capacity; });
  else
    fill([&](uint32_t pos, long long t) { return (long long)pos < ws.bin_capacity && ws.tile_off[t] != kNoBin; });
}

}  // namespace

cudaError_t launch_binning(const SceneDev& S, const Workspace& ws, const ViewList& vl, cudaStream_t st, bool prune,
                           bool defer_prune) {
  int nt = n_tiles(S);
  cudaError_t e = cudaMemsetAsync(ws.tile_count, 0, sizeof(uint32_t) * (size_t)vl.n * nt, st);
  if (e != cudaSuccess) return e;
  dim3 grid((S.nt + 255) / 256, vl.n);
  // (only the pruning reads the records: three projections and 32 B a triangle and view less without it)
  Workspace counted = ws;
  if (!prune) counted.tri_rec = nullptr;
  k_bin_rect_count<<<grid, 256, 0, st>>>(S, counted, vl);
  k_bin_place<<<(vl.n * nt + 1023) / 1024, 1024, 0, st>>>(ws, vl.n * nt, S.nt);
  k_bin_fill<<<grid, 256, 0, st>>>(S, ws);
  e = cudaGetLastError();
  if (e == cudaSuccess && prune && !defer_prune) e = launch_prune(S, ws, vl, st);
  return e;
}

}  // namespace sge
