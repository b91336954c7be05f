// Device building blocks shared by the estimator, staged and binning kernels.
//
// Bit-exactness: every float operation whose result decides an integer (the
// snapped screen position, the depth that picks the visible triangle, the UV
// that picks texels) is written with an explicit round-to-nearest intrinsic
// (__fmul_rn, __fadd_rn, __fdiv_rn, ...), which the compiler never fuses into an
// FMA, so the result is the same whichever kernel evaluates it.  Coverage uses
// exact 64-bit integer edge functions.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "sge_internal.h"

namespace sge {

// ---------------------------------------------------------------- range checks (checked build)
// Is 0 <= i < n?  The unchecked build assumes so (the host validates what it can); the checked
// build tests it and, when it fails, records SGE_ERR_BOUNDS in the status word so that the caller
// skips the access.
// The first failing check also records its site (file id * 100000 + line) and the index.
__device__ __forceinline__ bool chk(const SceneDev& S, long long i, long long n, int site) {
#if SGE_CHECKED
  if (i >= 0 && i < n) return true;
  atomicCAS(S.chk.status, 0u, (uint32_t)SGE_ERR_BOUNDS);
  if (S.chk.where && atomicCAS(S.chk.where, 0u, (uint32_t)site) == 0u) S.chk.where[1] = (uint32_t)i;
  return false;
#else
  (void)S;
  (void)i;
  (void)n;
  (void)site;
  return true;
#endif
}
#ifndef SGE_FILE_ID
#define SGE_FILE_ID 0
#endif
#define CHK(S_, i_, n_) chk(S_, i_, n_, SGE_FILE_ID * 100000 + __LINE__)
#define CHK_H(S_, i_, n_) chk(S_, i_, n_, 900000 + __LINE__)

// Vertex / UV index k of triangle tri (a failing check reads as index 0).
__device__ __forceinline__ int vert_of(const SceneDev& S, int tri, int k) {
  const int v = __ldg(S.pidx + 3 * tri + k);
  return CHK_H(S, v, S.chk.nv) ? v : 0;
}
__device__ __forceinline__ int uv_of(const SceneDev& S, int tri, int k) {
  const int t = __ldg(S.uvidx + 3 * tri + k);
  return CHK_H(S, t, S.chk.nuv) ? t : 0;
}

// Bin entry i (a failing check reads as triangle 0).
__device__ __forceinline__ uint32_t bin_at(const SceneDev& S, const Workspace& ws, long long i) {
  return CHK_H(S, i, S.chk.bins) ? ws.bins[i] : 0u;
}


// ---------------------------------------------------------------- sign hash (Algorithm 1)
// The paper draws s_i with a hash function it does not name.  This uses
// SplitMix64 (Steele, Lea & Flood 2014): mix64 is its output function; one
// generator step adds the golden-ratio increment and mixes.  The key of an
// estimate chains four steps over (seed, iteration, view, pair); s_i is bit
// (i mod 64) of the (floor(i / 64) + 1)-th output of the generator seeded with
// that key: one output gives the signs of 64 consecutive parameters.
constexpr uint64_t kGamma = 0x9E3779B97F4A7C15ull;

__host__ __device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__host__ __device__ __forceinline__ uint64_t pair_key(uint64_t seed, uint32_t iter, uint32_t view,
                                                      uint32_t pair) {
  uint64_t k = mix64(seed + kGamma);
  k = mix64((k ^ iter) + kGamma);
  k = mix64((k ^ view) + kGamma);
  return mix64((k ^ pair) + kGamma);
}

// true when s_i = -1
__device__ __forceinline__ bool sign_neg(uint64_t key, uint64_t i) {
  return ((mix64(key + ((i >> 6) + 1) * kGamma) >> (i & 63)) & 1) != 0;
}

// Bits 0..n-1 (n <= 32): s_{i0 + j} = -1, from the one or two generator outputs they lie in.
__device__ __forceinline__ uint32_t sign_bits(uint64_t key, uint64_t i0, int n) {
  const uint64_t blk = i0 >> 6;
  const int sh = (int)(i0 & 63);
  uint64_t x = mix64(key + (blk + 1) * kGamma) >> sh;
  if (sh + n > 64) x |= mix64(key + (blk + 2) * kGamma) << (64 - sh);
  return (uint32_t)x;
}

// ---------------------------------------------------------------- projection
// clip = M (x,y,z,1); screen = ((x/w)/2 + 1/2) W, (1/2 - (y/w)/2) H; snapped to
// 1/256 pixel with round-half-even.  A vertex needs w > near_w and |screen| < 2^15 px.
constexpr float kGuard = 8388608.0f;  // 2^23 fixed-point units

struct PVert {
  int X, Y;
  float z, iw;
  bool ok;
};

__device__ __forceinline__ float dot4_rn(const float* m, float x, float y, float z) {
  return __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(m[0], x), __fmul_rn(m[1], y)), __fmul_rn(m[2], z)),
                   m[3]);
}

__device__ __forceinline__ PVert project(const float* m, float x, float y, float z, int W, int H,
                                         float near_w) {
  PVert v;
  float cx = dot4_rn(m + 0, x, y, z), cy = dot4_rn(m + 4, x, y, z);
  float cz = dot4_rn(m + 8, x, y, z), cw = dot4_rn(m + 12, x, y, z);
  v.ok = cw > near_w;
  v.iw = __fdiv_rn(1.0f, cw);
  float xn = __fmul_rn(cx, v.iw), yn = __fmul_rn(cy, v.iw);
  v.z = __fmul_rn(cz, v.iw);
  float xs = __fmul_rn(__fadd_rn(__fmul_rn(xn, 0.5f), 0.5f), (float)W);
  float ys = __fmul_rn(__fsub_rn(0.5f, __fmul_rn(yn, 0.5f)), (float)H);
  float xf = __fmul_rn(xs, 256.0f), yf = __fmul_rn(ys, 256.0f);
  if (!(fabsf(xf) < kGuard) || !(fabsf(yf) < kGuard)) v.ok = false;
  v.X = v.ok ? __float2int_rn(xf) : 0;
  v.Y = v.ok ? __float2int_rn(yf) : 0;
  return v;
}

// int64 -> float, correctly rounded; values that fit 32 bits take the cheaper
// 32-bit conversion, which rounds the same value to the same float.
__device__ __forceinline__ float ll2f_rn(long long v) {
  return (v == (long long)(int)v) ? __int2float_rn((int)v) : __ll2float_rn(v);
}

// ---------------------------------------------------------------- triangle setup
// Edge function of the edge opposite vertex k (a = k+1, b = k+2 mod 3):
//   E_k(P) = (Xb-Xa)(Py-Ya) - (Yb-Ya)(Px-Xa),   E_0+E_1+E_2 = twice the signed area.
// After orienting to positive area, E_k = E_k(origin) + A_k dx + B_k dy exactly, with
// A_k = Ya-Yb, B_k = Xb-Xa (times the orientation).  Pixel centres inside: every
// E_k > 0, or E_k == 0 on a top or left edge (y grows downwards: left = A_k > 0,
// top = A_k == 0 && B_k > 0).
struct Tri {
  long long e0[3];  // oriented edge functions at the reference pixel centre
  int a[3], b[3];   // oriented per-unit steps in x and y (fixed-point units)
  int bias[3];      // 0 on top/left edges, -1 elsewhere: inside <=> e + bias >= 0
  float inv_area;   // 1 / (float)area
  float z[3], iw[3];
  int ok;
};

__device__ __forceinline__ long long edge_at(int Xa, int Ya, int Xb, int Yb, long long px,
                                             long long py) {
  return (long long)(Xb - Xa) * (py - Ya) - (long long)(Yb - Ya) * (px - Xa);
}

// Set up a triangle from its three projected vertices; (rx, ry) is the fixed-point
// reference point (a pixel centre) the edge functions are stored at.
__device__ __forceinline__ void setup_tri(const PVert& v0, const PVert& v1, const PVert& v2,
                                          long long rx, long long ry, Tri& t) {
  t.ok = v0.ok && v1.ok && v2.ok;
  if (!t.ok) return;
  long long area = edge_at(v0.X, v0.Y, v1.X, v1.Y, v2.X, v2.Y);
  if (area == 0) {
    t.ok = 0;
    return;
  }
  int sg = area > 0 ? 1 : -1;
  const PVert* v[3] = {&v0, &v1, &v2};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const PVert& A = *v[(k + 1) % 3];
    const PVert& B = *v[(k + 2) % 3];
    t.e0[k] = sg * edge_at(A.X, A.Y, B.X, B.Y, rx, ry);
    t.a[k] = sg * (A.Y - B.Y);
    t.b[k] = sg * (B.X - A.X);
    t.bias[k] = (t.a[k] > 0 || (t.a[k] == 0 && t.b[k] > 0)) ? 0 : -1;
  }
  t.inv_area = __fdiv_rn(1.0f, ll2f_rn(area > 0 ? area : -area));
  t.z[0] = v0.z; t.z[1] = v1.z; t.z[2] = v2.z;
  t.iw[0] = v0.iw; t.iw[1] = v1.iw; t.iw[2] = v2.iw;
}

__device__ __forceinline__ uint32_t ordered_bits(float z) {
  uint32_t b = __float_as_uint(z);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// Barycentric weights lambda_k = E_k / area as floats.
__device__ __forceinline__ void lambdas(const long long e[3], float inv_area, float l[3]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) l[k] = __fmul_rn(ll2f_rn(e[k]), inv_area);
}

__device__ __forceinline__ float interp_depth(const float l[3], const float z[3]) {
  return __fadd_rn(__fadd_rn(__fmul_rn(l[0], z[0]), __fmul_rn(l[1], z[1])), __fmul_rn(l[2], z[2]));
}

// Perspective-correct interpolation: q_k = lambda_k / w_k, value = sum q_k a_k / sum q_k.
struct PerspW {
  float q[3], qs;
};
__device__ __forceinline__ PerspW persp(const float l[3], const float iw[3]) {
  PerspW p;
#pragma unroll
  for (int k = 0; k < 3; ++k) p.q[k] = __fmul_rn(l[k], iw[k]);
  p.qs = __fadd_rn(__fadd_rn(p.q[0], p.q[1]), p.q[2]);
  return p;
}
__device__ __forceinline__ float persp_interp(const PerspW& p, float a0, float a1, float a2) {
  return __fdiv_rn(
      __fadd_rn(__fadd_rn(__fmul_rn(p.q[0], a0), __fmul_rn(p.q[1], a1)), __fmul_rn(p.q[2], a2)), p.qs);
}

// ---------------------------------------------------------------- texture footprint
// Texel centres at half-integers: x = u W - 1/2, x0 = floor(x), fx = x - x0; u wraps, v clamps.
struct Foot {
  int x0, x1, y0, y1;  // wrapped / clamped texel coordinates
  float fx, fy;
  int ix;              // floor(u W - 1/2) before wrapping (x0 = ix mod W, x1 = (ix + 1) mod W)
  int nearest;         // texel id of the nearest texel (set where SceneDev::foot_nearest asks for it)
};

// i mod n in [0, n); one add or subtract for the i in [-n, 2n) a texel lookup produces
__device__ __forceinline__ int wrap_i(int i, int n) {
  int r = i < 0 ? i + n : (i >= n ? i - n : i);
  if (r < 0 || r >= n) {
    r = i % n;
    r = r < 0 ? r + n : r;
  }
  return r;
}
__device__ __forceinline__ int clamp_i(int i, int n) { return i < 0 ? 0 : (i > n - 1 ? n - 1 : i); }

__device__ __forceinline__ Foot footprint(float u, float v, int W, int H) {
  Foot f;
  float x = __fsub_rn(__fmul_rn(u, (float)W), 0.5f);
  float y = __fsub_rn(__fmul_rn(v, (float)H), 0.5f);
  float xf = floorf(x), yf = floorf(y);
  f.fx = __fsub_rn(x, xf);
  f.fy = __fsub_rn(y, yf);
  int ix = (int)xf, iy = (int)yf;
  f.ix = ix;
  f.x0 = wrap_i(ix, W);
  f.x1 = wrap_i(ix + 1, W);
  f.y0 = clamp_i(iy, H);
  f.y1 = clamp_i(iy + 1, H);
  return f;
}

// The texels of the footprint named by a code, its first texel's id and kOneRow where its rows are clamped to
// one (w: the texture's width): columns x0, x1, rows y0, y1 (equal where it has one column or row).
constexpr uint32_t kOneRow = 1u << 28;
struct Quad {
  int x0, x1, y0, y1;
  __device__ __forceinline__ Quad(uint32_t cr, int w) {
    const int id = (int)(cr & 0x0FFFFFFFu);
    y0 = id / w;
    x0 = id - y0 * w;
    x1 = x0 + 1 == w ? 0 : x0 + 1;
    y1 = (cr & kOneRow) ? y0 : y0 + 1;
  }
  __device__ __forceinline__ int texel(int q, int w) const { return (q & 2 ? y1 : y0) * w + (q & 1 ? x1 : x0); }
  __device__ __forceinline__ bool repeats(int q) const { return ((q & 2) && y1 == y0) || ((q & 1) && x1 == x0); }
  __device__ __forceinline__ bool holds(const Quad& o, int q) const {
    const int x = q & 1 ? o.x1 : o.x0, y = q & 2 ? o.y1 : o.y0;
    return (x == x0 || x == x1) && (y == y0 || y == y1);
  }
};

// The texel whose square holds the sample point, (floor(u W) wrapped, floor(v H) clamped): the one
// texel Section 4.4 credits ("nearest" footprint); its id y W + x.
__device__ __forceinline__ int nearest_texel(float u, float v, int W, int H) {
  const int x = wrap_i((int)floorf(__fmul_rn(u, (float)W)), W);
  const int y = clamp_i((int)floorf(__fmul_rn(v, (float)H)), H);
  return y * W + x;
}

// ---------------------------------------------------------------- device scene view
// Sample all channels of perturbed texture T at footprint f (bilinear), float32.
__device__ __forceinline__ void sample_tex(const TexDev& T, const Foot& f, uint64_t key, int side,
                                           float out[4]) {
  float w[4] = {(1.0f - f.fx) * (1.0f - f.fy), f.fx * (1.0f - f.fy), (1.0f - f.fx) * f.fy,
                f.fx * f.fy};
  int tx[4] = {f.x0, f.x1, f.x0, f.x1};
  int ty[4] = {f.y0, f.y0, f.y1, f.y1};
#pragma unroll
  for (int c = 0; c < 4; ++c) out[c] = 0.0f;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    long long t = (long long)ty[j] * T.w + tx[j];
    const float* src = T.ptr + t * T.c;
    uint32_t sb = 0;
    float eps = 0.0f;
    if (side != 0) {
      sb = sign_bits(key, (uint64_t)(T.offset + t * T.c), T.c);
      eps = side < 0 ? -T.eps : T.eps;
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (c < T.c) {
        const float th = __ldg(src + c);
        out[c] += w[j] * (side == 0 ? th : __fadd_rn(th, ((sb >> c) & 1) ? -eps : eps));
      }
  }
  if (T.c == 1) out[1] = out[2] = out[0];
}

__device__ __forceinline__ float3 f3(float x, float y, float z) { return make_float3(x, y, z); }
__device__ __forceinline__ float3 sub3(float3 a, float3 b) { return f3(a.x - b.x, a.y - b.y, a.z - b.z); }
__device__ __forceinline__ float dot3(float3 a, float3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ float3 cross3(float3 a, float3 b) {
  return f3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}
__device__ __forceinline__ float3 norm3(float3 a) {
  float n = sqrtf(dot3(a, a));
  return n > 0.0f ? f3(a.x / n, a.y / n, a.z / n) : a;
}

// GGX colour for the shading normal n, light direction L and surface point P.
__device__ __forceinline__ float3 shade_ggx(const SceneDev& S, int view, float3 n, float3 L, const float* alb,
                                            float rough, float metal, float3 P) {
  // Cook-Torrance: GGX distribution, Smith-Schlick geometry (k = alpha/2), Schlick Fresnel.
  const float ndl = fmaxf(dot3(n, L), 0.0f);
  const float* cp = S.cam_pos + 3 * view;
  float3 V = norm3(f3(__ldg(cp) - P.x, __ldg(cp + 1) - P.y, __ldg(cp + 2) - P.z));
  float3 Hh = norm3(f3(L.x + V.x, L.y + V.y, L.z + V.z));
  float ndv = fmaxf(dot3(n, V), 1e-4f), ndh = fmaxf(dot3(n, Hh), 0.0f), vdh = fmaxf(dot3(V, Hh), 0.0f);
  float r = fminf(fmaxf(rough, 0.02f), 1.0f);
  float a = r * r, a2 = a * a;
  float dd = ndh * ndh * (a2 - 1.0f) + 1.0f;
  float D = a2 / (3.14159265358979f * dd * dd);
  float kk = 0.5f * a;
  float G = (ndl / (ndl * (1.0f - kk) + kk)) * (ndv / (ndv * (1.0f - kk) + kk));
  float mt = metal, om = 1.0f - vdh;
  float om5 = om * om * om * om * om;
  float out[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    float F0 = 0.04f * (1.0f - mt) + alb[c] * mt;
    float F = F0 + (1.0f - F0) * om5;
    float diff = (1.0f - F) * (1.0f - mt) * alb[c] * ndl * 0.318309886183791f;
    float spec = D * G * F / (4.0f * ndv);
    out[c] = S.light_rgb[c] * (diff + spec) + S.ambient * alb[c];
  }
  return f3(out[0], out[1], out[2]);
}

// Colour of a covered pixel of a lit model.  The shading normal is the tangent-space normal-map vector
// (2 t - 1) in the frame of the triangle's own perturbed geometry and UVs: N face normal, T along +u
// (Gram-Schmidt against N), B = N x T (tri_frame).  P: the surface point (GGX).
template <int SH>
__device__ __forceinline__ float3 shade_lit(const SceneDev& S, int view, const float* alb, const float* nm, float rough,
                                            float metal, float3 N, float3 T, float3 P) {
  const float3 B = cross3(N, T);
  const float mx = 2.0f * nm[0] - 1.0f, my = 2.0f * nm[1] - 1.0f, mz = 2.0f * nm[2] - 1.0f;
  float3 n = f3(T.x * mx + B.x * my + N.x * mz, T.y * mx + B.y * my + N.y * mz, T.z * mx + B.z * my + N.z * mz);
  if (dot3(n, n) == 0.0f) n = N;
  n = norm3(n);
  const float3 L = f3(S.light_dir[0], S.light_dir[1], S.light_dir[2]);
  if (SH == SHADE_LAMBERT) {
    const float ndl = fmaxf(dot3(n, L), 0.0f);
    return f3(alb[0] * (S.ambient + S.light_rgb[0] * ndl), alb[1] * (S.ambient + S.light_rgb[1] * ndl),
              alb[2] * (S.ambient + S.light_rgb[2] * ndl));
  }
  return shade_ggx(S, view, n, L, alb, rough, metal, P);
}

// ---------------------------------------------------------------- one visible surface sample
// Everything about a pixel seen through one triangle on one side: UV, colour,
// footprints of the textures the shading reads.
struct Surf {
  float u, v;
  float3 rgb;
  Foot foot[MAX_READ];  // footprint of each read texture, in read_k order
};

// Perturbed world position of welded vertex vi.
__device__ __forceinline__ float3 perturbed_pos(const SceneDev& S, int vi, uint64_t key, int side) {
  const float* p = S.pos + 3ll * vi;
  const float x = __ldg(p), y = __ldg(p + 1), z = __ldg(p + 2);
  if (side == 0) return f3(x, y, z);
  const uint32_t sb = sign_bits(key, 3ull * (uint64_t)vi, 3);
  const float e = side < 0 ? -S.eps_pos : S.eps_pos;
  return f3(__fadd_rn(x, (sb & 1) ? -e : e), __fadd_rn(y, (sb & 2) ? -e : e), __fadd_rn(z, (sb & 4) ? -e : e));
}

// Face normal N and u tangent T of a triangle : the same for every pixel.
__device__ __forceinline__ void tri_frame(const float3 p[3], const float* uv, float* out) {
  const float3 e1 = sub3(p[1], p[0]), e2 = sub3(p[2], p[0]);
  const float3 N = norm3(cross3(e1, e2));
  const float du1 = uv[2] - uv[0], dv1 = uv[3] - uv[1], du2 = uv[4] - uv[0], dv2 = uv[5] - uv[1];
  const float det = du1 * dv2 - du2 * dv1;
  float3 T = det != 0.0f ? f3((e1.x * dv2 - e2.x * dv1) / det, (e1.y * dv2 - e2.y * dv1) / det,
                              (e1.z * dv2 - e2.z * dv1) / det)
                         : e1;
  const float nt = dot3(N, T);
  T = norm3(f3(T.x - N.x * nt, T.y - N.y * nt, T.z - N.z * nt));
  out[0] = N.x, out[1] = N.y, out[2] = N.z;
  out[3] = T.x, out[4] = T.y, out[5] = T.z;
}

// The three UVs of triangle tri.
__device__ __forceinline__ void load_uvs(const SceneDev& S, int tri, float* uv) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int t = uv_of(S, tri, k);
    uv[2 * k] = __ldg(S.uvs + 2 * t);
    uv[2 * k + 1] = __ldg(S.uvs + 2 * t + 1);
  }
}

// Shade triangle `tri` at a pixel with barycentric weights l (iw: 1 / w of its vertices, uv: its UVs, fr:
// its frame for the lit models).
__device__ __forceinline__ void surface(const SceneDev& S, int view, int tri, const float l[3], const float iw[3],
                                        const float* uv, const float* fr, uint64_t key, int side, Surf& out) {
  PerspW pw = persp(l, iw);
  out.u = persp_interp(pw, uv[0], uv[2], uv[4]);
  out.v = persp_interp(pw, uv[1], uv[3], uv[5]);
  // (read textures come in role order: albedo, normal, roughness, metallic)
  float val[MAX_READ][4];
#pragma unroll
  for (int r = 0; r < MAX_READ; ++r) {
    if (r >= S.nread) break;
    const TexDev& T = S.rtex[r];
    out.foot[r] = footprint(out.u, out.v, T.w, T.h);
    if (S.foot_nearest) out.foot[r].nearest = nearest_texel(out.u, out.v, T.w, T.h);
    sample_tex(T, out.foot[r], key, side, val[r]);
  }
  if (S.shading == SHADE_UNLIT) {
    out.rgb = f3(val[0][0], val[0][1], val[0][2]);
    return;
  }
  const float3 N = f3(fr[0], fr[1], fr[2]), T = f3(fr[3], fr[4], fr[5]);
  if (S.shading == SHADE_LAMBERT) {
    out.rgb = shade_lit<SHADE_LAMBERT>(S, view, val[0], val[1], 0.5f, 0.0f, N, T, f3(0.f, 0.f, 0.f));
    return;
  }
  float3 p[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) p[k] = perturbed_pos(S, vert_of(S, tri, k), key, side);
  const float b[3] = {pw.q[0] / pw.qs, pw.q[1] / pw.qs, pw.q[2] / pw.qs};
  const float3 P = f3(b[0] * p[0].x + b[1] * p[1].x + b[2] * p[2].x, b[0] * p[0].y + b[1] * p[1].y + b[2] * p[2].y,
                      b[0] * p[0].z + b[1] * p[1].z + b[2] * p[2].z);
  out.rgb = shade_lit<SHADE_GGX>(S, view, val[0], val[1], val[2][0], val[3][0], N, T, P);
}

// The UVs and (lit models) the frame that surface() takes, for one side of an estimate.
__device__ __forceinline__ void load_surface(const SceneDev& S, int tri, uint64_t key, int side, float* uv, float* fr) {
  load_uvs(S, tri, uv);
  if (S.shading == SHADE_UNLIT) return;
  float3 p[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) p[k] = perturbed_pos(S, vert_of(S, tri, k), key, side);
  tri_frame(p, uv, fr);
}

// ---------------------------------------------------------------- signs of one estimate, precomputed
// The fused estimators read s_i from what the vertex pass stored (3 bits per welded vertex) and
// from the texel sign planes (4 bits per texel) instead of hashing: the same values sign_neg gives.
struct PairSigns {
  const uint32_t* planes;  // this estimate's texel sign planes
  const uint8_t* vbits;    // this estimate's vertex sign bits (bits 0-2: x, y, z have s = -1)
  const int* sgn_off;      // word offset of texture k's plane (Workspace::sgn_off)
#if SGE_CHECKED
  const SceneDev* S;       // range checks of the plane words
#endif
};

__device__ __forceinline__ PairSigns pair_signs(const SceneDev& S, const Workspace& ws, int slot, int pb) {
  const long long e = (long long)slot * ws.max_pairs + pb;
#if SGE_CHECKED
  return PairSigns{ws.tsign + e * ws.sgn_words, ws.vbits + e * S.nv, ws.sgn_off, &S};
#else
  return PairSigns{ws.tsign + e * ws.sgn_words, ws.vbits + e * S.nv, ws.sgn_off};
#endif
}

// Sign bits of texel t of texture k (bit c: channel c has s = -1).
__device__ __forceinline__ uint32_t texel_signs(const PairSigns& ps, int k, long long t) {
  const long long w = ps.sgn_off[k] + (t >> 3);
#if SGE_CHECKED
  if (ps.S && !CHK_H(*ps.S, w, ps.S->chk.sign_words)) return 0u;
#endif
  return (__ldg(ps.planes + w) >> (4 * (t & 7))) & 0xFu;
}

// Sign bits of welded vertex v (bit c: coordinate c has s = -1).
__device__ __forceinline__ uint32_t vertex_signs(const PairSigns& ps, int v) { return __ldg(ps.vbits + v) & 7u; }

// sample_tex with the signs of ps.
__device__ __forceinline__ void sample_tex_ps(const TexDev& T, const Foot& f, const PairSigns& ps, int side,
                                              float out[4]) {
  float w[4] = {(1.0f - f.fx) * (1.0f - f.fy), f.fx * (1.0f - f.fy), (1.0f - f.fx) * f.fy, f.fx * f.fy};
  int tx[4] = {f.x0, f.x1, f.x0, f.x1};
  int ty[4] = {f.y0, f.y0, f.y1, f.y1};
#pragma unroll
  for (int c = 0; c < 4; ++c) out[c] = 0.0f;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    long long t = (long long)ty[j] * T.w + tx[j];
    const float* src = T.ptr + t * T.c;
    uint32_t sb = texel_signs(ps, T.index, t);
    if (side < 0) sb = ~sb;
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (c < T.c) out[c] += w[j] * __fadd_rn(__ldg(src + c), ((sb >> c) & 1) ? -T.eps : T.eps);
  }
  if (T.c == 1) out[1] = out[2] = out[0];
}

// Project the three perturbed vertices of `tri` and set it up at reference point (rx, ry).
__device__ __forceinline__ void setup_from_scene(const SceneDev& S, const float* m, int tri, uint64_t key,
                                                 int side, long long rx, long long ry, Tri& t) {
  PVert v[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    int vi = vert_of(S, tri, k);
    float3 q = perturbed_pos(S, vi, key, side);
    v[k] = project(m, q.x, q.y, q.z, S.W, S.H, S.near_w);
  }
  setup_tri(v[0], v[1], v[2], rx, ry, t);
}

// The tile's columns (bits 0-15) and rows (bits 16-31) whose pixel centres lie in the bounding
// box of the projected vertices v grown by `grow` fixed-point units per axis (rx, ry: the tile's
// first pixel centre).  Every perturbed version of a triangle lies in its box grown by the margin
// (each snapped vertex moves at most that far per axis), and a pixel inside the triangle in its
// box: a pre-filter for maybe_visible and surely_covers, which decide inside it.
__device__ __forceinline__ uint32_t box_span(const PVert (&v)[3], long long rx, long long ry, long long grow) {
  const long long xl = (long long)min(v[0].X, min(v[1].X, v[2].X)) - rx - grow;
  const long long xh = (long long)max(v[0].X, max(v[1].X, v[2].X)) - rx + grow;
  const long long yl = (long long)min(v[0].Y, min(v[1].Y, v[2].Y)) - ry - grow;
  const long long yh = (long long)max(v[0].Y, max(v[1].Y, v[2].Y)) - ry + grow;
  // pixel (dx, dy) sits at (256 dx, 256 dy): columns ceil(xl / 256) .. floor(xh / 256)
  const long long x0 = -((-xl) >> 8), x1 = xh >> 8, y0 = -((-yl) >> 8), y1 = yh >> 8;
  if (x0 > 15 || x1 < 0 || y0 > 15 || y1 < 0 || x0 > x1 || y0 > y1) return 0u;
  const int xa = (int)max(x0, 0ll), xb = (int)min(x1, 15ll), ya = (int)max(y0, 0ll), yb = (int)min(y1, 15ll);
  const uint32_t xm = ((2u << xb) - 1u) & ~((1u << xa) - 1u);
  const uint32_t ym = ((2u << yb) - 1u) & ~((1u << ya) - 1u);
  return xm | (ym << 16);
}

__device__ __forceinline__ bool in_span(uint32_t span, int dx, int dy) {
  return ((span >> dx) & (span >> (16 + dy)) & 1u) != 0;
}

// ---------------------------------------------------------------- a triangle set up for one tile
// 64 bytes in shared memory.
// Small (every edge function over the tile fits 32 bits: |a|, |b| < 2^16, |e0| < 2^29, so
// |e| < 2^30 at the offsets 0..15 * 256): e = (E_0, E_1, area, flags) with E_k at the tile's first
// pixel centre and area = E_0 + E_1 + E_2, which is the same everywhere, so edge 2 follows from the
// other two; ab = (a_0, a_1, b_0, b_1).  Otherwise (kBig) the same with 64-bit edge functions: e = (E_0 low, E_0 high,
// E_1 low, flags), iw.w the bits of E_1 high; the area is |a_0 b_1 - a_1 b_0|.  (Kept as vertices and multiplied out at
// each test, a full-image call of 8 pairs of 2,048 triangles of half a 512^2 image took 20.4 ms, this 17.4 ms.)  Not drawn: E_0 = -1
// everywhere.  kVerts: big ones as vertices relative to the first pixel centre all the same, e = (X0, Y0, X1, flags), ab =
// (Y1, X2, Y2, -), which leaves the transparent kernel, bound by registers, fewer spills (8 views x 16 pairs 5,490 us, 5,566 us otherwise).
struct __align__(16) SideTri {
  int4 e, ab;
  float4 z;   // z_0..2, 1 / area
  float4 iw;  // 1 / w_0..2, -
};
static_assert(sizeof(SideTri) == 64, "SideTri layout");
constexpr int kBig = 8, kFlip = 16;  // flags; bits 0-2: edge k is not a top/left edge

// Set up one side of a triangle from its projected vertices (rx, ry: the tile's first pixel centre).
template <bool kVerts = false>
__device__ __forceinline__ void set_up_side(SideTri& d, const PVert (&v)[3], int rx, int ry) {
  if (!(v[0].ok && v[1].ok && v[2].ok)) {
    d.e = make_int4(-1, 0, 0, 0);
    d.ab = make_int4(0, 0, 0, 0);
    return;
  }
  const int x0 = v[0].X - rx, x1 = v[1].X - rx, x2 = v[2].X - rx, y0 = v[0].Y - ry, y1 = v[1].Y - ry, y2 = v[2].Y - ry;
  const int far = max(max(max(abs(x0), abs(x1)), abs(x2)), max(max(abs(y0), abs(y1)), abs(y2)));
  float inv;
  int e1_high = 0;
  if (far < (1 << 14)) {
    // vertices within 64 pixels of the tile's corner: E_k = x_a y_b - x_b y_a there, all in 32 bits
    // (|E_k| < 2^29, |a|, |b| < 2^15)
    int e0 = x1 * y2 - x2 * y1, e1 = x2 * y0 - x0 * y2, area = e0 + e1 + (x0 * y1 - x1 * y0);
    int a0 = y1 - y2, a1 = y2 - y0, a2 = y0 - y1, b0 = x2 - x1, b1 = x0 - x2, b2 = x1 - x0;
    if (area == 0) {
      d.e = make_int4(-1, 0, 0, 0);
      d.ab = make_int4(0, 0, 0, 0);
      return;
    }
    if (area < 0) {
      e0 = -e0, e1 = -e1, area = -area;
      a0 = -a0, a1 = -a1, a2 = -a2, b0 = -b0, b1 = -b1, b2 = -b2;
    }
    const int flags = (a0 > 0 || (a0 == 0 && b0 > 0) ? 0 : 1) | (a1 > 0 || (a1 == 0 && b1 > 0) ? 0 : 2) |
                      (a2 > 0 || (a2 == 0 && b2 > 0) ? 0 : 4);
    d.e = make_int4(e0, e1, area, flags);
    d.ab = make_int4(a0, a1, b0, b1);
    inv = __fdiv_rn(1.0f, __int2float_rn(area));
  } else {
    Tri t;
    setup_tri(v[0], v[1], v[2], rx, ry, t);
    if (!t.ok) {
      d.e = make_int4(-1, 0, 0, 0);
      d.ab = make_int4(0, 0, 0, 0);
      return;
    }
    int flags = 0;
    bool small = true;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      flags |= (t.bias[k] ? 1 : 0) << k;
      small = small && abs(t.a[k]) < (1 << 16) && abs(t.b[k]) < (1 << 16) && t.e0[k] > -(1ll << 29) &&
              t.e0[k] < (1ll << 29);
    }
    if (small) {
      d.e = make_int4((int)t.e0[0], (int)t.e0[1], (int)(t.e0[0] + t.e0[1] + t.e0[2]), flags);
      d.ab = make_int4(t.a[0], t.a[1], t.b[0], t.b[1]);
    } else if constexpr (kVerts) {
      const bool flip = (long long)(x1 - x0) * (y2 - y0) < (long long)(y1 - y0) * (x2 - x0);
      d.e = make_int4(x0, y0, x1, flags | kBig | (flip ? kFlip : 0));
      d.ab = make_int4(y1, x2, y2, 0);
    } else {
      d.e = make_int4((int)t.e0[0], (int)(t.e0[0] >> 32), (int)t.e0[1], flags | kBig);
      d.ab = make_int4(t.a[0], t.a[1], t.b[0], t.b[1]);
      e1_high = (int)(t.e0[1] >> 32);
    }
    inv = t.inv_area;
  }
  d.z = make_float4(v[0].z, v[1].z, v[2].z, inv);
  d.iw = make_float4(v[0].iw, v[1].iw, v[2].iw, __int_as_float(e1_high));
}

// Coverage of the tile's pixel whose centre lies (X, Y) fixed-point units (whole pixels) from its first one, and
// (covered) the barycentric weights E_k / area there as lambdas() forms them.
template <bool kVerts = false>
__device__ __forceinline__ bool cover_lambdas(const SideTri& t, int X, int Y, float l[3], float4& z) {
  const int4 e = t.e, ab = t.ab;
  if (!(e.w & kBig)) {
    const int e0 = e.x + ab.x * X + ab.z * Y, e1 = e.y + ab.y * X + ab.w * Y, e2 = e.z - e0 - e1;
    const int lo = min(min(e0, e1), e2);
    if (lo < 0) return false;
    if (lo == 0 && (((e.w & 1) && e0 == 0) || ((e.w & 2) && e1 == 0) || ((e.w & 4) && e2 == 0))) return false;
    z = t.z;
    l[0] = __fmul_rn(__int2float_rn(e0), z.w);
    l[1] = __fmul_rn(__int2float_rn(e1), z.w);
    l[2] = __fmul_rn(__int2float_rn(e2), z.w);
    return true;
  }
  if constexpr (kVerts) {
    const int vx[3] = {e.x, e.z, ab.y}, vy[3] = {e.y, ab.x, ab.z};
    long long E[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int a = (k + 1) % 3, b = (k + 2) % 3;
      E[k] = edge_at(vx[a], vy[a], vx[b], vy[b], X, Y);
      if (e.w & kFlip) E[k] = -E[k];
      if (E[k] - ((e.w >> k) & 1) < 0) return false;
    }
    z = t.z;
    lambdas(E, z.w, l);
    return true;
  }
  // steps in whole pixels: |a|, |b| <= 2^24 (vertices lie within 2^15 pixels), so 15 of each fit 32 bits
  const int dx = X >> 8, dy = Y >> 8;
  auto wide = [](int lo, int hi) { return (long long)((unsigned long long)(uint32_t)hi << 32 | (uint32_t)lo); };
  long long E[3];
  E[0] = wide(e.x, e.y) + 256ll * (ab.x * dx + ab.z * dy);
  if (E[0] - (e.w & 1) < 0) return false;
  E[1] = wide(e.z, __float_as_int(t.iw.w)) + 256ll * (ab.y * dx + ab.w * dy);
  if (E[1] - ((e.w >> 1) & 1) < 0) return false;
  const long long area = (long long)ab.x * ab.w - (long long)ab.y * ab.z;  // (a and b are both turned: its sign is not)
  E[2] = (area < 0 ? -area : area) - E[0] - E[1];
  if (E[2] - ((e.w >> 2) & 1) < 0) return false;
  z = t.z;
  lambdas(E, z.w, l);
  return true;
}

// The pixel centres of the tile in a projected triangle's vertex box; false: none, or the triangle is not drawn.
__device__ __forceinline__ bool tri_box(const int4& q0, const int4& q1, const int4& q2, int rx, int ry, int& c0, int& c1,
                                        int& r0, int& r1) {
  if (q0.x == kNotDrawn || q1.x == kNotDrawn || q2.x == kNotDrawn) return false;
  c0 = max((min(q0.x, min(q1.x, q2.x)) - rx + 255) >> 8, 0), c1 = min((max(q0.x, max(q1.x, q2.x)) - rx) >> 8, TILE - 1);
  r0 = max((min(q0.y, min(q1.y, q2.y)) - ry + 255) >> 8, 0), r1 = min((max(q0.y, max(q1.y, q2.y)) - ry) >> 8, TILE - 1);
  return c0 <= c1 && r0 <= r1;
}

// A key (depth, id) into a pixel's nearest.
__device__ __forceinline__ void put_key(unsigned long long* out, const float (&l)[3], float z0, float z1, float z2, int id) {
  const float z[3] = {z0, z1, z2};
  const unsigned long long key = ((unsigned long long)ordered_bits(interp_depth(l, z)) << 32) | (uint32_t)id;
  if (key < *(volatile unsigned long long*)out) atomicMin(out, key);
}

// A projected triangle (records as the vertex pass writes them) into the tile's keys: the nearest (depth bits << 32 |
// id) of each pixel centre it covers, columns c0..c1 and rows r0..r1 of its box.  The arithmetic of set_up_side,
// cover_lambdas and interp_depth, with the division left until a pixel is covered (most triangles of a dense tile cover
// none or one).
__device__ __forceinline__ void raster_tri(const int4& q0, const int4& q1, const int4& q2, int id, int rx, int ry, int c0,
                                           int c1, int r0, int r1, unsigned long long* keys) {
  const int x0 = q0.x - rx, x1 = q1.x - rx, x2 = q2.x - rx, y0 = q0.y - ry, y1 = q1.y - ry, y2 = q2.y - ry;
  const int xl = min(x0, min(x1, x2)), xh = max(x0, max(x1, x2)), yl = min(y0, min(y1, y2)), yh = max(y0, max(y1, y2));
  auto put = [&](int x, int y, const float (&l)[3]) {
    put_key(keys + y * TILE + x, l, __int_as_float(q0.z), __int_as_float(q1.z), __int_as_float(q2.z), id);
  };
  if (max(max(xh, yh), -min(xl, yl)) < (1 << 14)) {
    int e0 = x1 * y2 - x2 * y1, e1 = x2 * y0 - x0 * y2, e2 = x0 * y1 - x1 * y0, area = e0 + e1 + e2;
    int a0 = y1 - y2, a1 = y2 - y0, a2 = y0 - y1, b0 = x2 - x1, b1 = x0 - x2, b2 = x1 - x0;
    if (area == 0) return;
    if (area < 0) {
      e0 = -e0, e1 = -e1, e2 = -e2, area = -area;
      a0 = -a0, a1 = -a1, a2 = -a2, b0 = -b0, b1 = -b1, b2 = -b2;
    }
    // a pixel at an edge belongs to the triangle if the edge is top or left: the tests E_k >= 0 of the others
    // become E_k >= 1
    const int n0 = a0 > 0 || (a0 == 0 && b0 > 0) ? 0 : 1, n1 = a1 > 0 || (a1 == 0 && b1 > 0) ? 0 : 1,
              n2 = a2 > 0 || (a2 == 0 && b2 > 0) ? 0 : 1;
    float inv = 0.0f;
    int E0 = e0 + (a0 * c0 + b0 * r0) * 256, E1 = e1 + (a1 * c0 + b1 * r0) * 256;
    const int w = c1 - c0, d0 = (b0 - a0 * w) * 256, d1 = (b1 - a1 * w) * 256;
    // one loop over the box (rows in turn), so that lanes with boxes of other shapes keep together
    for (int x = c0, y = r0; y <= r1;) {
      const int E2 = area - E0 - E1;
      if (min(min(E0 - n0, E1 - n1), E2 - n2) >= 0) {
        if (inv == 0.0f) inv = __fdiv_rn(1.0f, __int2float_rn(area));
        const float l[3] = {__fmul_rn(__int2float_rn(E0), inv), __fmul_rn(__int2float_rn(E1), inv),
                            __fmul_rn(__int2float_rn(E2), inv)};
        put(x, y, l);
      }
      const bool turn = x == c1;
      x = turn ? c0 : x + 1;
      y += turn ? 1 : 0;
      E0 += turn ? d0 : a0 * 256;
      E1 += turn ? d1 : a1 * 256;
    }
    return;
  }
  PVert v[3];
  const int4 q[3] = {q0, q1, q2};
#pragma unroll
  for (int k = 0; k < 3; ++k) v[k] = PVert{q[k].x, q[k].y, __int_as_float(q[k].z), __int_as_float(q[k].w), true};
  SideTri d;
  set_up_side(d, v, rx, ry);
  for (int y = r0; y <= r1; ++y)
    for (int x = c0; x <= c1; ++x) {
      float l[3];
      float4 z;
      if (cover_lambdas(d, x * 256, y * 256, l, z)) put(x, y, l);
    }
}

// f(j) for every triangle j < cnt, in order, whose pixel span `which` reaches the warp's block of the
// tile (columns bits 0-15, rows bits 16-31 of block) and holds this thread's pixel.
template <typename F>
__device__ __forceinline__ void for_spans(const uint32_t (*span)[2], int which, int cnt, uint32_t block, int dx, int dy,
                                          F&& f) {
  const int lane = threadIdx.x & 31;
  for (int j0 = 0; j0 < cnt; j0 += 32) {
    const uint32_t s = j0 + lane < cnt ? span[j0 + lane][which] & block : 0u;
    for (uint32_t hit = __ballot_sync(0xffffffffu, (s & 0xFFFFu) && (s >> 16)); hit; hit &= hit - 1) {
      const int j = j0 + __ffs((int)hit) - 1;
      if (in_span(span[j][which], dx, dy)) f(j);
    }
  }
}

// Evaluate the oriented edge functions of t at offset (dx, dy) pixels from its reference point.
__device__ __forceinline__ bool cover(const Tri& t, int dx, int dy, long long e[3]) {
  bool in = true;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    e[k] = t.e0[k] + (long long)t.a[k] * (dx * 256) + (long long)t.b[k] * (dy * 256);
    in = in && (e[k] + t.bias[k] >= 0);
  }
  return in;
}

// ---------------------------------------------------------------- contributor set (Algorithm 2)
// Keys name a parameter group member: kind << 28 | index; kind 0 = welded vertex
// (its x, y, z), kind k+1 = texel of texture k (all its channels).
__device__ __forceinline__ uint32_t vkey(int v) { return (uint32_t)v; }
__device__ __forceinline__ uint32_t tkey(int k, int texel) { return ((uint32_t)(k + 1) << 28) | (uint32_t)texel; }

__device__ __forceinline__ void key_params(const SceneDev& S, uint32_t key, long long& base, int& nch) {
  uint32_t kind = key >> 28, idx = key & 0x0FFFFFFFu;
  if (kind == 0) {
    base = 3ll * idx;
    nch = 3;
  } else {
    const TexDev& T = S.tex[kind - 1];
    base = T.offset + (long long)idx * T.c;
    nch = T.c;
  }
}

// Call f(key) once for every key of the pixel's contributor set: the union over
// both sides (tris[0] = side +, tris[1] = side -, -1 = background) of the visible
// triangle's three welded vertices and the bilinear 2x2 footprint of each read
// texture.  foot[sd][r] is side sd's footprint of the r-th read texture.
template <typename F>
__device__ __forceinline__ void for_each_contrib(const SceneDev& S, const int tris[2],
                                                 const Foot (&foot)[2][MAX_READ], F&& f) {
  int vid[2][3];
#pragma unroll
  for (int sd = 0; sd < 2; ++sd) {
    if (tris[sd] < 0) continue;
#pragma unroll
    for (int k = 0; k < 3; ++k) vid[sd][k] = vert_of(S, tris[sd], k);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      bool dup = false;
      if (sd == 1 && tris[0] >= 0) dup = vid[1][k] == vid[0][0] || vid[1][k] == vid[0][1] || vid[1][k] == vid[0][2];
      if (!dup) f(vkey(vid[sd][k]));
    }
  }
#pragma unroll
  for (int r = 0; r < MAX_READ; ++r) {
    if (r >= S.nread) break;
    const int k = S.read_k[r];
    const int tw = S.tex[k].w;
    if (S.foot_nearest) {
      // one texel per side: the nearest one (Section 4.4), each once
      const int n0 = tris[0] >= 0 ? foot[0][r].nearest : -1;
      if (n0 >= 0) f(tkey(k, n0));
      if (tris[1] >= 0 && foot[1][r].nearest != n0) f(tkey(k, foot[1][r].nearest));
      continue;
    }
    int ids[2][4];
#pragma unroll
    for (int sd = 0; sd < 2; ++sd) {
      if (tris[sd] < 0) continue;
      const Foot& ft = foot[sd][r];
      ids[sd][0] = ft.y0 * tw + ft.x0;
      ids[sd][1] = ft.y0 * tw + ft.x1;
      ids[sd][2] = ft.y1 * tw + ft.x0;
      ids[sd][3] = ft.y1 * tw + ft.x1;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        bool dup = false;
#pragma unroll
        for (int o = 0; o < q; ++o) dup = dup || ids[sd][o] == ids[sd][q];
        if (sd == 1 && tris[0] >= 0) {
#pragma unroll
          for (int o = 0; o < 4; ++o) dup = dup || ids[0][o] == ids[1][q];
        }
        if (!dup) f(tkey(k, ids[sd][q]));
      }
    }
  }
}

// Loss difference f+ - f- of one pixel written without cancellation (Table 1, Algorithm 2):
// sum_c (I+_c - I-_c)(I+_c + I-_c - 2 I_c); also returns f+ and f-.
__device__ __forceinline__ float loss_diff(float3 ip, float3 im, float3 t, float& fp, float& fm) {
  float a[3] = {ip.x, ip.y, ip.z}, b[3] = {im.x, im.y, im.z}, c[3] = {t.x, t.y, t.z};
  float df = 0.0f;
  fp = fm = 0.0f;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    float dp = a[k] - c[k], dm = b[k] - c[k];
    fp += dp * dp;
    fm += dm * dm;
    df += (a[k] - b[k]) * (a[k] + b[k] - 2.0f * c[k]);
  }
  return df;
}

// One asset of a batched launch as the per-scene code expects it, in shared memory.
struct BatchSmem {
  AssetDesc d;
  ViewList vl;
  EstimateArgs a;
};

// Load asset ai of P into b (all threads of the CTA; the caller synchronises around it).
__device__ __forceinline__ void load_asset(const BatchArgs& P, int ai, BatchSmem& b) {
  const BatchAsset& A = P.as[ai];
  const int4* src = reinterpret_cast<const int4*>(A.desc);
  int4* dst = reinterpret_cast<int4*>(&b.d);
  for (int i = threadIdx.x; i < (int)(sizeof(AssetDesc) / 16); i += blockDim.x) dst[i] = src[i];
  if (threadIdx.x == 0) {
    b.vl.n = A.n_views;
    b.a = EstimateArgs{P.seed, P.iter, P.pairs, P.pairs_per_item, P.pair_begin, P.pair_count,
                       A.grad, A.counts, A.loss, nullptr, P.iter_dev};
  }
  if (threadIdx.x < SGE_MAX_BATCH_VIEWS) b.vl.id[threadIdx.x] = A.view[threadIdx.x];
}

}  // namespace sge
