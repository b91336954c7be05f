// Descent step D (Section 5): gradient estimate of Eq. 9 from the accumulated
// sums, SGD or Adam (Kingma & Ba 2015) per parameter, then the sums and counts
// are zeroed for the next iteration.  Memory bound.
#include <cuda_runtime.h>

#include <cfloat>
#include <cmath>

#include "sge_device.cuh"

namespace sge {

namespace {

struct StepGroups {
  int n;
  long long begin[SGE_MAX_TEXTURES + 2];  // flat parameter index where each group starts (+ end)
  float* theta[SGE_MAX_TEXTURES + 1];
  float eps[SGE_MAX_TEXTURES + 1];
  float lr[SGE_MAX_TEXTURES + 1];
};

// Group of parameter i.
__device__ __forceinline__ int group_of(const StepGroups& G, long long i) {
  int g = 0;
#pragma unroll 1
  while (g + 1 < G.n && i >= G.begin[g + 1]) ++g;
  return g;
}

__device__ __forceinline__ bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// Four consecutive parameters per thread: HBM bound, 20 B read and 20 B written per parameter (Adam), each
// flat array (sums, counts, m, v) as one 16-byte access and theta as one where its group starts on a
// multiple of four parameters (else four 4-byte ones).  One parameter per thread and grid-stride
// iteration reached 5.2 TB/s on 52 M parameters (394 us); this 6.6 TB/s (313 us).  Steps of few parameters last as long as a
// thread's chain, which four make longer (2,214 parameters 2.0 us with one a thread, 4.6 us with four; 198 K 3.8 and 5.1, 395 K 5.1
// and 5.4, 556 K 6.2 and 5.8): they keep one parameter a thread and iteration (kPer = 1).
template <int kPer>
__global__ void __launch_bounds__(256) k_step(StepGroups G, int kind, float* grad, uint32_t* counts, float inv_n,
                                              float b1, float b2, int t_host, float aeps, float* m, float* v,
                                              const int32_t* t_dev) {
  const long long d = G.begin[G.n], i0 = kPer * ((long long)blockIdx.x * blockDim.x + threadIdx.x);
  if (i0 >= d) return;
  // Adam's bias corrections 1 - beta^t for the step number t (from device memory in a replayed
  // graph's step), formed as -expm1(t log beta): no cancellation when beta^t is close to 1
  float c1 = 1.0f, c2 = 1.0f;
  if (kind == SGE_STEP_ADAM) {
    const float t = (float)(t_dev ? *t_dev : t_host);
    c1 = -expm1f(t * logf(b1));
    c2 = -expm1f(t * logf(b2));
  }
  // group g's |lr| 2^30 / (c1 adam_eps): |m| times it below |theta| means a step below 2^-30 |theta| (no bound, infinity,
  // where a factor is not positive or the product leaves the normal range)
  auto bound = [&](int g) {
    const float lr = fabsf(G.lr[g]);
    const float k = lr * (aeps > 0.0f && c1 > 0.0f && c2 > 0.0f ? 1.07374182e9f / (c1 * aeps) : INFINITY);
    return lr == 0.0f || k >= FLT_MIN ? k : INFINITY;
  };
  // one parameter of group g: theta, m, v updated
  auto update = [&](int g, float kg, float s, uint32_t cn, float& th, float& mm, float& vv) {
    const float scale = kind == SGE_STEP_SGD_MEAN ? 1.0f / (float)(cn > 0 ? cn : 1u) : inv_n;
    const float gr = s * scale / (2.0f * G.eps[g]);
    if (kind == SGE_STEP_ADAM) {
      mm = b1 * mm + (1.0f - b1) * gr;
      vv = b2 * vv + (1.0f - b2) * gr * gr;
      // the step is at most lr |m| / (c1 adam_eps): below theta's rounding by 2^-30 it leaves theta as it
      // is, and the divisions, which take a slow path for the denormal moments of parameters that nothing
      // touches any more, are left out (52 M such parameters: 460 -> 305 us)
      if (vv >= 0.0f && fabsf(mm) * kg < fabsf(th)) return;
      th -= G.lr[g] * (mm / c1) / (sqrtf(vv / c2) + aeps);
    } else {
      th -= G.lr[g] * gr;
    }
  };
  const int g = group_of(G, i0);
  const bool moments = kind == SGE_STEP_ADAM;
  if (kPer == 4 && i0 + 4 <= G.begin[g + 1] && aligned16(grad) && aligned16(counts) && (!moments || (aligned16(m) && aligned16(v)))) {
    const float4 s4 = __ldcs(reinterpret_cast<const float4*>(grad + i0));
    const uint4 n4 = __ldcs(reinterpret_cast<const uint4*>(counts + i0));
    float4 m4 = make_float4(0.f, 0.f, 0.f, 0.f), v4 = m4;
    if (moments) {
      m4 = __ldcs(reinterpret_cast<const float4*>(m + i0));
      v4 = __ldcs(reinterpret_cast<const float4*>(v + i0));
    }
    float* theta = G.theta[g] + (i0 - G.begin[g]);
    const bool vec = aligned16(theta);
    float th[4];
    if (vec) {
      const float4 t4 = *reinterpret_cast<const float4*>(theta);
      th[0] = t4.x, th[1] = t4.y, th[2] = t4.z, th[3] = t4.w;
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) th[k] = theta[k];
    }
    const float kg = bound(g);
    update(g, kg, s4.x, n4.x, th[0], m4.x, v4.x);
    update(g, kg, s4.y, n4.y, th[1], m4.y, v4.y);
    update(g, kg, s4.z, n4.z, th[2], m4.z, v4.z);
    update(g, kg, s4.w, n4.w, th[3], m4.w, v4.w);
    if (moments) {
      __stcs(reinterpret_cast<float4*>(m + i0), m4);
      __stcs(reinterpret_cast<float4*>(v + i0), v4);
    }
    if (vec) {
      *reinterpret_cast<float4*>(theta) = make_float4(th[0], th[1], th[2], th[3]);
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) theta[k] = th[k];
    }
    __stcs(reinterpret_cast<float4*>(grad + i0), make_float4(0.f, 0.f, 0.f, 0.f));
    __stcs(reinterpret_cast<uint4*>(counts + i0), make_uint4(0u, 0u, 0u, 0u));
    return;
  }
  // a quad across two groups, the last parameters, or arrays that do not start on 16 bytes; with one a thread, all
  const long long end = kPer == 4 && i0 + 4 < d ? i0 + 4 : d, by = kPer == 4 ? 1 : (long long)gridDim.x * blockDim.x;
  for (long long i = i0; i < end; i += by) {
    const int gi = group_of(G, i);
    float* theta = G.theta[gi] + (i - G.begin[gi]);
    float th = *theta, mm = moments ? m[i] : 0.0f, vv = moments ? v[i] : 0.0f;
    update(gi, bound(gi), grad[i], counts[i], th, mm, vv);
    if (moments) {
      m[i] = mm;
      v[i] = vv;
    }
    *theta = th;
    grad[i] = 0.0f;
    counts[i] = 0u;
  }
}

// Moves a captured loop's iteration state on: the iteration index and Adam's step number.
__global__ void k_iter_advance(uint32_t* state, int d_iter, int d_t) {
  state[0] += (uint32_t)d_iter;
  state[1] = (uint32_t)((int)state[1] + d_t);
}

// g_i = scale * grad_i / (2 eps_i n_total): the estimate of Eq. 9 (scale: device scalar or NULL).
// Four parameters per thread or one, as k_step (2,214 parameters 1.4 us with one, 2.1 us with four; 395 K 2.3 and 2.4).
template <int kPer>
__global__ void __launch_bounds__(256) k_gradient(StepGroups G, const float* grad, float inv_n, const float* scale,
                                                  float* out) {
  const long long d = G.begin[G.n], i0 = kPer * ((long long)blockIdx.x * blockDim.x + threadIdx.x);
  if (i0 >= d) return;
  const float sc = scale ? *scale : 1.0f;
  const int g = group_of(G, i0);
  if (kPer == 4 && i0 + 4 <= G.begin[g + 1] && aligned16(grad) && aligned16(out)) {
    const float4 s = *reinterpret_cast<const float4*>(grad + i0);
    const float e = 2.0f * G.eps[g];
    *reinterpret_cast<float4*>(out + i0) =
        make_float4(sc * (s.x * inv_n / e), sc * (s.y * inv_n / e), sc * (s.z * inv_n / e), sc * (s.w * inv_n / e));
    return;
  }
  const long long end = kPer == 4 && i0 + 4 < d ? i0 + 4 : d, by = kPer == 4 ? 1 : (long long)gridDim.x * blockDim.x;
  for (long long i = i0; i < end; i += by) out[i] = sc * (grad[i] * inv_n / (2.0f * G.eps[group_of(G, i)]));
}

StepGroups groups_of(const SceneDev& S) {
  StepGroups G;
  G.n = 1 + S.ntex;
  G.begin[0] = 0;
  G.theta[0] = const_cast<float*>(S.pos);
  G.eps[0] = S.eps_pos;
  G.lr[0] = 0.0f;
  for (int k = 0; k < S.ntex; ++k) {
    G.begin[k + 1] = S.tex[k].offset;
    G.theta[k + 1] = const_cast<float*>(S.tex[k].ptr);
    G.eps[k + 1] = S.tex[k].eps;
    G.lr[k + 1] = 0.0f;
  }
  G.begin[G.n] = S.n_params;
  return G;
}

// Steps and gradients of at most so many parameters take one a thread, in at most eight CTAs per SM.
constexpr long long kStepOne = 450000;
unsigned grid_one(long long n) { return (unsigned)(n > 256ll * 8 * 152 ? 8 * 152 : (n + 255) / 256); }

// CTAs of 256 threads, four parameters each.
unsigned grid_for(long long n) { return (unsigned)((n + 1023) / 1024); }

// Full-image estimator (Eq. 4), accumulation: every parameter i gets sum_e dF_e s_i(e) over
// the call's estimates e (signs from each estimate's key) and one count per estimate.  The
// estimates' keys and differences are staged in shared memory once per CTA; one thread per
// parameter (grid-stride).
__global__ void k_full_image_grad(long long d, int n_est, int pairs, ViewList vl, uint64_t seed, uint32_t iter,
                                  const float* dF, float* grad, uint32_t* counts) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint64_t* keys = reinterpret_cast<uint64_t*>(smem_raw);
  float* dfs = reinterpret_cast<float*>(keys + n_est);
  for (int e = threadIdx.x; e < n_est; e += blockDim.x) {
    keys[e] = pair_key(seed, iter, (uint32_t)vl.id[e / pairs], (uint32_t)(e % pairs));
    dfs[e] = dF[e];
  }
  __syncthreads();
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < d; i += (long long)gridDim.x * blockDim.x) {
    float acc = 0.0f;
    for (int e = 0; e < n_est; ++e) acc += sign_neg(keys[e], (uint64_t)i) ? -dfs[e] : dfs[e];
    grad[i] += acc;
    counts[i] += (uint32_t)n_est;
  }
}

// y[r] (+)= sum_j w_j x[col_j] for 3-vectors (xyz per row), rows of a CSR matrix in fixed order:
// the refine matrix of a subdivision (fine = R control) or its transpose (control gradient =
// R^T fine gradient).  One thread per row.
__global__ void k_csr_vec3(const int32_t* ptr, const int32_t* col, const float* w, int n_rows, const float* x,
                           float* y, int accumulate) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n_rows) return;
  float a0 = 0.0f, a1 = 0.0f, a2 = 0.0f;
  for (int j = ptr[r]; j < ptr[r + 1]; ++j) {
    const float wj = w[j];
    const long long c = 3ll * col[j];
    a0 += wj * x[c];
    a1 += wj * x[c + 1];
    a2 += wj * x[c + 2];
  }
  if (accumulate) {
    y[3ll * r] += a0;
    y[3ll * r + 1] += a1;
    y[3ll * r + 2] += a2;
  } else {
    y[3ll * r] = a0;
    y[3ll * r + 1] = a1;
    y[3ll * r + 2] = a2;
  }
}

}  // namespace

cudaError_t launch_gradient(const SceneDev& S, const float* grad, long long n_total, const float* scale, float* out,
                            cudaStream_t st) {
  const float inv_n = (float)(1.0 / (double)n_total);
  if (S.n_params <= kStepOne)
    k_gradient<1><<<grid_one(S.n_params), 256, 0, st>>>(groups_of(S), grad, inv_n, scale, out);
  else
    k_gradient<4><<<grid_for(S.n_params), 256, 0, st>>>(groups_of(S), grad, inv_n, scale, out);
  return cudaGetLastError();
}

cudaError_t launch_step(const SceneDev& S, const sge_opt& o, float* grad, uint32_t* counts, long long n_total,
                        float* m, float* v, cudaStream_t st, const int32_t* t_dev) {
  StepGroups G;
  G.n = 1 + S.ntex;
  G.begin[0] = 0;
  G.theta[0] = const_cast<float*>(S.pos);
  G.eps[0] = S.eps_pos;
  G.lr[0] = o.lr_pos;
  for (int k = 0; k < S.ntex; ++k) {
    G.begin[k + 1] = S.tex[k].offset;
    G.theta[k + 1] = const_cast<float*>(S.tex[k].ptr);
    G.eps[k + 1] = S.tex[k].eps;
    G.lr[k + 1] = o.lr_tex[k];
  }
  G.begin[G.n] = S.n_params;
  const float inv_n = (float)(1.0 / (double)n_total);
  if (S.n_params <= kStepOne)
    k_step<1><<<grid_one(S.n_params), 256, 0, st>>>(G, o.kind, grad, counts, inv_n, o.beta1, o.beta2, o.t, o.adam_eps, m, v,
                                                    t_dev);
  else
    k_step<4><<<grid_for(S.n_params), 256, 0, st>>>(G, o.kind, grad, counts, inv_n, o.beta1, o.beta2, o.t, o.adam_eps, m, v,
                                                    t_dev);
  return cudaGetLastError();
}

cudaError_t launch_iter_advance(uint32_t* state, int d_iter, int d_t, cudaStream_t st) {
  k_iter_advance<<<1, 1, 0, st>>>(state, d_iter, d_t);
  return cudaGetLastError();
}

cudaError_t launch_full_image_grad(const SceneDev& S, const ViewList& vl, int pairs, uint64_t seed, uint32_t iter,
                                   const float* dF, float* grad, uint32_t* counts, cudaStream_t st) {
  const int n_est = vl.n * pairs;
  const size_t smem = (size_t)n_est * (sizeof(uint64_t) + sizeof(float));
  long long blocks = (S.n_params + 255) / 256;
  if (blocks > 152 * 8) blocks = 152 * 8;
  k_full_image_grad<<<(unsigned)blocks, 256, smem, st>>>(S.n_params, n_est, pairs, vl, seed, iter, dF, grad, counts);
  return cudaGetLastError();
}

cudaError_t launch_csr_vec3(const int32_t* ptr, const int32_t* col, const float* w, int n_rows, const float* x,
                            float* y, int accumulate, cudaStream_t st) {
  if (n_rows > 0) k_csr_vec3<<<(n_rows + 255) / 256, 256, 0, st>>>(ptr, col, w, n_rows, x, y, accumulate);
  return cudaGetLastError();
}

}  // namespace sge
