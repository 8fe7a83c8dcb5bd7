// Training-step kernels (Sec. 5.1 "Optimization" and "Densification"): Adam over every parameter array in
// one launch, the accumulation of each Gaussian's positional-gradient magnitude, and split / prune
// compaction into new arrays.
//
// Adam (Kingma and Ba): m = b1 m + (1 - b1) g, v = b2 v + (1 - b2) g^2, step = lr m^ / (sqrt(v^) + eps) with
// the bias-corrected m^ = m / (1 - b1^t), v^ = v / (1 - b2^t); "bounded": the step is clipped to [-lr, lr].
//
// Densification: Gaussian i is pruned when sigmoid(logit) < min_opacity or max_k exp(s_k) < min_scale; else
// split when its mean positional-gradient magnitude accum / count exceeds the threshold (count > 0); else
// kept. Splits are granted in index order while the total stays within max_gaussians. A split replaces the
// Gaussian by two children at mu +- (sigma_a / 2) r_a along its longest axis a (r_a the rotation's column,
// sigma_a = exp(s_a)), with sigma_a scaled by sqrt(3)/2 so that the pair keeps the parent's variance along
// r_a (sigma_a'^2 + (sigma_a / 2)^2 = sigma_a^2); the other scales, the rotation, the opacity and the SH are
// the parent's. Kept Gaussians keep their Adam moments; children start from zero.
#include <math.h>

#include <algorithm>

#include "ngs_internal.cuh"

namespace ngs {
namespace {

struct ParamPtrs {
  float* p[5];
};

struct AdamArgs {
  ParamPtrs param, grad, m, v;
  int64_t count[5];       // elements of each array
  uint32_t first[5];      // first block of each array
  bool vec[5];            // its four pointers are 16-byte aligned
  float lr[5];
  float b1, b2, eps, c1, c2;  // c1 = 1 / (1 - b1^t), c2 = 1 / (1 - b2^t)
  int bounded;
};

__device__ __forceinline__ void adam_update(const AdamArgs& a, float lr, float g, float& m, float& v, float& p) {
  m = fmaf(a.b1, m, (1.f - a.b1) * g);
  v = fmaf(a.b2, v, (1.f - a.b2) * g * g);
  float step = lr * (m * a.c1) / (sqrtf(v * a.c2) + a.eps);
  if (a.bounded) step = fminf(fmaxf(step, -lr), lr);
  p -= step;
}

// A block works on one array, kAdamVecs 16-byte vectors of each of the four arrays per thread, all loaded before the
// first is used. Bound by HBM (28 B per element): 397 us with 4-byte loads and a search for the array per element,
// 236 us so (7.0 TB/s), at one million Gaussians of 59 parameters on GB300.
constexpr int kAdamThreads = 256, kAdamVecs = 2;
constexpr int64_t kAdamBlock = (int64_t)kAdamThreads * kAdamVecs * 4;  // elements
__global__ void __launch_bounds__(kAdamThreads) adam_kernel(AdamArgs a) {
  pdl_wait();
  int gi = 0;
  while (gi < 4 && blockIdx.x >= a.first[gi + 1]) ++gi;
  const int64_t base = (int64_t)(blockIdx.x - a.first[gi]) * kAdamBlock, count = a.count[gi];
  float *const param = a.param.p[gi], *const grad = a.grad.p[gi], *const ma = a.m.p[gi], *const va = a.v.p[gi];
  const float lr = a.lr[gi];
  if (a.vec[gi] && base + kAdamBlock <= count) {
    float4 g[kAdamVecs], m[kAdamVecs], v[kAdamVecs], p[kAdamVecs];
    const int64_t i0 = base / 4 + threadIdx.x;
#pragma unroll
    for (int k = 0; k < kAdamVecs; ++k) {
      const int64_t i = i0 + k * kAdamThreads;
      g[k] = __ldcs(reinterpret_cast<const float4*>(grad) + i);
      m[k] = __ldcs(reinterpret_cast<const float4*>(ma) + i);
      v[k] = __ldcs(reinterpret_cast<const float4*>(va) + i);
      p[k] = reinterpret_cast<const float4*>(param)[i];
    }
#pragma unroll
    for (int k = 0; k < kAdamVecs; ++k) {
      const int64_t i = i0 + k * kAdamThreads;
      adam_update(a, lr, g[k].x, m[k].x, v[k].x, p[k].x);
      adam_update(a, lr, g[k].y, m[k].y, v[k].y, p[k].y);
      adam_update(a, lr, g[k].z, m[k].z, v[k].z, p[k].z);
      adam_update(a, lr, g[k].w, m[k].w, v[k].w, p[k].w);
      __stcs(reinterpret_cast<float4*>(ma) + i, m[k]);
      __stcs(reinterpret_cast<float4*>(va) + i, v[k]);
      reinterpret_cast<float4*>(param)[i] = p[k];
    }
    return;
  }
  const int64_t end = base + kAdamBlock < count ? base + kAdamBlock : count;
  for (int64_t i = base + threadIdx.x; i < end; i += kAdamThreads) {
    float m = ma[i], v = va[i], p = param[i];
    adam_update(a, lr, grad[i], m, v, p);
    ma[i] = m;
    va[i] = v;
    param[i] = p;
  }
}

__global__ void accumulate_kernel(const float* __restrict__ d_means, int64_t n, float* __restrict__ accum,
                                  float* __restrict__ count) {
  pdl_wait();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float x = d_means[3 * i], y = d_means[3 * i + 1], z = d_means[3 * i + 2];
    const float norm = sqrtf(x * x + y * y + z * z);
    if (norm > 0.f) {
      accum[i] += norm;
      count[i] += 1.f;
    }
  }
}

// decision per Gaussian: 0 prune, 1 keep, 2 split candidate
__global__ void densify_decide_kernel(const float* __restrict__ logits, const float* __restrict__ log_scales,
                                      const float* __restrict__ accum, const float* __restrict__ count, int64_t n,
                                      ngs_densify_cfg cfg, uint32_t* __restrict__ decision,
                                      uint32_t* __restrict__ is_split) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float op = 1.f / (1.f + expf(-logits[i]));
  const float smax = expf(fmaxf(log_scales[3 * i], fmaxf(log_scales[3 * i + 1], log_scales[3 * i + 2])));
  uint32_t d = 1;
  if (cfg.prune && (op < cfg.min_opacity || smax < cfg.min_scale)) d = 0;
  else if (cfg.split && count[i] > 0.f && accum[i] / count[i] > cfg.grad_threshold) d = 2;
  decision[i] = d;
  is_split[i] = d == 2 ? 1u : 0u;
}

__device__ __forceinline__ void quat_axis(const float* q, int a, float* r) {
  const float n = rsqrtf(q[0] * q[0] + q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
  const float w = q[0] * n, x = q[1] * n, y = q[2] * n, z = q[3] * n;
  // column a of the rotation matrix of the unit quaternion (w, x, y, z)
  if (a == 0) {
    r[0] = 1.f - 2.f * (y * y + z * z);
    r[1] = 2.f * (x * y + w * z);
    r[2] = 2.f * (x * z - w * y);
  } else if (a == 1) {
    r[0] = 2.f * (x * y - w * z);
    r[1] = 1.f - 2.f * (x * x + z * z);
    r[2] = 2.f * (y * z + w * x);
  } else {
    r[0] = 2.f * (x * z + w * y);
    r[1] = 2.f * (y * z - w * x);
    r[2] = 1.f - 2.f * (x * x + y * y);
  }
}

struct DensifyArgs {
  ParamPtrs src, src_m, src_v, dst, dst_m, dst_v;
  int K3;  // 3 (sh_degree + 1)^2
};

__global__ void iota_kernel(uint32_t* __restrict__ out, int64_t n) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) out[i] = (uint32_t)i;
}

// splits allowed under the cap: min(candidates, max(0, cap - survivors)); survivors = n - pruned
__global__ void densify_allowed_kernel(const uint64_t* __restrict__ cand_total,
                                       const uint64_t* __restrict__ prune_total, int64_t n, int64_t cap,
                                       uint32_t* __restrict__ allowed) {
  const int64_t survivors = n - (int64_t)*prune_total;
  const int64_t room = cap > survivors ? cap - survivors : 0;
  *allowed = (uint32_t)min((int64_t)*cand_total, room);
}

// number of pruned Gaussians (decision 0), one atomic per warp
__global__ void count_pruned_kernel(const uint32_t* __restrict__ decision, int64_t n, uint64_t* __restrict__ pruned) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const uint32_t b = __ballot_sync(0xFFFFFFFFu, i < n && decision[i] == 0);
  if ((threadIdx.x & 31) == 0 && b) atomicAdd(reinterpret_cast<unsigned long long*>(pruned), (unsigned long long)__popc(b));
}

// output count per Gaussian: 0 pruned, 2 a granted split, else 1
__global__ void densify_count_kernel(const uint32_t* __restrict__ decision, const uint32_t* __restrict__ rank,
                                     const uint32_t* __restrict__ allowed, int64_t n, uint32_t* __restrict__ outc) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint32_t d = decision[i];
  outc[i] = d == 0 ? 0u : (d == 2 && rank[i] < *allowed ? 2u : 1u);
}

// Array gi (W floats per Gaussian) of kApplyRows Gaussians from i0 on: a thread per float, so that reads and writes
// are coalesced (a thread per Gaussian moved 59-float rows one float at a time: a split / prune of 100k Gaussians took
// 310 us on GB300, 203 us so).
constexpr int kApplyThreads = 256, kApplyRows = 64;
template <int W>
__device__ __forceinline__ void apply_array(const DensifyArgs& a, int gi, const uint32_t* __restrict__ outc,
                                            const uint32_t* __restrict__ pos, int64_t i0, int64_t n) {
  const int rows = (int)(n - i0 < kApplyRows ? n - i0 : kApplyRows);
  for (int e = threadIdx.x; e < rows * W; e += kApplyThreads) {
    const int r = e / W, k = e - r * W;
    const int64_t i = i0 + r, from = i * W + k;
    const uint32_t c = outc[i];
    if (c == 0) continue;
    const int64_t to = (int64_t)pos[i] * W + k;
    const float val = a.src.p[gi][from];
    if (c == 1) {
      a.dst.p[gi][to] = val;
      a.dst_m.p[gi][to] = a.src_m.p[gi][from];
      a.dst_v.p[gi][to] = a.src_v.p[gi][from];
      continue;
    }
    float v0 = val, v1 = val;
    if (gi <= 1) {  // split along the longest axis
      const float* ls = a.src.p[1] + 3 * i;
      const int ax = ls[0] >= ls[1] ? (ls[0] >= ls[2] ? 0 : 2) : (ls[1] >= ls[2] ? 1 : 2);
      if (gi == 0) {
        float r3[3];
        quat_axis(a.src.p[2] + 4 * i, ax, r3);
        const float half = 0.5f * expf(ls[ax]);
        const float d = half * (k == 0 ? r3[0] : (k == 1 ? r3[1] : r3[2]));
        v0 = val + d;
        v1 = val - d;
      } else if (k == ax) {
        v0 = v1 = val + logf(0.8660254037844386f);  // sigma_a sqrt(3)/2
      }
    }
    a.dst.p[gi][to] = v0;
    a.dst.p[gi][to + W] = v1;
    a.dst_m.p[gi][to] = a.dst_m.p[gi][to + W] = 0.f;
    a.dst_v.p[gi][to] = a.dst_v.p[gi][to + W] = 0.f;
  }
}

__global__ void __launch_bounds__(kApplyThreads) densify_apply_kernel(DensifyArgs a, const uint32_t* __restrict__ outc,
                                                                      const uint32_t* __restrict__ pos, int64_t n) {
  const int64_t i0 = (int64_t)blockIdx.x * kApplyRows;
  apply_array<3>(a, 0, outc, pos, i0, n);
  apply_array<3>(a, 1, outc, pos, i0, n);
  apply_array<4>(a, 2, outc, pos, i0, n);
  apply_array<1>(a, 3, outc, pos, i0, n);
  switch (a.K3) {
    case 3: apply_array<3>(a, 4, outc, pos, i0, n); break;
    case 12: apply_array<12>(a, 4, outc, pos, i0, n); break;
    case 27: apply_array<27>(a, 4, outc, pos, i0, n); break;
    default: apply_array<48>(a, 4, outc, pos, i0, n);
  }
}

ParamPtrs ptrs(const ngs_grads& g) { return ParamPtrs{{g.d_means, g.d_log_scales, g.d_quats, g.d_opacity_logits, g.d_sh}}; }

bool complete(const ngs_grads* g) {
  return g && g->d_means && g->d_log_scales && g->d_quats && g->d_opacity_logits && g->d_sh;
}

unsigned grid_for(int64_t n) { return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 1 << 20)); }

}  // namespace
}  // namespace ngs

using namespace ngs;

extern "C" {

NGS_API int ngs_adam_step(ngs_ctx* ctx, int64_t n, int32_t sh_degree, const ngs_grads* params, const ngs_grads* grads,
                          const ngs_grads* m, const ngs_grads* v, const ngs_adam* cfg, void* stream) {
  if (!ctx) return NGS_ERR_INVALID_ARG;
  if (n < 0 || sh_degree < 0 || sh_degree > 3 || !cfg || cfg->step < 1 || !(cfg->beta1 >= 0.f && cfg->beta1 < 1.f) ||
      !(cfg->beta2 >= 0.f && cfg->beta2 < 1.f) || !(cfg->eps > 0.f))
    return fail(ctx, NGS_ERR_INVALID_ARG, "adam: n, sh_degree or the configuration out of range");
  if (n == 0) return NGS_OK;
  if (!complete(params) || !complete(grads) || !complete(m) || !complete(v))
    return fail(ctx, NGS_ERR_INVALID_ARG, "adam: null array");
  const int K3 = 3 * (sh_degree + 1) * (sh_degree + 1);
  AdamArgs a;
  a.param = ptrs(*params);
  a.grad = ptrs(*grads);
  a.m = ptrs(*m);
  a.v = ptrs(*v);
  const int64_t width[5] = {3, 3, 4, 1, K3};
  int64_t blocks = 0;
  for (int gi = 0; gi < 5; ++gi) {
    a.count[gi] = width[gi] * n;
    a.first[gi] = (uint32_t)blocks;
    blocks += (a.count[gi] + kAdamBlock - 1) / kAdamBlock;
    a.vec[gi] = (((uintptr_t)a.param.p[gi] | (uintptr_t)a.grad.p[gi] | (uintptr_t)a.m.p[gi] | (uintptr_t)a.v.p[gi]) & 15) == 0;
    a.lr[gi] = cfg->lr[gi];
  }
  if (blocks >= (1ll << 31)) return fail(ctx, NGS_ERR_INVALID_ARG, "adam: more than 2^42 parameters");
  a.b1 = cfg->beta1;
  a.b2 = cfg->beta2;
  a.eps = cfg->eps;
  a.c1 = (float)(1.0 / (1.0 - pow((double)cfg->beta1, (double)cfg->step)));
  a.c2 = (float)(1.0 / (1.0 - pow((double)cfg->beta2, (double)cfg->step)));
  a.bounded = cfg->bounded != 0;
  launch_pdl(adam_kernel, (unsigned)blocks, kAdamThreads, 0, (cudaStream_t)stream, a);
  ctx->launches += 1;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(ctx, NGS_ERR_CUDA, std::string("adam launch: ") + cudaGetErrorString(e));
  return NGS_OK;
}

NGS_API int ngs_accumulate_grad_norm(ngs_ctx* ctx, int64_t n, const float* d_means, float* accum, float* count,
                                     void* stream) {
  if (!ctx) return NGS_ERR_INVALID_ARG;
  if (n < 0 || (n > 0 && (!d_means || !accum || !count)))
    return fail(ctx, NGS_ERR_INVALID_ARG, "accumulate: null array or n < 0");
  if (n == 0) return NGS_OK;
  launch_pdl(accumulate_kernel, grid_for(n), 256, 0, (cudaStream_t)stream, d_means, n, accum, count);
  ctx->launches += 1;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(ctx, NGS_ERR_CUDA, std::string("accumulate launch: ") + cudaGetErrorString(e));
  return NGS_OK;
}

NGS_API int ngs_densify(ngs_ctx* ctx, int64_t n, int32_t sh_degree, const ngs_grads* params, const ngs_grads* m,
                        const ngs_grads* v, const float* accum, const float* count, const ngs_densify_cfg* cfg,
                        int64_t capacity, const ngs_grads* out_params, const ngs_grads* out_m, const ngs_grads* out_v,
                        int64_t* n_out, void* stream) {
  if (!ctx) return NGS_ERR_INVALID_ARG;
  if (!cfg || !n_out || n < 0 || n >= (1ll << 30) || sh_degree < 0 || sh_degree > 3 || cfg->max_gaussians < 0)
    return fail(ctx, NGS_ERR_INVALID_ARG, "densify: null argument or n, sh_degree, max_gaussians out of range");
  const int64_t needed = std::min<int64_t>(2 * n, std::max<int64_t>(n, cfg->max_gaussians));
  if (capacity < needed)
    return fail(ctx, NGS_ERR_INVALID_ARG, "densify: output capacity below min(2 n, max(n, max_gaussians))");
  *n_out = 0;
  if (n == 0) return NGS_OK;
  if (!complete(params) || !complete(m) || !complete(v) || !complete(out_params) || !complete(out_m) ||
      !complete(out_v) || !accum || !count)
    return fail(ctx, NGS_ERR_INVALID_ARG, "densify: null array");
  cudaStream_t s = (cudaStream_t)stream;
  const uint32_t un = (uint32_t)n;
  // scratch: decision, candidate flags, their scan, output counts, their scan, identity order (u32 each),
  // allowed count; the scan's block sums and totals in the context's scan scratch
  const size_t words = 6 * ((size_t)un + 1) + 4;
  int rc = ensure(ctx, ctx->densify_tmp, sizeof(uint32_t) * words);
  if (rc == NGS_OK) rc = ensure(ctx, ctx->scan_tmp, sizeof(uint64_t) * scan_tmp_words(un));
  if (rc == NGS_OK) rc = ensure(ctx, ctx->densify_totals, 3 * sizeof(uint64_t));
  if (rc != NGS_OK) return rc;
  uint32_t* decision = ctx->densify_tmp.as<uint32_t>();
  uint32_t* cand = decision + (un + 1);
  uint32_t* rank = cand + (un + 1);
  uint32_t* outc = rank + (un + 1);
  uint32_t* pos = outc + (un + 1);
  uint32_t* iota = pos + (un + 1);
  uint32_t* allowed = iota + (un + 1);
  uint64_t* totals = ctx->densify_totals.as<uint64_t>();
  const unsigned blocks = (un + 255) / 256;
  int launches = 0;
  iota_kernel<<<blocks, 256, 0, s>>>(iota, n);
  densify_decide_kernel<<<blocks, 256, 0, s>>>(params->d_opacity_logits, params->d_log_scales, accum, count, n, *cfg,
                                               decision, cand);
  launches += 2;
  cudaError_t me = launch_scan_counts(cand, iota, un, rank, ctx->scan_tmp.as<uint64_t>(), &totals[0], s, &launches);
  if (me == cudaSuccess) me = cudaMemsetAsync(&totals[1], 0, sizeof(uint64_t), s);
  if (me != cudaSuccess) return fail(ctx, NGS_ERR_CUDA, std::string("densify: ") + cudaGetErrorString(me));
  count_pruned_kernel<<<blocks, 256, 0, s>>>(decision, n, &totals[1]);
  densify_allowed_kernel<<<1, 1, 0, s>>>(&totals[0], &totals[1], n, cfg->max_gaussians, allowed);
  densify_count_kernel<<<blocks, 256, 0, s>>>(decision, rank, allowed, n, outc);
  launches += 3;
  me = launch_scan_counts(outc, iota, un, pos, ctx->scan_tmp.as<uint64_t>(), &totals[2], s, &launches);
  if (me != cudaSuccess) return fail(ctx, NGS_ERR_CUDA, std::string("densify: ") + cudaGetErrorString(me));
  DensifyArgs da;
  da.src = ptrs(*params);
  da.src_m = ptrs(*m);
  da.src_v = ptrs(*v);
  da.dst = ptrs(*out_params);
  da.dst_m = ptrs(*out_m);
  da.dst_v = ptrs(*out_v);
  da.K3 = 3 * (sh_degree + 1) * (sh_degree + 1);
  densify_apply_kernel<<<(unsigned)((n + kApplyRows - 1) / kApplyRows), kApplyThreads, 0, s>>>(da, outc, pos, n);
  launches += 1;
  ctx->launches += launches;
  publish_words(ctx, &totals[2], 1, kMirrorDensify, s);  // the new count, through the mapped mirror
  ctx->launches += 1;
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return fail(ctx, NGS_ERR_CUDA, std::string("densify: ") + cudaGetErrorString(e));
  *n_out = (int64_t)static_cast<volatile uint64_t*>(ctx->h_total)[kMirrorDensify];
  return NGS_OK;
}

}  // extern "C"
