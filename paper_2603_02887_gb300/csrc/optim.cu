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

// ---- split / prune: one kernel decides and counts, one moves the rows -------------------------------------
//
// A Gaussian's place among the new ones is the number of survivors before it plus that of the granted splits before it,
// and the granted ones are the first `allowed` candidates: so one scan of (survivors, candidates) gives every place
// once the totals are known: two launches, where a scan for the candidates' ranks and one for the places took 13. A call for
// 100k Gaussians of degree 3, the counts read back: 206 -> 135 us.

constexpr int kPlanThreads = 256, kPlanBlock = 4 * kPlanThreads;
// A Gaussian's plan word: the survivors (11 bits) and candidates (11 bits) before it in its block of kPlanBlock, and
// its decision: 0 prune, 1 keep, 2 split candidate.
constexpr uint32_t kPlanBits = 11, kPlanMask = (1u << kPlanBits) - 1u;
static_assert(kPlanBlock <= (int)kPlanMask + 1, "the counts before an item of its block");

struct DensifyTotals {
  uint64_t blocks_done;  // zero before and after a launch
  uint64_t allowed;      // granted splits
};

__device__ __forceinline__ uint32_t densify_decision(const float* __restrict__ logits, const float* __restrict__ log_scales,
                                                     const float* __restrict__ accum, const float* __restrict__ count,
                                                     int64_t i, const ngs_densify_cfg& cfg) {
  const float op = 1.f / (1.f + expf(-logits[i]));
  const float smax = expf(fmaxf(log_scales[3 * i], fmaxf(log_scales[3 * i + 1], log_scales[3 * i + 2])));
  if (cfg.prune && (op < cfg.min_opacity || smax < cfg.min_scale)) return 0;
  return cfg.split && count[i] > 0.f && accum[i] / count[i] > cfg.grad_threshold ? 2 : 1;
}

// Inclusive prefix sum over the warp.
template <typename T>
__device__ __forceinline__ T warp_inclusive(T x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T y = __shfl_up_sync(0xFFFFFFFFu, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

// Plan words, and bases[b] = (survivors | candidates << 32) before block b: the block that finishes last scans the blocks'
// counts (no block waits on another), grants the splits and publishes the new number of Gaussians.
__global__ void __launch_bounds__(kPlanThreads) densify_plan_kernel(const float* __restrict__ logits,
                                                                    const float* __restrict__ log_scales,
                                                                    const float* __restrict__ accum,
                                                                    const float* __restrict__ count, int64_t n,
                                                                    ngs_densify_cfg cfg, uint32_t* __restrict__ plan,
                                                                    uint64_t* bases, DensifyTotals* totals,
                                                                    uint64_t* mirror) {
  pdl_wait();
  __shared__ uint64_t s_warp[kPlanThreads / 32];
  __shared__ bool s_last;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t i0 = (int64_t)blockIdx.x * kPlanBlock + 4 * tid;
  uint32_t d[4], mine = 0;  // survivors | candidates << 16
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    d[k] = i0 + k < n ? densify_decision(logits, log_scales, accum, count, i0 + k, cfg) : 0u;
    mine += (d[k] != 0 ? 1u : 0u) + (d[k] == 2 ? 1u << 16 : 0u);
  }
  const uint32_t incl = warp_inclusive(mine);
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  uint32_t run = incl - mine, all = 0;
#pragma unroll
  for (int w = 0; w < kPlanThreads / 32; ++w) {
    if (w < warp) run += (uint32_t)s_warp[w];
    all += (uint32_t)s_warp[w];
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (i0 + k < n) plan[i0 + k] = (run & 0xFFFFu) | (run >> 16) << kPlanBits | d[k] << (2 * kPlanBits);
    run += (d[k] != 0 ? 1u : 0u) + (d[k] == 2 ? 1u << 16 : 0u);
  }
  if (tid == 0) {
    bases[blockIdx.x] = (uint64_t)(all & 0xFFFFu) | (uint64_t)(all >> 16) << 32;
    __threadfence();
    s_last = atomicAdd(reinterpret_cast<unsigned long long*>(&totals->blocks_done), 1ull) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  uint64_t carry = 0;  // both counts stay below 2^30
  for (uint32_t b = 0; b < gridDim.x; b += kPlanThreads) {
    const uint32_t at = b + tid;
    const uint64_t v = at < gridDim.x ? __ldcg(reinterpret_cast<unsigned long long*>(bases) + at) : 0ull;
    const uint64_t in = warp_inclusive(v);
    __syncthreads();  // the previous use of s_warp is over
    if (lane == 31) s_warp[warp] = in;
    __syncthreads();
    uint64_t before = carry + in - v;
#pragma unroll
    for (int w = 0; w < kPlanThreads / 32; ++w) {
      if (w < warp) before += s_warp[w];
      carry += s_warp[w];
    }
    if (at < gridDim.x) bases[at] = before;
  }
  if (tid == 0) {
    const int64_t survivors = (int64_t)(carry & 0xFFFFFFFFu), candidates = (int64_t)(carry >> 32);
    const int64_t room = cfg.max_gaussians > survivors ? cfg.max_gaussians - survivors : 0;
    totals->allowed = (uint64_t)min(candidates, room);
    totals->blocks_done = 0;
    *mirror = (uint64_t)survivors + totals->allowed;
    __threadfence_system();
  }
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
  bool vec[5];  // the array's six pointers are 16-byte aligned
  int K3;       // 3 (sh_degree + 1)^2
};

// What becomes of each of a CTA's kApplyRows Gaussians: `copies` (0 pruned, 1 kept, 2 split) from row `to` on; a split's
// longest axis, half its extent along it and its direction.
constexpr int kApplyThreads = 256, kApplyRows = 64;
struct ApplyRows {
  uint32_t copies[kApplyRows], to[kApplyRows];
  int axis[kApplyRows];
  float half[kApplyRows], along[kApplyRows][3];
};

// Array gi (W floats per Gaussian, moved as VW at a time): a thread per element, so that reads and writes are coalesced.
template <int W, typename V>
__device__ __forceinline__ void apply_array(const DensifyArgs& a, int gi, const ApplyRows& rows, int64_t i0, int n_rows) {
  constexpr int E = W / (int)(sizeof(V) / sizeof(float));  // elements of a row
  const V *const src = reinterpret_cast<const V*>(a.src.p[gi]) + i0 * E;
  const V *const src_m = reinterpret_cast<const V*>(a.src_m.p[gi]) + i0 * E;
  const V *const src_v = reinterpret_cast<const V*>(a.src_v.p[gi]) + i0 * E;
  V *const dst = reinterpret_cast<V*>(a.dst.p[gi]), *const dst_m = reinterpret_cast<V*>(a.dst_m.p[gi]);
  V* const dst_v = reinterpret_cast<V*>(a.dst_v.p[gi]);
  for (int e = threadIdx.x; e < n_rows * E; e += kApplyThreads) {
    const int r = e / E, k = e - r * E;
    const uint32_t c = rows.copies[r];
    if (c == 0) continue;
    const int64_t to = (int64_t)rows.to[r] * E + k;
    const V val = src[e];
    if (c == 1) {
      const V vm = src_m[e], vv = src_v[e];
      dst[to] = val;
      dst_m[to] = vm;
      dst_v[to] = vv;
      continue;
    }
    V v0 = val, v1 = val;
    if constexpr (W == 3) {  // (means and log-scales; degree-0 colours are copied)
      if (gi == 0) {
        v0 = fmaf(rows.half[r], rows.along[r][k], val);
        v1 = fmaf(-rows.half[r], rows.along[r][k], val);
      } else if (gi == 1 && k == rows.axis[r]) {
        v0 = v1 = val + logf(0.8660254037844386f);  // sigma_a sqrt(3)/2
      }
    }
    dst[to] = v0;
    dst[to + E] = v1;
    dst_m[to] = dst_m[to + E] = V{};
    dst_v[to] = dst_v[to + E] = V{};
  }
}

// Bound by HBM: three arrays read and written, 59 floats a Gaussian at degree 3.
__global__ void __launch_bounds__(kApplyThreads) densify_apply_kernel(DensifyArgs a, const uint32_t* __restrict__ plan,
                                                                      const uint64_t* __restrict__ bases,
                                                                      const DensifyTotals* __restrict__ totals, int64_t n) {
  static_assert(kPlanBlock % kApplyRows == 0, "a CTA's rows lie in one block of the plan");
  pdl_wait();
  __shared__ ApplyRows rows;
  const int64_t i0 = (int64_t)blockIdx.x * kApplyRows;
  const int n_rows = (int)(n - i0 < kApplyRows ? n - i0 : kApplyRows);
  if ((int)threadIdx.x < n_rows) {
    const int r = threadIdx.x;
    const int64_t i = i0 + r;
    const uint32_t word = plan[i], d = word >> (2 * kPlanBits);
    const uint64_t base = bases[i0 / kPlanBlock];
    const uint32_t allowed = (uint32_t)totals->allowed;
    const uint32_t candidates = (uint32_t)(base >> 32) + (word >> kPlanBits & kPlanMask);
    const uint32_t copies = d == 0 ? 0u : (d == 2 && candidates < allowed ? 2u : 1u);
    rows.copies[r] = copies;
    rows.to[r] = (uint32_t)base + (word & kPlanMask) + min(candidates, allowed);
    if (copies == 2) {  // along the longest axis
      const float* ls = a.src.p[1] + 3 * i;
      const int ax = ls[0] >= ls[1] ? (ls[0] >= ls[2] ? 0 : 2) : (ls[1] >= ls[2] ? 1 : 2);
      float r3[3];
      quat_axis(a.src.p[2] + 4 * i, ax, r3);
      rows.axis[r] = ax;
      rows.half[r] = 0.5f * expf(ls[ax]);
      for (int k = 0; k < 3; ++k) rows.along[r][k] = r3[k];
    }
  }
  __syncthreads();
  apply_array<3, float>(a, 0, rows, i0, n_rows);
  apply_array<3, float>(a, 1, rows, i0, n_rows);
  if (a.vec[2]) apply_array<4, float4>(a, 2, rows, i0, n_rows);
  else apply_array<4, float>(a, 2, rows, i0, n_rows);
  apply_array<1, float>(a, 3, rows, i0, n_rows);
  switch (a.K3) {
    case 3: apply_array<3, float>(a, 4, rows, i0, n_rows); break;
    case 12:
      if (a.vec[4]) apply_array<12, float4>(a, 4, rows, i0, n_rows);
      else apply_array<12, float>(a, 4, rows, i0, n_rows);
      break;
    case 27: apply_array<27, float>(a, 4, rows, i0, n_rows); break;
    default:
      if (a.vec[4]) apply_array<48, float4>(a, 4, rows, i0, n_rows);
      else apply_array<48, float>(a, 4, rows, i0, n_rows);
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
  // scratch: the plan words; the totals and the blocks' first places
  const unsigned plan_blocks = (un + kPlanBlock - 1) / kPlanBlock;
  int rc = ensure(ctx, ctx->densify_tmp, sizeof(uint32_t) * (size_t)un);
  const size_t had = ctx->densify_totals.cap;
  if (rc == NGS_OK) rc = ensure(ctx, ctx->densify_totals, sizeof(DensifyTotals) + sizeof(uint64_t) * plan_blocks);
  if (rc != NGS_OK) return rc;
  uint32_t* plan = ctx->densify_tmp.as<uint32_t>();
  DensifyTotals* totals = ctx->densify_totals.as<DensifyTotals>();
  uint64_t* bases = reinterpret_cast<uint64_t*>(totals + 1);
  const cudaError_t me = ctx->densify_totals.cap == had ? cudaSuccess : cudaMemsetAsync(totals, 0, sizeof(DensifyTotals), s);
  if (me != cudaSuccess) return fail(ctx, NGS_ERR_CUDA, std::string("densify: ") + cudaGetErrorString(me));
  launch_pdl(densify_plan_kernel, plan_blocks, kPlanThreads, 0, s, params->d_opacity_logits, params->d_log_scales, accum,
             count, n, *cfg, plan, bases, totals, ctx->d_h_total + kMirrorDensify);
  DensifyArgs da;
  da.src = ptrs(*params);
  da.src_m = ptrs(*m);
  da.src_v = ptrs(*v);
  da.dst = ptrs(*out_params);
  da.dst_m = ptrs(*out_m);
  da.dst_v = ptrs(*out_v);
  for (int k = 0; k < 5; ++k)
    da.vec[k] = (((uintptr_t)da.src.p[k] | (uintptr_t)da.src_m.p[k] | (uintptr_t)da.src_v.p[k] | (uintptr_t)da.dst.p[k] |
                  (uintptr_t)da.dst_m.p[k] | (uintptr_t)da.dst_v.p[k]) & 15) == 0;
  da.K3 = 3 * (sh_degree + 1) * (sh_degree + 1);
  launch_pdl(densify_apply_kernel, (unsigned)((n + kApplyRows - 1) / kApplyRows), kApplyThreads, 0, s, da, plan, bases,
             totals, n);
  ctx->launches += 2;
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return fail(ctx, NGS_ERR_CUDA, std::string("densify: ") + cudaGetErrorString(e));
  *n_out = (int64_t)static_cast<volatile uint64_t*>(ctx->h_total)[kMirrorDensify];
  return NGS_OK;
}

}  // extern "C"
