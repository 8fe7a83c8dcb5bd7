// Image loss of the training step (Sec. 5.1 "Loss"): L = (1 - lambda) L1 + lambda (1 - SSIM), with L1 the
// mean absolute difference and SSIM the mean structural similarity (Wang et al. 2004) over pixels and
// channels, with the 11 x 11 Gaussian window (sigma 1.5) and zero padding of 3D Gaussian splatting, and
// its gradient w.r.t. the rendered image.
//
// Per channel, with windowed moments mx = G * x, my = G * y, sxx = G * x^2, syy = G * y^2, sxy = G * xy:
//   s = (2 mx my + C1)(2 (sxy - mx my) + C2) / ((mx^2 + my^2 + C1)((sxx - mx^2) + (syy - my^2) + C2)).
// Since x enters s(p) only through mx(p), sxx(p) and sxy(p) of the windows that contain it,
//   dSSIM/dx(q) = [G * a](q) + 2 x(q) [G * b](q) + y(q) [G * c](q),
//   a = ds/dmx, b = ds/dsxx, c = ds/dsxy (per pixel, zero outside the image), G symmetric,
// divided by the 3 H W terms of the mean.
//
// Two kernels, one per convolution: the moments and from them s and a / b / c, then the gradient. A CTA takes 64 pixels x
// 32 rows of all channels, four input rows at a time: the rows are staged in shared memory (the next four are on
// their way meanwhile), each thread convolves four neighbouring pixels of one channel horizontally into a ring of 16
// rows, and each thread then convolves one column vertically for four output rows. Pairs of values (x and y, their
// squares) go through packed FP32x2 instructions together. Only a / b / c pass through memory (36 B per pixel), where
// four separable passes moved 24 planes of moments and partials; every sum has the order of those passes.
// 282 -> 144 us at 1920 x 1080 on GB300 (map 76, gradient 68), bound by FP32 issue: seven IEEE divisions per channel
// of a pixel are half of the map's instructions.
#include <math.h>
#include <string.h>

#include "ngs_internal.cuh"

namespace ngs {
namespace {

constexpr int kRadius = 5, kTaps = 2 * kRadius + 1;
constexpr float kC1 = 0.01f * 0.01f, kC2 = 0.03f * 0.03f;

// The normalised 11-tap Gaussian of sigma 1.5, passed by value (it lands in the constant bank).
struct Window {
  float2 g[kTaps];  // {w, w}
};

constexpr int kTileW = 64, kTileH = 32, kRows = 4;    // pixels of a CTA, rows at a time
constexpr int kHaloW = kTileW + 2 * kRadius;          // 74 columns per channel
constexpr int kStage = 76;                            // of a channel's row in the staging buffer
constexpr int kRing = 16;                             // rows of convolved values
constexpr int kRingW = 70;                            // of a channel's row in the ring (against bank conflicts)
constexpr int kSteps = kTileH / kRows + 3;            // groups of input rows, from row -6 of the tile on
constexpr int kLossThreads = 224;                     // 3 channels x 74 columns
constexpr int kOutThreads = 3 * kTileW;               // 192
static_assert(3 * kHaloW <= kLossThreads && kRows * 3 * (kTileW / 4) == kOutThreads, "threads");

// The horizontal convolution of four neighbouring outputs.
__device__ __forceinline__ void conv4(const Window& win, const float2 (&v)[14], float2 (&acc)[4]) {
#pragma unroll
  for (int o = 0; o < 4; ++o) {
    acc[o] = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < kTaps; ++k) acc[o] = __ffma2_rn(win.g[k], v[o + k], acc[o]);
  }
}
__device__ __forceinline__ void conv4(const Window& win, const float (&v)[14], float (&acc)[4]) {
#pragma unroll
  for (int o = 0; o < 4; ++o) {
    acc[o] = 0.f;
#pragma unroll
    for (int k = 0; k < kTaps; ++k) acc[o] = fmaf(win.g[k].x, v[o + k], acc[o]);
  }
}
__device__ __forceinline__ void load14(const float2* __restrict__ row, float2 (&v)[14]) {
  const float4* r4 = reinterpret_cast<const float4*>(row);
#pragma unroll
  for (int k = 0; k < 7; ++k) {
    const float4 q = r4[k];
    v[2 * k] = make_float2(q.x, q.y);
    v[2 * k + 1] = make_float2(q.z, q.w);
  }
}

// Windowed moments, the SSIM map's partials a, b, c (9 planes [channel][a b c] of H W floats) and the CTA's sums of s and
// |x - y|.
struct MapSmem {
  float2 in[kRows][3][kStage];    // {x, y}
  float2 m[kRing][3][kRingW];     // horizontally convolved {x, y}
  float2 q[kRing][3][kRingW];     // {x^2, y^2}
  float c[kRing][3][kRingW + 2];  // x y
};
__global__ void __launch_bounds__(kLossThreads, 3)
    ssim_map_kernel(Window win, const float* __restrict__ x, const float* __restrict__ y, int W, int H,
                    float* __restrict__ abc, double2* __restrict__ partial) {
  pdl_wait();
  extern __shared__ __align__(16) unsigned char smem[];
  MapSmem& sm = *reinterpret_cast<MapSmem*>(smem);
  __shared__ double2 s_sum[kLossThreads / 32];
  const int tid = threadIdx.x;
  const int x0 = blockIdx.x * kTileW, y0 = blockIdx.y * kTileH;
  // staging: neighbouring threads on neighbouring floats
  const int xs = tid / 3, ch = tid - 3 * xs, col = x0 - kRadius + xs;
  const bool live = tid < 3 * kHaloW && col >= 0 && col < W;
  const bool inside = live && xs >= kRadius && xs < kRadius + kTileW;
  const float* px = x + 3 * (ptrdiff_t)col + ch;
  const float* py = y + 3 * (ptrdiff_t)col + ch;
  const size_t stride = 3 * (size_t)W;
  auto load = [&](int row) {
    const bool ok = live && row >= 0 && row < H;
    return ok ? make_float2(px[(size_t)row * stride], py[(size_t)row * stride]) : make_float2(0.f, 0.f);
  };
  // horizontal: four pixels of a row of a channel; vertical: a column of a channel
  const int hrow = tid / 48, hch = (tid / 16) % 3, hx = 4 * (tid & 15);
  const int vch = tid / kTileW, vx = tid & (kTileW - 1);
  float2 next[kRows];
#pragma unroll
  for (int r = 0; r < kRows; ++r) next[r] = load(y0 - 6 + r);
  float s_acc = 0.f, l1_acc = 0.f;
  for (int step = 0; step < kSteps; ++step) {
    const int in0 = y0 - 6 + kRows * step;  // the first of this step's input rows
    if (in0 - 6 >= H) break;                // (its output rows would be below the image)
    if (tid < 3 * kHaloW) {
#pragma unroll
      for (int r = 0; r < kRows; ++r) {
        sm.in[r][ch][xs] = next[r];
        if (inside && in0 + r >= y0 && in0 + r < y0 + kTileH) l1_acc += fabsf(next[r].x - next[r].y);
      }
    }
    if (step + 1 < kSteps) {
#pragma unroll
      for (int r = 0; r < kRows; ++r) next[r] = load(in0 + kRows + r);
    }
    __syncthreads();
    const int slot = (step & 3) * kRows;
    if (tid < kOutThreads) {
      float2 v[14], sq[14], mo[4], qo[4];
      float xy[14], co[4];
      load14(&sm.in[hrow][hch][hx], v);
#pragma unroll
      for (int k = 0; k < 14; ++k) {
        sq[k] = __fmul2_rn(v[k], v[k]);
        xy[k] = v[k].x * v[k].y;
      }
      conv4(win, v, mo);
      conv4(win, sq, qo);
      conv4(win, xy, co);
      float4* pm = reinterpret_cast<float4*>(&sm.m[slot + hrow][hch][hx]);
      float4* pq = reinterpret_cast<float4*>(&sm.q[slot + hrow][hch][hx]);
      pm[0] = make_float4(mo[0].x, mo[0].y, mo[1].x, mo[1].y);
      pm[1] = make_float4(mo[2].x, mo[2].y, mo[3].x, mo[3].y);
      pq[0] = make_float4(qo[0].x, qo[0].y, qo[1].x, qo[1].y);
      pq[1] = make_float4(qo[2].x, qo[2].y, qo[3].x, qo[3].y);
      *reinterpret_cast<float4*>(&sm.c[slot + hrow][hch][hx]) = make_float4(co[0], co[1], co[2], co[3]);
    }
    __syncthreads();
    const int out0 = in0 - 6;  // output rows [out0, out0 + 4) need input rows out0 - 5 .. out0 + 8 = in0 - 11 .. in0 + 2
    if (step < 3 || tid >= kOutThreads || x0 + vx >= W) continue;
    float2 m[kRows], q[kRows];
    float c[kRows];
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      m[r] = q[r] = make_float2(0.f, 0.f);
      c[r] = 0.f;
    }
#pragma unroll
    for (int j = 0; j < 14; ++j) {
      const int rr = (slot + 5 + j) & (kRing - 1);  // ring row of input row out0 - 5 + j
      const float2 vm = sm.m[rr][vch][vx], vq = sm.q[rr][vch][vx];
      const float vc = sm.c[rr][vch][vx];
#pragma unroll
      for (int r = 0; r < kRows; ++r) {
        const int k = j - r;
        if (k < 0 || k >= kTaps) continue;
        m[r] = __ffma2_rn(win.g[k], vm, m[r]);
        q[r] = __ffma2_rn(win.g[k], vq, q[r]);
        c[r] = fmaf(win.g[k].x, vc, c[r]);
      }
    }
    const size_t npix = (size_t)W * H;
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      if (out0 + r >= H) break;
      const float mx = m[r].x, my = m[r].y, sxx = q[r].x, syy = q[r].y, sxy = c[r];
      const float n1 = 2.f * mx * my + kC1, n2 = 2.f * (sxy - mx * my) + kC2;
      const float d1 = mx * mx + my * my + kC1, d2 = (sxx - mx * mx) + (syy - my * my) + kC2;
      const float s = (n1 * n2) / (d1 * d2);
      s_acc += s;
      float* const out = abc + 3 * vch * npix + (size_t)(out0 + r) * W + x0 + vx;
      out[0] = s * (2.f * my / n1 - 2.f * my / n2 - 2.f * mx / d1 + 2.f * mx / d2);
      out[npix] = -s / d2;
      out[2 * npix] = 2.f * s / n2;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s_acc += __shfl_xor_sync(0xFFFFFFFFu, s_acc, o);
    l1_acc += __shfl_xor_sync(0xFFFFFFFFu, l1_acc, o);
  }
  if ((tid & 31) == 0) s_sum[tid >> 5] = make_double2(s_acc, l1_acc);
  __syncthreads();
  if (tid == 0) {
    double2 t = make_double2(0., 0.);
    for (int w = 0; w < kLossThreads / 32; ++w) {
      t.x += s_sum[w].x;
      t.y += s_sum[w].y;
    }
    partial[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = t;
  }
}

// The convolution of a, b, c and the gradient.
struct GradSmem {
  float2 ab[kRows][3][kStage];
  float c[kRows][3][kStage];
  float2 hab[kRing][3][kRingW];
  float hc[kRing][3][kRingW + 2];
};
__global__ void __launch_bounds__(kLossThreads, 4)
    ssim_grad_kernel(Window win, const float* __restrict__ abc, const float* __restrict__ x, const float* __restrict__ y,
                     int W, int H, float w_l1, float w_ssim, float* __restrict__ dl) {
  pdl_wait();
  extern __shared__ __align__(16) unsigned char smem[];
  GradSmem& sm = *reinterpret_cast<GradSmem*>(smem);
  const int tid = threadIdx.x;
  const int x0 = blockIdx.x * kTileW, y0 = blockIdx.y * kTileH;
  const int ch = tid / kHaloW, xs = tid - ch * kHaloW, col = x0 - kRadius + xs;
  const bool live = tid < 3 * kHaloW && col >= 0 && col < W;
  const size_t npix = (size_t)W * H;
  const float* pa = abc + 3 * (ptrdiff_t)ch * (ptrdiff_t)npix + col;
  const int hrow = tid / 48, hch = (tid / 16) % 3, hx = 4 * (tid & 15);
  const int vx = tid / 3, vch = tid - 3 * vx;  // interleaved, as the image is
  float2 nab[kRows];
  float nc[kRows];
  auto load = [&](int row0) {
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const bool ok = live && row0 + r >= 0 && row0 + r < H;
      const float* p = pa + (ptrdiff_t)(row0 + r) * W;
      nab[r] = ok ? make_float2(p[0], p[npix]) : make_float2(0.f, 0.f);
      nc[r] = ok ? p[2 * npix] : 0.f;
    }
  };
  load(y0 - 6);
  for (int step = 0; step < kSteps; ++step) {
    const int in0 = y0 - 6 + kRows * step;
    if (in0 - 6 >= H) break;
    if (tid < 3 * kHaloW) {
#pragma unroll
      for (int r = 0; r < kRows; ++r) {
        sm.ab[r][ch][xs] = nab[r];
        sm.c[r][ch][xs] = nc[r];
      }
    }
    if (step + 1 < kSteps) load(in0 + kRows);
    __syncthreads();
    const int slot = (step & 3) * kRows;
    if (tid < kOutThreads) {
      float2 v[14], to[4];
      float c[14], eo[4];
      load14(&sm.ab[hrow][hch][hx], v);
      const float4* c4 = reinterpret_cast<const float4*>(&sm.c[hrow][hch][hx]);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float4 t = c4[k];
        c[4 * k] = t.x;
        c[4 * k + 1] = t.y;
        if (k < 3) c[4 * k + 2] = t.z, c[4 * k + 3] = t.w;
      }
      conv4(win, v, to);
      conv4(win, c, eo);
      float4* pab = reinterpret_cast<float4*>(&sm.hab[slot + hrow][hch][hx]);
      pab[0] = make_float4(to[0].x, to[0].y, to[1].x, to[1].y);
      pab[1] = make_float4(to[2].x, to[2].y, to[3].x, to[3].y);
      *reinterpret_cast<float4*>(&sm.hc[slot + hrow][hch][hx]) = make_float4(eo[0], eo[1], eo[2], eo[3]);
    }
    __syncthreads();
    const int out0 = in0 - 6;
    if (step < 3 || tid >= kOutThreads || x0 + vx >= W) continue;
    const size_t at0 = ((size_t)out0 * W + x0) * 3 + tid;
    float2 t[kRows], xy[kRows];  // (the pixels are on their way during the convolution)
    float e[kRows];
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const size_t at = at0 + (size_t)r * 3 * W;
      xy[r] = out0 + r < H ? make_float2(x[at], y[at]) : make_float2(0.f, 0.f);
      t[r] = make_float2(0.f, 0.f);
      e[r] = 0.f;
    }
#pragma unroll
    for (int j = 0; j < 14; ++j) {
      const int rr = (slot + 5 + j) & (kRing - 1);
      const float2 vt = sm.hab[rr][vch][vx];
      const float ve = sm.hc[rr][vch][vx];
#pragma unroll
      for (int r = 0; r < kRows; ++r) {
        const int k = j - r;
        if (k < 0 || k >= kTaps) continue;
        t[r] = __ffma2_rn(win.g[k], vt, t[r]);
        e[r] = fmaf(win.g[k].x, ve, e[r]);
      }
    }
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      if (out0 + r >= H) break;
      const float a = xy[r].x, b = xy[r].y;
      const float dssim = t[r].x + 2.f * a * t[r].y + b * e[r];
      const float d = a - b;
      const float sgn = d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f);
      dl[at0 + (size_t)r * 3 * W] = w_l1 * sgn - w_ssim * dssim;
    }
  }
}

// The sums of all CTAs into the host mirror.
__global__ void __launch_bounds__(1024) loss_sum_kernel(const double2* __restrict__ partial, int n, uint64_t* mirror) {
  pdl_wait();
  __shared__ double2 s_sum[32];
  double2 t = make_double2(0., 0.);
  for (int i = threadIdx.x; i < n; i += 1024) {
    t.x += partial[i].x;
    t.y += partial[i].y;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    t.x += __shfl_xor_sync(0xFFFFFFFFu, t.x, o);
    t.y += __shfl_xor_sync(0xFFFFFFFFu, t.y, o);
  }
  if ((threadIdx.x & 31) == 0) s_sum[threadIdx.x >> 5] = t;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 32; ++w) {
      t.x += s_sum[w].x;
      t.y += s_sum[w].y;
    }
    mirror[0] = (uint64_t)__double_as_longlong(t.x);
    mirror[1] = (uint64_t)__double_as_longlong(t.y);
    __threadfence_system();
  }
}

}  // namespace
}  // namespace ngs

using namespace ngs;

extern "C" NGS_API int ngs_loss_l1_ssim(ngs_ctx* ctx, const float* image, const float* target, int32_t width,
                                        int32_t height, float lambda, float* dl_dimage, double* loss_out,
                                        void* stream) {
  if (!ctx) return NGS_ERR_INVALID_ARG;
  if (!image || !target || width < 1 || height < 1 || width > 16384 || height > 16384 || !(lambda >= 0.f) ||
      !(lambda <= 1.f))
    return fail(ctx, NGS_ERR_INVALID_ARG, "loss: null image/target, size outside 1..16384 or lambda outside [0, 1]");
  cudaStream_t s = (cudaStream_t)stream;
  const size_t npix = (size_t)width * height;
  Window win;
  {
    double g[kTaps], sum = 0.0;
    for (int i = 0; i < kTaps; ++i) {
      const double d = (double)(i - kRadius);
      g[i] = exp(-d * d / (2.0 * 1.5 * 1.5));
      sum += g[i];
    }
    for (int i = 0; i < kTaps; ++i) win.g[i] = make_float2((float)(g[i] / sum), (float)(g[i] / sum));
  }
  const dim3 grid((width + kTileW - 1) / kTileW, (height + kTileH - 1) / kTileH);
  const size_t abc_bytes = (sizeof(float) * 9 * npix + 15) & ~(size_t)15;
  const int rc = ensure(ctx, ctx->loss_tmp, abc_bytes + sizeof(double2) * (size_t)grid.x * grid.y);
  if (rc != NGS_OK) return rc;
  // 74 KB of shared memory: more than the default limit of a kernel (an attribute of the function, set on each call:
  // it is per device, and the call takes well under a microsecond)
  if (cudaFuncSetAttribute(ssim_map_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(MapSmem)) != cudaSuccess ||
      cudaFuncSetAttribute(ssim_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GradSmem)) != cudaSuccess)
    return fail(ctx, NGS_ERR_CUDA, "loss: setting the kernels' shared memory failed");
  float* abc = ctx->loss_tmp.as<float>();
  double2* partial = reinterpret_cast<double2*>(ctx->loss_tmp.as<char>() + abc_bytes);
  launch_pdl(ssim_map_kernel, grid, kLossThreads, sizeof(MapSmem), s, win, image, target, width, height, abc, partial);
  int launches = 1;
  if (dl_dimage) {
    const float nterms = 3.f * (float)npix;
    launch_pdl(ssim_grad_kernel, grid, kLossThreads, sizeof(GradSmem), s, win, abc, image, target, width, height,
               (1.f - lambda) / nterms, lambda / nterms, dl_dimage);
    launches += 1;
  }
  ctx->launches += launches;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(ctx, NGS_ERR_CUDA, std::string("loss launch: ") + cudaGetErrorString(e));
  if (loss_out) {  // one synchronisation: the scalar loss to the host (through the mapped mirror)
    launch_pdl(loss_sum_kernel, 1, 1024, 0, s, partial, (int)(grid.x * grid.y), ctx->d_h_total + kMirrorLoss);
    ctx->launches += 1;
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return fail(ctx, NGS_ERR_CUDA, std::string("loss read-back: ") + cudaGetErrorString(e));
    const volatile uint64_t* mirror = ctx->h_total + kMirrorLoss;
    const uint64_t w[2] = {mirror[0], mirror[1]};
    double h[2];
    memcpy(h, w, sizeof h);
    const double n = 3.0 * (double)npix;
    loss_out[0] = (1.0 - lambda) * (h[1] / n) + lambda * (1.0 - h[0] / n);
    loss_out[1] = h[1] / n;  // L1
    loss_out[2] = h[0] / n;  // SSIM
  }
  return NGS_OK;
}
