// Per-tile front-to-back compositing (forward) and its path-replay adjoint (backward).
//
// One CTA per screen tile of any view of the batch (global tile index -> view by binary search over the
// views' first tiles), or persistent CTAs over a work list. The tile's depth-sorted splat list is walked in
// chunks of records staged in shared memory (half, one or two per pixel).
// Replay, and the forward of the exponential model (and of the quadratic ones on tiles of >= 256 pixels):
// two pixels per thread, (x, y) and (x, y + 4), so that a warp covers an 8 x 8 block; the two step through
// each entry together in packed FP32x2 instructions (add / mul / fma .rn.f32x2), each lane rounding like
// the one-pixel form, with splat operands staged in duplicated pairs. The replay sums its contributions over
// the 64 pixels for eight entries at a time. Other forwards: one thread per pixel, warps on 8 x 4 pixel blocks
// whose pixels are close and tend to saturate together.
//
// Forward, per pixel (Eq. generalized_gaussian with pbar_i from Eq. nexp_p and Table 1):
//   alpha_i = min(alpha_max, aleph_i K_i(p)), skipped when alpha_i < alpha_min;
//   quadratic:   pt = [alpha_i (1 + c taubar_i)]_+; if S + pt >= 1 the splat is k: pbar_k = 1 - S, the
//                ray has saturated and stops; else pbar_i = pt, S += pt, taubar += alpha_i;
//   exponential: stop before the splat that would take T below t_eps; pbar_i = alpha_i T, T *= 1 - alpha_i;
//   blended:     as quadratic with pt = alpha_i (1 - g + g P_i), P_i = prod_{j<i}(1 - alpha_j);
//   Vicini:      pbar_i = (1 - g) pbar_i^lin + g pbar_i^exp, the linear list saturating and the exponential
//                list stopping on their own; the ray stops once both have.
// A warp whose 32 pixels have all stopped leaves the chunk loop (ballot), and the CTA leaves the tile once
// every pixel has stopped (__syncthreads_count), which is where the faster-than-exponential models win.
//
// Backward (App. C), per pixel, replaying the same list front to back with identical FP32 arithmetic:
//   quadratic:   dL0/dalpha_i = DeltaE_i (1 + c taubar_i) + c Theta_i for i < k, Theta running down from
//                Theta_{-1} = A - E_k taubar_k (A = sum_{i<k} E_i alpha_i saved by the forward pass);
//                dL0/dE_i = pbar_i; dL0/dalpha_k = 0;
//   exponential: dL0/dalpha_i = T_i E_i - R_i / (1 - alpha_i), R_i = L0 - sum_{j<=i} E_j pbar_j;
//   blended:     dL0/dalpha_i = DeltaE_i (1 - g + g P_i) - g (B - B_i) / (1 - alpha_i), B_i the prefix sums
//                of DeltaE_l alpha_l P_l and B their total (saved by the forward pass);
//   Vicini:      (1 - g) x the linear adjoint + g x the exponential adjoint, each over its own list;
// then w = dL/d(log2 alpha) and its moments w, w dx, w dy, w dx^2, w dx dy, w dy^2 (which determine the
// gradient of the splat record, see the projection backward) and dL/dE: a warp gathers the w and pbar of eight
// entries in shared memory, sums them over its pixels four lanes to an entry, and adds the totals to the
// per-Gaussian buffer.
#include <algorithm>

#include <type_traits>

#include "ngs_internal.cuh"

namespace ngs {
namespace {

constexpr uint32_t kFull = 0xFFFFFFFFu;

// Stage splat record `id` in shared memory. An index outside [0, n_records) (which a correct binning never
// produces) is not read: the entry gets log2(aleph) = -inf, so no pixel composites it, and
// the device error word records the event.
__device__ __forceinline__ void stage_record(const float4* __restrict__ rec, uint32_t id, const RenderParams& rp,
                                             float4& r0, float4& r1, float& e2) {
  if (id < rp.n_records) {
    r0 = rec[3 * (size_t)id];
    r1 = rec[3 * (size_t)id + 1];
    e2 = rec[3 * (size_t)id + 2].x;
  } else {
    r0 = make_float4(0.f, 0.f, 0.f, 0.f);
    r1 = make_float4(0.f, -INFINITY, 0.f, 0.f);
    e2 = 0.f;
    atomicOr(rp.check, kCheckIndex);
  }
}

template <int TW, int TH, int PPT>
struct TileGeom {
  static constexpr int kPix = PPT;  // pixels per thread
  static constexpr int kThreads = TW * TH / kPix;
  static constexpr int kWarpsX = TW / 8;
  static_assert(TW % 8 == 0 && TH % (4 * PPT) == 0, "tile must be a multiple of 8 x (4 PPT)");
  // warp w covers the 8 x (4 PPT) block (w % kWarpsX, w / kWarpsX) of the tile; lane l owns its pixels
  // (l & 7, (l >> 3) + 4 k), k < PPT
  __device__ static void pixel(int tid, int k, int tile_x0, int tile_y0, int& x, int& y) {
    int warp = tid >> 5, lane = tid & 31;
    x = tile_x0 + (warp % kWarpsX) * 8 + (lane & 7);
    y = tile_y0 + (warp / kWarpsX) * 4 * PPT + (lane >> 3) + 4 * k;
  }
};

// The forward keeps one pixel per thread (a thread retires with its pixel); the replay takes two, so that
// the warp reduces once per 64 pixels.
constexpr int kBwdPix = 2;

// ---- forward ---------------------------------------------------------------------------------------

// Shared-memory staging of one chunk of CH splat records.
template <int CH>
struct StageBuf {
  float4 r0[CH];
  float4 r1[CH];
  float e2[CH];
};

// Stage list entries [base, base + CH) of the tile (those below `end`): slot k by thread k mod B.
template <int B, int CH>
__device__ __forceinline__ void stage_chunk(const float4* __restrict__ rec, const uint32_t* __restrict__ ids,
                                            const RenderParams& rp, uint32_t base, uint32_t end, StageBuf<CH>& sb,
                                            uint32_t* s_id) {
#pragma unroll
  for (int k = 0; k < (CH + B - 1) / B; ++k) {
    const int slot = k * B + (int)threadIdx.x;
    const uint32_t i = base + (uint32_t)slot;
    if (slot < CH && i < end) {
      const uint32_t id = ids[i];
      if (s_id) s_id[slot] = id < rp.n_records ? id : 0u;
      stage_record(rec, id, rp, sb.r0[slot], sb.r1[slot], sb.e2[slot]);
    }
  }
}

// Persistent schedule: the next tile of a CTA, the next entry of the work list taken with one atomic per
// CTA. Returns n_tiles when none is left.
__device__ __forceinline__ uint32_t next_tile(const uint32_t* __restrict__ work, uint32_t* counter, uint32_t n_tiles,
                                              uint32_t* s_next) {
  __syncthreads();  // every thread has read the previous s_next and is done with the staging buffers
  if (threadIdx.x == 0) *s_next = atomicAdd(counter, 1u);
  __syncthreads();
  const uint32_t w = *s_next;
  return w < n_tiles ? (work ? work[w] : w) : n_tiles;
}

// Staging of one chunk for the packed (two pixels per thread) forward and replay. The operands of FP32x2 instructions
// are duplicated: one 16-byte shared load gives the operand pairs {a, a, b, b} of two instructions. The replay
// keeps only C' and L so, and takes its other operands single, in scalar instructions (see kSlots).
template <int CH, bool REPLAY>
struct PairStageBuf {  // (the first arrays have an entry that is read ahead but never used)
  float4 r0[REPLAY ? CH + 1 : 1];  // replay: {u, v, A', B'}
  float4 q0[REPLAY ? 1 : CH + 1];  // forward: {-u, -u, -v, -v}
  float4 q1[REPLAY ? 1 : CH + 1];  // forward: {A', A', B', B'}
  float4 q2[CH + 1];  // {C', C', L, L}
  float4 q3[CH];  // forward: {E0, E0, E1, E1}; replay: {E0, E1, E2, record index (bits)}
  float2 q4[REPLAY ? 1 : CH];  // forward: {E2, E2}
};

// The packed form (exponential and quadratic models) is used while the forward's staging (72 B per record) stays
// within 40 KB of static shared memory.
template <int KIND, int CH>
constexpr bool kPairForm = (KIND == NGS_MODEL_EXP || KIND == NGS_MODEL_QUAD) && sizeof(PairStageBuf<CH, false>) <= 41248;

template <int B, int CH, bool REPLAY>
__device__ __forceinline__ void stage_chunk_pairs(const float4* __restrict__ rec, const uint32_t* __restrict__ ids,
                                                  const RenderParams& rp, uint32_t base, uint32_t end,
                                                  PairStageBuf<CH, REPLAY>& sb) {
#pragma unroll
  for (int k = 0; k < (CH + B - 1) / B; ++k) {
    const int slot = k * B + (int)threadIdx.x;
    const uint32_t i = base + (uint32_t)slot;
    if (slot < CH && i < end) {
      const uint32_t id = ids[i];
      float4 r0, r1;
      float e2;
      stage_record(rec, id, rp, r0, r1, e2);
      if constexpr (REPLAY) {
        sb.r0[slot] = r0;
      } else {
        sb.q0[slot] = make_float4(-r0.x, -r0.x, -r0.y, -r0.y);
        sb.q1[slot] = make_float4(r0.z, r0.z, r0.w, r0.w);
      }
      sb.q2[slot] = make_float4(r1.x, r1.x, r1.y, r1.y);
      if constexpr (REPLAY) {
        sb.q3[slot] = make_float4(r1.z, r1.w, e2, __uint_as_float(id < rp.n_records ? id : 0u));
      } else {
        sb.q3[slot] = make_float4(r1.z, r1.z, r1.w, r1.w);
        sb.q4[slot] = make_float2(e2, e2);
      }
    }
  }
}

__device__ __forceinline__ float2 lo_hi(float4 q, bool hi) { return hi ? make_float2(q.z, q.w) : make_float2(q.x, q.y); }

template <int TW, int TH, int KIND, int CH>
__device__ __forceinline__ void forward_tile(const float4* __restrict__ rec, const uint32_t* __restrict__ ids,
                                             const uint2* __restrict__ ranges, const RenderParams& rp,
                                             const ViewParams* __restrict__ views, float* __restrict__ image,
                                             int32_t* __restrict__ overdraw, float4* __restrict__ state,
                                             uint32_t tile, StageBuf<CH>& sb) {
  using G = TileGeom<TW, TH, 1>;
  constexpr int B = G::kThreads;
  const TileView tv = tile_view(rp, views, (uint32_t)tile);
  const int W = tv.W, H = tv.H;
  const int tx = tv.local % tv.tiles_x, ty = tv.local / tv.tiles_x;
  int tid = threadIdx.x;
  int x, y;
  G::pixel(tid, 0, tx * TW, ty * TH, x, y);
  bool inside = x < W && y < H;
  float px = (float)x + 0.5f, py = (float)y + 0.5f;
  uint2 range = ranges[tile];
  bool done = !inside;
  int od = 0;
  uint32_t stop = range.y - range.x;  // entries walked (n of the replay state)
  bool saturated = false;  // quadratic / blended: the ray saturated; Vicini: its linear list did
  float C0 = 0.f, C1 = 0.f, C2 = 0.f;  // Vicini: the linear list's sum
  // quadratic (A = sum E alpha, tau) and blended (A = sum E alpha P, X = sum alpha P, P) state
  float S = 0.f, tau = 0.f, A0 = 0.f, A1 = 0.f, A2 = 0.f, Ek0 = rp.bg[0], Ek1 = rp.bg[1], Ek2 = rp.bg[2];
  float P = 1.f, X = 0.f;
  // exponential state (Vicini: its exponential list, with its own colour sum)
  float T = 1.f;
  bool stop_e = false;
  float Ce0 = 0.f, Ce1 = 0.f, Ce2 = 0.f;
  const float amax = rp.alpha_max, l2min = rp.log2_alpha_min, c = rp.c;
  for (uint32_t base = range.x; base < range.y; base += CH) {
    if (__syncthreads_count(done) == B) break;
    stage_chunk<B, CH>(rec, ids, rp, base, range.y, sb, nullptr);
    __syncthreads();
    int cnt = (int)min((uint32_t)CH, range.y - base);
    if (__any_sync(kFull, !done)) {
      for (int j = 0; j < cnt && !done; ++j) {
        float4 r0 = sb.r0[j], r1 = sb.r1[j];
        float dx, dy;
        float e = splat_log2_alpha(px, py, r0, r1, dx, dy);
        if (e < l2min) continue;
        float alpha = fminf(amax, fast_exp2(e));
        float E0 = r1.z, E1 = r1.w, E2 = sb.e2[j];
        if constexpr (KIND == NGS_MODEL_QUAD || KIND == NGS_MODEL_BLEND) {
          const float pt = KIND == NGS_MODEL_QUAD ? quad_slope(alpha, c, tau) : blend_slope(alpha, c, rp.c1, P);
          float Sn = __fadd_rn(S, pt);
          ++od;
          if (Sn >= 1.0f) {  // the saturating splat k: pbar_k = 1 - S (Eq. nexp_p)
            float pk = 1.0f - S;
            C0 = fmaf(E0, pk, C0);
            C1 = fmaf(E1, pk, C1);
            C2 = fmaf(E2, pk, C2);
            Ek0 = E0;
            Ek1 = E1;
            Ek2 = E2;
            saturated = true;
            done = true;
            stop = base + j + 1 - range.x;
            break;
          }
          C0 = fmaf(E0, pt, C0);
          C1 = fmaf(E1, pt, C1);
          C2 = fmaf(E2, pt, C2);
          const float w = KIND == NGS_MODEL_QUAD ? alpha : __fmul_rn(alpha, P);
          A0 = fmaf(E0, w, A0);
          A1 = fmaf(E1, w, A1);
          A2 = fmaf(E2, w, A2);
          S = Sn;
          if (KIND == NGS_MODEL_QUAD) {
            tau = __fadd_rn(tau, alpha);
          } else {
            X = __fadd_rn(X, w);
            P = __fmul_rn(P, __fsub_rn(1.0f, alpha));
          }
        } else if constexpr (KIND == NGS_MODEL_VICINI) {
          // the exponential list (own t_eps stop) and the linear list (own saturation), lerped by gamma
          float pe = 0.f;
          if (!stop_e) {
            const float testT = __fmul_rn(T, __fsub_rn(1.0f, alpha));
            if (testT < rp.t_eps) {
              stop_e = true;
            } else {
              pe = alpha * T;
              T = testT;
            }
          }
          if (saturated && stop_e) {  // both lists have stopped before this splat
            done = true;
            stop = base + j - range.x;
            break;
          }
          float pl = 0.f;
          if (!saturated) {
            const float Sn = __fadd_rn(S, alpha);
            if (Sn >= 1.0f) {
              pl = 1.0f - S;
              S = 1.0f;
              saturated = true;
              Ek0 = E0;
              Ek1 = E1;
              Ek2 = E2;
            } else {
              pl = alpha;
              S = Sn;
            }
          }
          C0 = fmaf(E0, pl, C0);
          C1 = fmaf(E1, pl, C1);
          C2 = fmaf(E2, pl, C2);
          Ce0 = fmaf(E0, pe, Ce0);
          Ce1 = fmaf(E1, pe, Ce1);
          Ce2 = fmaf(E2, pe, Ce2);
          ++od;
          if (saturated && stop_e) {
            done = true;
            stop = base + j + 1 - range.x;
            break;
          }
        } else {
          float testT = __fmul_rn(T, __fsub_rn(1.0f, alpha));
          if (testT < rp.t_eps) {
            done = true;
            stop = base + j - range.x;
            break;
          }
          float w = alpha * T;
          C0 = fmaf(E0, w, C0);
          C1 = fmaf(E1, w, C1);
          C2 = fmaf(E2, w, C2);
          T = testT;
          ++od;
        }
        if (rp.max_splats > 0 && od == rp.max_splats) {
          done = true;
          stop = base + j + 1 - range.x;
          break;
        }
      }
    }
  }
  if (!inside) return;  // (the caller's next barrier is reached by every thread)
  const size_t lpix = (size_t)y * W + x;                         // pixel within the view
  const size_t pix = view_pix_base(rp, views, tv.view) + lpix;  // packed pixel of the replay state
  float* const out_image = view_image(rp, views, tv.view, image);
  int32_t* const out_overdraw = view_overdraw(rp, views, tv.view, overdraw);
  float L0, L1, L2, Tend;
  if constexpr (KIND == NGS_MODEL_VICINI) {
    Tend = fmaf(rp.c1, 1.0f - S, c * T);  // lerp(1 - S, T_exp, gamma)
    L0 = fmaf(rp.c1, C0, fmaf(c, Ce0, rp.bg[0] * Tend));
    L1 = fmaf(rp.c1, C1, fmaf(c, Ce1, rp.bg[1] * Tend));
    L2 = fmaf(rp.c1, C2, fmaf(c, Ce2, rp.bg[2] * Tend));
  } else {
    Tend = KIND == NGS_MODEL_EXP ? T : (saturated ? 0.f : 1.f - S);
    L0 = C0 + rp.bg[0] * Tend;
    L1 = C1 + rp.bg[1] * Tend;
    L2 = C2 + rp.bg[2] * Tend;
  }
  out_image[3 * lpix] = L0;
  out_image[3 * lpix + 1] = L1;
  out_image[3 * lpix + 2] = L2;
  if (out_overdraw) out_overdraw[lpix] = od;
  uint32_t nbits = stop | (saturated ? 0x80000000u : 0u);
  if constexpr (KIND == NGS_MODEL_QUAD) {
    state[2 * pix] = make_float4(__uint_as_float(nbits), Ek0, Ek1, Ek2);
    state[2 * pix + 1] = make_float4(A0, A1, A2, tau);
  } else if constexpr (KIND == NGS_MODEL_BLEND) {
    state[2 * pix] = make_float4(__uint_as_float(nbits), Ek0, Ek1, Ek2);
    state[2 * pix + 1] = make_float4(A0, A1, A2, X);
  } else if constexpr (KIND == NGS_MODEL_VICINI) {
    state[2 * pix] = make_float4(__uint_as_float(nbits), Ek0, Ek1, Ek2);
    state[2 * pix + 1] = make_float4(fmaf(rp.bg[0], T, Ce0), fmaf(rp.bg[1], T, Ce1), fmaf(rp.bg[2], T, Ce2), 0.f);
  } else {
    state[2 * pix] = make_float4(__uint_as_float(nbits), L0, L1, L2);
    state[2 * pix + 1] = make_float4(Tend, 0.f, 0.f, 0.f);
  }
}

// Packed forward (exponential and quadratic): two pixels per thread, (x, y) and (x, y + 4), stepping through
// each entry together in FP32x2 instructions. Each lane rounds exactly like the one-pixel form above, so
// the image, the stop index and the replay state are the same bits. A pixel that has stopped, or that
// does not composite the entry, gets alpha = 0, which leaves its sums exactly unchanged.
template <int TW, int TH, int KIND, int CH, bool AHEAD>
__device__ __forceinline__ void forward_tile_pairs(const float4* __restrict__ rec, const uint32_t* __restrict__ ids,
                                                   const uint2* __restrict__ ranges, const RenderParams& rp,
                                                   const ViewParams* __restrict__ views, float* __restrict__ image,
                                                   int32_t* __restrict__ overdraw, float4* __restrict__ state,
                                                   uint32_t tile, PairStageBuf<CH, false>& sb) {
  using G = TileGeom<TW, TH, 2>;
  constexpr int B = G::kThreads;
  const TileView tv = tile_view(rp, views, (uint32_t)tile);
  const int W = tv.W, H = tv.H;
  const int tx = tv.local % tv.tiles_x, ty = tv.local / tv.tiles_x;
  int x, y;
  G::pixel(threadIdx.x, 0, tx * TW, ty * TH, x, y);  // the second pixel is (x, y + 4)
  const bool in0 = x < W && y < H, in1 = x < W && y + 4 < H;
  const float2 one = make_float2(1.f, 1.f), neg = make_float2(-1.f, -1.f), zero = make_float2(0.f, 0.f);
  const float2 px = make_float2((float)x + 0.5f, (float)x + 0.5f);
  const float2 py = make_float2((float)y + 0.5f, (float)(y + 4) + 0.5f);
  const uint2 range = ranges[tile];
  bool done0 = !in0, done1 = !in1;
  int od0 = 0, od1 = 0;
  uint32_t stop0 = range.y - range.x, stop1 = stop0;  // entries walked (n of the replay state)
  bool sat0 = false, sat1 = false;
  float2 C0 = zero, C1 = zero, C2 = zero;
  float2 S = zero, tau = zero, A0 = zero, A1 = zero, A2 = zero;  // quadratic
  float Ek[2][3] = {{rp.bg[0], rp.bg[1], rp.bg[2]}, {rp.bg[0], rp.bg[1], rp.bg[2]}};
  float2 T = one;  // exponential
  const float amax = rp.alpha_max, l2min = rp.log2_alpha_min;
  const float2 c2 = make_float2(rp.c, rp.c);
  for (uint32_t base = range.x; base < range.y; base += CH) {
    if (__syncthreads_count(done0 && done1) == B) break;
    stage_chunk_pairs<B, CH>(rec, ids, rp, base, range.y, sb);
    __syncthreads();
    const int cnt = (int)min((uint32_t)CH, range.y - base);
    if (__any_sync(kFull, !(done0 && done1))) {
      auto exponent = [&](int j) {
        const float4 q0 = sb.q0[j], q1 = sb.q1[j], q2 = sb.q2[j];
        const float2 dx = __fadd2_rn(px, lo_hi(q0, false));
        const float2 adx = __fmul2_rn(lo_hi(q1, false), dx);
        const float2 dy = __fadd2_rn(py, lo_hi(q0, true));
        const float2 t = __ffma2_rn(lo_hi(q1, true), dy, adx);
        const float2 cdd = __fmul2_rn(__fmul2_rn(lo_hi(q2, false), dy), dy);
        return __fadd2_rn(lo_hi(q2, true), __ffma2_rn(dx, t, cdd));
      };
      float2 e_next;
      if constexpr (AHEAD) e_next = exponent(0);
      for (int j = 0; j < cnt; ++j) {
        float2 e;
        if constexpr (AHEAD) {  // the next entry's, while this one is composited
          e = e_next;
          e_next = exponent(j + 1);
        } else {
          e = exponent(j);
        }
        const bool on0 = !done0 && e.x >= l2min, on1 = !done1 && e.y >= l2min;
        // warp-uniform: a lane that does not composite the entry (or has stopped) runs the step with
        // alpha = 0, which leaves its sums exactly as they were; the warp leaves the chunk once all of its
        // pixels have stopped
        if (__ballot_sync(kFull, on0 || on1) == 0u) {
          if (__all_sync(kFull, done0 && done1)) break;
          continue;
        }
        const float4 q3 = sb.q3[j];
        const float2 E0 = lo_hi(q3, false), E1 = lo_hi(q3, true), E2 = sb.q4[j];
        const float2 alpha = make_float2(on0 ? fminf(amax, fast_exp2(e.x)) : 0.f, on1 ? fminf(amax, fast_exp2(e.y)) : 0.f);
        const uint32_t pos = base + j - range.x;
        bool c0, c1;  // composited (the overdraw count)
        if constexpr (KIND == NGS_MODEL_QUAD) {
          const float2 ptr = __fmul2_rn(alpha, __ffma2_rn(c2, tau, one));
          const float2 pt = make_float2(fmaxf(ptr.x, 0.f), fmaxf(ptr.y, 0.f));
          const float2 Sn = __fadd2_rn(S, pt);
          const bool s0 = on0 && Sn.x >= 1.0f, s1 = on1 && Sn.y >= 1.0f;  // the saturating splat k
          const float2 oms = __ffma2_rn(S, neg, one);                     // pbar_k = 1 - S (Eq. nexp_p)
          const float2 wc = make_float2(s0 ? oms.x : pt.x, s1 ? oms.y : pt.y);
          const float2 wa = make_float2(s0 ? 0.f : alpha.x, s1 ? 0.f : alpha.y);
          C0 = __ffma2_rn(E0, wc, C0);
          C1 = __ffma2_rn(E1, wc, C1);
          C2 = __ffma2_rn(E2, wc, C2);
          A0 = __ffma2_rn(E0, wa, A0);
          A1 = __ffma2_rn(E1, wa, A1);
          A2 = __ffma2_rn(E2, wa, A2);
          S = make_float2(s0 ? S.x : Sn.x, s1 ? S.y : Sn.y);
          tau = __fadd2_rn(tau, wa);
          if (s0) {
            Ek[0][0] = E0.x, Ek[0][1] = E1.x, Ek[0][2] = E2.x;
            sat0 = done0 = true;
            stop0 = pos + 1;
          }
          if (s1) {
            Ek[1][0] = E0.y, Ek[1][1] = E1.y, Ek[1][2] = E2.y;
            sat1 = done1 = true;
            stop1 = pos + 1;
          }
          c0 = on0;
          c1 = on1;
        } else {
          // stop before the splat that would take T below t_eps (only a pixel that composites can; it happens at most
          // once per pixel, so the warp tests for it together)
          float2 testT = __fmul2_rn(T, __ffma2_rn(alpha, neg, one)), a = alpha;
          c0 = on0;
          c1 = on1;
          const bool st0 = testT.x < rp.t_eps, st1 = testT.y < rp.t_eps;
          if (__any_sync(kFull, st0 || st1)) {
            if (st0) {
              done0 = true;
              stop0 = pos;
              c0 = false;
              a.x = 0.f;
              testT.x = T.x;
            }
            if (st1) {
              done1 = true;
              stop1 = pos;
              c1 = false;
              a.y = 0.f;
              testT.y = T.y;
            }
          }
          const float2 w = __fmul2_rn(a, T);
          C0 = __ffma2_rn(E0, w, C0);
          C1 = __ffma2_rn(E1, w, C1);
          C2 = __ffma2_rn(E2, w, C2);
          T = testT;
        }
        od0 += c0;
        od1 += c1;
        if (rp.max_splats > 0) {
          if (c0 && !done0 && od0 == rp.max_splats) {
            done0 = true;
            stop0 = pos + 1;
          }
          if (c1 && !done1 && od1 == rp.max_splats) {
            done1 = true;
            stop1 = pos + 1;
          }
        }
      }
    }
  }
  const size_t pbase = view_pix_base(rp, views, tv.view);
  float* const out_image = view_image(rp, views, tv.view, image);
  int32_t* const out_overdraw = view_overdraw(rp, views, tv.view, overdraw);
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    if (!(k ? in1 : in0)) continue;
    const size_t lpix = (size_t)(y + 4 * k) * W + x;  // pixel within the view
    const size_t pix = pbase + lpix;                  // packed pixel of the replay state
    const float c0v = k ? C0.y : C0.x, c1v = k ? C1.y : C1.x, c2v = k ? C2.y : C2.x;
    const bool sat = k ? sat1 : sat0;
    const float Tend = KIND == NGS_MODEL_EXP ? (k ? T.y : T.x) : (sat ? 0.f : 1.f - (k ? S.y : S.x));
    const float L0 = c0v + rp.bg[0] * Tend, L1 = c1v + rp.bg[1] * Tend, L2 = c2v + rp.bg[2] * Tend;
    out_image[3 * lpix] = L0;
    out_image[3 * lpix + 1] = L1;
    out_image[3 * lpix + 2] = L2;
    if (out_overdraw) out_overdraw[lpix] = k ? od1 : od0;
    const uint32_t nbits = (k ? stop1 : stop0) | (sat ? 0x80000000u : 0u);
    if constexpr (KIND == NGS_MODEL_QUAD) {
      state[2 * pix] = make_float4(__uint_as_float(nbits), Ek[k][0], Ek[k][1], Ek[k][2]);
      state[2 * pix + 1] = make_float4(k ? A0.y : A0.x, k ? A1.y : A1.x, k ? A2.y : A2.x, k ? tau.y : tau.x);
    } else {
      state[2 * pix] = make_float4(__uint_as_float(nbits), L0, L1, L2);
      state[2 * pix + 1] = make_float4(Tend, 0.f, 0.f, 0.f);
    }
  }
}

// The packed forward pays where pixels walk long lists: always for the exponential model; for the quadratic
// models (rays saturate after ~8 splats, and a thread runs until the later of its two pixels stops) only on
// tiles of 256 pixels or more (measured on GB300 at 500k / 1080p: exponential 8x8 forward -10 %,
// quadratic 16x16 -1 %, quadratic 8x8 +3 % to +30 %).
template <int TW, int TH, int KIND, int CH>
constexpr bool kPairFwd = kPairForm<KIND, CH> && (KIND == NGS_MODEL_EXP || TW * TH >= 256);
template <int TW, int TH, int KIND, int CH>
constexpr int kFwdThreads = TW * TH / (kPairFwd<TW, TH, KIND, CH> ? 2 : 1);
// The packed quadratic forward on 16x16 tiles: nine CTAs of 128 threads per SM (at most 56 registers)
// instead of the eight its 64 registers would allow.
template <int TW, int TH, int KIND, int CH>
constexpr int kFwdMinBlocks = (kPairFwd<TW, TH, KIND, CH> && KIND == NGS_MODEL_QUAD && TW * TH == 256) ? 9 : 1;

// How a launch walks the tiles: one CTA per tile; persistent CTAs over the work list; or one CTA per tile that reads
// ahead, for frames of so few tiles that each warp's own latency is the time. Reading ahead takes the next entry's
// exponent off the chain of dependent instructions of an entry, at the price of a few more instructions (1k Gaussians,
// 128x128, exponential: 24.9 + 29.0 -> 22.6 + 26.9 us; 50k, 640x360, c = +0.5: 63 + 45 -> 56 + 42; but 500k, 1920x1080,
// exponential: 187 + 349 -> 195 + 365).
enum Walk { kTiles, kPersistent, kAhead };

template <int TW, int TH, int KIND, int CH, Walk WALK>
__global__ void __launch_bounds__(kFwdThreads<TW, TH, KIND, CH>, kFwdMinBlocks<TW, TH, KIND, CH>)
    composite_forward_kernel(const float4* __restrict__ rec,
                                                                   const uint32_t* __restrict__ ids,
                                                                   const uint2* __restrict__ ranges, RenderParams rp,
                                                                   const ViewParams* __restrict__ views,
                                                                   float* __restrict__ image,
                                                                   int32_t* __restrict__ overdraw,
                                                                   float4* __restrict__ state,
                                                                   const uint32_t* __restrict__ work,
                                                                   uint32_t* counter) {
  pdl_wait();
  using Buf = std::conditional_t<kPairFwd<TW, TH, KIND, CH>, PairStageBuf<CH, false>, StageBuf<CH>>;
  __shared__ Buf sb;
  auto one_tile = [&](uint32_t tile) {
    if constexpr (kPairFwd<TW, TH, KIND, CH>)
      forward_tile_pairs<TW, TH, KIND, CH, WALK == kAhead>(rec, ids, ranges, rp, views, image, overdraw, state, tile, sb);
    else
      forward_tile<TW, TH, KIND, CH>(rec, ids, ranges, rp, views, image, overdraw, state, tile, sb);
  };
  if constexpr (WALK == kPersistent) {
    __shared__ uint32_t s_next;
    for (;;) {
      const uint32_t tile = next_tile(work, counter, rp.n_tiles, &s_next);
      if (tile >= rp.n_tiles) break;
      one_tile(tile);
    }
  } else {
    one_tile(blockIdx.x);
  }
}

// ---- backward (path replay) --------------------------------------------------------------------------

struct BwdPixel {
  float px, py;
  uint32_t last;        // replay entries [range.x, last)
  float g0, g1, g2;
  float gEk, gTh, gL0;  // quadratic: g.E_k, g.Theta; exponential: g.L0; Vicini: both lists' (gEk, gL0)
  float S, tau, T, gacc;
  float P, gB, gBi;     // blended: prod (1 - alpha), g.B and its running prefix
  bool sat, stop_e;     // Vicini: the linear list saturated / the exponential list stopped
};

// ---- replay: sums over a warp's pixels ----------------------------------------------------------------
//
// A warp holds each composited entry's w = dL/d(log2 alpha) (over ln 2) and wE = dL0/dE of its 64 pixels, 16 B per
// lane, until kSlots entries have gathered; then lane (r, e) sums entry e over the pixel rows r and r + 4, and the four
// lanes of an entry add their sums. About 16 instructions an entry, and 9 atomics in two instructions. Reducing each
// entry by itself took about 50: nine sums through twelve shuffles, or up to 16 lanes' own atomics, whichever were fewer.
// Eight entries are the most whose words leave the registers, not shared memory, to limit a multiprocessor's warps (28).
// What bounds the walk now are the shared-memory pipe (82 % busy) and the issue slots (70 %): a 16-byte load takes two of the pipe's cycles
// even where all lanes read the same words, which is why the replay stages its operands single (273 us; duplicated for
// the packed instructions as in the forward: 326 us). Replay before -> now: 500k, 1920x1080, exponential on 8 x 8 tiles
// 326 -> 273 us, c = -0.5 on 16 x 16 147 -> 133 us; 1M, 1297x840, c = 0 101 -> 96 us; 32 views of 3M 9.29 -> 8.2 ms;
// 1k, 128x128 27 -> 22 us.
constexpr int kSlots = 8;
constexpr int kSlotStride = 33;  // float4: eight lanes read eight entries without bank conflicts

struct ReplayWarp {
  float4 w[kSlots * kSlotStride];  // [entry][lane]: {w, w, wE, wE} of pixels (x, y) and (x, y + 4)
  float4 g01[32];                  // [lane]: {g0, g0, g1, g1} of the two pixels
  float2 g2[32];
};

// The entry in slot lane % kSlots, held by each of its four lanes.
struct ReplaySlot {
  float u, v;
  uint32_t id;  // record index
};

// The replay of a warp's 8 x 8 block starts: the upstream gradients of the thread's two pixels. A lane with one that
// is not finite (returned) adds its own products to dL/dE (replay_odd_lane), so that it reaches only the entries it composites.
__device__ __forceinline__ bool replay_begin(ReplayWarp& rw, const float (&ga)[3], const float (&gb)[3], int lane) {
  const bool odd = !(isfinite(ga[0]) && isfinite(ga[1]) && isfinite(ga[2]) && isfinite(gb[0]) && isfinite(gb[1]) &&
                     isfinite(gb[2]));
  rw.g01[lane] = odd ? make_float4(0.f, 0.f, 0.f, 0.f) : make_float4(ga[0], gb[0], ga[1], gb[1]);
  rw.g2[lane] = odd ? make_float2(0.f, 0.f) : make_float2(ga[2], gb[2]);
  return odd;
}

__device__ __forceinline__ void replay_odd_lane(float* dst, float g0, float g1, float g2, float wE) {
  atomicAdd(dst + 6, g0 * wE);
  atomicAdd(dst + 7, g1 * wE);
  atomicAdd(dst + 8, g2 * wE);
}

// Adds the sums of the first `count` gathered entries to grad2d: the moments w dx, w dy, w dx^2, w dx dy, w dy^2, w
// and the three of dL/dE. (bx, by): the centre of the block's first pixel.
__device__ __forceinline__ void replay_flush(const ReplayWarp& rw, const ReplaySlot& slot, uint32_t count, float bx,
                                             float by, float4* __restrict__ grad2d, int lane) {
  __syncwarp();
  const uint32_t e = lane & 7, r = lane >> 3;
  const float2 one = make_float2(1.f, 1.f), zero = make_float2(0.f, 0.f);
  const float2 dy = __fadd2_rn(make_float2(by + (float)r, by + (float)(r + 4)), make_float2(-slot.v, -slot.v));
  float2 dx = __fadd2_rn(make_float2(bx, bx), make_float2(-slot.u, -slot.u));
  float2 s0 = zero, s1 = zero, s2 = zero, c0 = zero, c1 = zero, c2 = zero;
  const float4* w = rw.w + e * kSlotStride + 8 * r;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const float4 ww = w[c], g01 = rw.g01[8 * r + c];
    const float2 g2 = rw.g2[8 * r + c];
    const float2 wgt = lo_hi(ww, false), wE = lo_hi(ww, true);
    const float2 t = __fmul2_rn(wgt, dx);
    s0 = __fadd2_rn(s0, wgt);
    s1 = __fadd2_rn(s1, t);
    s2 = __ffma2_rn(t, dx, s2);
    c0 = __ffma2_rn(lo_hi(g01, false), wE, c0);
    c1 = __ffma2_rn(lo_hi(g01, true), wE, c1);
    c2 = __ffma2_rn(g2, wE, c2);
    if (c < 7) dx = __fadd2_rn(dx, one);
  }
  const float2 wdy = __fmul2_rn(s0, dy), wdxdy = __fmul2_rn(s1, dy), wdydy = __fmul2_rn(wdy, dy);
  const float v[9] = {s1.x + s1.y,       wdy.x + wdy.y, s2.x + s2.y, wdxdy.x + wdxdy.y, wdydy.x + wdydy.y,
                      s0.x + s0.y,       c0.x + c0.y,   c1.x + c1.y, c2.x + c2.y};
  // over the entry's four lanes, transposing: lane r ends with the totals 2 r and 2 r + 1
  const bool b1 = r & 2, b0 = r & 1;
  float x[4], y[2];
#pragma unroll
  for (int k = 0; k < 4; ++k) x[k] = (b1 ? v[k + 4] : v[k]) + __shfl_xor_sync(kFull, b1 ? v[k] : v[k + 4], 16);
#pragma unroll
  for (int k = 0; k < 2; ++k) y[k] = (b0 ? x[k + 2] : x[k]) + __shfl_xor_sync(kFull, b0 ? x[k] : x[k + 2], 8);
  float z = v[8] + __shfl_xor_sync(kFull, v[8], 16);
  z += __shfl_xor_sync(kFull, z, 8);
  if (e < count) {
    float* dst = reinterpret_cast<float*>(grad2d + 3 * (size_t)slot.id);
    atomicAdd(reinterpret_cast<float2*>(dst + 2 * r), make_float2(y[0], y[1]));
    if (r == 0) atomicAdd(dst + 8, z);
  }
  __syncwarp();  // the slots are free
}

// One list entry for one pixel of the replay: its w and wE (untouched where it does not composite the splat), and
// whether it does.
template <int KIND>
__device__ __forceinline__ bool bwd_step(BwdPixel& p, float dx, float adx, float4 r0, float4 r1, const float& e2,
                                         uint32_t pos, const RenderParams& rp, float& w_out, float& wE_out) {
  if (pos >= p.last) return false;
  float dy;
  float e = splat_log2_alpha_col(dx, adx, p.py, r0, r1, dy);
  if (e < rp.log2_alpha_min) return false;
  float raw = fast_exp2(e);
  float alpha = fminf(rp.alpha_max, raw);
  float E0 = r1.z, E1 = r1.w, E2 = e2;
  float gE = fmaf(p.g2, E2, fmaf(p.g1, E1, p.g0 * E0));  // g.E_i
  float dLda, wE;
  if constexpr (KIND == NGS_MODEL_BLEND) {
    // L0 = sum_{i<k} DeltaE_i alpha_i (1 - g + g P_i) + E_k; with B = sum_{l<k} DeltaE_l alpha_l P_l and its
    // prefix B_i = sum_{l<=i}: dL0/dalpha_i = DeltaE_i (1 - g + g P_i) - g (B - B_i) / (1 - alpha_i)
    const float pt = blend_slope(alpha, rp.c, rp.c1, p.P);
    const float Sn = __fadd_rn(p.S, pt);
    if (Sn >= 1.0f) {
      wE = 1.0f - p.S;
      dLda = 0.f;
    } else {
      const float gd = gE - p.gEk;
      p.gBi = fmaf(gd, __fmul_rn(alpha, p.P), p.gBi);
      dLda = fmaf(gd, __fmaf_rn(rp.c, p.P, rp.c1), -rp.c * (p.gB - p.gBi) * fast_rcp(1.0f - alpha));
      wE = pt;
      p.S = Sn;
      p.P = __fmul_rn(p.P, __fsub_rn(1.0f, alpha));
    }
  } else if constexpr (KIND == NGS_MODEL_VICINI) {
    // (1 - g) x the linear list's adjoint + g x the exponential list's, each up to its own stop
    float pe = 0.f, dexp = 0.f;
    if (!p.stop_e) {
      const float testT = __fmul_rn(p.T, __fsub_rn(1.0f, alpha));
      if (testT < rp.t_eps) {
        p.stop_e = true;
      } else {
        pe = alpha * p.T;
        p.gacc = fmaf(gE, pe, p.gacc);
        dexp = fmaf(p.T, gE, -fast_rcp(1.0f - alpha) * (p.gL0 - p.gacc));
        p.T = testT;
      }
    }
    float pl = 0.f, dlin = 0.f;
    if (!p.sat) {
      const float Sn = __fadd_rn(p.S, alpha);
      if (Sn >= 1.0f) {
        pl = 1.0f - p.S;
        p.S = 1.0f;
        p.sat = true;
      } else {
        pl = alpha;
        p.S = Sn;
        dlin = gE - p.gEk;
      }
    }
    dLda = fmaf(rp.c1, dlin, rp.c * dexp);
    wE = fmaf(rp.c1, pl, rp.c * pe);
  } else if constexpr (KIND == NGS_MODEL_QUAD) {
    float pt = quad_slope(alpha, rp.c, p.tau);
    float Sn = __fadd_rn(p.S, pt);
    if (Sn >= 1.0f) {  // the saturating splat k: pbar_k = 1 - S, no dependence on alpha_k
      wE = 1.0f - p.S;
      dLda = 0.f;
    } else {
      // g.dL0/dalpha_i = g.DeltaE_i (1 + c taubar_i) + c g.Theta_i, Theta_i = Theta_{i-1} - DeltaE_i alpha_i
      float gd = gE - p.gEk;
      p.gTh = fmaf(-gd, alpha, p.gTh);
      dLda = fmaf(gd, fmaf(rp.c, p.tau, 1.0f), rp.c * p.gTh);
      wE = pt;
      p.S = Sn;
      p.tau = __fadd_rn(p.tau, alpha);
    }
  } else {
    // g.dL0/dalpha_i = T_i g.E_i - (g.L0 - g.sum_{j<=i} E_j pbar_j) / (1 - alpha_i)
    wE = alpha * p.T;
    p.gacc = fmaf(gE, wE, p.gacc);
    dLda = fmaf(p.T, gE, -fast_rcp(1.0f - alpha) * (p.gL0 - p.gacc));
    p.T = __fmul_rn(p.T, __fsub_rn(1.0f, alpha));
  }
  // alpha = 2^e with e = L + dx (A' dx + B' dy) + C' dy^2, unless clamped at alpha_max. With
  // w = dL/de, de/dA' = dx^2, de/dB' = dx dy, de/dC' = dy^2, de/dL = 1 and de/du = -(2A' dx + B' dy),
  // de/dv = -(B' dx + 2C' dy): the per-splat sums of w, w dx, w dy, w dx^2, w dx dy, w dy^2 carry
  // everything; the projection backward applies the per-splat A', B', C' (and ln 2) once.
  w_out = raw >= rp.alpha_max ? 0.f : dLda * alpha;  // dL/de / ln 2
  wE_out = wE;
  return true;
}

// ---- backward, packed form (exponential and quadratic) -----------------------------------------------
//
// The thread's two pixels (x, y) and (x, y + 4) step through each list entry together in FP32x2
// instructions (add / mul / fma .f32x2, one instruction for both pixels). Each lane rounds exactly like
// the scalar forward, so alpha and every compositing decision are bit-identical. A pixel that does not
// composite the entry (past its stop, or alpha < alpha_min) gets alpha = 0, which leaves its running sums
// exactly as they were and contributes zero.

// Both pixels' replay state, lane 0 = pixel (x, y), lane 1 = pixel (x, y + 4).
struct BwdPair {
  float px;
  float2 py;
  uint32_t last0, last1;  // replay entries [range.x, last)
  float2 g0, g1, g2;
  float2 T, gacc, gL0;    // exponential: T_i, g.sum_{j<i} E_j pbar_j, g.L0
  float2 S, tau, nEk, nTh;  // quadratic: S, taubar, -g.E_k, -g.Theta
};

// The quadratic form of an entry at both pixels (as splat_log2_alpha_col computes it per pixel): e = log2
// of aleph K.
__device__ __forceinline__ float2 pair_log2_alpha(const BwdPair& p, float4 r0, float4 q2) {
  const float dx = __fsub_rn(p.px, r0.x), adx = __fmul_rn(r0.z, dx);
  const float2 dy = make_float2(__fsub_rn(p.py.x, r0.y), __fsub_rn(p.py.y, r0.y));
  const float2 cdd = __fmul2_rn(__fmul2_rn(lo_hi(q2, false), dy), dy);
  const float2 q = make_float2(__fmaf_rn(dx, __fmaf_rn(r0.w, dy.x, adx), cdd.x),
                               __fmaf_rn(dx, __fmaf_rn(r0.w, dy.y, adx), cdd.y));
  return __fadd2_rn(lo_hi(q2, true), q);
}

// One list entry for both pixels, given the quadratic form (e, dx, dy) and which pixels composite it
// (on0 / on1: not past their stop, alpha >= alpha_min): {w, w, wE, wE}. A pixel that does not composite it gets
// alpha = 0, which leaves its running sums exactly as they were, and zeros, so the warp runs the step
// whenever any lane is on.
template <int KIND>
__device__ __forceinline__ float4 bwd_pair_step(BwdPair& p, float2 e, float4 q3, bool on0, bool on1,
                                                const RenderParams& rp) {
  const float2 one = make_float2(1.f, 1.f), neg = make_float2(-1.f, -1.f);
  const float raw0 = fast_exp2(e.x), raw1 = fast_exp2(e.y);
  const float2 alpha = make_float2(on0 ? fminf(rp.alpha_max, raw0) : 0.f, on1 ? fminf(rp.alpha_max, raw1) : 0.f);
  // w = dL/de: zero where alpha is clamped at alpha_max (it no longer depends on e) or not composited
  bool live0 = on0 && raw0 < rp.alpha_max, live1 = on1 && raw1 < rp.alpha_max;
  const float2 gE = make_float2(fmaf(p.g2.x, q3.z, fmaf(p.g1.x, q3.y, p.g0.x * q3.x)),
                                fmaf(p.g2.y, q3.z, fmaf(p.g1.y, q3.y, p.g0.y * q3.x)));
  float2 dLda, wE;
  if constexpr (KIND == NGS_MODEL_QUAD) {
    const float2 ct = __ffma2_rn(make_float2(rp.c, rp.c), p.tau, one);  // 1 + c taubar_i
    const float2 ptr = __fmul2_rn(alpha, ct);
    const float2 pt = make_float2(fmaxf(ptr.x, 0.f), fmaxf(ptr.y, 0.f));
    const float2 Sn = __fadd2_rn(p.S, pt);
    const bool sat0 = Sn.x >= 1.0f, sat1 = Sn.y >= 1.0f;  // the saturating splat k: pbar_k = 1 - S
    const float2 oms = __ffma2_rn(p.S, neg, one);
    wE = make_float2(sat0 ? oms.x : pt.x, sat1 ? oms.y : pt.y);
    live0 = live0 && !sat0;
    live1 = live1 && !sat1;
    // -g.Theta_i = -g.Theta_{i-1} + g.DeltaE_i alpha_i; dL0/dalpha_i = g.DeltaE_i (1 + c taubar_i) + c g.Theta_i
    const float2 gd = __fadd2_rn(gE, p.nEk);
    p.nTh = __ffma2_rn(gd, alpha, p.nTh);
    dLda = __ffma2_rn(gd, ct, __fmul2_rn(make_float2(-rp.c, -rp.c), p.nTh));
    p.S = make_float2(sat0 ? p.S.x : Sn.x, sat1 ? p.S.y : Sn.y);  // S stays below 1 for later entries
    p.tau = __fadd2_rn(p.tau, alpha);
  } else {
    // dL0/dalpha_i = T_i g.E_i - (g.L0 - g.sum_{j<=i} E_j pbar_j) / (1 - alpha_i)
    wE = __fmul2_rn(alpha, p.T);
    p.gacc = __ffma2_rn(gE, wE, p.gacc);
    const float2 oma = __ffma2_rn(alpha, neg, one);
    const float2 rcp = make_float2(fast_rcp(oma.x), fast_rcp(oma.y));
    dLda = __ffma2_rn(p.T, gE, __fmul2_rn(rcp, __ffma2_rn(p.gL0, neg, p.gacc)));
    p.T = __fmul2_rn(p.T, oma);
  }
  const float2 wgt = __fmul2_rn(dLda, make_float2(live0 ? alpha.x : 0.f, live1 ? alpha.y : 0.f));
  return make_float4(on0 ? wgt.x : 0.f, on1 ? wgt.y : 0.f, wE.x, wE.y);
}

template <int TW, int TH, int KIND, int CH, bool AHEAD>
__device__ __forceinline__ void backward_tile_pairs(const float4* __restrict__ rec, const uint32_t* __restrict__ ids,
                                                    const uint2* __restrict__ ranges, const RenderParams& rp,
                                                    const ViewParams* __restrict__ views,
                                                    const float* __restrict__ dl_dimage,
                                                    const float4* __restrict__ state, float4* __restrict__ grad2d,
                                                    uint32_t tile, PairStageBuf<CH, true>& sb, ReplayWarp& rw) {
  using G = TileGeom<TW, TH, kBwdPix>;
  constexpr int B = G::kThreads;
  const TileView tv = tile_view(rp, views, (uint32_t)tile);
  const int W = tv.W, H = tv.H;
  const size_t pix_base = view_pix_base(rp, views, tv.view);
  const int tx = tv.local % tv.tiles_x, ty = tv.local / tv.tiles_x;
  const int tid = threadIdx.x, lane = tid & 31;
  const uint2 range = ranges[tile];
  BwdPair p;
  float px[2], py[2], g[2][3], gEk[2], gThe[2], gL0[2];
  uint32_t last[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    int x, y;
    G::pixel(tid, k, tx * TW, ty * TH, x, y);
    px[k] = (float)x + 0.5f;
    py[k] = (float)y + 0.5f;
    last[k] = range.x;
    g[k][0] = g[k][1] = g[k][2] = 0.f;
    gEk[k] = gThe[k] = gL0[k] = 0.f;
    if (x < W && y < H) {
      const size_t pix = pix_base + (size_t)y * W + x;
      const float4 s0 = state[2 * pix], s1 = state[2 * pix + 1];
      last[k] = range.x + (__float_as_uint(s0.x) & 0x7FFFFFFFu);
      g[k][0] = dl_dimage[3 * pix];
      g[k][1] = dl_dimage[3 * pix + 1];
      g[k][2] = dl_dimage[3 * pix + 2];
      if constexpr (KIND == NGS_MODEL_QUAD) {
        gEk[k] = g[k][0] * s0.y + g[k][1] * s0.z + g[k][2] * s0.w;
        // Theta_{-1} = A - E_k taubar_k
        gThe[k] = g[k][0] * (s1.x - s0.y * s1.w) + g[k][1] * (s1.y - s0.z * s1.w) + g[k][2] * (s1.z - s0.w * s1.w);
      } else {
        gL0[k] = g[k][0] * s0.y + g[k][1] * s0.z + g[k][2] * s0.w;
      }
      if (g[k][0] == 0.f && g[k][1] == 0.f && g[k][2] == 0.f) last[k] = range.x;
    }
  }
  const bool odd = replay_begin(rw, g[0], g[1], lane), odd_warp = __any_sync(kFull, odd);
  const float bx = __shfl_sync(kFull, px[0], 0), by = __shfl_sync(kFull, py[0], 0);
  ReplaySlot slot = {0.f, 0.f, 0u};
  uint32_t slots = 0;
  p.px = px[0];  // one column: px[1] == px[0]
  p.py = make_float2(py[0], py[1]);
  p.last0 = last[0];
  p.last1 = last[1];
  p.g0 = make_float2(g[0][0], g[1][0]);
  p.g1 = make_float2(g[0][1], g[1][1]);
  p.g2 = make_float2(g[0][2], g[1][2]);
  p.T = make_float2(1.f, 1.f);
  p.gacc = make_float2(0.f, 0.f);
  p.gL0 = make_float2(gL0[0], gL0[1]);
  p.S = p.tau = make_float2(0.f, 0.f);
  p.nEk = make_float2(-gEk[0], -gEk[1]);
  p.nTh = make_float2(-gThe[0], -gThe[1]);
  const uint32_t my_last = max(p.last0, p.last1);
  const uint32_t warp_last = __reduce_max_sync(kFull, my_last);
  for (uint32_t base = range.x; base < range.y; base += CH) {
    if (__syncthreads_count(base >= my_last) == B) break;
    stage_chunk_pairs<B, CH>(rec, ids, rp, base, range.y, sb);
    __syncthreads();
    if (base < warp_last) {
      const int cnt = (int)(min(warp_last, min(base + (uint32_t)CH, range.y)) - base);
      float2 e_next;
      if constexpr (AHEAD) e_next = pair_log2_alpha(p, sb.r0[0], sb.q2[0]);
      for (int j = 0; j < cnt; ++j) {
        const float4 r0 = sb.r0[j];
        float2 e;
        if constexpr (AHEAD) {  // the next entry's, while this one is differentiated
          e = e_next;
          e_next = pair_log2_alpha(p, sb.r0[j + 1], sb.q2[j + 1]);
        } else {
          e = pair_log2_alpha(p, r0, sb.q2[j]);
        }
        const uint32_t pos = base + j;
        const bool on0 = pos < p.last0 && e.x >= rp.log2_alpha_min;
        const bool on1 = pos < p.last1 && e.y >= rp.log2_alpha_min;
        if (__any_sync(kFull, on0 || on1)) {  // the step is exact for the pixels that are off
          const float4 q3 = sb.q3[j];
          const float4 w = bwd_pair_step<KIND>(p, e, q3, on0, on1, rp);
          rw.w[slots * kSlotStride + lane] = w;
          if ((uint32_t)(lane & (kSlots - 1)) == slots) slot = {r0.x, r0.y, __float_as_uint(q3.w)};
          if (odd_warp && odd) {
            float* dst = reinterpret_cast<float*>(grad2d + 3 * (size_t)__float_as_uint(q3.w));
            if (on0) replay_odd_lane(dst, p.g0.x, p.g1.x, p.g2.x, w.z);
            if (on1) replay_odd_lane(dst, p.g0.y, p.g1.y, p.g2.y, w.w);
          }
          if (++slots == kSlots) {
            replay_flush(rw, slot, kSlots, bx, by, grad2d, lane);
            slots = 0;
          }
        }
      }
    }
  }
  if (slots) replay_flush(rw, slot, slots, bx, by, grad2d, lane);
}

template <int TW, int TH, int KIND, int CH>
__device__ __forceinline__ void backward_tile(const float4* __restrict__ rec, const uint32_t* __restrict__ ids,
                                              const uint2* __restrict__ ranges, const RenderParams& rp,
                                              const ViewParams* __restrict__ views,
                                              const float* __restrict__ dl_dimage, const float4* __restrict__ state,
                                              float4* __restrict__ grad2d, uint32_t tile, StageBuf<CH>& sb,
                                              uint32_t* s_id, ReplayWarp& rw) {
  using G = TileGeom<TW, TH, kBwdPix>;
  constexpr int B = G::kThreads;
  static_assert(kBwdPix == 2, "the replay below is written for two pixels per thread");
  const TileView tv = tile_view(rp, views, (uint32_t)tile);
  const int W = tv.W, H = tv.H;
  const size_t pix_base = view_pix_base(rp, views, tv.view);
  const int tx = tv.local % tv.tiles_x, ty = tv.local / tv.tiles_x;
  const int tid = threadIdx.x, lane = tid & 31;
  const uint2 range = ranges[tile];
  BwdPixel p[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    int x, y;
    G::pixel(tid, k, tx * TW, ty * TH, x, y);
    BwdPixel& q = p[k];
    q.px = (float)x + 0.5f;
    q.py = (float)y + 0.5f;
    q.last = range.x;
    q.g0 = q.g1 = q.g2 = 0.f;
    // everything the adjoint needs is a dot product with g: quadratic keeps g.E_k and g.Theta,
    // exponential keeps g.L0 and the running g.sum_{j<=i} E_j pbar_j
    q.gEk = q.gTh = q.gL0 = 0.f;
    q.S = q.tau = q.gacc = 0.f;
    q.T = 1.f;
    q.P = 1.f;
    q.gB = q.gBi = 0.f;
    q.sat = q.stop_e = false;
    if (x < W && y < H) {
      size_t pix = pix_base + (size_t)y * W + x;
      float4 s0 = state[2 * pix], s1 = state[2 * pix + 1];
      q.last = range.x + (__float_as_uint(s0.x) & 0x7FFFFFFFu);
      q.g0 = dl_dimage[3 * pix];
      q.g1 = dl_dimage[3 * pix + 1];
      q.g2 = dl_dimage[3 * pix + 2];
      if constexpr (KIND == NGS_MODEL_QUAD) {
        q.gEk = q.g0 * s0.y + q.g1 * s0.z + q.g2 * s0.w;
        // Theta_{-1} = A - E_k taubar_k
        q.gTh = q.g0 * (s1.x - s0.y * s1.w) + q.g1 * (s1.y - s0.z * s1.w) + q.g2 * (s1.z - s0.w * s1.w);
      } else if constexpr (KIND == NGS_MODEL_BLEND) {
        q.gEk = q.g0 * s0.y + q.g1 * s0.z + q.g2 * s0.w;
        // B = sum_{l<k} E_l alpha_l P_l - E_k sum_{l<k} alpha_l P_l
        q.gB = q.g0 * s1.x + q.g1 * s1.y + q.g2 * s1.z - q.gEk * s1.w;
      } else if constexpr (KIND == NGS_MODEL_VICINI) {
        q.gEk = q.g0 * s0.y + q.g1 * s0.z + q.g2 * s0.w;  // E_k of the linear list
        q.gL0 = q.g0 * s1.x + q.g1 * s1.y + q.g2 * s1.z;  // L0 of the exponential list
      } else {
        q.gL0 = q.g0 * s0.y + q.g1 * s0.z + q.g2 * s0.w;
      }
      if (q.g0 == 0.f && q.g1 == 0.f && q.g2 == 0.f) q.last = range.x;
    }
  }
  const float ga[3] = {p[0].g0, p[0].g1, p[0].g2}, gb[3] = {p[1].g0, p[1].g1, p[1].g2};
  const bool odd = replay_begin(rw, ga, gb, lane), odd_warp = __any_sync(kFull, odd);
  const float bx = __shfl_sync(kFull, p[0].px, 0), by = __shfl_sync(kFull, p[0].py, 0);
  ReplaySlot slot = {0.f, 0.f, 0u};
  uint32_t slots = 0;
  // the warp walks entries up to the largest stop of its pixels
  const uint32_t warp_last = __reduce_max_sync(kFull, max(p[0].last, p[1].last));
  for (uint32_t base = range.x; base < range.y; base += CH) {
    const bool done = base >= max(p[0].last, p[1].last);
    if (__syncthreads_count(done) == B) break;
    stage_chunk<B, CH>(rec, ids, rp, base, range.y, sb, s_id);
    __syncthreads();
    if (base < warp_last) {
      const int cnt = (int)(min(warp_last, min(base + (uint32_t)CH, range.y)) - base);
      for (int j = 0; j < cnt; ++j) {
        const uint32_t pos = base + j;
        const float4 r0 = sb.r0[j], r1 = sb.r1[j];
        // both pixels of the thread lie in one column: dx and A' dx are shared
        const float dx = __fsub_rn(p[0].px, r0.x), adx = __fmul_rn(r0.z, dx);
        float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
        const bool on0 = bwd_step<KIND>(p[0], dx, adx, r0, r1, sb.e2[j], pos, rp, w.x, w.z);
        const bool on1 = bwd_step<KIND>(p[1], dx, adx, r0, r1, sb.e2[j], pos, rp, w.y, w.w);
        if (__any_sync(kFull, on0 || on1)) {
          rw.w[slots * kSlotStride + lane] = w;
          if ((uint32_t)(lane & (kSlots - 1)) == slots) slot = {r0.x, r0.y, s_id[j]};
          if (odd_warp && odd) {
            float* dst = reinterpret_cast<float*>(grad2d + 3 * (size_t)s_id[j]);
            if (on0) replay_odd_lane(dst, p[0].g0, p[0].g1, p[0].g2, w.z);
            if (on1) replay_odd_lane(dst, p[1].g0, p[1].g1, p[1].g2, w.w);
          }
          if (++slots == kSlots) {
            replay_flush(rw, slot, kSlots, bx, by, grad2d, lane);
            slots = 0;
          }
        }
      }
    }
  }
  if (slots) replay_flush(rw, slot, slots, bx, by, grad2d, lane);
}

// Shared memory of a replay CTA: the staged chunk, then each warp's gathered entries.
template <int TW, int TH, int KIND, int CH>
struct ReplayShared {
  std::conditional_t<kPairForm<KIND, CH>, PairStageBuf<CH, true>, StageBuf<CH>> sb;
  uint32_t id[kPairForm<KIND, CH> ? 4 : CH];  // the packed form carries the index in its q4
  ReplayWarp warps[TW * TH / 64];
};

// 28 warps per SM: 72 registers, which the kernels just need (four bytes of spills in some).
template <int TW, int TH, int KIND, int CH, Walk WALK>
__global__ void __launch_bounds__(TW* TH / kBwdPix, 28 * 64 / (TW * TH)) composite_backward_kernel(const float4* __restrict__ rec,
                                                                        const uint32_t* __restrict__ ids,
                                                                        const uint2* __restrict__ ranges,
                                                                        RenderParams rp,
                                                                        const ViewParams* __restrict__ views,
                                                                        const float* __restrict__ dl_dimage,
                                                                        const float4* __restrict__ state,
                                                                        float4* __restrict__ grad2d,
                                                                        const uint32_t* __restrict__ work,
                                                                        uint32_t* counter) {
  pdl_wait();
  extern __shared__ __align__(16) unsigned char s_replay[];
  ReplayShared<TW, TH, KIND, CH>& sh = *reinterpret_cast<ReplayShared<TW, TH, KIND, CH>*>(s_replay);
  ReplayWarp& rw = sh.warps[threadIdx.x >> 5];
  auto one_tile = [&](uint32_t tile) {
    if constexpr (kPairForm<KIND, CH>)
      backward_tile_pairs<TW, TH, KIND, CH, WALK == kAhead>(rec, ids, ranges, rp, views, dl_dimage, state, grad2d, tile, sh.sb, rw);
    else
      backward_tile<TW, TH, KIND, CH>(rec, ids, ranges, rp, views, dl_dimage, state, grad2d, tile, sh.sb, sh.id, rw);
  };
  if constexpr (WALK == kPersistent) {
    __shared__ uint32_t s_next;
    for (;;) {
      const uint32_t tile = next_tile(work, counter, rp.n_tiles, &s_next);
      if (tile >= rp.n_tiles) break;
      one_tile(tile);
    }
  } else {
    one_tile(blockIdx.x);
  }
}

// Launch configuration of a composite launch: chunk factor (records staged per round = tile pixels x
// {1/2, 1, 2}) and schedule (one CTA per tile, or persistent CTAs over the work list).
struct Launch {
  int chunk_code;                   // 0: half, 1: equal, 2: double the tile's pixel count
  const uint32_t* work;             // persistent schedule: tile order (null: identity)
  uint32_t* counter;                // persistent schedule: zeroed work counter (null: one CTA per tile)
  int num_sms;
};

// One CTA per tile, or one wave of persistent CTAs (SM count x resident CTAs per SM).
template <typename Kernel>
static unsigned grid_for(Kernel k, int threads, size_t shared, const Launch& L, uint32_t n_tiles) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, threads, shared) != cudaSuccess || per_sm < 1) per_sm = 1;
  return (unsigned)std::min<uint64_t>((uint64_t)per_sm * (uint64_t)L.num_sms, n_tiles);
}

// Few tiles: at most 32 warps per SM in all (one 8 x 8 pixel block per warp).
template <int TW, int TH>
static bool few_tiles(const Launch& L, uint32_t n_tiles) {
  return (uint64_t)n_tiles * (TW * TH / 64) <= 32ull * (uint64_t)std::max(L.num_sms, 1);
}

template <int TW, int TH, int KIND, int CH>
void forward_launch(const float4* rec, const uint32_t* ids, const uint2* ranges, const RenderParams& rp,
                    const ViewParams* views, float* image, int32_t* overdraw, float4* state, const Launch& L,
                    cudaStream_t s) {
  constexpr int threads = kFwdThreads<TW, TH, KIND, CH>;
  auto k = composite_forward_kernel<TW, TH, KIND, CH, kTiles>;
  unsigned grid = rp.n_tiles;
  if (kPairFwd<TW, TH, KIND, CH> && few_tiles<TW, TH>(L, rp.n_tiles)) {
    k = composite_forward_kernel<TW, TH, KIND, CH, kPairFwd<TW, TH, KIND, CH> ? kAhead : kTiles>;
  } else if (L.counter) {
    k = composite_forward_kernel<TW, TH, KIND, CH, kPersistent>;
    grid = grid_for(k, threads, 0, L, rp.n_tiles);
  }
  launch_pdl(k, grid, threads, 0, s, rec, ids, ranges, rp, views, image, overdraw, state, L.work, L.counter);
}

template <int TW, int TH, int KIND, int CH>
void backward_launch(const float4* rec, const uint32_t* ids, const uint2* ranges, const RenderParams& rp,
                     const ViewParams* views, const float* dl, const float4* state, float4* grad2d, const Launch& L,
                     cudaStream_t s) {
  constexpr int threads = TileGeom<TW, TH, kBwdPix>::kThreads;
  auto k = composite_backward_kernel<TW, TH, KIND, CH, kTiles>;
  constexpr size_t shared = sizeof(ReplayShared<TW, TH, KIND, CH>);
  unsigned grid = rp.n_tiles;
  if (kPairForm<KIND, CH> && few_tiles<TW, TH>(L, rp.n_tiles)) {
    k = composite_backward_kernel<TW, TH, KIND, CH, kPairForm<KIND, CH> ? kAhead : kTiles>;
  } else if (L.counter) {
    k = composite_backward_kernel<TW, TH, KIND, CH, kPersistent>;
  }
  if (shared > 48 * 1024 &&
      cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shared) != cudaSuccess)
    return;  // the launch sequence's error check reports it
  if (k == composite_backward_kernel<TW, TH, KIND, CH, kPersistent>) {
    grid = grid_for(k, threads, shared, L, rp.n_tiles);
  }
  launch_pdl(k, grid, threads, shared, s, rec, ids, ranges, rp, views, dl, state, grad2d, L.work, L.counter);
}

template <int TW, int TH, int KIND>
void forward_chunk(const float4* rec, const uint32_t* ids, const uint2* ranges, const RenderParams& rp,
                   const ViewParams* views, float* image, int32_t* overdraw, float4* state, const Launch& L,
                   cudaStream_t s) {
  constexpr int P = TW * TH;
  if (L.chunk_code == 0) forward_launch<TW, TH, KIND, P / 2>(rec, ids, ranges, rp, views, image, overdraw, state, L, s);
  else if (L.chunk_code == 2) forward_launch<TW, TH, KIND, 2 * P>(rec, ids, ranges, rp, views, image, overdraw, state, L, s);
  else forward_launch<TW, TH, KIND, P>(rec, ids, ranges, rp, views, image, overdraw, state, L, s);
}

template <int TW, int TH, int KIND>
void backward_chunk(const float4* rec, const uint32_t* ids, const uint2* ranges, const RenderParams& rp,
                    const ViewParams* views, const float* dl, const float4* state, float4* grad2d, const Launch& L,
                    cudaStream_t s) {
  constexpr int P = TW * TH;
  if (L.chunk_code == 0) backward_launch<TW, TH, KIND, P / 2>(rec, ids, ranges, rp, views, dl, state, grad2d, L, s);
  else if (L.chunk_code == 2) backward_launch<TW, TH, KIND, 2 * P>(rec, ids, ranges, rp, views, dl, state, grad2d, L, s);
  else backward_launch<TW, TH, KIND, P>(rec, ids, ranges, rp, views, dl, state, grad2d, L, s);
}

template <int TW, int TH>
void forward_kind(const float4* rec, const uint32_t* ids, const uint2* ranges, const RenderParams& rp,
                  const ViewParams* views, float* image, int32_t* overdraw, float4* state, const Launch& L,
                  cudaStream_t s) {
  switch (rp.kind) {
    case NGS_MODEL_QUAD:
      forward_chunk<TW, TH, NGS_MODEL_QUAD>(rec, ids, ranges, rp, views, image, overdraw, state, L, s);
      break;
    case NGS_MODEL_BLEND:
      forward_chunk<TW, TH, NGS_MODEL_BLEND>(rec, ids, ranges, rp, views, image, overdraw, state, L, s);
      break;
    case NGS_MODEL_VICINI:
      forward_chunk<TW, TH, NGS_MODEL_VICINI>(rec, ids, ranges, rp, views, image, overdraw, state, L, s);
      break;
    default:
      forward_chunk<TW, TH, NGS_MODEL_EXP>(rec, ids, ranges, rp, views, image, overdraw, state, L, s);
  }
}

template <int TW, int TH>
void backward_kind(const float4* rec, const uint32_t* ids, const uint2* ranges, const RenderParams& rp,
                   const ViewParams* views, const float* dl, const float4* state, float4* grad2d, const Launch& L,
                   cudaStream_t s) {
  switch (rp.kind) {
    case NGS_MODEL_QUAD:
      backward_chunk<TW, TH, NGS_MODEL_QUAD>(rec, ids, ranges, rp, views, dl, state, grad2d, L, s);
      break;
    case NGS_MODEL_BLEND:
      backward_chunk<TW, TH, NGS_MODEL_BLEND>(rec, ids, ranges, rp, views, dl, state, grad2d, L, s);
      break;
    case NGS_MODEL_VICINI:
      backward_chunk<TW, TH, NGS_MODEL_VICINI>(rec, ids, ranges, rp, views, dl, state, grad2d, L, s);
      break;
    default:
      backward_chunk<TW, TH, NGS_MODEL_EXP>(rec, ids, ranges, rp, views, dl, state, grad2d, L, s);
  }
}

int chunk_code(const RenderParams& rp) {
  const int P = rp.tile_w * rp.tile_h;
  return rp.chunk == P / 2 ? 0 : rp.chunk == 2 * P ? 2 : 1;
}

}  // namespace

void launch_composite_forward(const float4* rec, const uint32_t* ids, const uint2* ranges, const RenderParams& rp,
                              const ViewParams* views, float* image, int32_t* overdraw, float4* state,
                              const uint32_t* work, uint32_t* counter, int num_sms, cudaStream_t s) {
  const Launch L{chunk_code(rp), work, counter, num_sms};
  if (rp.tile_w == 8 && rp.tile_h == 8)
    forward_kind<8, 8>(rec, ids, ranges, rp, views, image, overdraw, state, L, s);
  else if (rp.tile_w == 16 && rp.tile_h == 16)
    forward_kind<16, 16>(rec, ids, ranges, rp, views, image, overdraw, state, L, s);
  else
    forward_kind<16, 32>(rec, ids, ranges, rp, views, image, overdraw, state, L, s);
}

void launch_composite_backward(const float4* rec, const uint32_t* ids, const uint2* ranges, const RenderParams& rp,
                               const ViewParams* views, const float* dl_dimage, const float4* state, float4* grad2d,
                               const uint32_t* work, uint32_t* counter, int num_sms, cudaStream_t s) {
  const Launch L{chunk_code(rp), work, counter, num_sms};
  if (rp.tile_w == 8 && rp.tile_h == 8)
    backward_kind<8, 8>(rec, ids, ranges, rp, views, dl_dimage, state, grad2d, L, s);
  else if (rp.tile_w == 16 && rp.tile_h == 16)
    backward_kind<16, 16>(rec, ids, ranges, rp, views, dl_dimage, state, grad2d, L, s);
  else
    backward_kind<16, 32>(rec, ids, ranges, rp, views, dl_dimage, state, grad2d, L, s);
}

}  // namespace ngs
