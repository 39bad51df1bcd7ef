// Per-tile front-to-back compositing (Sec. 3.2, Eq. 6 of arXiv 2412.20720)
// and its reverse-mode derivative, plus the photometric L1 loss (Sec. 3.3).
//
// Forward: one CTA per (view, 16x16 tile).  A thread owns a vertical strip of
// kPPT pixels of one column, so the per-entry work that does not depend on the
// row (shared-memory loads, dx, (a1 dx)^2, b1 dx) is done once for kPPT pixels.
// The tile's depth-sorted list is staged through shared memory in batches of
// 128 or 256 records; the CTA stops loading once every pixel has reached the
// transmittance cutoff (__syncthreads_count).  alpha = min(0.99, a 2^-q),
// skip when alpha < 1/255, stop before the entry that would take T below 1e-4
// -- evaluated by pixel_alpha, shared with the backward pass so both take
// bit-identical decisions.  The power > 0 skip of the reference rasteriser is
// not taken: q is a positive definite form, so q < 0 only arises by rounding
// next to the Gaussian's centre, where skipping would drop the entry.
//
// Backward: the same tiles traversed back to front from each pixel's last
// composited entry, recomputing T_i = T_{i+1} / (1 - alpha_i) from the final
// transmittance.  A thread first sums its strip's contributions; the lanes' sums
// then meet in shared memory (render_bwd_kernel) and are added with one atomic
// per sum, warp and entry.
#include <algorithm>
#include <type_traits>

#include "fgs4d_internal.cuh"

namespace fgs4d {

namespace {


struct RenderArgs {
  const uint2 *ranges;
  const uint32_t *inst_val;
  const float4 *rec_geom, *rec_color;  // rec_geom: (u, v, a1, b1); rec_color: (b2, log2 a, r, g)
  const float *rec_blue;
  const float4 *rec_aux;  // auxiliary mode only
  uint32_t vis_cap;
  float *out_rgb, *out_T;
  float *out_aux;  // [views][4][H][W]: depth, opacity, flow_u, flow_v (auxiliary mode only)
  float *pix_T;
  uint32_t *pix_last;
  float bg0, bg1, bg2;
};

struct RenderBwdArgs {
  const uint2 *ranges;
  const uint32_t *inst_val;
  const float4 *rec_geom, *rec_color;
  const float *rec_blue;
  const float4 *rec_aux;  // auxiliary mode only
  uint32_t vis_cap;
  const float *pix_T;
  const uint32_t *pix_last;
  const float *dL_drgb;
  const float *dL_daux;  // [views][4][H][W] (depth, opacity used), auxiliary mode only
  float4 *slot_grad;
  float bg0, bg1, bg2;
};

// Pixels per thread of the compositor kernels (the autotuned block shape):
// 16x16 tiles take 2, 4 or 8, 8x8 tiles 1 or 2.  Defaults for 16x16 tiles: 4;
// with few tiles, whose lists too few warps would walk, 2; with many tiles the
// adjoint of the image, whose per-entry work (moments and reduction rows) is
// shared by a strip, 8 -- unless the instance capacity says that the lists are
// short, where a block's set-up counts.  Measured forward / adjoint (us)
// with 2, 4 and 8 rows a thread: 48 tiles 12.0 / 26.7, 18.5 / 39.2, 35.0 /
// 63.5; 690 tiles 26.8 / 63.7, 38.9 / 84.0, 70.6 / 123; 1200 tiles 32.3 / 76.4,
// 33.1 / 74.6, 59.1 / 107; 3978 tiles 54.5 / 155, 56.7 / 139, 77.5 / 146; 5440
// tiles of 308 entries 190 / 561, 186 / 438, 267 / 411.  Adjoint with 4 and 8
// rows at 21,760 tiles and more, by entries a tile: 1.7 110 / 121, 2.7 151 /
// 162, 9.8 111 / 114, 19 178 / 174, 39 321 / 303, 77 605 / 552 (capacities are
// some twice that).
constexpr int64_t kFewTiles = 1024, kManyTiles = 5000, kLongListCap = 32;
inline int render_ppt(const fgs4d_settings *s, const Layout &L, bool adjoint) {
  if (s->tile == 8) return s->pixels_per_thread == 1 ? 1 : 2;
  if (s->pixels_per_thread) return s->pixels_per_thread;
  if (L.total_tiles < kFewTiles) return 2;
  return adjoint && L.total_tiles >= kManyTiles && L.inst_cap >= kLongListCap * L.total_tiles ? 8 : 4;
}


// Magnitudes up to which products of gradients with colours and depths, and
// their sums, stay far below the largest float (render_bwd_kernel).
constexpr float kMagMax = 1152921504606846976.0f;  // 2^60

// What the records a thread staged ask of the pixel loop.
struct StagedFlags {
  bool clamp;  // some entry can reach the 0.99 clamp
  bool large;  // some colour or depth is above kMagMax (or not a number)
};

// Stages records [base, min(base + kBatch, end)) of the tile list into shared
// memory; slots out of range (only possible after a recorded timeout) stage a
// record that every pixel skips.  Without kFlags (the image-only forward) the
// records go straight to shared memory and the caller looks for clamping
// entries there: 549 us for 4 views of 1352x1014 against 553; the others gain
// from the flags (627 -> 625, with the auxiliary channels 245 -> 229).
template <int NT, int kBatch, bool kFlags = true>
__device__ __forceinline__ StagedFlags stage_batch(const uint32_t *inst_val, const float4 *rec_geom,
                                                   const float4 *rec_color, const float *rec_blue, uint32_t vis_cap,
                                                   uint32_t base, uint32_t end, float4 *s_geom, float4 *s_col,
                                                   float *s_blue, uint32_t *s_slot, const float4 *rec_aux = nullptr,
                                                   float4 *s_aux = nullptr) {
  StagedFlags f = {false, false};
#pragma unroll
  for (int i = 0; i < kBatch / NT; ++i) {
    const int k = threadIdx.x + i * NT;
    const uint32_t idx = base + k;
    if (idx < end) {
      const uint32_t s = inst_val[idx];
      if (s_slot) s_slot[k] = s;
      if constexpr (!kFlags) {
        if (s < vis_cap) {
          s_geom[k] = rec_geom[s];
          s_col[k] = rec_color[s];
          s_blue[k] = rec_blue[s];
        } else {
          s_geom[k] = make_float4(0.f, 0.f, 0.f, 0.f);
          s_col[k] = make_float4(0.f, kLogAlphaNone, 0.f, 0.f);
          s_blue[k] = 0.f;
        }
      } else {
        float4 geom = make_float4(0.f, 0.f, 0.f, 0.f), col = make_float4(0.f, kLogAlphaNone, 0.f, 0.f), aux = geom;
        float blue = 0.f;
        if (s < vis_cap) {
          geom = rec_geom[s];
          col = rec_color[s];
          blue = rec_blue[s];
          if (s_aux) aux = rec_aux[s];
        }
        s_geom[k] = geom;
        s_col[k] = col;
        s_blue[k] = blue;
        if (s_aux) s_aux[k] = aux;
        f.clamp = f.clamp || entry_clamps(col.y);
        f.large = f.large || !(fabsf(col.z) + fabsf(col.w) + fabsf(blue) + fabsf(aux.x) <= kMagMax);
      }
    }
  }
  return f;
}

// kMode 0: image (and the per-pixel state of the backward pass); 3: image
// only -- no last-contributor index is tracked (the plane is written as 0);
// 1 (kStats): also counts the pixel-entry alpha evaluations, the composited
// entries and the evaluations up to each pixel's last composited entry (the
// ones the backward pass repeats) -- a diagnostic variant used to state the
// algorithmic work; 2 (kAux): also blends the per-slot depth and flow with
// the colour weights and writes depth, opacity 1 - T and flow planes.
// A pixel that has stopped is marked by a negative T (its final transmittance
// negated; a live pixel always has T >= 1e-4) and by the row offset +inf,
// which makes every later alpha fail the 1/255 test, so the inner loop tests
// no flag.  The update stays a branch: whole warps skip it for entries that
// miss all their pixels.
// Resident blocks per SM asked of the compiler for the image-only form of the
// 64-thread 4-pixel-strip blocks: 18 (56 registers, no spills).  At 20 (48
// registers) the pixel pairs spill: 16 views, 8 frames in flight, 3.32 ms
// against 3.07.
template <int TILE, int PPT, int kMode>
constexpr int fwd_min_blocks() {
  return (TILE == 16 && PPT == 4 && kMode == 3) ? 18 : 1;
}

template <int MAXV, int TILE, int PPT, int kMode, int kBatch>
__global__ void __launch_bounds__(TILE *TILE / PPT, (fwd_min_blocks<TILE, PPT, kMode>()))
    render_fwd_kernel(RenderArgs A, RasterViews<MAXV> rv, unsigned long long *stats) {
  grid_dependency_sync();
  constexpr bool kStats = kMode == 1, kAux = kMode == 2, kTrack = kMode != 3;
  constexpr int NT = TILE * TILE / PPT;
  __shared__ float4 s_geom[kBatch];
  __shared__ float4 s_col[kBatch];
  __shared__ float s_blue[kBatch];
  __shared__ float4 s_aux[kAux ? kBatch : 1];
  const int32_t gt = blockIdx.x;
  const RasterView &V = rv.v[find_view<MAXV>(rv, gt)];
  const int32_t lt = gt - V.tile_base;
  const int32_t tx = lt % V.gw, ty = lt / V.gw;
  const int32_t px = tx * TILE + (threadIdx.x & (TILE - 1));
  const int32_t py0 = ty * TILE + (threadIdx.x / TILE) * PPT;
  const uint2 range = tile_range(A.ranges, gt);
  const float pxc = (float)px + 0.5f;
  // Row groups of the strip (one for strips of up to 4 rows, which never
  // straddle a group; PPT / 4 otherwise) and each pixel's row offset.
  constexpr int kGroups = (PPT + 3) / 4;
  float gyc[kGroups];
#pragma unroll
  for (int g = 0; g < kGroups; ++g) gyc[g] = row_group_centre(py0 + 4 * g);
  // Pixel k is lane k & 1 of pair k >> 1 (a 1-pixel strip leaves the second
  // lane outside the image).
  constexpr int kPairs = (PPT + 1) / 2;
  float2 T[kPairs], C0[kPairs], C1[kPairs], C2[kPairs], off[kPairs];
  float2 X0[kAux ? kPairs : 1], X1[kAux ? kPairs : 1], X2[kAux ? kPairs : 1];  // depth, flow_u, flow_v sums
  uint32_t last[2 * kPairs];
  uint32_t pend[kStats ? 2 * kPairs : 1];  // evaluations since the pixel's last composited entry
  int nlive = 0;  // pixels of this thread still compositing
#pragma unroll
  for (int k = 0; k < 2 * kPairs; ++k) {
    const bool in = k < PPT && px < V.width && py0 + k < V.height;
    const int q = k >> 1;
    if (kStats) pend[k] = 0u;
    const float t = in ? 1.0f : -1.0f, o = in ? row_offset(py0 + k) : stopped_offset();
    if (k & 1) {
      T[q].y = t;
      off[q].y = o;
    } else {
      T[q].x = t;
      off[q].x = o;
      C0[q] = C1[q] = C2[q] = make_float2(0.f, 0.f);
      if (kAux) X0[q] = X1[q] = X2[q] = make_float2(0.f, 0.f);
    }
    last[k] = 0u;
    nlive += in;
  }
  uint32_t n_eval = 0u, n_comp = 0u, n_evb = 0u;
  for (uint32_t base = range.x; base < range.y; base += kBatch) {
    if (__syncthreads_count(nlive > 0) == 0) break;
    const StagedFlags staged =
        stage_batch<NT, kBatch, kTrack>(A.inst_val, A.rec_geom, A.rec_color, A.rec_blue, A.vis_cap, base, range.y, s_geom, s_col,
                                s_blue, nullptr, kAux ? A.rec_aux : nullptr, kAux ? s_aux : nullptr);
    const int nb = (int)min(range.y - base, (uint32_t)kBatch);
    // Whether any staged entry can reach the 0.99 clamp (opacity > 0.98, rare):
    // the barrier that publishes the batch ORs the threads' answers.
    bool my_clamp = staged.clamp;
    if (!kTrack) {
#pragma unroll
      for (int i = 0; i < kBatch / NT; ++i) {
        const int k = threadIdx.x + i * NT;
        if (k < nb) my_clamp = my_clamp || entry_clamps(s_col[k].y);
      }
    }
    const bool clamp_any = __syncthreads_or(my_clamp) != 0;
    const uint32_t pos0 = base - range.x + 1u;
    // One entry of the list at every pixel of the thread, two pixels at a time
    // with two-lane FP32 instructions (each lane rounds as the scalar one
    // does); a skipped pixel takes part with alpha = 0, which changes nothing.
    // The clamp case is a separate copy of the pixel loop.
    auto entry = [&](int j, auto clamp_tag) {
      constexpr bool kClamp = decltype(clamp_tag)::value;
      const float4 geom = s_geom[j];
      const float4 col = s_col[j];
      const float blue = s_blue[j];
      const float4 xa = kAux ? s_aux[j] : make_float4(0.f, 0.f, 0.f, 0.f);  // depth and flow of the entry
      const ColumnTerms ct = column_terms(geom, pxc, col.y);
      float w4[kGroups];
#pragma unroll
      for (int g = 0; g < kGroups; ++g) w4[g] = group_w(ct, geom.y, col.x, gyc[g]);
#pragma unroll
      for (int q = 0; q < kPairs; ++q) {
        // the two lanes of pixel_alpha
        const float wg = w4[q >> 1];
        const float2 w2 = __ffma2_rn(make_float2(col.x, col.x), off[q], make_float2(wg, wg));
        const float2 q2 = __ffma2_rn(w2, w2, make_float2(ct.adx2, ct.adx2));
        const float aG0 = ex2_approx(-q2.x), aG1 = ex2_approx(-q2.y);
        const float al0 = kClamp ? min_nan(0.99f, aG0) : aG0, al1 = kClamp ? min_nan(0.99f, aG1) : aG1;
        if (kStats) {
          n_eval += (T[q].x > 0.0f) + (T[q].y > 0.0f);
          pend[2 * q] += T[q].x > 0.0f;
          pend[2 * q + 1] += T[q].y > 0.0f;
        }
        // false for stopped pixels (row offset +inf)
        const bool v0 = al0 >= kAlphaMin, v1 = al1 >= kAlphaMin;
        if (v0 || v1) {
          float2 w = __fmul2_rn(make_float2(v0 ? al0 : 0.0f, v1 ? al1 : 0.0f), T[q]);
          float2 Tn = __ffma2_rn(w, make_float2(-1.0f, -1.0f), T[q]);  // T - w
          bool c0 = v0, c1 = v1;
          if ((v0 && Tn.x < kTMin) || (v1 && Tn.y < kTMin)) {
            if (v0 && Tn.x < kTMin) {
              Tn.x = -T[q].x;
              w.x = 0.0f;
              off[q].x = stopped_offset();
              --nlive;
              c0 = false;
            }
            if (v1 && Tn.y < kTMin) {
              Tn.y = -T[q].y;
              w.y = 0.0f;
              off[q].y = stopped_offset();
              --nlive;
              c1 = false;
            }
          }
          C0[q] = __ffma2_rn(make_float2(col.z, col.z), w, C0[q]);
          C1[q] = __ffma2_rn(make_float2(col.w, col.w), w, C1[q]);
          C2[q] = __ffma2_rn(make_float2(blue, blue), w, C2[q]);
          if (kAux) {
            // a depth or flow may overflow to infinity and must not meet a zero weight
            if (c0) {
              X0[q].x = __fmaf_rn(xa.x, w.x, X0[q].x);
              X1[q].x = __fmaf_rn(xa.y, w.x, X1[q].x);
              X2[q].x = __fmaf_rn(xa.z, w.x, X2[q].x);
            }
            if (c1) {
              X0[q].y = __fmaf_rn(xa.x, w.y, X0[q].y);
              X1[q].y = __fmaf_rn(xa.y, w.y, X1[q].y);
              X2[q].y = __fmaf_rn(xa.z, w.y, X2[q].y);
            }
          }
          T[q] = Tn;
          if (kTrack) {
            if (c0) last[2 * q] = pos0 + (uint32_t)j;
            if (c1) last[2 * q + 1] = pos0 + (uint32_t)j;
          }
          if (kStats) {
            if (c0) {
              ++n_comp;
              n_evb += pend[2 * q];
              pend[2 * q] = 0u;
            }
            if (c1) {
              ++n_comp;
              n_evb += pend[2 * q + 1];
              pend[2 * q + 1] = 0u;
            }
          }
        }
      }
    };
    if (clamp_any) {
      for (int j = 0; j < nb && nlive > 0; ++j) {
        if (entry_clamps(s_col[j].y)) entry(j, std::true_type());
        else entry(j, std::false_type());
      }
    } else {
      // No entry of the batch can clamp: two entries per iteration, the
      // liveness test once per pair (a pixel that stopped at the first
      // takes no alpha from the second: its row offset is +inf).
      int j = 0;
      for (; j + 1 < nb && nlive > 0; j += 2) {
        entry(j, std::false_type());
        entry(j + 1, std::false_type());
      }
      if (j < nb && nlive > 0) entry(j, std::false_type());
    }
  }
  if (kStats) {
    unsigned long long ev = n_eval, co = n_comp, eb = n_evb;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      ev += __shfl_xor_sync(0xffffffffu, ev, o);
      co += __shfl_xor_sync(0xffffffffu, co, o);
      eb += __shfl_xor_sync(0xffffffffu, eb, o);
    }
    if ((threadIdx.x & 31) == 0) {
      atomicAdd(&stats[0], ev);
      atomicAdd(&stats[1], co);
      atomicAdd(&stats[2], eb);
    }
  }
  const int64_t HW = (int64_t)V.width * V.height;
  float *img = A.out_rgb + V.pix_base * 3;
#pragma unroll
  for (int k = 0; k < PPT; ++k) {
    if (!(px < V.width && py0 + k < V.height)) continue;
    const int64_t p = (int64_t)(py0 + k) * V.width + px;
    auto lane = [k](const float2 *v) { return k & 1 ? v[k >> 1].y : v[k >> 1].x; };
    const float Tend = fabsf(lane(T));
    img[p] = lane(C0) + Tend * A.bg0;
    img[HW + p] = lane(C1) + Tend * A.bg1;
    img[2 * HW + p] = lane(C2) + Tend * A.bg2;
    A.pix_T[V.pix_base + p] = Tend;
    A.pix_last[V.pix_base + p] = kTrack ? last[k] : 0u;
    if (A.out_T) A.out_T[V.pix_base + p] = Tend;
    if (kAux) {
      float *aux = A.out_aux + V.pix_base * 4;
      aux[p] = lane(X0);
      aux[HW + p] = 1.0f - Tend;
      aux[2 * HW + p] = lane(X1);
      aux[3 * HW + p] = lane(X2);
    }
  }
}

// 1/x to within an ulp or so (MUFU reciprocal); the backward pass only needs
// T recovered to the accuracy of its own accumulated rounding.
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Gradient sums of one (warp, entry): kRedSums rows of 32 lanes, in the order
// S_x0, S_1, S_xx, S_x1, S_2, S_0 (moments of gp, below), dr, dg, db, [dz].
template <bool kAux>
__host__ __device__ constexpr int red_sums() {
  return kAux ? 10 : 9;
}
constexpr int kRedEntries = 3;  // entries per reduction: 3 x 9 or 10 sums, one per lane
constexpr int kRedStride = 36;  // floats per row: 16-byte rows whose float4 reads by 8 lanes hit 32 banks

// Resident blocks asked of the compiler for strips on 16x16 tiles: 4 pixels,
// 16 blocks of 64 threads (64 registers, 4 to 8 bytes spilled outside the
// pixel loop; 12 at 80 with the auxiliary channels); 8 pixels, 18 of 32 threads
// (96 registers, 4 to 12 bytes spilled, instead of 117 and 17 blocks).
template <int TILE, int PPT, bool kAux>
constexpr int bwd_min_blocks() {
  if (TILE != 16) return 1;
  return PPT == 4 ? (kAux ? 12 : 16) : (PPT == 8 && !kAux ? 18 : 1);
}

// Reverse traversal of a tile's list.  The kernel is bound by instruction
// issue (86 % of the slots at 4 views of 1352x1014), so a thread's pixels are
// taken in pairs with two-lane FP32 instructions: a skipped pixel takes part
// with alpha = 0, which leaves its T and its sums unchanged (1/(1 - 0) = 1),
// and a pair is skipped when neither pixel composites the entry.  The sums
// over the warp's pixels go through shared memory: the lanes' partial sums of
// kRedEntries entries are rows, and each lane then adds up one row (8 float4
// loads) and adds it with one atomic -- about 25 warp instructions an entry
// where the transposed shuffle butterfly and its operands took about 70.
// 4 views of 1352x1014, 349k visible, 6.3M instances: 1.755 -> 1.343 ms (8 rows
// a thread).  Ordinary batches take a copy of the pixel loop that tests neither
// the clamp nor the range of the products (1.403 -> 1.343 ms).
//
// kAux: the loss also has gradients dL/dD, dL/dO with respect to the depth
// and opacity channels (zero background, x_i = z_i resp. 1 in the colour
// rule); adds dL/dz_i = sum dL/dD alpha_i T_i per slot.
template <int MAXV, int TILE, int kPPT, bool kAux, int kBatch>
__global__ void __launch_bounds__(TILE *TILE / kPPT, (bwd_min_blocks<TILE, kPPT, kAux>())) render_bwd_kernel(RenderBwdArgs A, RasterViews<MAXV> rv) {
  grid_dependency_sync();
  constexpr int kRenderThreads = TILE * TILE / kPPT;
  constexpr int kPairs = (kPPT + 1) / 2;  // a 1-pixel strip leaves its second lane empty
  constexpr int kSums = red_sums<kAux>();
  __shared__ float4 s_geom[kBatch];
  __shared__ float4 s_col[kBatch];
  __shared__ float s_blue[kBatch];
  __shared__ float4 s_aux[kAux ? kBatch : 1];
  __shared__ uint32_t s_slot[kBatch];
  __shared__ uint32_t s_maxlast;
  __shared__ int s_jb[kRenderThreads / 32][kRedEntries];
  __shared__ __align__(16) float s_red[kRenderThreads / 32][kRedEntries * kSums][kRedStride];
  const int32_t gt = blockIdx.x;
  const RasterView &V = rv.v[find_view<MAXV>(rv, gt)];
  const int32_t lt = gt - V.tile_base;
  const int32_t tx = lt % V.gw, ty = lt / V.gw;
  const int32_t px = tx * TILE + (threadIdx.x & (TILE - 1));
  const int32_t py0 = ty * TILE + (threadIdx.x / TILE) * kPPT;
  const uint2 range = tile_range(A.ranges, gt);
  if (range.x == range.y) return;  // nothing was composited: no gradient, and its planes need no reading
  const float pxc = (float)px + 0.5f;
  const int64_t HW = (int64_t)V.width * V.height;
  constexpr int kGroups = (kPPT + 3) / 4;  // row groups of the strip (see group_w)
  float gyc[kGroups];
#pragma unroll
  for (int g = 0; g < kGroups; ++g) gyc[g] = row_group_centre(py0 + 4 * g);
  // Row offset of the strip's first pixel within its group: 0 when the strip
  // starts a group (4 and 8 rows), else -(py0 mod 4).
  const float base_off = row_offset(py0);
  // Dr = sum over channels of dL/dX * (X composited behind the current
  // entry), X = R, G, B (and depth, opacity): the "behind" terms of
  // dL/dalpha enter only through this sum, which grows by w * (dL/dX . x_i).
  // nC0, nC1, nC2, nD, nO: the upstream gradients, negated (see entry()).
  float2 T[kPairs], nC0[kPairs], nC1[kPairs], nC2[kPairs], Dr[kPairs];
  float2 nD[kAux ? kPairs : 1], nO[kAux ? kPairs : 1];
  uint32_t last[2 * kPairs];
  uint32_t my_max = 0u;
  const float *g = A.dL_drgb + V.pix_base * 3;
  // Whether no product of the thread's (then the warp's) upstream gradients can
  // overflow: a skipped pixel takes part with weight 0, which must not meet an
  // infinity (see entry()).  With gradients, colours and depths up to kMagMax
  // the sums below stay under 2^124.
  bool tame = true;
#pragma unroll
  for (int k = 0; k < 2 * kPairs; ++k) {
    float t = 1.0f, c0 = 0.f, c1 = 0.f, c2 = 0.f, d = 0.f, o = 0.f;
    last[k] = 0u;
    if (k < kPPT && px < V.width && py0 + k < V.height) {
      const int64_t p = (int64_t)(py0 + k) * V.width + px;
      t = A.pix_T[V.pix_base + p];
      last[k] = A.pix_last[V.pix_base + p];
      c0 = g[p];
      c1 = g[HW + p];
      c2 = g[2 * HW + p];
      if (kAux) {
        const float *ga = A.dL_daux + V.pix_base * 4;
        d = ga[p];
        o = ga[HW + p];
      }
    }
    const float dr = t * (c0 * A.bg0 + c1 * A.bg1 + c2 * A.bg2);  // the background behind all
    tame = tame && fabsf(c0) <= kMagMax && fabsf(c1) <= kMagMax && fabsf(c2) <= kMagMax && fabsf(d) <= kMagMax &&
           fabsf(o) <= kMagMax && fabsf(dr) <= kMagMax * kMagMax;
    auto lane = [k](float2 &v, float x) { (k & 1 ? v.y : v.x) = x; };
    lane(T[k >> 1], t);
    lane(nC0[k >> 1], -c0);
    lane(nC1[k >> 1], -c1);
    lane(nC2[k >> 1], -c2);
    lane(Dr[k >> 1], dr);
    if (kAux) {
      lane(nD[k >> 1], -d);
      lane(nO[k >> 1], -o);
    }
    my_max = max(my_max, last[k]);
  }
  if (threadIdx.x == 0) s_maxlast = 0u;
  __syncthreads();
  if (my_max) atomicMax(&s_maxlast, my_max);
  __syncthreads();
  const uint32_t end = range.x + min(s_maxlast, range.y - range.x);
  const uint32_t warp_max = __reduce_max_sync(0xffffffffu, my_max);  // past the last entry of the warp's pixels
  tame = __all_sync(0xffffffffu, tame);
  const int lane = threadIdx.x & 31;
  float(*red)[kRedStride] = s_red[threadIdx.x >> 5];
  int buffered = 0;  // entries in `red` (the same in every lane)
  int *jb = s_jb[threadIdx.x >> 5];  // their positions in the batch
  // Sums the buffered rows and adds them to the slots.  Lane e kSums + r sums
  // row r of entry e; the centre and conic gradients follow from the moments
  // with the natural-log conic (An, Bn, Cn) of the record's factors (A' =
  // a1^2 + b1^2, B' = 2 b1 b2, C' = b2^2 in base 2):
  //   du = -(An S_x0 + Bn S_1)   dv = -(Cn S_1 + Bn S_x0)
  //   dA = -S_xx / 2   dB = -S_x1   dC = -S_2 / 2   da = S_0 / a
  auto flush = [&]() {
    __syncwarp();
    const int e = lane / kSums, r = lane - e * kSums;
    const bool on = e < buffered;
    float own = 0.f;
    if (on) {  // pairwise, lanes 16, 8, 4, 2 and 1 apart
      const float4 *row = reinterpret_cast<const float4 *>(red[lane]);
      float2 y[8];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 u = row[q], v = row[q + 4];
        y[2 * q] = __fadd2_rn(make_float2(u.x, u.y), make_float2(v.x, v.y));
        y[2 * q + 1] = __fadd2_rn(make_float2(u.z, u.w), make_float2(v.z, v.w));
      }
#pragma unroll
      for (int h = 4; h >= 1; h >>= 1)
#pragma unroll
        for (int q = 0; q < h; ++q) y[q] = __fadd2_rn(y[q], y[q + h]);
      own = y[0].x + y[0].y;
    }
    const float other = __shfl_sync(0xffffffffu, own, r == 0 ? lane + 1 : (r == 1 ? lane - 1 : lane));
    if (on) {
      const int j = jb[e];
      const float4 geom = s_geom[j];
      const float2 ca = *reinterpret_cast<const float2 *>(&s_col[j]);
      const float k2 = -2.0f * kLn2;
      float m = r == 5 ? ex2_approx(-ca.y) : 1.0f;
      if (r == 0) m = k2 * __fmaf_rn(geom.z, geom.z, geom.w * geom.w);
      if (r == 1) m = k2 * (ca.x * ca.x);
      if (r == 2 || r == 4) m = -0.5f;
      if (r == 3) m = -1.0f;
      float out = m * own;
      if (r < 2) out = __fmaf_rn(k2 * (geom.w * ca.x), other, out);
      const uint32_t slot = s_slot[j];
      if (slot < A.vis_cap) atomicAdd(reinterpret_cast<float *>(A.slot_grad + 3 * (size_t)slot) + r, out);
    }
    __syncwarp();  // the rows may be overwritten
    buffered = 0;
  };
  const int nbatch = (int)((end - range.x + kBatch - 1) / kBatch);
  for (int bi = nbatch - 1; bi >= 0; --bi) {
    const uint32_t base = range.x + (uint32_t)bi * kBatch;
    __syncthreads();
    const StagedFlags staged =
        stage_batch<kRenderThreads, kBatch>(A.inst_val, A.rec_geom, A.rec_color, A.rec_blue, A.vis_cap, base, end, s_geom,
                                            s_col, s_blue, s_slot, kAux ? A.rec_aux : nullptr, kAux ? s_aux : nullptr);
    const int nb = (int)min(end - base, (uint32_t)kBatch);
    // Whether any staged entry can reach the 0.99 clamp (rare): then the batch
    // takes the careful copy of the pixel loop, which gives the entries that
    // cannot clamp the same alpha.  So does every batch of a warp whose
    // products may overflow: from its upstream gradients, or from the first
    // batch on that holds a colour or depth above kMagMax.
    const bool clamp_any = __syncthreads_or(staged.clamp || staged.large) != 0;
    if (clamp_any && __syncthreads_or(staged.large)) tame = false;
    // One list entry.
    auto entry = [&](int j, uint32_t pos, auto clamp_tag) {
      constexpr bool kClamp = decltype(clamp_tag)::value;
      const float4 geom = s_geom[j];
      const float4 col = s_col[j];
      const float blue = s_blue[j];
      const ColumnTerms ct = column_terms(geom, pxc, col.y);
      // group_w, keeping v - (group row centre) for the pixels' dy
      float dy4[kGroups], w4[kGroups];
#pragma unroll
      for (int g = 0; g < kGroups; ++g) {
        dy4[g] = __fsub_rn(geom.y, gyc[g]);
        w4[g] = __fmaf_rn(col.x, dy4[g], ct.bdx);
      }
      const float zj = kAux ? s_aux[j].x : 0.f;
      // gp = dL/d(natural-log power) of each pixel; a pixel that is not
      // skipped has alpha = a 2^-q (below the clamp), so gp = g_alpha a 2^-q
      // is also the opacity term: dL/da = S_0 / a.
      float2 gp[kPairs], gr = make_float2(0.f, 0.f), gg = gr, gb = gr, gz = gr;
      bool contrib = false;  // the same in every lane
#pragma unroll
      for (int q = 0; q < kPairs; ++q) {
        gp[q] = make_float2(0.f, 0.f);
        const int k0 = 2 * q, k1 = 2 * q + 1;
        // the two lanes of pixel_alpha
        const float2 offs = kPPT >= 4 ? make_float2(-(float)(k0 & 3), -(float)(k1 & 3))
                                      : make_float2(base_off - (float)k0, base_off - (float)k1);
        const float wg = w4[k0 >> 2];
        const float2 w2 = __ffma2_rn(make_float2(col.x, col.x), offs, make_float2(wg, wg));
        const float2 q2 = __ffma2_rn(w2, w2, make_float2(ct.adx2, ct.adx2));
        const float aG0 = ex2_approx(-q2.x), aG1 = ex2_approx(-q2.y);
        const float al0 = kClamp ? min_nan(0.99f, aG0) : aG0, al1 = kClamp ? min_nan(0.99f, aG1) : aG1;
        // the forward's skip decision, NaN included, up to the pixel's last entry
        const bool v0 = pos < last[k0] && al0 >= kAlphaMin, v1 = pos < last[k1] && al1 >= kAlphaMin;
        if (!__any_sync(0xffffffffu, v0 || v1)) continue;
        contrib = true;
        if (kClamp && !tame) {  // an infinity or NaN of a skipped pixel must not meet its zero weight: one at a time
          auto pixel = [&](bool v, float al, float aG, float &t, float &dr, float n0, float n1, float n2, float nd,
                           float no, float &sr, float &sg, float &sb, float &sz, float &gpk) {
            if (!v) return;
            const float io = rcp_approx(__fsub_rn(1.0f, al));
            t = t * io;
            const float nw = -al * t;
            sr = __fmaf_rn(n0, nw, sr);
            sg = __fmaf_rn(n1, nw, sg);
            sb = __fmaf_rn(n2, nw, sb);
            float nDc = __fmaf_rn(n2, blue, __fmaf_rn(n0, col.z, n1 * col.w));
            if (kAux) {
              nDc += __fmaf_rn(nd, zj, no);
              sz = __fmaf_rn(nd, nw, sz);
            }
            if (!(kClamp && aG > 0.99f)) gpk = __fmaf_rn(t, nDc, io * dr) * -al;
            dr = __fmaf_rn(nw, nDc, dr);
          };
          const float2 nd = kAux ? nD[q] : gz, no = kAux ? nO[q] : gz;
          pixel(v0, al0, aG0, T[q].x, Dr[q].x, nC0[q].x, nC1[q].x, nC2[q].x, nd.x, no.x, gr.x, gg.x, gb.x, gz.x, gp[q].x);
          pixel(v1, al1, aG1, T[q].y, Dr[q].y, nC0[q].y, nC1[q].y, nC2[q].y, nd.y, no.y, gr.y, gg.y, gb.y, gz.y, gp[q].y);
          continue;
        }
        const float2 na = make_float2(v0 ? -al0 : 0.0f, v1 ? -al1 : 0.0f);  // -alpha
        const float2 om = __fadd2_rn(make_float2(1.0f, 1.0f), na);
        const float2 io = make_float2(rcp_approx(om.x), rcp_approx(om.y));
        T[q] = __fmul2_rn(T[q], io);               // transmittance in front of this entry
        const float2 nw = __fmul2_rn(na, T[q]);    // -alpha T
        gr = __ffma2_rn(nC0[q], nw, gr);
        gg = __ffma2_rn(nC1[q], nw, gg);
        gb = __ffma2_rn(nC2[q], nw, gb);
        // -(dL/dX . x_i)
        float2 nDc = __ffma2_rn(nC2[q], make_float2(blue, blue),
                                __ffma2_rn(nC0[q], make_float2(col.z, col.z), __fmul2_rn(nC1[q], make_float2(col.w, col.w))));
        if (kAux) {
          nDc = __fadd2_rn(nDc, __ffma2_rn(nD[q], make_float2(zj, zj), nO[q]));
          gz = __ffma2_rn(nD[q], nw, gz);
        }
        const float2 nga = __ffma2_rn(T[q], nDc, __fmul2_rn(io, Dr[q]));  // -dL/dalpha
        Dr[q] = __ffma2_rn(nw, nDc, Dr[q]);
        gp[q] = __fmul2_rn(nga, na);
        if (kClamp) {  // min(0.99, .) is locally constant when clamped
          if (aG0 > 0.99f) gp[q].x = 0.0f;
          if (aG1 > 0.99f) gp[q].y = 0.0f;
        }
      }
      if (!contrib) return;
      // Moments S_0 = sum gp, S_1 = sum gp dy, S_2 = sum gp dy^2 of the strip.
      // Per row group dy = dyb - o with o the pixel's row in the group, so
      // with P_n = sum o^n gp: S_1 = dyb P_0 - P_1, S_2 = dyb (dyb P_0 - 2
      // P_1) + P_2.
      float S0 = 0.f, S1 = 0.f, S2 = 0.f;
#pragma unroll
      for (int g = 0; g < kGroups; ++g) {
        const float dyb = dy4[g] + base_off;  // dy of the group's first row in the strip
        float P0, P1, P2;
        if (kPPT >= 4) {
          const float2 ga = gp[2 * g], gc = gp[2 * g + 1 < kPairs ? 2 * g + 1 : 0];
          P0 = ((ga.x + ga.y) + gc.x) + gc.y;
          P1 = __fmaf_rn(3.0f, gc.y, __fmaf_rn(2.0f, gc.x, ga.y));
          P2 = __fmaf_rn(9.0f, gc.y, __fmaf_rn(4.0f, gc.x, ga.y));
        } else {
          P0 = gp[0].x + gp[0].y;
          P1 = P2 = gp[0].y;
        }
        S0 += P0;
        S1 += __fmaf_rn(dyb, P0, -P1);
        S2 += __fmaf_rn(dyb, __fmaf_rn(dyb, P0, -2.0f * P1), P2);
      }
      float *dst = &red[buffered * kSums][lane];
      dst[0 * kRedStride] = ct.dx * S0;
      dst[1 * kRedStride] = S1;
      dst[2 * kRedStride] = (ct.dx * ct.dx) * S0;
      dst[3 * kRedStride] = ct.dx * S1;
      dst[4 * kRedStride] = S2;
      dst[5 * kRedStride] = S0;
      dst[6 * kRedStride] = gr.x + gr.y;
      dst[7 * kRedStride] = gg.x + gg.y;
      dst[8 * kRedStride] = gb.x + gb.y;
      if (kAux) dst[(kSums - 1) * kRedStride] = gz.x + gz.y;
      if (lane == 0) jb[buffered] = j;
      ++buffered;
    };
    const uint32_t pos0 = base - range.x;  // entry index of the batch's first entry
    const int first = warp_max > pos0 ? (int)min(warp_max - pos0, (uint32_t)nb) - 1 : -1;
    if (clamp_any || !tame) {
      for (int j = first; j >= 0; --j) {
        entry(j, pos0 + j, std::true_type());
        if (buffered == kRedEntries) flush();
      }
    } else {
      for (int j = first; j >= 0; --j) {
        entry(j, pos0 + j, std::false_type());
        if (buffered == kRedEntries) flush();
      }
    }
    if (buffered) flush();  // the batch's records are about to be replaced
  }
}

__global__ void l1_loss_kernel(const float *__restrict__ img, const float *__restrict__ target, int64_t count,
                               float inv_count, float *loss, float *grad) {
  grid_dependency_sync();
  float acc = 0.f;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
    const float d = img[i] - target[i];
    acc += fabsf(d);
    grad[i] = d > 0.f ? inv_count : (d < 0.f ? -inv_count : 0.f);
  }
  acc = warp_sum(acc);
  __shared__ float s[32];
  if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    float v = threadIdx.x < (blockDim.x >> 5) ? s[threadIdx.x] : 0.f;
    v = warp_sum(v);
    if (threadIdx.x == 0) atomicAdd(loss, v * inv_count);
  }
}

// Adam (the optimiser of the training step): with t the device step count,
// m = b1 m + (1 - b1) g, v = b2 v + (1 - b2) g^2,
// p -= lr / (1 - b1^t) * m / (sqrt(v) / sqrt(1 - b2^t) + eps).
struct AdamArgs {
  float *p;
  const float *g;
  float *m, *v;
  int64_t count;
  float lr, b1, b2, eps;
  const int32_t *step;
};

__device__ __forceinline__ float adam_one(float &p, float g, float &m, float &v, float b1, float b2, float eps,
                                          float step_size, float inv_sqrt_bc2) {
  m = b1 * m + (1.0f - b1) * g;
  v = b2 * v + (1.0f - b2) * g * g;
  p -= step_size * m / (sqrtf(v) * inv_sqrt_bc2 + eps);
  return p;
}

__global__ void adam_kernel(AdamArgs A) {
  grid_dependency_sync();
  const float t = (float)*A.step;
  const float bc1 = 1.0f - powf(A.b1, t), bc2 = 1.0f - powf(A.b2, t);
  const float step_size = A.lr / bc1, inv_sqrt_bc2 = rsqrtf(bc2);
  const int64_t n4 = A.count / 4;
  float4 *p4 = reinterpret_cast<float4 *>(A.p);
  const float4 *g4 = reinterpret_cast<const float4 *>(A.g);
  float4 *m4 = reinterpret_cast<float4 *>(A.m);
  float4 *v4 = reinterpret_cast<float4 *>(A.v);
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += stride) {
    float4 p = p4[i], m = m4[i], v = v4[i];
    const float4 g = g4[i];
    adam_one(p.x, g.x, m.x, v.x, A.b1, A.b2, A.eps, step_size, inv_sqrt_bc2);
    adam_one(p.y, g.y, m.y, v.y, A.b1, A.b2, A.eps, step_size, inv_sqrt_bc2);
    adam_one(p.z, g.z, m.z, v.z, A.b1, A.b2, A.eps, step_size, inv_sqrt_bc2);
    adam_one(p.w, g.w, m.w, v.w, A.b1, A.b2, A.eps, step_size, inv_sqrt_bc2);
    p4[i] = p;
    m4[i] = m;
    v4[i] = v;
  }
  for (int64_t i = 4 * n4 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < A.count; i += stride)
    adam_one(A.p[i], A.g[i], A.m[i], A.v[i], A.b1, A.b2, A.eps, step_size, inv_sqrt_bc2);
}

// Adam over a set of tensors in one launch: unit u of the set is float4 u -
// first[k] of tensor k (the last unit of a tensor whose count is not a
// multiple of 4 takes its 1-3 trailing scalars).  Each element gets exactly
// adam_one, as in adam_kernel; with zero the gradient is cleared after it is
// read, so the next step accumulates into zeros without a separate fill.
struct AdamSetArgs {
  AdamTensorDev t[kAdamMaxTensors];
  int64_t first[kAdamMaxTensors + 1];  // prefix of the tensors' unit counts
  int32_t n;
  float b1, b2, eps;
  const int32_t *step;
  int32_t zero;
};

__global__ void adam_set_kernel(AdamSetArgs A) {
  grid_dependency_sync();
  const float t = (float)*A.step;
  const float bc1 = 1.0f - powf(A.b1, t), bc2 = 1.0f - powf(A.b2, t);
  const float inv_sqrt_bc2 = rsqrtf(bc2);
  const int64_t total = A.first[A.n];
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  int k = 0;
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < total; u += stride) {
    while (u >= A.first[k + 1]) ++k;  // units only grow along the loop
    const AdamTensorDev &T = A.t[k];
    const float step_size = T.lr / bc1;
    const int64_t i = u - A.first[k];
    if (4 * i + 4 <= T.count) {
      float4 *p4 = reinterpret_cast<float4 *>(T.p) + i;
      float4 *g4 = reinterpret_cast<float4 *>(T.g) + i;
      float4 *m4 = reinterpret_cast<float4 *>(T.m) + i;
      float4 *v4 = reinterpret_cast<float4 *>(T.v) + i;
      float4 p = *p4, m = *m4, v = *v4;
      const float4 g = *g4;
      adam_one(p.x, g.x, m.x, v.x, A.b1, A.b2, A.eps, step_size, inv_sqrt_bc2);
      adam_one(p.y, g.y, m.y, v.y, A.b1, A.b2, A.eps, step_size, inv_sqrt_bc2);
      adam_one(p.z, g.z, m.z, v.z, A.b1, A.b2, A.eps, step_size, inv_sqrt_bc2);
      adam_one(p.w, g.w, m.w, v.w, A.b1, A.b2, A.eps, step_size, inv_sqrt_bc2);
      *p4 = p;
      *m4 = m;
      *v4 = v;
      if (A.zero) *g4 = make_float4(0.f, 0.f, 0.f, 0.f);
    } else {
      for (int64_t e = 4 * i; e < T.count; ++e) {
        adam_one(T.p[e], T.g[e], T.m[e], T.v[e], A.b1, A.b2, A.eps, step_size, inv_sqrt_bc2);
        if (A.zero) T.g[e] = 0.f;
      }
    }
  }
}

// Clears a set of tensors in one launch (units as in adam_set_kernel): six
// fills of a small model's gradients took six launches of the host's time.
struct ZeroSetArgs {
  float *p[kAdamMaxTensors];
  int64_t count[kAdamMaxTensors], first[kAdamMaxTensors + 1];
  int32_t n;
};

__global__ void zero_set_kernel(ZeroSetArgs A) {
  grid_dependency_sync();
  const int64_t total = A.first[A.n], stride = (int64_t)gridDim.x * blockDim.x;
  int k = 0;
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < total; u += stride) {
    while (u >= A.first[k + 1]) ++k;  // units only grow along the loop
    const int64_t i = 4 * (u - A.first[k]);
    if (i + 4 <= A.count[k]) {
      *reinterpret_cast<float4 *>(A.p[k] + i) = make_float4(0.f, 0.f, 0.f, 0.f);
    } else {
      for (int64_t e = i; e < A.count[k]; ++e) A.p[k][e] = 0.f;
    }
  }
}

__global__ void adam_tick_kernel(int32_t *step) {
  grid_dependency_sync();
  if (threadIdx.x == 0) *step += 1;
}

// Mask compression loss (Sec. 4.3): L = mean sigmoid(m), dL/dm = M (1 - M) / n.
__global__ void mask_loss_kernel(const float *__restrict__ m, int64_t n, float inv_n, float *loss, float *grad) {
  grid_dependency_sync();
  float acc = 0.f;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float M = 1.0f / (1.0f + expf(-m[i]));
    acc += M;
    grad[i] += M * (1.0f - M) * inv_n;
  }
  acc = warp_sum(acc);
  __shared__ float s[32];
  if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    float v = threadIdx.x < (blockDim.x >> 5) ? s[threadIdx.x] : 0.f;
    v = warp_sum(v);
    if (threadIdx.x == 0) atomicAdd(loss, v * inv_n);
  }
}

template <int MAXV, int TILE, int PPT, int B>
cudaError_t launch_fwd_batch(const RenderArgs &A, const RasterViews<MAXV> &rv, unsigned grid,
                             unsigned long long *stats, bool image_only, cudaStream_t st) {
  constexpr unsigned NT = TILE * TILE / PPT;
  if (image_only)
    return launch_pdl(render_fwd_kernel<MAXV, TILE, PPT, 3, B>, grid, NT, st, A, rv, (unsigned long long *)nullptr);
  if (stats) return launch_pdl(render_fwd_kernel<MAXV, TILE, PPT, 1, B>, grid, NT, st, A, rv, stats);
  if (A.out_aux)
    return launch_pdl(render_fwd_kernel<MAXV, TILE, PPT, 2, B>, grid, NT, st, A, rv, (unsigned long long *)nullptr);
  return launch_pdl(render_fwd_kernel<MAXV, TILE, PPT, 0, B>, grid, NT, st, A, rv, (unsigned long long *)nullptr);
}

template <int MAXV, int TILE, int PPT>
cudaError_t launch_fwd_ppt(const RenderArgs &A, const RasterViews<MAXV> &rv, unsigned grid,
                           unsigned long long *stats, int batch, bool image_only, cudaStream_t st) {
  if (batch == 128) return launch_fwd_batch<MAXV, TILE, PPT, 128>(A, rv, grid, stats, image_only, st);
  return launch_fwd_batch<MAXV, TILE, PPT, 256>(A, rv, grid, stats, image_only, st);
}

template <int MAXV>
cudaError_t render_fwd_typed(const Layout &L, const fgs4d_settings *s, const fgs4d_view *views, int32_t nviews,
                             unsigned char *ws, float *out_rgb, float *out_T, unsigned long long *stats,
                             float *out_aux, bool image_only, cudaStream_t st) {
  RasterViews<MAXV> rv;
  if (!make_raster_views<MAXV>(L, views, nviews, &rv)) return cudaErrorInvalidValue;
  RenderArgs A;
  A.ranges = reinterpret_cast<const uint2 *>(ws + L.ranges);
  A.inst_val = reinterpret_cast<const uint32_t *>(ws + L.inst_val[L.tile_passes & 1]);
  A.rec_geom = reinterpret_cast<const float4 *>(ws + L.rec_geom);
  A.rec_color = reinterpret_cast<const float4 *>(ws + L.rec_color);
  A.rec_blue = reinterpret_cast<const float *>(ws + L.rec_blue);
  A.rec_aux = reinterpret_cast<const float4 *>(ws + L.rec_aux);
  A.vis_cap = (uint32_t)L.vis_cap;
  A.out_rgb = out_rgb;
  A.out_T = out_T;
  A.out_aux = out_aux;
  A.pix_T = reinterpret_cast<float *>(ws + L.pix_T);
  A.pix_last = reinterpret_cast<uint32_t *>(ws + L.pix_last);
  A.bg0 = s->bg[0];
  A.bg1 = s->bg[1];
  A.bg2 = s->bg[2];
  if (L.total_tiles == 0) return cudaSuccess;
  const unsigned grid = (unsigned)L.total_tiles;
  if (s->tile == 8) {
    if (render_ppt(s, L, false) == 1) return launch_fwd_ppt<MAXV, 8, 1>(A, rv, grid, stats, s->shared_batch, image_only, st);
    return launch_fwd_ppt<MAXV, 8, 2>(A, rv, grid, stats, s->shared_batch, image_only, st);
  }
  switch (render_ppt(s, L, false)) {
    case 2: return launch_fwd_ppt<MAXV, 16, 2>(A, rv, grid, stats, s->shared_batch, image_only, st);
    case 8: return launch_fwd_ppt<MAXV, 16, 8>(A, rv, grid, stats, s->shared_batch, image_only, st);
    default: return launch_fwd_ppt<MAXV, 16, 4>(A, rv, grid, stats, s->shared_batch, image_only, st);
  }
}

template <int MAXV, int TILE, int PPT, int B>
cudaError_t launch_bwd_batch(const RenderBwdArgs &A, const RasterViews<MAXV> &rv, unsigned grid, cudaStream_t st) {
  constexpr unsigned NT = TILE * TILE / PPT;
  if (A.dL_daux) return launch_pdl(render_bwd_kernel<MAXV, TILE, PPT, true, B>, grid, NT, st, A, rv);
  return launch_pdl(render_bwd_kernel<MAXV, TILE, PPT, false, B>, grid, NT, st, A, rv);
}

template <int MAXV, int TILE, int PPT>
cudaError_t launch_bwd_ppt(const RenderBwdArgs &A, const RasterViews<MAXV> &rv, unsigned grid, int batch,
                           cudaStream_t st) {
  // Default 128: with the reduction rows a block of 64 threads then takes 13
  // KB of shared memory instead of 18, so that shared memory does not bound
  // the resident blocks below the registers' 16.
  if (batch == 256) return launch_bwd_batch<MAXV, TILE, PPT, 256>(A, rv, grid, st);
  return launch_bwd_batch<MAXV, TILE, PPT, 128>(A, rv, grid, st);
}

template <int MAXV>
cudaError_t render_bwd_typed(const Layout &L, const fgs4d_settings *s, const fgs4d_view *views, int32_t nviews,
                             unsigned char *ws, const float *dL_drgb, const float *dL_daux, cudaStream_t st) {
  RasterViews<MAXV> rv;
  if (!make_raster_views<MAXV>(L, views, nviews, &rv)) return cudaErrorInvalidValue;
  cudaError_t e = cudaMemsetAsync(ws + L.slot_grad, 0, (size_t)L.vis_cap * kSlotGradFloats * sizeof(float), st);
  if (e != cudaSuccess) return e;
  RenderBwdArgs A;
  A.ranges = reinterpret_cast<const uint2 *>(ws + L.ranges);
  A.inst_val = reinterpret_cast<const uint32_t *>(ws + L.inst_val[L.tile_passes & 1]);
  A.rec_geom = reinterpret_cast<const float4 *>(ws + L.rec_geom);
  A.rec_color = reinterpret_cast<const float4 *>(ws + L.rec_color);
  A.rec_blue = reinterpret_cast<const float *>(ws + L.rec_blue);
  A.vis_cap = (uint32_t)L.vis_cap;
  A.pix_T = reinterpret_cast<const float *>(ws + L.pix_T);
  A.pix_last = reinterpret_cast<const uint32_t *>(ws + L.pix_last);
  A.dL_drgb = dL_drgb;
  A.dL_daux = dL_daux;
  A.rec_aux = reinterpret_cast<const float4 *>(ws + L.rec_aux);
  A.slot_grad = reinterpret_cast<float4 *>(ws + L.slot_grad);
  A.bg0 = s->bg[0];
  A.bg1 = s->bg[1];
  A.bg2 = s->bg[2];
  if (L.total_tiles == 0) return cudaSuccess;
  const unsigned grid = (unsigned)L.total_tiles;
  if (s->tile == 8) {
    if (render_ppt(s, L, dL_daux == nullptr) == 1) return launch_bwd_ppt<MAXV, 8, 1>(A, rv, grid, s->shared_batch, st);
    return launch_bwd_ppt<MAXV, 8, 2>(A, rv, grid, s->shared_batch, st);
  }
  switch (render_ppt(s, L, dL_daux == nullptr)) {
    case 2: return launch_bwd_ppt<MAXV, 16, 2>(A, rv, grid, s->shared_batch, st);
    case 8: return launch_bwd_ppt<MAXV, 16, 8>(A, rv, grid, s->shared_batch, st);
    default: return launch_bwd_ppt<MAXV, 16, 4>(A, rv, grid, s->shared_batch, st);
  }
}

}  // namespace

cudaError_t launch_render_fwd(const Layout &L, const fgs4d_settings *s, const fgs4d_view *views, int32_t nviews,
                              unsigned char *ws, float *out_rgb, float *out_T, unsigned long long *stats,
                              float *out_aux, cudaStream_t stream, bool image_only) {
  if (nviews == 1)
    return render_fwd_typed<1>(L, s, views, nviews, ws, out_rgb, out_T, stats, out_aux, image_only, stream);
  return render_fwd_typed<FGS4D_MAX_VIEWS>(L, s, views, nviews, ws, out_rgb, out_T, stats, out_aux, image_only,
                                           stream);
}

cudaError_t launch_render_bwd(const Layout &L, const fgs4d_settings *s, const fgs4d_view *views, int32_t nviews,
                              unsigned char *ws, const float *dL_drgb, const float *dL_daux, cudaStream_t stream) {
  if (nviews == 1) return render_bwd_typed<1>(L, s, views, nviews, ws, dL_drgb, dL_daux, stream);
  return render_bwd_typed<FGS4D_MAX_VIEWS>(L, s, views, nviews, ws, dL_drgb, dL_daux, stream);
}

cudaError_t launch_adam(float *p, const float *g, float *m, float *v, int64_t count, float lr, float b1, float b2,
                        float eps, const int32_t *step, cudaStream_t stream) {
  if (count <= 0) return cudaSuccess;
  AdamArgs A{p, g, m, v, count, lr, b1, b2, eps, step};
  const int blocks = (int)std::min<int64_t>((count / 4 + 255) / 256 + 1, 152 * 8);
  return launch_pdl(adam_kernel, (unsigned)blocks, 256u, stream, A);
}

cudaError_t launch_adam_set(const AdamTensorDev *tensors, int32_t n, float b1, float b2, float eps,
                            const int32_t *step, bool zero_grad, cudaStream_t stream) {
  AdamSetArgs A{};
  A.n = n;
  A.first[0] = 0;
  for (int32_t k = 0; k < n; ++k) {
    A.t[k] = tensors[k];
    A.first[k + 1] = A.first[k] + (tensors[k].count + 3) / 4;
  }
  A.b1 = b1;
  A.b2 = b2;
  A.eps = eps;
  A.step = step;
  A.zero = zero_grad ? 1 : 0;
  const int64_t total = A.first[n];
  if (total == 0) return cudaSuccess;
  const int blocks = (int)std::min<int64_t>((total + 255) / 256, 152 * 8);
  return launch_pdl(adam_set_kernel, (unsigned)blocks, 256u, stream, A);
}

cudaError_t launch_zero_set(float *const *tensors, const int64_t *counts, int32_t n, cudaStream_t stream) {
  ZeroSetArgs A{};
  A.n = n;
  for (int32_t k = 0; k < n; ++k) {
    A.p[k] = tensors[k];
    A.count[k] = counts[k];
    A.first[k + 1] = A.first[k] + (counts[k] + 3) / 4;
  }
  if (A.first[n] == 0) return cudaSuccess;
  const int blocks = (int)std::min<int64_t>((A.first[n] + 255) / 256, 152 * 8);
  return launch_pdl(zero_set_kernel, (unsigned)blocks, 256u, stream, A);
}

cudaError_t launch_adam_tick(int32_t *step, cudaStream_t stream) {
  return launch_pdl(adam_tick_kernel, 1u, 32u, stream, step);
}

cudaError_t launch_mask_loss(const float *mask_logit, int64_t n, float *loss, float *grad, cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  const int blocks = (int)std::min<int64_t>((n + 255) / 256, 152 * 8);
  return launch_pdl(mask_loss_kernel, (unsigned)blocks, 256u, stream, mask_logit, n, 1.0f / (float)n, loss, grad);
}

cudaError_t launch_l1_loss(const float *img, const float *target, int64_t count, int64_t mean_count, float *loss,
                           float *grad, cudaStream_t stream) {
  if (count <= 0) return cudaSuccess;
  const int blocks = (int)std::min<int64_t>((count + 255) / 256, 152 * 8);
  return launch_pdl(l1_loss_kernel, (unsigned)blocks, 256u, stream, img, target, count, 1.0f / (float)mean_count,
                    loss, grad);
}

}  // namespace fgs4d
