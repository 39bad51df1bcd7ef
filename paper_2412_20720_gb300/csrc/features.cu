// Scale-gated feature rendering for 4D segmentation (Sec. 7 of arXiv
// 2412.20720, "Scale-gated features"): each Gaussian carries a feature
// f in R^D; at a scale s the gate vector S(s) in [0,1]^D gives
// f^s = S(s) (.) f, which is normalised and composited exactly like the
// colour of Eq. 6 (zero background).  The geometry is that of a pre-trained
// 4DGS, so the backward pass returns dL/df and dL/dS(s) only.
//
// Both directions are contractions (short lists, and the map for D <= 16, take
// scalar kernels: launch_feat_typed): the map is F[p][c] = sum_j w[p][j]
// fhat[j][c], and the adjoint needs v[j][c] = sum_p w[p][j] dL/dF[p][c].  One
// CTA per (view, tile), one pixel per thread; a warp computes the weights of
// its 32 pixels for kChunk entries (pixel_alpha's skip/stop decisions, so the
// weights equal those of the colour compositor bit for bit), passes them
// through shared memory and multiplies on the tensor cores (mma.sync m16n8k8,
// TF32 operands split in two: x = hi + lo with 11 bits each, lo hi + hi lo + hi
// hi; with lo rounded to 2^-23 |x| and lo lo left out, up to 2^-22, a product
// is within 2^-21; the accumulators start at zero every chunk, take a chunk's
// small products before its large ones, as the matrix unit's sums lose bits at
// the size they have reached, and are added up in FP32).  The warp-level instruction is taken
// rather than tcgen05 because the weights come out of a per-pixel recurrence
// 32 pixels at a time and the contraction is the small part: 48 products of
// some 800 issued instructions per chunk of 16 entries and 32 pixels at D = 32.
//
// Backward: a warp's product sums over its own 32 pixels; the warps' sums of
// an entry are added through shared memory, the normalisation Jacobian is
// applied once per (tile, entry): dL/dg = (v - fhat (fhat . v)) / |g|,
// dL/df = S (.) dL/dg is added with one atomic per component, and dL/dS(s) =
// f (.) dL/dg is summed per block.
//
// Measured at 300k Gaussians, one 1352x1014 view, before (multiply-adds with a
// shuffle butterfly and D atomics per (warp, entry)) -> now, us: D = 32 forward
// 900 -> 726, backward 1490 -> 851; D = 16 backward 933 -> 574; D = 8 670 -> 465.
// Bound by issue; at D = 32 a quarter of the warps are resident (operands or
// accumulators take 128 registers a thread).
#include <algorithm>

#include "fgs4d_internal.cuh"

namespace fgs4d {

namespace {

constexpr int kChunk = 16;      // entries per matrix product (M of the adjoint, two K steps of the forward)
constexpr int kFeatBatch = 64;  // staged records
static_assert(kFeatBatch % kChunk == 0, "whole chunks per batch");

// One pixel per thread.
template <int TILE>
__host__ __device__ constexpr int feat_threads() {
  return TILE * TILE;
}
// Floats per row of the staged features: = 8 mod 32 (or 8, 24), so that the
// 4 x 8 lanes of an operand load hit 32 banks.
template <int D>
__host__ __device__ constexpr int feat_stride() {
  return D == 32 ? 40 : (D == 16 ? 24 : 8);
}
constexpr int kWFwd = 40;  // floats per entry row of the forward's weights (= 8 mod 32)
constexpr int kWBwd = 36;  // and of the adjoint's (= 4 mod 32)

struct FeatArgs {
  const uint2 *ranges;
  const uint32_t *inst_val;
  const float4 *rec_geom, *rec_color;
  const int4 *rec_meta;
  uint32_t vis_cap;
  int64_t n;
  const float *feat;  // [n][D]
  const float *gate;  // [D] or null (ones)
  float *out;         // [views][D][H][W]
  const float *dL_dF; // backward: [views][D][H][W]
  float *g_feat;      // backward: [n][D]
  float *g_gate;      // backward: [D] or null
};

// Pixels of a column per thread in the scalar kernels.  The adjoint reduces D
// sums per (warp, entry): with D <= 16 it takes 4 at 16x16 (64 threads), half
// the warps per tile and so half the reductions.
constexpr int kScalarPPT = 2;
template <int TILE, int D>
__host__ __device__ constexpr int scalar_bwd_ppt() {
  return (TILE == 16 && D <= 16) ? 4 : kScalarPPT;
}

// Stages entry `k` of the batch: geometry, opacity and normalised gated
// feature (rows padded to D + 1 floats against bank conflicts); for the
// adjoint also the raw feature, its gated norm and the Gaussian.
template <int D, bool kBwd>
__device__ __forceinline__ void stage_feature(const FeatArgs &A, const float *s_gate, uint32_t idx, int k,
                                              float4 *s_geom, float2 *s_ca, float *s_fhat, float *s_f, float *s_norm,
                                              int32_t *s_gi) {
  const uint32_t s = A.inst_val[idx];
  float4 geom = make_float4(0.f, 0.f, 0.f, 0.f);
  float2 ca = make_float2(0.f, kLogAlphaNone);  // (b2, log2 a): every pixel skips the entry
  int32_t gi = -1;
  if (s < A.vis_cap) {
    geom = A.rec_geom[s];
    const float4 c = A.rec_color[s];
    ca = make_float2(c.x, c.y);
    gi = A.rec_meta[s].x;
    if (gi < 0 || (int64_t)gi >= A.n) {
      gi = -1;
      ca.y = kLogAlphaNone;
    }
  }
  s_geom[k] = geom;
  s_ca[k] = ca;
  float g[D];
  float nn = 0.f;
  if (gi >= 0) {
    const float4 *row = reinterpret_cast<const float4 *>(A.feat + (int64_t)gi * D);
#pragma unroll
    for (int c4 = 0; c4 < D / 4; ++c4) {
      const float4 v = row[c4];
      g[4 * c4 + 0] = v.x;
      g[4 * c4 + 1] = v.y;
      g[4 * c4 + 2] = v.z;
      g[4 * c4 + 3] = v.w;
    }
  } else {
#pragma unroll
    for (int c = 0; c < D; ++c) g[c] = 0.f;
  }
#pragma unroll
  for (int c = 0; c < D; ++c) {
    if (kBwd) s_f[k * (D + 1) + c] = g[c];
    g[c] *= s_gate[c];
    nn += g[c] * g[c];
  }
  const float norm = sqrtf(nn);
  const float inv = norm > 0.f ? 1.0f / norm : 0.f;
#pragma unroll
  for (int c = 0; c < D; ++c) s_fhat[k * (D + 1) + c] = g[c] * inv;
  if (kBwd) {
    s_norm[k] = norm;
    s_gi[k] = gi;
  }
}

// Feature map with a multiply-add per component, pixel and entry, a thread on a
// vertical pair of pixels: for D <= 16, where the matrix form's weights cost a
// thread per pixel (300k Gaussians at 1352x1014, us, this / matrix form: D = 8
// 331 / 409, D = 16 486 / 488; a street view of 14 entries a tile D = 16 44 /
// 63), and for D = 32 on short lists (launch_feat_typed).
template <int MAXV, int TILE, int D>
__global__ void __launch_bounds__(TILE *TILE / kScalarPPT)
    render_features_scalar_kernel(FeatArgs A, RasterViews<MAXV> rv) {
  grid_dependency_sync();
  constexpr int kBatch = TILE * TILE / kScalarPPT;
  __shared__ float4 s_geom[kBatch];
  __shared__ float2 s_ca[kBatch];
  __shared__ float s_fhat[kBatch * (D + 1)];
  __shared__ float s_gate[D];
  const int32_t gt = blockIdx.x;
  const RasterView &V = rv.v[find_view<MAXV>(rv, gt)];
  const int32_t lt = gt - V.tile_base;
  const int32_t tx = lt % V.gw, ty = lt / V.gw;
  const int32_t px = tx * TILE + (threadIdx.x & (TILE - 1));
  const int32_t py0 = ty * TILE + (threadIdx.x / TILE) * kScalarPPT;
  const uint2 range = tile_range(A.ranges, gt);
  const float pxc = (float)px + 0.5f;
  if (threadIdx.x < D) s_gate[threadIdx.x] = A.gate ? A.gate[threadIdx.x] : 1.0f;
  static_assert(kScalarPPT <= 4, "a strip inside one row group");
  const float gyc = row_group_centre(py0);
  float T[kScalarPPT], off[kScalarPPT], F[kScalarPPT][D];
  bool live = false;
#pragma unroll
  for (int k = 0; k < kScalarPPT; ++k) {
    const bool in = px < V.width && py0 + k < V.height;
    T[k] = in ? 1.0f : -1.0f;
    off[k] = in ? row_offset(py0 + k) : stopped_offset();
#pragma unroll
    for (int c = 0; c < D; ++c) F[k][c] = 0.f;
    live = live || in;
  }
  for (uint32_t base = range.x; base < range.y; base += kBatch) {
    if (__syncthreads_count(live) == 0) break;
    if (base + threadIdx.x < range.y)
      stage_feature<D, false>(A, s_gate, base + threadIdx.x, threadIdx.x, s_geom, s_ca, s_fhat, nullptr, nullptr,
                              nullptr);
    __syncthreads();
    const int nb = (int)min(range.y - base, (uint32_t)kBatch);
    for (int j = 0; j < nb && live; ++j) {
      const float4 geom = s_geom[j];
      const float2 ca = s_ca[j];
      const ColumnTerms ct = column_terms(geom, pxc, ca.y);
      const float w4 = group_w(ct, geom.y, ca.x, gyc);
      const bool clamp = entry_clamps(ca.y);
#pragma unroll
      for (int k = 0; k < kScalarPPT; ++k) {
        const AlphaEval e = pixel_alpha(ct, w4, ca.x, off[k], clamp);
        if (e.alpha >= kAlphaMin) {  // false for stopped pixels (row offset +inf)
          const float w = __fmul_rn(e.alpha, T[k]);
          const float Tn = __fsub_rn(T[k], w);
          if (Tn < kTMin) {
            T[k] = -T[k];
            off[k] = stopped_offset();
          } else {
#pragma unroll
            for (int c = 0; c < D; ++c) F[k][c] = __fmaf_rn(s_fhat[j * (D + 1) + c], w, F[k][c]);
            T[k] = Tn;
          }
        }
      }
      live = false;
#pragma unroll
      for (int k = 0; k < kScalarPPT; ++k) live = live || T[k] > 0.0f;
    }
  }
  const int64_t HW = (int64_t)V.width * V.height;
  float *out = A.out + V.pix_base * D;
#pragma unroll
  for (int k = 0; k < kScalarPPT; ++k) {
    if (!(px < V.width && py0 + k < V.height)) continue;
    const int64_t p = (int64_t)(py0 + k) * V.width + px;
#pragma unroll
    for (int c = 0; c < D; ++c) out[c * HW + p] = F[k][c];
  }
}

// Sums D <= 32 per-lane values over the warp; on return a[0] of lane l holds
// the total of value l (lanes >= D hold totals of zero padding).
template <int D>
__device__ __forceinline__ float warp_transpose_sum(float (&a)[32], int lane) {
#pragma unroll
  for (int half = 16; half >= 1; half >>= 1) {
    const bool up = (lane & half) != 0;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const float send = up ? a[i] : a[i + half];
      const float keep = up ? a[i + half] : a[i];
      a[i] = keep + __shfl_xor_sync(0xffffffffu, send, half);
    }
  }
  return a[0];
}

// Adjoint with a multiply-add per component, pixel and entry and a butterfly
// of D sums per (warp, entry): for short lists, where a matrix block's upstream
// operands (split once per tile) and its barriers cost more than its products
// save (launch_feat_typed).
template <int MAXV, int TILE, int D>
__global__ void __launch_bounds__(TILE *TILE / scalar_bwd_ppt<TILE, D>())
    render_features_bwd_scalar_kernel(FeatArgs A, RasterViews<MAXV> rv) {
  grid_dependency_sync();
  constexpr int kPPT = scalar_bwd_ppt<TILE, D>();
  constexpr int kBatch = TILE * TILE / kPPT;
  __shared__ float4 s_geom[kBatch];
  __shared__ float2 s_ca[kBatch];
  __shared__ int32_t s_gi[kBatch];
  __shared__ float s_fhat[kBatch * (D + 1)];
  __shared__ float s_f[kBatch * (D + 1)];
  __shared__ float s_norm[kBatch];
  __shared__ float s_gate[D];
  __shared__ float s_ggate[D];
  const int32_t gt = blockIdx.x;
  const RasterView &V = rv.v[find_view<MAXV>(rv, gt)];
  const int32_t lt = gt - V.tile_base;
  const int32_t tx = lt % V.gw, ty = lt / V.gw;
  const int32_t px = tx * TILE + (threadIdx.x & (TILE - 1));
  const int32_t py0 = ty * TILE + (threadIdx.x / TILE) * kPPT;
  const uint2 range = tile_range(A.ranges, gt);
  if (range.x == range.y) return;  // nothing to add
  const float pxc = (float)px + 0.5f;
  const int lane = threadIdx.x & 31;
  if (threadIdx.x < D) {
    s_gate[threadIdx.x] = A.gate ? A.gate[threadIdx.x] : 1.0f;
    s_ggate[threadIdx.x] = 0.f;
  }
  const int64_t HW = (int64_t)V.width * V.height;
  const float *dF = A.dL_dF + V.pix_base * D;
  const float gyc = row_group_centre(py0);
  float T[kPPT], off[kPPT], G[kPPT][D];
  bool live = false;
#pragma unroll
  for (int k = 0; k < kPPT; ++k) {
    const bool in = px < V.width && py0 + k < V.height;
    T[k] = in ? 1.0f : -1.0f;
    off[k] = in ? row_offset(py0 + k) : stopped_offset();
    const int64_t p = (int64_t)(py0 + k) * V.width + px;
#pragma unroll
    for (int c = 0; c < D; ++c) G[k][c] = in ? dF[c * HW + p] : 0.f;
    live = live || in;
  }
  for (uint32_t base = range.x; base < range.y; base += kBatch) {
    if (__syncthreads_count(live) == 0) break;
    if (base + threadIdx.x < range.y)
      stage_feature<D, true>(A, s_gate, base + threadIdx.x, threadIdx.x, s_geom, s_ca, s_fhat, s_f, s_norm, s_gi);
    __syncthreads();
    const int nb = (int)min(range.y - base, (uint32_t)kBatch);
    for (int j = 0; j < nb; ++j) {
      if (!__any_sync(0xffffffffu, live)) break;  // the warp's pixels have all stopped
      const float4 geom = s_geom[j];
      const float2 ca = s_ca[j];
      const ColumnTerms ct = column_terms(geom, pxc, ca.y);
      const float w4 = group_w(ct, geom.y, ca.x, gyc);
      const bool clamp = entry_clamps(ca.y);
      float v[32];
#pragma unroll
      for (int c = 0; c < 32; ++c) v[c] = 0.f;
      bool contrib = false;
#pragma unroll
      for (int k = 0; k < kPPT; ++k) {
        const AlphaEval e = pixel_alpha(ct, w4, ca.x, off[k], clamp);
        if (e.alpha >= kAlphaMin) {  // false for stopped pixels (row offset +inf)
          const float w = __fmul_rn(e.alpha, T[k]);
          const float Tn = __fsub_rn(T[k], w);
          if (Tn < kTMin) {
            T[k] = -T[k];
            off[k] = stopped_offset();
          } else {
            contrib = true;
#pragma unroll
            for (int c = 0; c < D; ++c) v[c] = __fmaf_rn(G[k][c], w, v[c]);
            T[k] = Tn;
          }
        }
      }
      live = false;
#pragma unroll
      for (int k = 0; k < kPPT; ++k) live = live || T[k] > 0.0f;
      if (!__any_sync(0xffffffffu, contrib)) continue;
      const int32_t gi = s_gi[j];
      const float vc = warp_transpose_sum<D>(v, lane);  // lane c: component c of the warp's sum
      const float fh = lane < D ? s_fhat[j * (D + 1) + lane] : 0.f;
      const float dot = warp_sum(fh * vc);
      const float norm = s_norm[j];
      if (gi >= 0 && norm > 0.f && lane < D) {
        const float dg = (vc - fh * dot) / norm;
        atomicAdd(&A.g_feat[(int64_t)gi * D + lane], s_gate[lane] * dg);
        if (A.g_gate) atomicAdd(&s_ggate[lane], s_f[j * (D + 1) + lane] * dg);
      }
    }
  }
  __syncthreads();
  if (A.g_gate && threadIdx.x < D && s_ggate[threadIdx.x] != 0.f) atomicAdd(&A.g_gate[threadIdx.x], s_ggate[threadIdx.x]);
}

__device__ __forceinline__ float tf32_round(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

// x = hi + lo (+ about 2^-23 |x|), both with TF32 significands.
__device__ __forceinline__ void tf32_split(float x, uint32_t *hi, uint32_t *lo) {
  const float h = tf32_round(x);
  *hi = __float_as_uint(h);
  *lo = __float_as_uint(tf32_round(__fsub_rn(x, h)));
}

// The same for values up to the largest float: where hi would round to
// infinity it is cut off instead (x = hi + lo to about 2^-21 there).
__device__ __forceinline__ void tf32_split_any(float x, uint32_t *hi, uint32_t *lo) {
  float h = tf32_round(x);
  if (isinf(h)) h = __uint_as_float(__float_as_uint(x) & 0xffffe000u);
  *hi = __float_as_uint(h);
  *lo = __float_as_uint(tf32_round(__fsub_rn(x, h)));
}

// c += a b: a 16 x 8 (row = lane / 4, + 8; column = lane % 4, + 4), b 8 x 8
// (row = lane % 4, + 4; column = lane / 4), c 16 x 8 (row = lane / 4, + 8;
// columns 2 (lane % 4), + 1).
__device__ __forceinline__ void mma_tf32(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Per-entry part of a staged batch.
struct FeatEntries {
  float4 geom[kFeatBatch];
  float2 ca[kFeatBatch];     // (b2, log2 a)
  uint32_t bad[kFeatBatch];  // components of the normalised feature that are not finite
  int32_t gi[kFeatBatch];
  float norm[kFeatBatch];
};

// Stages records [base, base + nb) of a tile's list, four threads per entry,
// each with D / 4 components: `put(k, c, f, fhat)` receives component c of the
// raw feature and of the normalised gated one (0 where it is
// not finite; `bad` then has the component's bit).  Entries up to the next
// multiple of kChunk are staged as skipped by every pixel with zero features.
// Returns whether any component of the thread's entries was not finite.
template <int NT, int D, typename Put>
__device__ __forceinline__ bool stage_features(const FeatArgs &A, const float *s_gate, uint32_t base, int nb,
                                               FeatEntries &S, Put put) {
  constexpr int kPer = D / 4;
  const int sub = threadIdx.x & 3;
  const int padded = (nb + kChunk - 1) / kChunk * kChunk;
  bool any_bad = false;
  for (int k0 = 0; k0 < padded; k0 += NT / 4) {  // the trip count is the same for the whole warp
    const int k = k0 + (int)threadIdx.x / 4;
    float4 geom = make_float4(0.f, 0.f, 0.f, 0.f);
    float2 ca = make_float2(0.f, kLogAlphaNone);  // every pixel skips the entry
    int32_t gi = -1;
    if (k < nb) {
      const uint32_t s = A.inst_val[base + k];
      if (s < A.vis_cap) {
        gi = A.rec_meta[s].x;
        if (gi < 0 || (int64_t)gi >= A.n) {
          gi = -1;
        } else if (sub == 0) {
          geom = A.rec_geom[s];
          const float4 c = A.rec_color[s];
          ca = make_float2(c.x, c.y);
        }
      }
    }
    float f[kPer], g[kPer];
    float nn = 0.f;
    if (gi >= 0) {
      const float *row = A.feat + (int64_t)gi * D + sub * kPer;
      if (kPer >= 4) {
#pragma unroll
        for (int c4 = 0; c4 < kPer / 4; ++c4) {
          const float4 v = reinterpret_cast<const float4 *>(row)[c4];
          f[4 * c4 + 0] = v.x;
          f[4 * c4 + 1 < kPer ? 4 * c4 + 1 : 0] = v.y;
          f[4 * c4 + 2 < kPer ? 4 * c4 + 2 : 0] = v.z;
          f[4 * c4 + 3 < kPer ? 4 * c4 + 3 : 0] = v.w;
        }
      } else {
        const float2 v = *reinterpret_cast<const float2 *>(row);
        f[0] = v.x;
        f[1] = v.y;
      }
    } else {
#pragma unroll
      for (int c = 0; c < kPer; ++c) f[c] = 0.f;
    }
#pragma unroll
    for (int c = 0; c < kPer; ++c) {
      g[c] = f[c] * s_gate[sub * kPer + c];
      nn += g[c] * g[c];
    }
    nn += __shfl_xor_sync(0xffffffffu, nn, 1);
    nn += __shfl_xor_sync(0xffffffffu, nn, 2);
    const float norm = sqrtf(nn);
    const float inv = norm > 0.f ? 1.0f / norm : 0.f;
    uint32_t bad = 0u;
#pragma unroll
    for (int c = 0; c < kPer; ++c) {
      const float x = g[c] * inv;
      const bool ok = isfinite(x);
      if (!ok) bad |= 1u << (sub * kPer + c);
      if (k < padded) put(k, sub * kPer + c, f[c], ok ? x : 0.f);
    }
    bad |= __shfl_xor_sync(0xffffffffu, bad, 1);
    bad |= __shfl_xor_sync(0xffffffffu, bad, 2);
    any_bad = any_bad || bad != 0u;
    if (sub == 0 && k < padded) {
      S.geom[k] = geom;
      S.ca[k] = ca;
      S.bad[k] = bad;
      S.gi[k] = gi;
      S.norm[k] = norm;
    }
  }
  return any_bad;
}

// One pixel's front-to-back state.  A pixel that has stopped (or lies outside
// the image) has the row offset +inf, so that it takes no more alpha.
struct FeatPixel {
  float pxc, gyc, off, T;

  __device__ __forceinline__ FeatPixel(int32_t px, int32_t py, bool in) {
    pxc = (float)px + 0.5f;
    gyc = row_group_centre(py);
    off = in ? row_offset(py) : stopped_offset();
    T = 1.0f;
  }
  __device__ __forceinline__ bool live() const { return off < 1.0f; }
  // Weight of the entry at this pixel (0: skipped or stopped).  Every entry
  // takes the clamp: it changes no alpha of one that cannot reach it.
  __device__ __forceinline__ float weight(float4 geom, float2 ca) {
    const ColumnTerms ct = column_terms(geom, pxc, ca.y);
    const float alpha = pixel_alpha<true>(ct, group_w(ct, geom.y, ca.x, gyc), ca.x, off).alpha;
    float w = alpha >= kAlphaMin ? __fmul_rn(alpha, T) : 0.0f;  // 0 for NaN
    const float Tn = __fsub_rn(T, w);
    if (Tn < kTMin) {  // T itself is never below kTMin
      off = stopped_offset();
      w = 0.0f;
    } else {
      T = Tn;
    }
    return w;
  }
};

template <int MAXV, int TILE, int D>
__global__ void __launch_bounds__(feat_threads<TILE>()) render_features_kernel(FeatArgs A, RasterViews<MAXV> rv) {
  grid_dependency_sync();
  constexpr int NT = feat_threads<TILE>(), kStride = feat_stride<D>(), kN = D / 8;
  __shared__ FeatEntries S;
  __shared__ uint32_t s_hi[kFeatBatch * kStride], s_lo[kFeatBatch * kStride];
  __shared__ float s_w[NT / 32][kChunk * kWFwd];
  __shared__ float s_gate[D];
  const int32_t gt = blockIdx.x;
  const RasterView &V = rv.v[find_view<MAXV>(rv, gt)];
  const int32_t lt = gt - V.tile_base;
  const int32_t px = (lt % V.gw) * TILE + (threadIdx.x & (TILE - 1)), py = (lt / V.gw) * TILE + threadIdx.x / TILE;
  const bool in = px < V.width && py < V.height;
  const uint2 range = tile_range(A.ranges, gt);
  const int lane = threadIdx.x & 31, lr = lane >> 2, lc = lane & 3;
  float *w = s_w[threadIdx.x >> 5];
  if (threadIdx.x < D) s_gate[threadIdx.x] = A.gate ? A.gate[threadIdx.x] : 1.0f;
  FeatPixel P(px, py, in);
  uint32_t poison = 0u;  // components that took a feature value that is not finite
  float F[2][kN][4];     // pixels 16 m + lane / 4 (+ 8) of the warp, components 8 n + 2 (lane % 4) (+ 1)
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int n = 0; n < kN; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i) F[m][n][i] = 0.f;
  for (uint32_t base = range.x; base < range.y; base += kFeatBatch) {
    if (__syncthreads_count(P.live()) == 0) break;
    const int nb = (int)min(range.y - base, (uint32_t)kFeatBatch);
    const bool bad = stage_features<NT, D>(A, s_gate, base, nb, S, [&](int k, int c, float, float x) {
      tf32_split(x, &s_hi[k * kStride + c], &s_lo[k * kStride + c]);
    });
    const bool any_bad = __syncthreads_or(bad) != 0;
    for (int j0 = 0; j0 < nb; j0 += kChunk) {
      if (!__any_sync(0xffffffffu, P.live())) break;
      bool some = false;
      auto one = [&](int j) {
        const float x = P.weight(S.geom[j0 + j], S.ca[j0 + j]);
        if (any_bad && x > 0.f) poison |= S.bad[j0 + j];
        some = some || x > 0.f;
        w[j * kWFwd + lane] = x;
      };
      if (nb - j0 >= kChunk) {
#pragma unroll 4
        for (int j = 0; j < kChunk; ++j) one(j);
      } else {  // the rest of the last chunk has no weights
        for (int j = 0; j < nb - j0; ++j) one(j);
        for (int j = nb - j0; j < kChunk; ++j) w[j * kWFwd + lane] = 0.f;
      }
      __syncwarp();
      if (__any_sync(0xffffffffu, some)) {
        float acc[2][kN][4] = {};
        uint32_t ah[kChunk / 8][2][4];
        // the small products of both K steps first
#pragma unroll
        for (int ks = 0; ks < kChunk / 8; ++ks) {
          uint32_t al[2][4];
#pragma unroll
          for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int i = 0; i < 4; ++i)
              tf32_split(w[(8 * ks + lc + (i >> 1) * 4) * kWFwd + 16 * m + lr + (i & 1) * 8], &ah[ks][m][i], &al[m][i]);
          const int r0 = (j0 + 8 * ks + lc) * kStride + lr, r1 = r0 + 4 * kStride;
#pragma unroll
          for (int n = 0; n < kN; ++n) {
            const uint32_t bh0 = s_hi[r0 + 8 * n], bh1 = s_hi[r1 + 8 * n];
            const uint32_t bl0 = s_lo[r0 + 8 * n], bl1 = s_lo[r1 + 8 * n];
#pragma unroll
            for (int m = 0; m < 2; ++m) {
              mma_tf32(acc[m][n], al[m], bh0, bh1);
              mma_tf32(acc[m][n], ah[ks][m], bl0, bl1);
            }
          }
        }
#pragma unroll
        for (int ks = 0; ks < kChunk / 8; ++ks) {
          const int r0 = (j0 + 8 * ks + lc) * kStride + lr, r1 = r0 + 4 * kStride;
#pragma unroll
          for (int n = 0; n < kN; ++n) {
            const uint32_t bh0 = s_hi[r0 + 8 * n], bh1 = s_hi[r1 + 8 * n];
#pragma unroll
            for (int m = 0; m < 2; ++m) mma_tf32(acc[m][n], ah[ks][m], bh0, bh1);
          }
        }
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
          for (int n = 0; n < kN; ++n)
#pragma unroll
            for (int i = 0; i < 4; ++i) F[m][n][i] = __fadd_rn(F[m][n][i], acc[m][n][i]);
      }
      __syncwarp();  // the weights are overwritten by the next chunk
    }
  }
  // The map leaves through the weights' buffer, 8 components at a time: lane
  // = pixel, so a warp writes two rows of its tile per component.
  const int64_t HW = (int64_t)V.width * V.height, p = (int64_t)py * V.width + px;
  float *out = A.out + V.pix_base * D;
#pragma unroll
  for (int n = 0; n < kN; ++n) {
    __syncwarp();
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int i = 0; i < 4; ++i) w[(2 * lc + (i & 1)) * kWFwd + 16 * m + lr + (i >> 1) * 8] = F[m][n][i];
    __syncwarp();
    if (in) {
#pragma unroll
      for (int c = 0; c < 8; ++c)
        out[(8 * n + c) * HW + p] =
            (poison >> (8 * n + c)) & 1u ? __int_as_float(0x7fffffff) : w[c * kWFwd + lane];
    }
  }
}

// Resident blocks of 256 threads (or as many threads of 64) per SM: what the
// operands and accumulators allow without spills (64, 80 and 128 registers).
template <int TILE, int D>
constexpr int bwd_min_blocks() {
  return (D == 8 ? 4 : (D == 16 ? 3 : 2)) * (TILE == 16 ? 1 : 4);
}

template <int MAXV, int TILE, int D>
__global__ void __launch_bounds__(feat_threads<TILE>(), (bwd_min_blocks<TILE, D>()))
    render_features_bwd_kernel(FeatArgs A, RasterViews<MAXV> rv) {
  grid_dependency_sync();
  constexpr int NT = feat_threads<TILE>(), kWarps = NT / 32, kN = D / 8, kRow = D + 1;
  constexpr int kPart = feat_stride<D>();  // floats per entry row of a warp's sums
  constexpr int kBuf = kChunk * (kPart > kWBwd ? kPart : kWBwd);
  __shared__ FeatEntries S;
  __shared__ float s_fhat[kFeatBatch * kRow], s_f[kFeatBatch * kRow];
  __shared__ __align__(16) float s_buf[kWarps][kBuf];  // a warp's weights, then its sums
  __shared__ uint32_t s_has[2];  // warps that have sums (two words, for alternate chunks)
  // Entries of the chunk composited by a pixel whose gradient is not finite
  // (two words, for alternate chunks).
  __shared__ uint32_t s_poison[2];
  __shared__ float s_gate[D], s_ggate[D];
  const int32_t gt = blockIdx.x;
  const RasterView &V = rv.v[find_view<MAXV>(rv, gt)];
  const int32_t lt = gt - V.tile_base;
  const int32_t tx0 = (lt % V.gw) * TILE, ty0 = (lt / V.gw) * TILE;
  const int32_t px = tx0 + (threadIdx.x & (TILE - 1)), py = ty0 + threadIdx.x / TILE;
  const bool in = px < V.width && py < V.height;
  const uint2 range = tile_range(A.ranges, gt);
  if (range.x == range.y) return;  // nothing to add
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, lr = lane >> 2, lc = lane & 3;
  if (threadIdx.x < D) {
    s_gate[threadIdx.x] = A.gate ? A.gate[threadIdx.x] : 1.0f;
    s_ggate[threadIdx.x] = 0.f;
  }
  if (threadIdx.x < 2) s_poison[threadIdx.x] = s_has[threadIdx.x] = 0u;
  // Upstream gradients as operands: pixel 8 ks + lane % 4 (+ 4) of the warp,
  // component 8 n + lane / 4, from coalesced loads (lane = pixel) through the
  // warp's buffer.  A value that is not finite becomes 0 and marks its pixel.
  const int64_t HW = (int64_t)V.width * V.height, pixel = (int64_t)py * V.width + px;
  const float *dF = A.dL_dF + V.pix_base * D;
  uint32_t Gh[4][kN][2], Gl[4][kN][2];
  float up[D];  // all in flight before the first is used
#pragma unroll
  for (int c = 0; c < D; ++c) up[c] = in ? dF[c * HW + pixel] : 0.f;
  // The first batch is staged meanwhile.
  auto stage = [&](uint32_t base, int nb) {
    stage_features<NT, D>(A, s_gate, base, nb, S, [&](int k, int c, float f, float x) {
      s_f[k * kRow + c] = f;
      s_fhat[k * kRow + c] = x;
    });
  };
  __syncthreads();  // s_gate
  stage(range.x, (int)min(range.y - range.x, (uint32_t)kFeatBatch));
  bool bad = false;
#pragma unroll
  for (int n = 0; n < kN; ++n) {
    __syncwarp();
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const bool ok = isfinite(up[8 * n + c]);
      bad = bad || !ok;
      s_buf[warp][c * kWBwd + lane] = ok ? up[8 * n + c] : 0.f;
    }
    __syncwarp();
#pragma unroll
    for (int ks = 0; ks < 4; ++ks)
#pragma unroll
      for (int h = 0; h < 2; ++h)
        tf32_split_any(s_buf[warp][lr * kWBwd + 8 * ks + lc + 4 * h], &Gh[ks][n][h], &Gl[ks][n][h]);
  }
  const uint32_t bad_pixels = __ballot_sync(0xffffffffu, bad);  // of the warp
  __syncwarp();
  FeatPixel P(px, py, in);
  float ggate = 0.f;  // of component lane % D
  int buf = 0;
  for (uint32_t base = range.x; base < range.y; base += kFeatBatch) {
    const int nb = (int)min(range.y - base, (uint32_t)kFeatBatch);
    if (base != range.x) {
      if (__syncthreads_count(P.live()) == 0) break;
      stage(base, nb);
    }
    __syncthreads();
    for (int j0 = 0; j0 < nb; j0 += kChunk, buf ^= 1) {
      float *w = s_buf[warp];
      bool some = false;
      if (__any_sync(0xffffffffu, P.live())) {
        uint32_t hit = 0u;
        const int m = min(nb - j0, kChunk);  // the rest of the last chunk has no weights
        for (int j4 = 0; j4 < kChunk; j4 += 4) {
          if (j4 < m) {
#pragma unroll
            for (int j = j4; j < j4 + 4; ++j) {
              const float x = P.weight(S.geom[j0 + j], S.ca[j0 + j]);
              if (x > 0.f) hit |= 1u << j;
              w[j * kWBwd + lane] = x;
            }
          } else {
#pragma unroll
            for (int j = j4; j < j4 + 4; ++j) w[j * kWBwd + lane] = 0.f;
          }
        }
        if (bad_pixels) {
          const uint32_t e = __reduce_or_sync(0xffffffffu, bad ? hit : 0u);
          if (lane == 0 && e) atomicOr(&s_poison[buf], e);
        }
        some = __any_sync(0xffffffffu, hit != 0u);
      }
      __syncwarp();
      if (some) {
        float acc[kN][4] = {};
        uint32_t ah[4][4];
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
          uint32_t al[4];
#pragma unroll
          for (int i = 0; i < 4; ++i)
            tf32_split(w[(lr + (i & 1) * 8) * kWBwd + 8 * ks + lc + (i >> 1) * 4], &ah[ks][i], &al[i]);
#pragma unroll
          for (int n = 0; n < kN; ++n) {
            mma_tf32(acc[n], al, Gh[ks][n][0], Gh[ks][n][1]);
            mma_tf32(acc[n], ah[ks], Gl[ks][n][0], Gl[ks][n][1]);
          }
        }
#pragma unroll
        for (int ks = 0; ks < 4; ++ks)
#pragma unroll
          for (int n = 0; n < kN; ++n) mma_tf32(acc[n], ah[ks], Gh[ks][n][0], Gh[ks][n][1]);
        __syncwarp();  // the weights have been read
#pragma unroll
        for (int n = 0; n < kN; ++n)
#pragma unroll
          for (int h = 0; h < 2; ++h)
            *reinterpret_cast<float2 *>(&w[(lr + 8 * h) * kPart + 8 * n + 2 * lc]) =
                make_float2(acc[n][2 * h], acc[n][2 * h + 1]);
      }
      if (lane == 0 && some) atomicOr(&s_has[buf], 1u << warp);
      __syncthreads();
      // Entry e of the chunk on D lanes, one component each.
      constexpr int kPerWarp = 32 / D, kPass = kWarps * kPerWarp;
      const int c = lane % D;
      const uint32_t has = s_has[buf];
#pragma unroll
      for (int e0 = 0; e0 < kChunk; e0 += kPass) {
        const int e = e0 + warp * kPerWarp + lane / D, j = j0 + e;
        float v = 0.f;
        if (e < kChunk) {
#pragma unroll
          for (int k = 0; k < kWarps; ++k)
            if ((has >> k) & 1u) v += s_buf[k][e * kPart + c];
          if ((s_poison[buf] >> e) & 1u) v = __int_as_float(0x7fffffff);
        }
        if (!__any_sync(0xffffffffu, v != 0.f)) continue;  // (NaN != 0)
        const bool on = e < kChunk && j < nb;
        float fh = on ? s_fhat[j * kRow + c] : 0.f;
        if (on && (S.bad[j] >> c) & 1u) fh = __int_as_float(0x7fffffff);
        float dot = fh * v;
#pragma unroll
        for (int o = D / 2; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
        const int32_t gi = on ? S.gi[j] : -1;
        const float norm = on ? S.norm[j] : 0.f;
        if (gi >= 0 && norm > 0.f) {
          const float dg = (v - fh * dot) / norm;
          atomicAdd(&A.g_feat[(int64_t)gi * D + c], s_gate[c] * dg);
          ggate += s_f[j * kRow + c] * dg;
        }
      }
      if (threadIdx.x == 0) s_poison[buf ^ 1] = s_has[buf ^ 1] = 0u;  // read by the chunk before, written by the next
      __syncthreads();  // the sums have been read
    }
  }
  __syncthreads();
  if (A.g_gate) {
    if (ggate != 0.f) atomicAdd(&s_ggate[lane % D], ggate);
    __syncthreads();
    if (threadIdx.x < D && s_ggate[threadIdx.x] != 0.f) atomicAdd(&A.g_gate[threadIdx.x], s_ggate[threadIdx.x]);
  }
}

template <int MAXV, int TILE, int D>
cudaError_t launch_feat_tile(const FeatArgs &A, const RasterViews<MAXV> &rv, unsigned grid, bool backward,
                             bool short_lists, cudaStream_t st) {
  constexpr unsigned NT = feat_threads<TILE>();
  if (backward) {
    if (short_lists)
      return launch_pdl(render_features_bwd_scalar_kernel<MAXV, TILE, D>, grid,
                        (unsigned)(TILE * TILE / scalar_bwd_ppt<TILE, D>()), st, A, rv);
    return launch_pdl(render_features_bwd_kernel<MAXV, TILE, D>, grid, NT, st, A, rv);
  }
  if constexpr (D > 16) {
    if (!short_lists) return launch_pdl(render_features_kernel<MAXV, TILE, D>, grid, NT, st, A, rv);
  }
  return launch_pdl(render_features_scalar_kernel<MAXV, TILE, D>, grid, (unsigned)(TILE * TILE / kScalarPPT), st, A, rv);
}

// Calls whose lists are surely short take the scalar kernels: the instance
// capacity, an upper bound of the instances, is below this many a tile (twice
// the lists' length or more, as capacities have headroom).  Scalar / matrix
// (us) at 1352x1014, by instances a tile: adjoint D = 8 5.2 33 / 48, 10.6 50 /
// 56, 15 64 / 66, 20.5 81 / 76, 308 670 / 465; D = 32 78 / 113, 115 / 126, 146 /
// 142, 181 / 158, 1490 / 851; map D = 32 5.2 56 / 95, 10.6 74 / 105, 20.5 111 /
// 132, 31 154 / 160, 41 197 / 187, 308 902 / 726.  With fewer tiles than some
// 4000 one round of blocks holds most of a call and the longest list decides:
// the adjoint of 1200 tiles with 10 entries a tile takes 25 / 19 at D = 8.
constexpr int64_t kShortAdjointCap = 40, kShortAdjointMinTiles = 4096, kShortMapCap = 72;

template <int MAXV, int D>
cudaError_t launch_feat_typed(const Layout &L, const FeatArgs &A, const fgs4d_view *views, int32_t nviews,
                              bool backward, cudaStream_t st) {
  RasterViews<MAXV> rv;
  if (!make_raster_views<MAXV>(L, views, nviews, &rv)) return cudaErrorInvalidValue;
  if (L.total_tiles == 0) return cudaSuccess;
  const unsigned grid = (unsigned)L.total_tiles;
  const bool short_lists =
      backward ? L.total_tiles >= kShortAdjointMinTiles && L.inst_cap < kShortAdjointCap * L.total_tiles
               : L.inst_cap < kShortMapCap * L.total_tiles;
  if (L.tile == 8) return launch_feat_tile<MAXV, 8, D>(A, rv, grid, backward, short_lists, st);
  return launch_feat_tile<MAXV, 16, D>(A, rv, grid, backward, short_lists, st);
}

template <int D>
cudaError_t launch_feat_d(const Layout &L, const FeatArgs &A, const fgs4d_view *views, int32_t nviews,
                          bool backward, cudaStream_t st) {
  if (nviews == 1) return launch_feat_typed<1, D>(L, A, views, nviews, backward, st);
  return launch_feat_typed<FGS4D_MAX_VIEWS, D>(L, A, views, nviews, backward, st);
}

}  // namespace

bool feature_dim_supported(int32_t D) { return D == 8 || D == 16 || D == 32; }

cudaError_t launch_render_features(const Layout &L, const fgs4d_view *views, int32_t nviews, unsigned char *ws,
                                   int64_t n, const float *feat, int32_t D, const float *gate, float *out,
                                   const float *dL_dF, float *g_feat, float *g_gate, cudaStream_t st) {
  FeatArgs A;
  A.ranges = reinterpret_cast<const uint2 *>(ws + L.ranges);
  A.inst_val = reinterpret_cast<const uint32_t *>(ws + L.inst_val[L.tile_passes & 1]);
  A.rec_geom = reinterpret_cast<const float4 *>(ws + L.rec_geom);
  A.rec_color = reinterpret_cast<const float4 *>(ws + L.rec_color);
  A.rec_meta = reinterpret_cast<const int4 *>(ws + L.rec_meta);
  A.vis_cap = (uint32_t)L.vis_cap;
  A.n = n;
  A.feat = feat;
  A.gate = gate;
  A.out = out;
  A.dL_dF = dL_dF;
  A.g_feat = g_feat;
  A.g_gate = g_gate;
  const bool bwd = dL_dF != nullptr;
  switch (D) {
    case 8: return launch_feat_d<8>(L, A, views, nviews, bwd, st);
    case 16: return launch_feat_d<16>(L, A, views, nviews, bwd, st);
    default: return launch_feat_d<32>(L, A, views, nviews, bwd, st);
  }
}

}  // namespace fgs4d
