// Two-level tile binning for large instance lists (included by sort.cu).
//
// A cell is a square of kCellEdge x kCellEdge tiles.  Instead of emitting
// every (tile, Gaussian) instance and radix-sorting the instances by tile id,
// the depth-sorted slots emit (cell, slot) pairs with a 64-bit mask of the
// cell's tiles their 1/255 ellipse meets, the pairs (one for up to 64
// instances) are sorted by cell id, and each cell's list is expanded into its
// tiles' lists at positions known from per-segment bit counts:
//
//   pair scan     candidate (slot, cell) pairs of the depth-sorted slots
//   cell_emit     masks; pairs with an empty mask dropped; depth order kept
//   radix pass    stable, on the cell id (8 bits at up to 256 cells)
//   cell_count    per segment of kCellSeg sorted pairs: instances per tile
//   cell_prefix   per cell: prefix of its segments' counts and tile totals;
//                 the last block scans the totals into the tile ranges
//   cell_write    per segment: (tile id, slot) of every set bit, in list order
//
// The result -- instances ordered by (tile, depth, slot), and their ranges --
// is that of the instance sort, instance for instance.  Reads and writes per instance drop from the
// sort's 16 bytes a pass to the 8 bytes of the final list; the passes over
// pairs move 28 bytes a pair.

constexpr int kCellShift = 3;
constexpr int kCellEdge = 1 << kCellShift;
constexpr int kCellTiles = kCellEdge * kCellEdge;  // bits of a mask
static_assert(kCellTiles == 64, "one 64-bit mask per pair");

struct CellArgs {
  EmitArgs e;
  int32_t total_cells, cell_passes;
  uint32_t *key;         // cell id per pair, in depth order
  uint32_t *slot;        // slot per pair, in depth order
  uint2 *mask;           // tile mask per pair, in depth order (low word: tile rows 0-3)
  const uint32_t *skey;  // sorted cell ids
  const uint32_t *sidx;  // sorted pairs (indices into slot and mask)
  uint2 *cell_ranges;    // [start, end) of each cell's sorted pairs (entry c << kCellRangeShift)
  uint32_t *rows;        // instances per tile of each (segment, cell) run; after cell_prefix their exclusive prefix
};

// Cells a tile rect [x0, x1) x [y0, y1) touches, by row of cells.
__device__ __forceinline__ int cell_span(int lo, int hi) { return ((hi - 1) >> kCellShift) - (lo >> kCellShift) + 1; }

// sqrt within an ulp or two (the intervals below have room for that).
__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// The tiles [tx0, tx1) x [ty0, ty1) of one cell that ellipse_meets_box accepts
// for a record, as bits (ty & 7) * 8 + (tx & 7): the instance sort's test, bit
// for bit, mostly without making it.  Per row of tiles the ellipse's x extent
// over the row's band of pixel centres is an interval: with q = (a1 x)^2 +
// (b1 x + b2 y)^2 and n = a1^2 + b1^2, the rightmost point of q <= t lies at
// y = kx r / a1 (r^2 = t, kx = -b1 / b2); clamped to the band as y = Y its row
// ends at x = ky Y + sqrt((t - (a1 b2 Y)^2 / n) / n) (ky = -b1 b2 / n), and the
// left end is the mirror image.  With t = tau + margin and the interval
// widened by `slack` no tile outside it can pass the test; with t = tau -
// margin and the interval narrowed every tile that it meets does; the few
// between (about 0.1 % of a cell's tiles) are tested.  margin covers the FP32
// error of q, whose terms are up to |b1| / a1 times larger than tau, in the test
// and here; slack that of the coordinates and of the interval's terms.  Records
// outside the bounds for which that holds (or not finite) have all tiles
// tested.  A row costs about 45 instructions instead of up to 8 tests of 40.
__device__ __forceinline__ uint64_t cell_mask(float u, float v, float a1, float b1, float b2, float kx, float ky,
                                              float tau, const RasterView &V, int tx0, int tx1, int ty0, int ty1) {
  const float T = (float)V.tile, iT = 1.0f / T;
  const float xmax = (float)V.width - 0.5f - u, ymax = (float)V.height - 0.5f - v;  // last pixel centre
  const uint32_t cols = (((1u << (tx1 - tx0)) - 1u) << (tx0 & (kCellEdge - 1)));
  const float aspect = __fdividef(fabsf(b1), a1), ab = a1 * b2;
  const float margin = 2e-5f + 2e-6f * tau * (1.0f + aspect);
  const float t = tau + margin;
  const float n = __fmaf_rn(a1, a1, b1 * b1);
  const bool ok = tau >= 0.0f && t < 1e9f && a1 > 1e-12f && b2 > 1e-12f && b2 < 1e9f && ab > 1e-18f &&
                  aspect < 1e6f && n < 1e18f && fabsf(u) < 1e9f && fabsf(v) < 1e9f;
  uint64_t sure = 0ull, maybe = 0ull;
  if (ok) {
    // all corners inside: the whole (convex) box is
    const float lx = (float)tx0 * T + 0.5f - u, hx = fminf((float)tx1 * T - 0.5f - u, xmax);
    const float by0 = (float)ty0 * T + 0.5f - v, by1 = fminf((float)ty1 * T - 0.5f - v, ymax);
    const float tin = tau - margin;
    if (sum_sq(a1, b1, b2, lx, by0) <= tin && sum_sq(a1, b1, b2, hx, by0) <= tin &&
        sum_sq(a1, b1, b2, lx, by1) <= tin && sum_sq(a1, b1, b2, hx, by1) <= tin) {
      for (int ty = ty0; ty < ty1; ++ty) sure |= (uint64_t)cols << ((ty & (kCellEdge - 1)) * kCellEdge);
      return sure;
    }
    const float in = __fdividef(1.0f, n), r = sqrt_approx(t);
    const float ym = kx * __fdividef(r, a1);  // y of the rightmost point
    const float slack = 2e-7f * (fabsf(u) + fabsf(v) + (float)V.width + (float)V.height);
    const float ry = __fdividef(r * sqrt_approx(n), ab) * 1.00001f + slack;  // vertical half-extent
    const float c2 = ab * ab * in;
    // tile columns that [l, h] meets
    auto columns = [&](float l, float h) -> uint32_t {
      const float flo = ceilf((l + u - (T - 0.5f)) * iT), fhi = floorf((h + u - 0.5f) * iT);
      const int lo = (int)fmaxf(flo, (float)tx0), hi = (int)fminf(fhi, (float)(tx1 - 1));
      if (l > xmax || lo > hi || lo >= tx1 || hi < tx0) return 0u;
      return (((2u << (hi - lo)) - 1u) << (lo & (kCellEdge - 1))) & cols;
    };
    for (int ty = ty0; ty < ty1; ++ty) {
      const float ly = (float)ty * T + 0.5f - v, hy = fminf((float)ty * T + (T - 0.5f) - v, ymax);
      if (ly > ry || hy < -ry) continue;
      // right end: the rightmost point's y clamped to the band; left end: its mirror's
      const float yr = fminf(fmaxf(ym, ly), hy), yl = fminf(fmaxf(-ym, ly), hy);
      const float kr = ky * yr, kl = ky * yl;
      const float dr = __fmaf_rn(-c2 * yr, yr, t), dl = __fmaf_rn(-c2 * yl, yl, t);
      const float xr = kr + sqrt_approx(fmaxf(dr, 0.0f) * in), xl = kl - sqrt_approx(fmaxf(dl, 0.0f) * in);
      const float er = slack + 4e-6f * (fabsf(kr) + fabsf(xr)), el = slack + 4e-6f * (fabsf(kl) + fabsf(xl));
      const uint32_t outer = columns(xl - el, xr + er);
      const float ir = dr - 2.0f * margin, il = dl - 2.0f * margin;
      const float xri = kr + sqrt_approx(fmaxf(ir, 0.0f) * in) - er, xli = kl - sqrt_approx(fmaxf(il, 0.0f) * in) + el;
      const uint32_t inner = ir >= 0.0f && il >= 0.0f && xli <= xri ? columns(xli, xri) & outer : 0u;
      const int row = (ty & (kCellEdge - 1)) * kCellEdge;
      sure |= (uint64_t)inner << row;
      maybe |= (uint64_t)(outer & ~inner) << row;
    }
  } else {
    for (int ty = ty0; ty < ty1; ++ty) maybe |= (uint64_t)cols << ((ty & (kCellEdge - 1)) * kCellEdge);
  }
  while (maybe) {
    const int bit = __ffsll((long long)maybe) - 1;
    maybe &= maybe - 1ull;
    const int tx = (tx0 & ~(kCellEdge - 1)) + (bit & (kCellEdge - 1));
    const int ty = (ty0 & ~(kCellEdge - 1)) + (bit >> kCellShift);
    if (tile_meets(u, v, a1, b1, b2, kx, ky, tau, V, tx, ty)) sure |= 1ull << bit;
  }
  return sure;
}

// The tiles of all slots' rects: the instances that a call whose pairs
// outnumber the pair capacity may need.  Added up here, only then, so that the
// pair scan carries one sum.
__device__ __forceinline__ void add_rect_tiles(const EmitArgs &A, int64_t nvis) {
  uint64_t sum = 0ull;
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < nvis; j += (int64_t)gridDim.x * blockDim.x) {
    const int4 r = A.emit_rec[3 * j + 2];
    const int w = (r.w & 0xffff) - (r.z & 0xffff), h = (int)((uint32_t)r.w >> 16) - (int)((uint32_t)r.z >> 16);
    sum += (uint64_t)max(w, 0) * (uint64_t)max(h, 0);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if ((threadIdx.x & 31) == 0 && sum)
    atomicAdd(reinterpret_cast<unsigned long long *>(&A.counters[kCtrRectTiles64]), (unsigned long long)sum);
}

// Pair emission, one candidate (slot, cell) pair per thread and kCellChunk
// pairs per chunk: the pair's slot is found by a binary search of the pair
// prefix and its mask computed.  When the candidates fit the pair buffers (the
// instance capacity, as every kept pair holds an instance) each is written at
// its own index, empty masks included: no chunk waits for another.  Otherwise
// the chunks are taken by ticket and the pairs with a set bit compacted in
// depth order (block scan and decoupled look-back).  Clears the cell sort's
// look-back rows, sets the empty cell ranges, takes the cell-id digit
// histograms and counts the instances.
template <int MAXV>
__global__ void __launch_bounds__(kCellChunk) cell_emit_kernel(CellArgs C, RasterViews<MAXV> rv) {
  grid_dependency_sync();
  constexpr int kPrefCache = 2 * kCellChunk;
  __shared__ uint32_t s_pref[kPrefCache + 1];
  __shared__ uint32_t s_scan[kCellChunk / 32 + 1];
  __shared__ uint32_t s_hist[kMaxPasses][kRadixBins];
  __shared__ uint32_t s_ticket;
  __shared__ uint64_t s_prefix;
  const EmitArgs &A = C.e;
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < C.total_cells;
       r += (int64_t)gridDim.x * blockDim.x)
    C.cell_ranges[r << kCellRangeShift] = make_uint2(0xffffffffu, 0u);
  const int64_t nvis = min64((int64_t)A.counters[kCtrVisible], A.vis_cap);
  const uint32_t npairs = A.counters[kCtrPairs];
  const uint32_t nchunks = (uint32_t)min64(((int64_t)npairs + kCellChunk - 1) / kCellChunk, A.chunk_cap);
  if (nchunks == 0u) {
    if (blockIdx.x == 0 && threadIdx.x == 0) A.counters[kCtrCellPairs] = 0u;
    return;
  }
  if (A.counters[kCtrPairOverflow]) add_rect_tiles(A, nvis);
  for (int p = 0; p < C.cell_passes; ++p) s_hist[p][threadIdx.x] = 0u;
  const bool direct = (int64_t)npairs <= A.inst_cap;
  if (direct && blockIdx.x == 0 && threadIdx.x == 0) A.counters[kCtrCellPairs] = npairs;
  uint64_t kept = 0u;  // instances of this thread's pairs
  for (uint32_t c = blockIdx.x;; c += gridDim.x) {
    if (!direct) {
      if (threadIdx.x == 0) s_ticket = atomicAdd(&A.counters[kCtrTicketChunk], 1u);
      __syncthreads();
      c = s_ticket;
    }
    if (c >= nchunks) break;
    // radix tile rt of the pair sort is covered by the chunks' pairs (kept pairs never outnumber them)
    if (c % (kInstSortTile / kCellChunk) == 0u) {
      const int64_t rt = c / (kInstSortTile / kCellChunk);
      if (rt < A.tile_blocks)
        for (int p = 0; p < C.cell_passes; ++p)
          A.tile_state[((size_t)p * A.tile_blocks + rt) * kRadixBins + threadIdx.x] = 0u;
    }
    const uint32_t f = c * kCellChunk + threadIdx.x;
    // positions of the chunk's pairs (clamped: after a recorded timeout the marks may be stale)
    const int64_t j0 = min64(A.chunk_first[c], nvis - 1);
    const int64_t j1 = c + 1u == nchunks ? nvis - 1 : min64(A.chunk_first[c + 1], nvis - 1);
    const int64_t ns = max64(j1 - j0 + 1, 1);
    const bool cached = ns <= kPrefCache;
    if (cached)
      for (int k = threadIdx.x; k < (int)ns; k += kCellChunk) s_pref[k] = A.pair_prefix[j0 + k];
    __syncthreads();
    uint64_t mask = 0ull;
    uint32_t key = 0u, slot = 0u;
    if (f < npairs) {
      int64_t lo = 0, hi = ns - 1;
      while (lo < hi) {  // last position whose pair prefix is <= f
        const int64_t mid = (lo + hi + 1) >> 1;
        if ((cached ? s_pref[mid] : A.pair_prefix[j0 + mid]) <= f) lo = mid;
        else hi = mid - 1;
      }
      const uint32_t local = f - (cached ? s_pref[lo] : A.pair_prefix[j0 + lo]);
      const int4 *er = A.emit_rec + 3 * (j0 + lo);
      const int4 r0 = er[0], r1 = er[1], r2 = er[2];
      const RasterView &V = rv.v[MAXV == 1 ? 0 : r2.y];
      const int x0 = r2.z & 0xffff, y0 = (uint32_t)r2.z >> 16, x1 = r2.w & 0xffff, y1 = (uint32_t)r2.w >> 16;
      const uint32_t ncx = (uint32_t)max(cell_span(x0, x1), 1);
      const uint32_t qy = local / ncx;
      const int cx = (x0 >> kCellShift) + (int)(local - qy * ncx), cy = (y0 >> kCellShift) + (int)qy;
      slot = (uint32_t)r2.x;
      key = (uint32_t)(V.cell_base + cy * V.cgw + cx);
      const int tx0 = max(x0, cx << kCellShift), tx1 = min(x1, (cx + 1) << kCellShift);
      const int ty0 = max(y0, cy << kCellShift), ty1 = min(y1, (cy + 1) << kCellShift);
      if (tx0 < tx1 && ty0 < ty1)
        mask = cell_mask(__int_as_float(r0.x), __int_as_float(r0.y), __int_as_float(r0.z), __int_as_float(r0.w),
                         __int_as_float(r1.x), __int_as_float(r1.y), __int_as_float(r1.z), __int_as_float(r1.w), V,
                         tx0, tx1, ty0, ty1);
    }
    const bool keep = direct ? f < npairs : mask != 0ull;
    uint64_t pos = f;
    if (!direct) {
      uint32_t total;
      const uint32_t local_pos = block_exclusive_scan(keep ? 1u : 0u, s_scan, &total);
      if (threadIdx.x < 32) {
        const uint64_t prefix = lookback_u64_warp(A.lb_chunk, (int32_t)c, total, &A.counters[kCtrStatus]);
        if (threadIdx.x == 0) {
          s_prefix = prefix;
          if (c == nchunks - 1u) A.counters[kCtrCellPairs] = (uint32_t)umin64(prefix + total, (uint64_t)A.inst_cap);
        }
      }
      __syncthreads();
      pos = s_prefix + local_pos;
    }
    if (keep) {
      kept += (uint32_t)__popcll(mask);
      for (int p = 0; p < C.cell_passes; ++p) atomicAdd(&s_hist[p][(key >> (kRadixBits * p)) & (kRadixBins - 1)], 1u);
      if (pos < (uint64_t)A.inst_cap) {
        C.key[pos] = key;
        C.slot[pos] = slot;
        C.mask[pos] = make_uint2((uint32_t)mask, (uint32_t)(mask >> 32));
      }
    }
    __syncthreads();  // s_pref, s_ticket and s_prefix are reused by the next chunk
  }
  __syncthreads();
  for (int p = 0; p < C.cell_passes; ++p) {
    const uint32_t h = s_hist[p][threadIdx.x];
    if (h) atomicAdd(&A.hist_tile[p * kRadixBins + threadIdx.x], h);
  }
  uint64_t k64 = kept;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) k64 += __shfl_xor_sync(0xffffffffu, k64, o);
  if ((threadIdx.x & 31) == 0 && k64)
    atomicAdd(reinterpret_cast<unsigned long long *>(&A.counters[kCtrInstances64]), (unsigned long long)k64);
}

// A segment is kCellSeg consecutive sorted pairs; a run is the part of a
// segment that belongs to one cell.  The runs of segment s and cell c use row
// s + c of the counts: along the sorted list every new run advances s or c,
// so the rows are distinct.
//
// Transposes a 32 x 32 bit matrix held one row per lane: bit j of lane i
// becomes bit i of lane j.
__device__ __forceinline__ uint32_t warp_transpose_bits(uint32_t x, int lane) {
  constexpr uint32_t kLow[5] = {0x0000ffffu, 0x00ff00ffu, 0x0f0f0f0fu, 0x33333333u, 0x55555555u};
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    const int s = 16 >> i;
    const uint32_t m = kLow[i], y = __shfl_xor_sync(0xffffffffu, x, s);
    x = (lane & s) ? (x & ~m) | ((y >> s) & m) : (x & m) | ((y << s) & ~m);
  }
  return x;
}

// End of the run starting at position a of a segment of n sorted keys.
__device__ __forceinline__ int run_end(const uint32_t *key, int a, int n) {
  const uint32_t c = key[a];
  int lo = a + 1, hi = n;  // first position past the run
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (key[mid] == c) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// Walk over the segments of a persistent block, one pair per thread: the
// sorted key and index of the next segment are loaded while the current one
// is processed.
struct SegmentWalk {
  uint32_t key, idx;
  int64_t npairs;

  __device__ __forceinline__ void load(const CellArgs &C, int64_t s) {
    const int64_t i = s * kCellSeg + threadIdx.x;
    key = idx = 0xffffffffu;
    if (i < npairs) {
      idx = C.sidx[i];
      key = C.skey[i];
    }
  }

  // Stages the keys (and slots, if wanted) of the loaded segment s and returns
  // its pair count; *mask is the thread's pair's; loads segment `next`.
  __device__ __forceinline__ int stage(const CellArgs &C, int64_t s, int64_t next, uint32_t *s_key, uint32_t *s_slot,
                                       uint2 *mask) {
    const int n = (int)min64(kCellSeg, npairs - s * kCellSeg);
    *mask = make_uint2(0u, 0u);
    if ((int)threadIdx.x < n) {
      const bool ok = (int64_t)idx < npairs && (int64_t)key < C.total_cells;  // false only after a recorded timeout
      if (!ok) atomicOr(&C.e.counters[kCtrStatus], kStatusInternal);
      s_key[threadIdx.x] = ok ? key : 0u;
      if (ok) *mask = C.mask[idx];
      if (s_slot) s_slot[threadIdx.x] = ok ? C.slot[idx] : 0u;
    }
    load(C, next);
    __syncthreads();
    return n;
  }
};

// The masks of a run [a, b) as words of 32 pairs per tile: lane t of warp w
// gets the pairs 32 w .. 32 w + 31 of the segment that hold tile t (w0) and
// tile 32 + t (w1).  A transpose of the 32 x 64 bits costs about 50
// instructions where a ballot per tile and its unpacking took about 300.
__device__ __forceinline__ void run_words(uint2 mask, int a, int b, int lane, uint32_t *w0, uint32_t *w1) {
  const bool in = (int)threadIdx.x >= a && (int)threadIdx.x < b;
  *w0 = *w1 = 0u;
  if (!__any_sync(0xffffffffu, in)) return;
  *w0 = warp_transpose_bits(in ? mask.x : 0u, lane);
  *w1 = warp_transpose_bits(in ? mask.y : 0u, lane);
}

// Instances per tile of every run.
__global__ void __launch_bounds__(kCellBlock) cell_count_kernel(CellArgs C) {
  grid_dependency_sync();
  constexpr int kWarps = kCellBlock / 32;
  __shared__ uint32_t s_key[kCellSeg];
  __shared__ uint8_t s_cnt[kWarps][kCellTiles];
  const int64_t npairs = min64((int64_t)C.e.counters[kCtrCellPairs], C.e.inst_cap);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  SegmentWalk W;
  W.npairs = npairs;
  W.load(C, blockIdx.x);
  for (int64_t s = blockIdx.x; s * kCellSeg < npairs; s += gridDim.x) {
    uint2 mask;
    const int n = W.stage(C, s, s + gridDim.x, s_key, nullptr, &mask);
    for (int a = 0; a < n;) {
      const int b = run_end(s_key, a, n);
      uint32_t w0, w1;
      run_words(mask, a, b, lane, &w0, &w1);
      s_cnt[warp][lane] = (uint8_t)__popc(w0);
      s_cnt[warp][32 + lane] = (uint8_t)__popc(w1);
      __syncthreads();
      if (threadIdx.x < kCellTiles) {
        uint32_t cnt = 0u;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) cnt += s_cnt[w][threadIdx.x];
        C.rows[((size_t)s + s_key[a]) * kCellTiles + threadIdx.x] = cnt;
      }
      a = b;
      __syncthreads();  // s_cnt, s_key
    }
  }
}

// Cell -> its view (last view whose first cell is <= c).
template <int MAXV>
__device__ __forceinline__ int find_cell_view(const RasterViews<MAXV> &rv, int32_t c) {
  if (MAXV == 1) return 0;
  int lo = 0, hi = rv.nviews - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (rv.v[mid].cell_base <= c) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Per cell: exclusive prefix of its runs' counts and each tile's total (into
// ranges[tile].y); the block that finishes last scans the totals over the
// global tile order into [start, end) and sets the instance total.  One block
// per cell: kCellPrefixThreads / 64 groups of 64 tile threads share its rows.
template <int MAXV>
__global__ void __launch_bounds__(kCellPrefixThreads) cell_prefix_kernel(CellArgs C, RasterViews<MAXV> rv) {
  grid_dependency_sync();
  constexpr int kGroups = kCellPrefixThreads / kCellTiles, kWarps = kCellPrefixThreads / 32;
  __shared__ uint32_t s_sum[kGroups][kCellTiles];
  __shared__ uint32_t s_scan[kWarps + 1];
  __shared__ bool s_last;
  const EmitArgs &A = C.e;
  const int64_t npairs = min64((int64_t)A.counters[kCtrCellPairs], A.inst_cap);
  const int t = threadIdx.x & (kCellTiles - 1), g = threadIdx.x / kCellTiles;
  for (int32_t c = blockIdx.x; c < C.total_cells; c += gridDim.x) {
    const uint2 r = C.cell_ranges[(int64_t)c << kCellRangeShift];
    int64_t s0 = 0, s1 = 0;  // rows [s0, s1) of the cell
    if (r.x < r.y && (int64_t)r.y <= npairs) {
      s0 = (int64_t)(r.x / kCellSeg) + c;
      s1 = (int64_t)((r.y - 1u) / kCellSeg) + c + 1;
    }
    const int64_t per = (s1 - s0 + kGroups - 1) / kGroups;
    const int64_t ga = min64(s0 + g * per, s1), gb = min64(ga + per, s1);
    uint32_t sum = 0u;
    for (int64_t k = ga; k < gb; ++k) sum += C.rows[k * kCellTiles + t];
    s_sum[g][t] = sum;
    __syncthreads();
    uint32_t run = 0u, total = 0u;
#pragma unroll
    for (int k = 0; k < kGroups; ++k) {
      if (k < g) run += s_sum[k][t];
      total += s_sum[k][t];
    }
    for (int64_t k = ga; k < gb; ++k) {
      const uint32_t x = C.rows[k * kCellTiles + t];
      C.rows[k * kCellTiles + t] = run;
      run += x;
    }
    if (g == 0) {
      const RasterView &V = rv.v[find_cell_view<MAXV>(rv, c)];
      const int lc = c - V.cell_base;
      const int tx = (lc % V.cgw) * kCellEdge + (t & (kCellEdge - 1));
      const int ty = (lc / V.cgw) * kCellEdge + (t >> kCellShift);
      if (tx < V.gw && ty < V.gh) A.ranges[V.tile_base + ty * V.gw + tx].y = total;
    }
    __syncthreads();  // s_sum is reused by the next cell
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(&A.counters[kCtrCellDone], 1u) == gridDim.x - 1u;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  uint64_t base = 0ull;
  constexpr int kPer = 8;
  for (int64_t i0 = 0; i0 < A.total_tiles; i0 += kCellPrefixThreads * kPer) {
    const int64_t i = i0 + (int64_t)threadIdx.x * kPer;
    uint32_t x[kPer], sum = 0u, total;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      x[k] = i + k < A.total_tiles ? __ldcg(&A.ranges[i + k].y) : 0u;
      sum += x[k];
    }
    uint64_t p = base + block_exclusive_scan<kWarps>(sum, s_scan, &total);
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const uint64_t e = p + x[k];
      if (i + k < A.total_tiles)
        A.ranges[i + k] = make_uint2((uint32_t)umin64(p, (uint64_t)A.inst_cap), (uint32_t)umin64(e, (uint64_t)A.inst_cap));
      p = e;
    }
    base += total;
  }
  if (threadIdx.x == 0) {
    if (A.counters[kCtrPairOverflow])
      A.counters[kCtrNeedInstances] = (uint32_t)umin64(
          *reinterpret_cast<const volatile unsigned long long *>(&A.counters[kCtrRectTiles64]), 0xffffffffull);
    set_instance_total(A, *reinterpret_cast<const volatile unsigned long long *>(&A.counters[kCtrInstances64]));
  }
}

// Expands every run into its tiles' lists.  The run's (tile, pair) bits are
// placed in shared memory ordered by tile and pair -- lane t of warp w walks
// the set bits of its words, from the tile's offset in the run plus the counts
// of the warps before -- and then written, consecutive threads on consecutive
// staged bits, to each tile's place in the instance list (the tile's start
// plus the cell's earlier runs).  The explicit minimum of one resident block
// lets the compiler take more registers than its own choice: bin_sort (us)
// without / with it 725 / 664 at 2.3M visible slots and 15M instances (8
// views), 112 / 112 at 94k and 1.7M.  Walking words of many set bits by an
// unrolled loop over all 32 gave 4165 us without the minimum and 4219 with it
// at 741M instances; the plain walk with the minimum 4018.
template <int MAXV>
__global__ void __launch_bounds__(kCellBlock, 1) cell_write_kernel(CellArgs C, RasterViews<MAXV> rv) {
  grid_dependency_sync();
  constexpr int kWarps = kCellBlock / 32;
  static_assert(kCellSeg <= 256, "a pair's place in its segment fits a byte");
  __shared__ uint32_t s_key[kCellSeg], s_slot[kCellSeg];
  __shared__ uint16_t s_cnt[kWarps][kCellTiles];  // then: the warp's first staged position of the tile
  __shared__ uint32_t s_base[kCellTiles];  // the tile's place in the instance list less its first staged position
  __shared__ uint32_t s_total;
  __shared__ int32_t s_tile[kCellTiles];
  __shared__ uint16_t s_stage[kCellSeg * kCellTiles];  // (tile of the cell, pair of the segment)
  const EmitArgs &A = C.e;
  const int64_t npairs = min64((int64_t)A.counters[kCtrCellPairs], A.inst_cap);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  SegmentWalk W;
  W.npairs = npairs;
  W.load(C, blockIdx.x);
  for (int64_t s = blockIdx.x; s * kCellSeg < npairs; s += gridDim.x) {
    uint2 mask;
    const int n = W.stage(C, s, s + gridDim.x, s_key, s_slot, &mask);
    for (int a = 0; a < n;) {
      const int b = run_end(s_key, a, n);
      const int32_t c = (int32_t)s_key[a];
      if (warp == kWarps - 1) {  // places of the 64 tiles, two per lane
        const RasterView &V = rv.v[find_cell_view<MAXV>(rv, c)];
        const int lc = c - V.cell_base;
        const int tx0 = (lc % V.cgw) * kCellEdge, ty0 = (lc / V.cgw) * kCellEdge;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int t = 32 * h + lane;
          const int tx = tx0 + (t & (kCellEdge - 1)), ty = ty0 + (t >> kCellShift);
          const int32_t tile = tx < V.gw && ty < V.gh ? V.tile_base + ty * V.gw + tx : -1;
          s_tile[t] = tile;
          s_base[t] = tile < 0 ? 0u : A.ranges[tile].x + C.rows[((size_t)s + c) * kCellTiles + t];
        }
      }
      uint32_t w[2];
      run_words(mask, a, b, lane, &w[0], &w[1]);
      s_cnt[warp][lane] = (uint16_t)__popc(w[0]);
      s_cnt[warp][32 + lane] = (uint16_t)__popc(w[1]);
      __syncthreads();
      if (warp == 0) {  // exclusive prefix over tiles (lane: tiles 2 lane, 2 lane + 1), then over warps
        uint32_t t0 = 0u, t1 = 0u;
#pragma unroll
        for (int k = 0; k < kWarps; ++k) {
          t0 += s_cnt[k][2 * lane];
          t1 += s_cnt[k][2 * lane + 1];
        }
        uint32_t inc = t0 + t1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
          if (lane >= o) inc += y;
        }
        uint32_t p0 = inc - t0 - t1, p1 = inc - t1;
        s_base[2 * lane] -= p0;
        s_base[2 * lane + 1] -= p1;
        if (lane == 31) s_total = inc;
#pragma unroll
        for (int k = 0; k < kWarps; ++k) {
          const uint32_t c0 = s_cnt[k][2 * lane], c1 = s_cnt[k][2 * lane + 1];
          s_cnt[k][2 * lane] = (uint16_t)p0;  // at most 256 x 64 - 1
          s_cnt[k][2 * lane + 1] = (uint16_t)p1;
          p0 += c0;
          p1 += c1;
        }
      }
      __syncthreads();
      // (tile, pair) of this lane's first pair in each word
      const uint32_t v0 = (uint32_t)((lane << 8) | (32 * warp)), v1 = v0 + (32u << 8);
      uint32_t p0 = s_cnt[warp][lane], p1 = s_cnt[warp][32 + lane];
      for (uint32_t x = w[0]; x; x &= x - 1u) s_stage[p0++] = (uint16_t)(v0 + __ffs(x) - 1);
      for (uint32_t x = w[1]; x; x &= x - 1u) s_stage[p1++] = (uint16_t)(v1 + __ffs(x) - 1);
      __syncthreads();
      const uint32_t total = s_total;
#pragma unroll 4
      for (uint32_t q = threadIdx.x; q < total; q += kCellBlock) {
        const uint32_t v = s_stage[q], p = s_base[v >> 8] + q;
        if ((int64_t)p < A.inst_cap) {
          A.inst_key[p] = (uint32_t)s_tile[v >> 8];
          A.inst_val[p] = s_slot[v & 255u];
        }
      }
      a = b;
      __syncthreads();  // the staged run, s_key and s_slot are reused
    }
  }
}
