// Duplication and tile sort of the fused frame (Sec. II-A "Duplication with
// Tiles" and "Sorting", Identify Range of Sec. IV-B) as two stable splits of
// intervals.  The Gaussians arrive in depth order (view after view).  A
// Gaussian's tile rectangle is an interval of tile rows times an interval of
// tile columns, so the pairs need no sort of their own:
//   level 1  items = Gaussians in depth order, bins = tile rows: every
//            Gaussian goes, in order, to the list of each row it covers, as a
//            segment {depth bits, index} and its columns;
//   level 2  items = a row's segments in order, bins = tile columns: every
//            segment goes to the list of each column it covers, as the final
//            (tile << 32 | depth bits, index) pair.
// Rows are outer and columns inner in the tile id, so the rows' lists one
// after the other are the sorted pairs, and each tile's list keeps the depth
// order.  Only level 2 touches every pair, once: no pair is written or read
// in between.
//
// One level is three launches over tiles of 1024 items:
//   count  per tile and bin, how many items cover it (two shared atomics per
//          item into a difference array, then a prefix over the bins);
//   scan   per row: each tile's first position in each bin's list (level 2:
//          also the tile ranges);
//   split  ranks and writes the tile (k_split below).
//
// Ranks need no sort either.  A warp takes 32 items; per bin, the mask of its
// items that cover the bin is the prefix XOR over the bins of each item's bit
// toggled at its first bin and past its last one: two shared atomics per item
// and one XOR scan over the bins, whatever the intervals.  The rank of item i
// in a bin is the number of lower bits of that bin's mask, plus the bin's
// items in the warps before.
//
// Measured against the form this replaced (an expanding pass that wrote packed
// (tile, depth rank) elements and a second pass over them, both serial in a
// look-back chain), whole frames: 1M Gaussians at 1280x720 (10.6M pairs) 239
// to 145 us, 3M at 1080p 867 to 390 us, 16 views of 500,000 1410 to 832 us.  Two levels
// with counts and a scan in place of one pass with a look-back: the counts
// read 2 to 4 B per item where the look-back held every tile for the one
// before, and no launch waits inside.
#include "radix.cuh"

namespace tdgs {
namespace split {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kPerWarp = 2;                                 // 32-item batches per warp
constexpr int kBatches = kWarps * kPerWarp;
constexpr uint32_t kTile = kBatches * 32;                   // items per tile
constexpr uint32_t kStage = 8192;                           // pairs staged in shared memory at once
constexpr uint32_t kMaxBins = kSplitMaxBins;
constexpr int kCountThreads = 256;
constexpr uint32_t kEmptyRect = 0x00ff0000u;                // first row above the last: no rows
static_assert(kTile == kSplitTile, "the host sizes the tile tables");
static_assert(kMaxBins == 256, "bins and columns are packed in bytes");
static_assert(kTile <= kStage, "one bin of a tile fits the stage");

// Largest i < n with begin[i] <= x (begin ascending, begin[0] <= x), by the
// whole warp: 32 probes at a time.
__device__ __forceinline__ uint32_t warp_find(const uint32_t* begin, uint32_t n, uint32_t x) {
  uint32_t lo = 0, len = n;
  while (len > 1) {
    const uint32_t step = (len + 31) / 32, at = lane_id() * step;
    const bool le = at < len && __ldca(begin + lo + at) <= x;
    const uint32_t k = 31u - __clz(__ballot_sync(0xffffffffu, le) | 1u);
    lo += k * step;
    len = min(step, len - k * step);
  }
  return lo;
}

// 1 << n, 0 for n above 31, and the n lowest bits.
__device__ __forceinline__ uint32_t bit_or_none(uint32_t n) {
  uint32_t x;
  asm("shl.b32 %0, 1, %1;" : "=r"(x) : "r"(n));
  return x;
}
__device__ __forceinline__ uint32_t low_bits(uint32_t n) {
  uint32_t x;
  asm("bmsk.clamp.b32 %0, 0, %1;" : "=r"(x) : "r"(n));
  return x;
}

template <typename T>
__device__ __forceinline__ T warp_incl_scan(T x) {
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const T o = __shfl_up_sync(0xffffffffu, x, d);
    if (lane_id() >= static_cast<uint32_t>(d)) x += o;
  }
  return x;
}

// Inclusive sums over the block of two values at once (s_w: one per warp).
template <int kW, typename T>
__device__ __forceinline__ void block_incl_scan2(T& a, T& b, T (*s_w)[2]) {
  const uint32_t lane = lane_id(), warp = threadIdx.x >> 5;
  a = warp_incl_scan(a);
  b = warp_incl_scan(b);
  if (lane == 31) {
    s_w[warp][0] = a;
    s_w[warp][1] = b;
  }
  __syncthreads();
  T pa = 0, pb = 0;
#pragma unroll
  for (int w = 0; w < kW; ++w)
    if (w < static_cast<int>(warp)) {
      pa += s_w[w][0];
      pb += s_w[w][1];
    }
  a += pa;
  b += pb;
}

// Where view v's level-1 tiles, rows and counts lie among all views'.
struct Place {
  uint32_t tile0, tiles, row0, c10;
};
__device__ __forceinline__ Place place_of(const SplitArgs& a, uint32_t v) {
  if (a.vt.one.on) return Place{0u, a.ntiles1, 0u, 0u};
  const uint32_t t0 = __ldca(a.t1_begin + v);
  return Place{t0, __ldca(a.t1_begin + v + 1) - t0, __ldca(a.row_begin + v), __ldca(a.c1_begin + v)};
}

// A captured batch reads its view table when it is replayed: views may have
// other proportions or Gaussians by then, within the same totals.  The counts
// of tiles and rows come from the table, and a view that the launches or
// buffers have no room for is left out (k_row_scan reports it).
__device__ __forceinline__ uint32_t tiles1_of(const SplitArgs& a) {
  return a.vt.one.on ? a.ntiles1 : __ldca(a.t1_begin + a.vt.nv);
}
__device__ __forceinline__ uint32_t rows_of(const SplitArgs& a) {
  return a.vt.one.on ? a.nrows : min(a.nrows, __ldca(a.row_begin + a.vt.nv));
}
__device__ __forceinline__ bool has_room(const SplitArgs& a, const Place& pl, const FrameGeom& fg) {
  return static_cast<uint32_t>(fg.gx) <= a.pitch && static_cast<uint32_t>(fg.gy) <= a.max_gy &&
         pl.c10 + static_cast<uint64_t>(pl.tiles) * fg.gy <= a.c1_cap;
}

// ------------------------------------------------------------ level 1 count
// Per tile of 1024 depth positions: each Gaussian's {depth key, index} and
// rectangle in depth order (coalesced for the later launches; the records
// are gathered here, once), and per row its Gaussians and its pairs in the
// tile, as differences at the first row and past the last.
// Bound by the gather of 16 B records from L2 in depth order (four in flight
// per thread): 12.8 us for 1M Gaussians, 28.5 us for 3M (1.0 and 1.3 TB/s of
// 32 B sectors that hold two records).  Gathered here, the depth sort need
// carry no rectangle or count per Gaussian, and the split reads 12 B per item
// in order.
__global__ void __launch_bounds__(kCountThreads) k_row_count(SplitArgs a) {
  __shared__ int s_d[kMaxBins + 1][2];
  __shared__ uint32_t s_w[kCountThreads / 32][2];
  begin_launch();
  const uint32_t t = threadIdx.x;
  if (blockIdx.x >= tiles1_of(a)) return;
  const uint32_t v = a.vt.nv == 1 ? 0u : warp_find(a.t1_begin, a.vt.nv, blockIdx.x);
  const Place pl = place_of(a, v);
  const ViewOf vw = view_of(a.vt, v);
  if (!has_room(a, pl, vw.geom)) return;
  const uint32_t tl = blockIdx.x - pl.tile0, nt = pl.tiles, rec0 = vw.rec0, nrec = vw.nrec;
  const FrameGeom fg = vw.geom;
  const float4* g = vw.g;
  for (uint32_t b = t; b <= kMaxBins; b += kCountThreads) s_d[b][0] = s_d[b][1] = 0;
  __syncthreads();
  constexpr int kPer = kTile / kCountThreads;
  const uint32_t first = tl * kTile;
  float dmin = 0.0f, scale = 0.0f;
  if (a.norm) {
    dmin = __uint_as_float(__ldcg(a.norm));
    scale = norm_scale(dmin, __uint_as_float(__ldcg(a.norm + 1)));
  }
  uint32_t gi[kPer];
  float4 rec[kPer];
#pragma unroll
  for (int u = 0; u < kPer; ++u) {
    const uint32_t p = first + u * kCountThreads + t;
    gi[u] = p < nrec ? __ldca(a.sorder + rec0 + p) - rec0 : 0xffffffffu;
  }
#pragma unroll
  for (int u = 0; u < kPer; ++u)  // an order that is not a permutation is never followed out of bounds
    rec[u] = gi[u] < nrec ? __ldca(g + gi[u]) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int u = 0; u < kPer; ++u) {
    const uint32_t p = first + u * kCountThreads + t;
    if (p >= nrec) continue;
    const TileRect q = tile_rect(rec[u], fg);
    uint32_t pack = kEmptyRect;
    if (q.count) {
      const int w = q.x1 - q.x0;
      pack = static_cast<uint32_t>(q.x0) | (static_cast<uint32_t>(q.x1 - 1) << 8) |
             (static_cast<uint32_t>(q.y0) << 16) | (static_cast<uint32_t>(q.y1 - 1) << 24);
      atomicAdd(&s_d[q.y0][0], 1);
      atomicAdd(&s_d[q.y0][1], w);
      atomicAdd(&s_d[q.y1][0], -1);
      atomicAdd(&s_d[q.y1][1], -w);
    }
    a.rects[rec0 + p] = pack;
    // the low part of the pairs' keys: depth bits, or the normalised depth
    const uint32_t low = a.norm ? norm_depth(rec[u].z, dmin, scale) : __float_as_uint(rec[u].z);
    a.sdo[rec0 + p] = make_uint2(low, gi[u]);
  }
  __syncthreads();
  uint32_t c = static_cast<uint32_t>(s_d[t][0]), w = static_cast<uint32_t>(s_d[t][1]);
  block_incl_scan2<kCountThreads / 32>(c, w, s_w);
  if (t < static_cast<uint32_t>(fg.gy)) a.c1[pl.c10 + t * nt + tl] = make_uint2(c, w);
}

// ------------------------------------------------------------- level 1 scan
// One block per row (of all views): the row's Gaussians before each of its
// tiles, and the row's segments and pairs.  The last block then gives every
// row its first segment, first level-2 tile and first pair.  More pairs than
// the buffers hold (or than the depth order accounts for) latches
// TDGS_ERR_CAPACITY and leaves nothing for the later launches to do.
// Latency: a row's tiles in one or a few steps of 1024, one ticket, and the
// last block's scan of the rows: 5.5 us for 45 rows of 977 tiles, 8.4 us for
// 68 rows of 2930.
__global__ void __launch_bounds__(kCountThreads) k_row_scan(SplitArgs a) {
  __shared__ uint32_t s_w[kCountThreads / 32][2];
  __shared__ unsigned long long s_w64[kCountThreads / 32][2];
  __shared__ bool s_last;
  begin_launch();
  constexpr uint32_t kPer = 4;
  const uint32_t t = threadIdx.x, r = blockIdx.x;
  const uint32_t v = a.vt.nv == 1 ? 0u : warp_find(a.row_begin, a.vt.nv, r);
  const Place pl = place_of(a, v);
  const uint32_t nt = r < rows_of(a) && has_room(a, pl, view_of(a.vt, v).geom) ? pl.tiles : 0u;
  uint2* __restrict__ col = a.c1 + pl.c10 + static_cast<size_t>(r - pl.row0) * nt;
  uint32_t segs = 0, pairs = 0;
  for (uint32_t i0 = 0; i0 < nt; i0 += kCountThreads * kPer) {
    uint2 x[kPer];
    uint32_t sum = 0, w = 0;
#pragma unroll
    for (uint32_t u = 0; u < kPer; ++u) {
      const uint32_t i = i0 + t * kPer + u;
      x[u] = i < nt ? col[i] : make_uint2(0u, 0u);
      sum += x[u].x;
      w += x[u].y;
    }
    uint32_t run = sum;
    block_incl_scan2<kCountThreads / 32>(run, w, s_w);
    uint32_t before = segs + run - sum;
#pragma unroll
    for (uint32_t u = 0; u < kPer; ++u) {
      const uint32_t i = i0 + t * kPer + u;
      if (i < nt) col[i].y = before;
      before += x[u].x;
    }
    __syncthreads();  // s_w is read
    if (t == kCountThreads - 1) {
      s_w[0][0] = run;
      s_w[0][1] = w;
    }
    __syncthreads();
    segs += s_w[0][0];
    pairs += s_w[0][1];
    __syncthreads();
  }
  if (t == 0) {
    a.row_tot[r] = make_uint2(segs, pairs);  // (one entry per block)
    __threadfence();
    s_last = atomicAdd(a.ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  bool room = true;
  for (uint32_t i = t; i < a.vt.nv; i += kCountThreads) room &= has_room(a, place_of(a, i), view_of(a.vt, i).geom);
  const uint32_t nrows = gridDim.x;  // (rows beyond the table's have no segments)
  room = __syncthreads_and(room) && (a.vt.one.on || __ldca(a.row_begin + a.vt.nv) <= a.nrows);
  uint32_t seg0 = 0, tile0 = 0;
  unsigned long long pair0 = 0;
  for (uint32_t i0 = 0; i0 < nrows; i0 += kCountThreads) {
    const uint32_t i = i0 + t;
    const uint2 x = i < nrows ? __ldcg(a.row_tot + i) : make_uint2(0u, 0u);
    const uint32_t nt2 = (x.x + kTile - 1) / kTile;
    // segments and tiles side by side in 64 bits (neither reaches 2^32)
    unsigned long long st = (static_cast<unsigned long long>(nt2) << 32) | x.x, pr = x.y;
    block_incl_scan2<kCountThreads / 32>(st, pr, s_w64);
    if (i < nrows) {
      a.row_seg[i] = seg0 + static_cast<uint32_t>(st) - x.x;
      a.row_tile[i] = tile0 + static_cast<uint32_t>(st >> 32) - nt2;
      a.row_pair[i] = static_cast<uint32_t>(pair0 + pr - x.y);
    }
    __syncthreads();
    if (t == kCountThreads - 1) {
      s_w64[0][0] = st;
      s_w64[0][1] = pr;
    }
    __syncthreads();
    seg0 += static_cast<uint32_t>(s_w64[0][0]);
    tile0 += static_cast<uint32_t>(s_w64[0][0] >> 32);
    pair0 += s_w64[0][1];
    __syncthreads();
  }
  if (t == 0) {
    const bool fits = room && pair0 == *a.total && pair0 <= a.cap;
    if (!fits)
      latch_error(a.err, *a.total > 0xffffffffull ? TDGS_ERR_OVERFLOW : TDGS_ERR_CAPACITY, kSiteViewsDup);
    a.row_seg[nrows] = seg0;
    a.row_tile[nrows] = tile0;
    a.info[0] = fits ? tile0 : 0u;  // level-2 tiles to process
    a.info[1] = fits ? 1u : 0u;
    *a.ticket = 0u;
  }
}

// ------------------------------------------------------------ level 2 count
// Per tile of 1024 segments of one row: the segments that cover each column.
// Two shared atomics per segment and one 2 B read: 8.6 us for 2.6M segments,
// 18.8 us for 8.6M, half of it launch, search and the scan of the columns.
__global__ void __launch_bounds__(kCountThreads) k_col_count(SplitArgs a) {
  __shared__ int s_d[kMaxBins + 1];
  __shared__ uint32_t s_w[kCountThreads / 32];
  begin_launch();
  const uint32_t t = threadIdx.x, lane = lane_id(), warp = t >> 5;
  const uint32_t ntiles = __ldca(a.info);
  for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const uint32_t r = warp_find(a.row_tile, a.nrows, tile);
    const uint32_t beg = __ldca(a.row_seg + r) + (tile - __ldca(a.row_tile + r)) * kTile;
    const uint32_t end = min(beg + kTile, __ldca(a.row_seg + r + 1));
    constexpr int kPer = kTile / kCountThreads;
    uint32_t x[kPer];
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const uint32_t p = beg + u * kCountThreads + t;
      x[u] = p < end ? __ldca(a.cols + p) : 0xffffffffu;
    }
    for (uint32_t b = t; b <= kMaxBins; b += kCountThreads) s_d[b] = 0;
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      if (x[u] != 0xffffffffu) {
        atomicAdd(&s_d[x[u] & 0xffu], 1);
        atomicAdd(&s_d[(x[u] >> 8) + 1u], -1);
      }
    }
    __syncthreads();
    uint32_t c = warp_incl_scan(static_cast<uint32_t>(s_d[t]));
    if (lane == 31) s_w[warp] = c;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kCountThreads / 32; ++w)
      if (w < static_cast<int>(warp)) c += s_w[w];
    if (t < a.pitch) a.c2[static_cast<size_t>(tile) * a.pitch + t] = static_cast<uint16_t>(c);
    __syncthreads();
  }
}

// ------------------------------------------------------------- level 2 scan
// One block per row: the first output position of every tile and column, and
// the row's tile ranges (relative to the view's first pair; {0, 0} if
// empty).  Thread (g, c) walks column c over the g-th share of the row's
// tiles: once for the sums, once for the positions (the second time from L1
// or L2).  Latency of the two walks with eight loads in flight: 8.8 us for
// 45 rows of ~58 tiles, 10.8 us for 68 of ~125.  One block per row, not the
// count kernel's last block of a row: that made count and scan one launch,
// but 43 and 171 us of it where these two take 17 and 30: a block in a scan
// holds up its later tiles, so the rows end one after another.
constexpr int kScanThreads = 1024;
__global__ void __launch_bounds__(kScanThreads) k_col_scan(SplitArgs a) {
  __shared__ uint32_t s_sum[kScanThreads];
  __shared__ uint32_t s_w[kScanThreads / 32];
  begin_launch();
  if (__ldca(a.info + 1) == 0u) return;  // more pairs than the buffers hold
  const uint32_t t = threadIdx.x, r = blockIdx.x;
  if (r >= rows_of(a)) return;
  const uint32_t v = a.vt.nv == 1 ? 0u : warp_find(a.row_begin, a.vt.nv, r);
  const uint32_t gx = static_cast<uint32_t>(view_of(a.vt, v).geom.gx), y = r - place_of(a, v).row0;
  const uint32_t lp = gx <= 32 ? 5u : 32u - static_cast<uint32_t>(__clz(gx - 1));  // columns padded to 2^lp
  const uint32_t c = t & ((1u << lp) - 1u), g = t >> lp, groups = kScanThreads >> lp;
  const uint32_t tile0 = __ldca(a.row_tile + r), nt = __ldca(a.row_tile + r + 1) - tile0;
  const uint32_t per = (nt + groups - 1) / groups;
  const uint32_t lo = min(g * per, nt), hi = min(lo + per, nt);
  const uint16_t* cnt = a.c2 + static_cast<size_t>(tile0) * a.pitch + c;
  uint32_t sum = 0;
  if (c < gx) {
#pragma unroll 8
    for (uint32_t i = lo; i < hi; ++i) sum += __ldca(cnt + static_cast<size_t>(i) * a.pitch);
  }
  s_sum[t] = sum;
  __syncthreads();
  uint32_t before = 0, total = 0;
  for (uint32_t k = 0; k < groups; ++k) {
    const uint32_t x = s_sum[(k << lp) + c];
    if (k < g) before += x;
    total += x;
  }
  // columns in order: the first 2^lp threads hold each column once
  uint32_t incl = warp_incl_scan(t < (1u << lp) ? total : 0u);
  if (lane_id() == 31) s_w[t >> 5] = incl;
  __syncthreads();
  const uint32_t cw = c >> 5;  // the warp that holds column c
#pragma unroll
  for (uint32_t w = 0; w < kMaxBins / 32; ++w)
    if (w < cw && t < (1u << lp)) incl += s_w[w];
  __syncthreads();
  if (t < (1u << lp)) {
    const uint32_t start = __ldca(a.row_pair + r) + incl - total;
    s_sum[t] = start;
    if (c < gx) {
      const uint32_t pb = a.vt.pbeg[v];
      a.ranges[(a.vt.one.on ? 0u : __ldca(a.vt.tile_begin + v)) + y * gx + c] =
          total ? make_uint2(start - pb, start + total - pb) : make_uint2(0u, 0u);
    }
  }
  __syncthreads();
  uint32_t run = s_sum[c] + before;
  if (c < gx) {
    uint32_t* __restrict__ out = a.b2 + static_cast<size_t>(tile0) * a.pitch + c;
#pragma unroll 8
    for (uint32_t i = lo; i < hi; ++i) {
      out[static_cast<size_t>(i) * a.pitch] = run;
      run += __ldca(cnt + static_cast<size_t>(i) * a.pitch);
    }
  }
}

// ------------------------------------------------------------------- split
// One tile of up to 1024 items at a time.  kLevel 1: items are depth
// positions, bins the view's rows, the output segments; kLevel 2: items are
// a row's segments, bins the columns, the output final pairs.  Steps:
//   load     each lane its items' intervals and payloads; one warp the tile's
//            counts and positions per bin (their prefix over the bins is
//            where each bin's pairs start in the tile);
//   masks    per warp and batch of 32 items, by the XOR scan;
//   prefix   per bin over the batches, four threads per bin;
//   expand   the batch's pairs, 32 at a time, staged as {bin, item} at their
//            positions in bin order;
//   flush    the staged pairs in bin order: runs of consecutive addresses.
// A tile with more pairs than the stage holds takes windows of whole bins.
//
// Level 2 is the frame's longest kernel and bound by instruction issue and the
// shared-memory pipe together (10.6M pairs: 3.3 warp instructions per
// pair, issue 60 %, LSU data pipe 68 % busy, 69 % of the warps
// resident), not by its 127 MB of final pairs, of which 65 to 81 MB reach
// DRAM inside the launch: 51 us, 2.5 TB/s written; 166 us for the 36M pairs of
// a 3M-Gaussian frame, 2.6 TB/s.  Level 1: 18.6 us for 2.6M segments.  What it
// replaced took 154 us for the 10.6M pairs (expand + one tile pass).
// 512 threads and 1024 items, three blocks per SM, so that one block's flush
// overlaps another's ranks.  A frame of 1M / 3M Gaussians takes longer with 256
// threads and 512 items (1.2 / 13 us), 256 and 1024 (8 / 20), 512 and 512 (11 /
// 33: every tile pays for its bins, and its runs are half as long).  The owner
// search over the starts' word took the 1M column split from 75 us (each lane
// walking its own item's bins) to 57.
template <int kWords>  // 32 kWords bins; each lane scans kWords consecutive ones
struct Smem {
  static constexpr int kBinsP = 32 * kWords;
  static constexpr int kPitch = kBinsP + 1;  // odd: (batch, bin) lanes of the prefix step hit different banks
  uint2 pay[kTile];
  uint32_t stage[kStage];
  uint32_t mask[kBatches][kPitch];
  uint32_t lstart[kBinsP + 1];
  uint32_t off[kBinsP];
  uint16_t pos[kBatches][kPitch];
  uint16_t cols[kTile];  // level 1: the items' columns
};
static_assert(sizeof(Smem<9>) < 220 * 1024, "one CTA fits an SM");

// The steps after the load, for one tile whose counts and positions are in
// s.lstart and s.off.  row_tile: level 2, the row's first tile in its view.
// Starts and ends with a block barrier.
template <int kLevel, int kWords>
__device__ __forceinline__ void split_tile(Smem<kWords>& s, const SplitArgs& a, const uint32_t (&lo)[kPerWarp],
                                           const uint32_t (&hi)[kPerWarp], uint32_t bins, uint32_t row_tile) {
  constexpr int kBinsP = Smem<kWords>::kBinsP;
  const uint32_t t = threadIdx.x, lane = lane_id(), warp = t >> 5;
  const uint32_t lt = lanemask_lt(), le = lt | (1u << lane);
  // ---- masks
#pragma unroll
  for (int b = 0; b < kPerWarp; ++b) {
    uint32_t* m = s.mask[warp * kPerWarp + b];
#pragma unroll
    for (int k = 0; k < kWords; ++k) m[k * 32 + lane] = 0u;
    __syncwarp();
    if (hi[b] > lo[b]) {
      atomicXor(m + lo[b], 1u << lane);
      if (hi[b] < bins) atomicXor(m + hi[b], 1u << lane);
    }
    __syncwarp();
    uint32_t x[kWords], own = 0;  // inclusive over this lane's bins, then over the lanes before
#pragma unroll
    for (int k = 0; k < kWords; ++k) {
      own ^= m[lane * kWords + k];
      x[k] = own;
    }
    uint32_t before = own;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t o = __shfl_up_sync(0xffffffffu, before, d);
      if (lane >= static_cast<uint32_t>(d)) before ^= o;
    }
    before ^= own;
#pragma unroll
    for (int k = 0; k < kWords; ++k) m[lane * kWords + k] = x[k] ^ before;
  }
  __syncthreads();
  const uint32_t total = s.lstart[kBinsP];
  for (uint32_t b0 = 0; b0 < bins;) {
    // bins [b0, b1): the whole tile, or as many as the stage holds
    uint32_t b1 = bins;
    const uint32_t p0 = s.lstart[b0];
    if (total - p0 > kStage) {
      b1 = b0 + 1;
      while (b1 < bins && s.lstart[b1 + 1] - p0 <= kStage) ++b1;
    }
    const uint32_t np = s.lstart[b1] - p0;
    // ---- prefix over the batches
    for (uint32_t cw = b0 + warp * 8; cw < b1; cw += kWarps * 8) {  // eight bins a warp, four lanes each
      const uint32_t c = cw + (lane >> 2);
      constexpr int kEach = kBatches / 4;
      const uint32_t g = t & 3u, cc = min(c, b1 - 1u);
      uint32_t x[kEach], sum = 0;
#pragma unroll
      for (int i = 0; i < kEach; ++i) {
        x[i] = __popc(s.mask[g * kEach + i][cc]);
        sum += x[i];
      }
      uint32_t run = sum;
#pragma unroll
      for (int d = 1; d < 4; d <<= 1) {
        const uint32_t o = __shfl_up_sync(0xffffffffu, run, d, 4);
        if (g >= static_cast<uint32_t>(d)) run += o;
      }
      run += s.lstart[cc] - p0 - sum;
      if (c < b1) {
#pragma unroll
        for (int i = 0; i < kEach; ++i) {
          s.pos[g * kEach + i][c] = static_cast<uint16_t>(run);
          run += x[i];
        }
      }
    }
    __syncthreads();
    // ---- expand
#pragma unroll
    for (int b = 0; b < kPerWarp; ++b) {
      const uint32_t bat = warp * kPerWarp + b;
      const uint32_t* m = s.mask[bat];
      const uint16_t* ps = s.pos[bat];
      const uint32_t l = max(lo[b], b0), h = min(hi[b], b1);
      const uint32_t n = h > l ? h - l : 0u;
      const uint32_t item0 = bat * 32;
      const uint32_t full = __ballot_sync(0xffffffffu, n != 0u);
      if ((full & (full + 1u)) == 0u) {
        // Lane p of a step takes the batch's p-th pair: its owner is the
        // last item that starts at or before it.  The starts that fall into
        // the step's 32 pairs are one word, and the items are in lane order.
        const uint32_t end = warp_incl_scan(n), st = end - n;
        const uint32_t np_b = __shfl_sync(0xffffffffu, end, 31);
        const uint32_t shift = l - st;            // bin of pair p of this item, less p
        uint32_t at = n ? st : 0x80000000u;       // start relative to the step (never 0..31 if none)
        uint32_t seen = 0xffffffffu;              // items that start before the step, less one
        for (uint32_t p = lane; p < np_b + lane; p += 32, at -= 32) {
          const uint32_t starts = __reduce_or_sync(0xffffffffu, bit_or_none(at));
          const uint32_t src = seen + __popc(starts & le);
          seen += __popc(starts);
          const uint32_t c = p + __shfl_sync(0xffffffffu, shift, src);
          if (p < np_b) s.stage[ps[c] + __popc(m[c] & low_bits(src))] = c * 65536u + (item0 + src);
        }
      } else {  // a window left items without bins between others: each lane walks its own
        const uint32_t steps = __reduce_max_sync(0xffffffffu, n);
        for (uint32_t j = 0; j < steps; ++j) {
          const uint32_t c = l + j;
          if (j < n) s.stage[ps[c] + __popc(m[c] & lt)] = c * 65536u + (item0 + lane);
        }
      }
    }
    __syncthreads();
    // ---- flush
    if constexpr (kLevel == 1) {
#pragma unroll 2
      for (uint32_t p = t; p < np; p += kThreads) {
        const uint32_t e = s.stage[p], i = e & 0xffffu, dst = s.off[e >> 16] + p0 + p;
        a.segs[dst] = s.pay[i];
        a.cols[dst] = s.cols[i];
      }
    } else if (a.keys32) {
#pragma unroll 2
      for (uint32_t p = t; p < np; p += kThreads) {
        const uint32_t e = s.stage[p], c = e >> 16;
        const uint2 q = s.pay[e & 0xffffu];
        const uint32_t dst = s.off[c] + p0 + p;
        a.keys32[dst] = ((row_tile + c) << 10) | q.x;
        a.values[dst] = q.y;
      }
    } else {
#pragma unroll 2
      for (uint32_t p = t; p < np; p += kThreads) {
        const uint32_t e = s.stage[p], c = e >> 16;
        const uint2 q = s.pay[e & 0xffffu];
        const uint32_t dst = s.off[c] + p0 + p;
        a.keys[dst] = (static_cast<uint64_t>(row_tile + c) << 32) | q.x;
        a.values[dst] = q.y;
      }
    }
    __syncthreads();
    b0 = b1;
  }
}

template <int kLevel, int kWords>
__global__ void __launch_bounds__(kThreads, kWords > 5 ? 2 : 3) k_split(SplitArgs a) {
  using S = Smem<kWords>;
  constexpr int kBinsP = S::kBinsP;
  extern __shared__ __align__(16) unsigned char smem[];
  S& s = *reinterpret_cast<S*>(smem);
  begin_launch();
  const uint32_t t = threadIdx.x, lane = lane_id(), warp = t >> 5;
  if (__ldca(a.info + 1) == 0u) return;
  const uint32_t ntiles = kLevel == 1 ? tiles1_of(a) : __ldca(a.info);
  for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    uint32_t v, beg, cnt, bins, r = 0, tl = 0;
    Place pl;
    if constexpr (kLevel == 1) {
      v = a.vt.nv == 1 ? 0u : warp_find(a.t1_begin, a.vt.nv, tile);
      pl = place_of(a, v);
      const ViewOf vw = view_of(a.vt, v);
      tl = tile - pl.tile0;
      beg = vw.rec0 + tl * kTile;
      cnt = min(kTile, vw.nrec - tl * kTile);
      bins = static_cast<uint32_t>(vw.geom.gy);
    } else {
      r = warp_find(a.row_tile, a.nrows, tile);
      v = a.vt.nv == 1 ? 0u : warp_find(a.row_begin, a.vt.nv, r);
      pl = place_of(a, v);
      beg = __ldca(a.row_seg + r) + (tile - __ldca(a.row_tile + r)) * kTile;
      cnt = min(kTile, __ldca(a.row_seg + r + 1) - beg);
      bins = static_cast<uint32_t>(view_of(a.vt, v).geom.gx);
    }
    // ---- load
    uint32_t lo[kPerWarp], hi[kPerWarp];  // bins [lo, hi)
#pragma unroll
    for (int b = 0; b < kPerWarp; ++b) {
      const uint32_t i = (warp * kPerWarp + b) * 32 + lane;
      lo[b] = hi[b] = 0u;
      if (i < cnt) {
        if constexpr (kLevel == 1) {
          const uint32_t q = __ldca(a.rects + beg + i);
          lo[b] = (q >> 16) & 0xffu;
          hi[b] = (q >> 24) + 1u;
          if (hi[b] <= lo[b]) lo[b] = hi[b] = 0u;
          s.pay[i] = __ldca(a.sdo + beg + i);
          s.cols[i] = static_cast<uint16_t>(q);
        } else {
          const uint32_t q = __ldca(a.cols + beg + i);
          lo[b] = q & 0xffu;
          hi[b] = (q >> 8) + 1u;
          s.pay[i] = __ldca(a.segs + beg + i);
        }
      }
    }
    if (warp == kWarps - 1) {
      constexpr int kPer = kWords;
      uint32_t c[kPer], base[kPer], sum = 0;
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        const uint32_t b = lane * kPer + i;
        c[i] = base[i] = 0u;
        if (b < bins) {
          if constexpr (kLevel == 1) {
            const uint2 x = __ldca(a.c1 + pl.c10 + static_cast<size_t>(b) * pl.tiles + tl);
            c[i] = x.x;
            base[i] = x.y + __ldca(a.row_seg + pl.row0 + b);
          } else {
            c[i] = __ldca(a.c2 + static_cast<size_t>(tile) * a.pitch + b);
            base[i] = __ldca(a.b2 + static_cast<size_t>(tile) * a.pitch + b);
          }
        }
        sum += c[i];
      }
      uint32_t run = warp_incl_scan(sum) - sum;
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        const uint32_t b = lane * kPer + i;
        s.lstart[b] = run;
        s.off[b] = base[i] - run;
        run += c[i];
      }
      if (lane == 31) s.lstart[kBinsP] = run;  // (all pairs; every bin past the last starts here too)
    }
    split_tile<kLevel, kWords>(s, a, lo, hi, bins, kLevel == 2 ? (r - pl.row0) * bins : 0u);
  }
}

// ------------------------------------------------------------- small frames
// All of it for one small view in one cooperative launch: count, row split,
// column split, with a grid barrier between them.  The scans and the column
// counts need no phase of their own: every block sums the few tiles' counts of
// all rows for level 1, and counts all segments of its tile's row for level 2
// (at most kSplitSmall of them: the sums are kept in 16 bits).
// Bound by the latency of its phases and two barriers: for 10,000 Gaussians
// (57k pairs) one launch of ~20 us in place of six (34 us), the frame 57 to
// 46 us; 30,000 Gaussians 58 to 50 us.  From ~60,000 on the six launches are
// as fast, since every block of level 2 counts its whole row again: the line
// (kSplitSmall) lies below, where the 16-bit sums end too.
// What an earlier phase wrote is read through L2 (__ldcg).  A barrier that
// times out ends the block: the counts that size the staging are then not to
// be trusted.
__device__ __forceinline__ bool small_barrier(uint32_t* bar, uint32_t* err) {
  __shared__ bool s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    bool ok = true;
    const uint32_t gen = radix::ld_acquire32(bar + 1);
    if (radix::atom_add_acq_rel32(bar, 1u) == gridDim.x - 1) {
      bar[0] = 0u;  // ordered before the release below
      radix::st_release32(bar + 1, gen + 1);
    } else {
      uint32_t spins = 0;
      while (radix::ld_acquire32(bar + 1) == gen) {
        if (++spins > kSpinLimit) {
          latch_error(err, TDGS_ERR_TIMEOUT, kSiteBarrier);
          ok = false;
          break;
        }
        __nanosleep(20);
      }
    }
    s_ok = ok;
  }
  __syncthreads();
  return s_ok;
}

template <int kWords>
__global__ void __launch_bounds__(kThreads, 1) k_small(SplitArgs a) {
  using S = Smem<kWords>;
  constexpr int kBinsP = S::kBinsP;
  extern __shared__ __align__(16) unsigned char smem[];
  S& s = *reinterpret_cast<S*>(smem);
  __shared__ uint32_t s_seg[kMaxBins + 1], s_tile[kMaxBins + 1], s_pair[kMaxBins];  // of each row: the first
  __shared__ unsigned long long s_w[kWarps][2];
  __shared__ uint32_t s_w32[kWarps][2];
  int(*s_d)[2] = reinterpret_cast<int(*)[2]>(s.stage);  // differences of a count phase
  static_assert(sizeof(s.stage) >= (kMaxBins + 1) * sizeof(int[2]), "the differences fit the stage");
  static_assert(kThreads >= kMaxBins, "one bin per thread");
  const uint32_t t = threadIdx.x, lane = lane_id(), warp = t >> 5;
  const FrameGeom fg = a.vt.one.geom;
  const uint32_t n = a.vt.one.n, nt = a.ntiles1;
  const uint32_t gx = static_cast<uint32_t>(fg.gx), gy = static_cast<uint32_t>(fg.gy);
  const float4* g = a.vt.one.g;
  constexpr int kPer = kTile / kThreads;
  // ---- rectangles in depth order and the rows' counts
  float dmin = 0.0f, scale = 0.0f;
  if (a.norm) {
    dmin = __uint_as_float(__ldcg(a.norm));
    scale = norm_scale(dmin, __uint_as_float(__ldcg(a.norm + 1)));
  }
  for (uint32_t tile = blockIdx.x; tile < nt; tile += gridDim.x) {
    if (t <= kMaxBins) s_d[t][0] = s_d[t][1] = 0;
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const uint32_t p = tile * kTile + u * kThreads + t;
      if (p >= n) continue;
      const uint32_t gi = __ldca(a.sorder + p);
      const float4 rec = gi < n ? __ldca(g + gi) : make_float4(0.f, 0.f, 0.f, 0.f);
      const TileRect q = tile_rect(rec, fg);
      uint32_t pack = kEmptyRect;
      if (q.count) {
        const int w = q.x1 - q.x0;
        pack = static_cast<uint32_t>(q.x0) | (static_cast<uint32_t>(q.x1 - 1) << 8) |
               (static_cast<uint32_t>(q.y0) << 16) | (static_cast<uint32_t>(q.y1 - 1) << 24);
        atomicAdd(&s_d[q.y0][0], 1);
        atomicAdd(&s_d[q.y0][1], w);
        atomicAdd(&s_d[q.y1][0], -1);
        atomicAdd(&s_d[q.y1][1], -w);
      }
      a.rects[p] = pack;
      a.sdo[p] = make_uint2(a.norm ? norm_depth(rec.z, dmin, scale) : __float_as_uint(rec.z), gi);
    }
    __syncthreads();
    unsigned long long c = t < kMaxBins ? static_cast<uint32_t>(s_d[t][0]) : 0u;
    unsigned long long w = t < kMaxBins ? static_cast<uint32_t>(s_d[t][1]) : 0u;
    block_incl_scan2<kWarps>(c, w, s_w);  // (differences modulo 2^32)
    if (t < gy) a.c1[t * nt + tile] = make_uint2(static_cast<uint32_t>(c), static_cast<uint32_t>(w));
    __syncthreads();
  }
  if (!small_barrier(a.bar, a.err)) return;
  // ---- the rows' segments: every block finds all rows' starts, and its
  // tile's positions in them
  const uint64_t m = __ldcg(a.total);
  uint32_t tile = blockIdx.x;
  do {
    uint32_t cnt = 0, before = 0, segs = 0, pairs = 0;
    if (t < gy) {
      for (uint32_t k = 0; k < nt; ++k) {
        const uint2 x = __ldcg(a.c1 + t * nt + k);
        segs += x.x;
        pairs += x.y;
        if (k < tile) before += x.x;
        if (k == tile) cnt = x.x;
      }
    }
    const uint32_t nt2 = (segs + kTile - 1) / kTile;
    // two sums a word: {level-2 tiles, segments}, {items of this tile, pairs}
    const unsigned long long own0 = (static_cast<unsigned long long>(nt2) << 32) | segs;
    const unsigned long long own1 = (static_cast<unsigned long long>(cnt) << 40) | pairs;
    unsigned long long in0 = own0, in1 = own1;
    block_incl_scan2<kWarps>(in0, in1, s_w);
    const unsigned long long ex0 = in0 - own0, ex1 = in1 - own1;
    const uint32_t lstart = static_cast<uint32_t>(ex1 >> 40);
    if (t <= gy) {
      s_seg[t] = static_cast<uint32_t>(ex0);
      s_tile[t] = static_cast<uint32_t>(ex0 >> 32);
      if (t < gy) s_pair[t] = static_cast<uint32_t>(ex1);
    }
    if (t < kBinsP) {
      s.lstart[t] = lstart;
      s.off[t] = static_cast<uint32_t>(ex0) + before - lstart;
    }
    if (t == kThreads - 1) s.lstart[kBinsP] = static_cast<uint32_t>(in1 >> 40);
    const unsigned long long sum = in1 & ((1ull << 40) - 1);  // (the last thread's: all pairs)
    if (__syncthreads_or(t == kThreads - 1 && (sum != m || m > a.cap))) {
      if (t == 0 && blockIdx.x == 0)
        latch_error(a.err, m > 0xffffffffull ? TDGS_ERR_OVERFLOW : TDGS_ERR_CAPACITY, kSiteViewsDup);
      return;  // in every block: all see the same sums
    }
    if (tile < nt) {
      uint32_t lo[kPerWarp], hi[kPerWarp];
#pragma unroll
      for (int b = 0; b < kPerWarp; ++b) {
        const uint32_t i = (warp * kPerWarp + b) * 32 + lane, p = tile * kTile + i;
        lo[b] = hi[b] = 0u;
        if (p < n) {
          const uint32_t q = __ldcg(a.rects + p);
          lo[b] = (q >> 16) & 0xffu;
          hi[b] = (q >> 24) + 1u;
          if (hi[b] <= lo[b]) lo[b] = hi[b] = 0u;
          s.pay[i] = __ldcg(a.sdo + p);
          s.cols[i] = static_cast<uint16_t>(q);
        }
      }
      split_tile<1, kWords>(s, a, lo, hi, gy, 0u);
    }
    tile += gridDim.x;
  } while (tile < nt);
  if (!small_barrier(a.bar, a.err)) return;
  const uint32_t ntiles2 = s_tile[gy];
  auto row_of = [&](uint32_t x) {  // the last row that starts at or before tile x
    uint32_t lo = 0, len = gy;
    while (len > 1) {
      const uint32_t half = len >> 1;
      if (s_tile[lo + half] <= x) {
        lo += half;
        len -= half;
      } else {
        len = half;
      }
    }
    return lo;
  };
  // ---- the ranges of rows without tiles, then the pairs: a tile's positions
  // from the columns of all its row's segments
  for (uint32_t r = blockIdx.x; r < gy; r += gridDim.x)
    if (s_tile[r] == s_tile[r + 1] && t < gx) a.ranges[r * gx + t] = make_uint2(0u, 0u);
  for (uint32_t x = blockIdx.x; x < ntiles2; x += gridDim.x) {
    const uint32_t r = row_of(x), k0 = x - s_tile[r];
    const uint32_t beg = s_seg[r] + k0 * kTile, cnt_items = min(kTile, s_seg[r + 1] - beg);
    uint32_t lo[kPerWarp], hi[kPerWarp];
#pragma unroll
    for (int b = 0; b < kPerWarp; ++b) {
      const uint32_t i = (warp * kPerWarp + b) * 32 + lane;
      lo[b] = hi[b] = 0u;
      if (i < cnt_items) {
        const uint32_t q = __ldcg(a.cols + beg + i);
        lo[b] = q & 0xffu;
        hi[b] = (q >> 8) + 1u;
        s.pay[i] = __ldcg(a.segs + beg + i);
      }
    }
    // per column, as differences: [0] segments in the row (low half) and in
    // its tiles before this one (high half), [1] in this tile
    if (t <= kMaxBins) s_d[t][0] = s_d[t][1] = 0;
    __syncthreads();
    for (uint32_t p = s_seg[r] + t; p < s_seg[r + 1]; p += kThreads) {
      const uint32_t q = __ldcg(a.cols + p), c0 = q & 0xffu, c1 = (q >> 8) + 1u;
      const int one = p < beg ? 0x10001 : 1;
      atomicAdd(&s_d[c0][0], one);
      atomicAdd(&s_d[c1][0], -one);
      if (p - beg < cnt_items) {
        atomicAdd(&s_d[c0][1], 1);
        atomicAdd(&s_d[c1][1], -1);
      }
    }
    __syncthreads();
    uint32_t both = t < kMaxBins ? static_cast<uint32_t>(s_d[t][0]) : 0u;
    uint32_t cnt = t < kMaxBins ? static_cast<uint32_t>(s_d[t][1]) : 0u;
    block_incl_scan2<kWarps>(both, cnt, s_w32);
    const uint32_t total = t < gx ? both & 0xffffu : 0u, before = both >> 16;
    if (t >= gx) cnt = 0u;
    unsigned long long in0 = total, in1 = cnt;
    block_incl_scan2<kWarps>(in0, in1, s_w);
    const uint32_t start = s_pair[r] + static_cast<uint32_t>(in0) - total, lstart = static_cast<uint32_t>(in1) - cnt;
    if (t < kBinsP) {
      s.lstart[t] = lstart;
      s.off[t] = start + before - lstart;
    }
    if (t == kThreads - 1) s.lstart[kBinsP] = static_cast<uint32_t>(in1);
    if (k0 == 0 && t < gx) a.ranges[r * gx + t] = total ? make_uint2(start, start + total) : make_uint2(0u, 0u);
    __syncthreads();
    split_tile<2, kWords>(s, a, lo, hi, gx, r * gx);
  }
}

// ---------------------------------------------------------------- host side
template <int kWords>
cudaError_t launch_small_form(const SplitArgs& a, uint32_t tiles, cudaStream_t s) {
  const size_t smem = sizeof(Smem<kWords>);
  const void* fn = reinterpret_cast<const void*>(&k_small<kWords>);
  const uint32_t resident = radix::resident_ctas(radix::Kernel{fn, 0, kThreads, 0, smem, 1});
  if (resident == 0) return cudaErrorInvalidConfiguration;
  SplitArgs args = a;
  void* params[] = {(void*)&args};
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(tiles < resident ? tiles : resident);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelExC(&cfg, fn, params);
}

template <int kLevel, int kWords>
cudaError_t launch_split_form(const SplitArgs& a, uint32_t tiles, int ctas_per_sm, cudaStream_t s) {
  const size_t smem = sizeof(Smem<kWords>);
  const radix::Kernel k{reinterpret_cast<const void*>(&k_split<kLevel, kWords>), 0, kThreads, 0, smem, 4};
  const uint32_t resident = radix::resident_ctas(k, ctas_per_sm);
  if (resident == 0) return cudaErrorInvalidConfiguration;
  return launch_after(k_split<kLevel, kWords>, tiles < resident ? tiles : resident, kThreads, smem, s, a);
}

template <int kLevel>
cudaError_t launch_split(const SplitArgs& a, uint32_t bins, uint32_t tiles, int ctas_per_sm, cudaStream_t s) {
  // an odd number of words keeps the lanes' consecutive bins in different banks
  if (bins <= 32) return launch_split_form<kLevel, 1>(a, tiles, ctas_per_sm, s);
  if (bins <= 64) return launch_split_form<kLevel, 2>(a, tiles, ctas_per_sm, s);
  if (bins <= 96) return launch_split_form<kLevel, 3>(a, tiles, ctas_per_sm, s);
  if (bins <= 160) return launch_split_form<kLevel, 5>(a, tiles, ctas_per_sm, s);
  if (bins <= 224) return launch_split_form<kLevel, 7>(a, tiles, ctas_per_sm, s);
  return launch_split_form<kLevel, 9>(a, tiles, ctas_per_sm, s);
}

}  // namespace split

cudaError_t launch_small_split(const SplitArgs& a, uint32_t max_bins, uint32_t max_tiles, cudaStream_t s) {
  if (!a.vt.one.on || a.ntiles1 == 0) return cudaErrorInvalidValue;
  const uint32_t tiles = a.ntiles1 > max_tiles ? a.ntiles1 : max_tiles;
  if (max_bins <= 64) return split::launch_small_form<2>(a, tiles, s);
  if (max_bins <= 96) return split::launch_small_form<3>(a, tiles, s);
  if (max_bins <= 160) return split::launch_small_form<5>(a, tiles, s);
  return split::launch_small_form<9>(a, tiles, s);
}
cudaError_t launch_row_count(const SplitArgs& a, cudaStream_t s) {
  if (a.ntiles1 == 0) return cudaSuccess;
  return launch_after(split::k_row_count, a.ntiles1, split::kCountThreads, 0, s, a);
}
cudaError_t launch_row_scan(const SplitArgs& a, cudaStream_t s) {
  return launch_after(split::k_row_scan, a.nrows, split::kCountThreads, 0, s, a);
}
cudaError_t launch_row_split(const SplitArgs& a, uint32_t max_rows, int ctas_per_sm, cudaStream_t s) {
  if (a.ntiles1 == 0) return cudaSuccess;
  return split::launch_split<1>(a, max_rows, a.ntiles1, ctas_per_sm, s);
}
cudaError_t launch_col_count(const SplitArgs& a, uint32_t max_tiles, cudaStream_t s) {
  if (max_tiles == 0) return cudaSuccess;
  const uint32_t cap = 152u * 8u;
  return launch_after(split::k_col_count, max_tiles < cap ? max_tiles : cap, split::kCountThreads, 0, s, a);
}
cudaError_t launch_col_scan(const SplitArgs& a, cudaStream_t s) {
  return launch_after(split::k_col_scan, a.nrows, split::kScanThreads, 0, s, a);
}
cudaError_t launch_col_split(const SplitArgs& a, uint32_t max_cols, uint32_t max_tiles, int ctas_per_sm,
                             cudaStream_t s) {
  if (max_tiles == 0) return cudaSuccess;
  return split::launch_split<2>(a, max_cols, max_tiles, ctas_per_sm, s);
}

}  // namespace tdgs
