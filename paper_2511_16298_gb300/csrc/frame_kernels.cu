// Per-frame kernels: tile count, exclusive scan, pair duplication and tile
// ranges (Sec. II-A "Duplication with Tiles"; Table III PrefixSum and
// DuplicateWithTile; Table VI Scan / Duplicate with tiles / Identify Range).
#include "tdgs_internal.cuh"

namespace tdgs {

// ------------------------------------------------------------ tile count
// One Gaussian per thread; one 128-bit load per record (Table IV packs the
// mean, depth and radius into one 16-byte record for exactly this read).
__global__ void __launch_bounds__(256) k_count_tiles(const float4* g, uint32_t n,
                                                     FrameGeom fg, uint32_t* __restrict__ counts,
                                                     uint32_t* err) {
  begin_launch();
  bool bad = false;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i = next_of(i, gridDim.x * blockDim.x, n)) {
    const TileRect q = tile_rect(__ldca(g + i), fg);
    bad |= q.invalid;
    counts[i] = q.count;
  }
  if (__any_sync(0xffffffffu, bad) && lane_id() == 0) latch_error(err, TDGS_ERR_INVALID_ARGUMENT, kSiteCount);
}

cudaError_t launch_count_tiles(const float4* g, uint32_t n, FrameGeom fg, uint32_t* counts,
                               uint32_t* err, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const uint32_t blocks = ceil_div(n, 256);
  const uint32_t grid = blocks < 152u * 16u ? blocks : 152u * 16u;
  return launch_after(k_count_tiles, grid, 256, 0, s, g, n, fg, counts, err);
}

// --------------------------------------------------------- exclusive scan
// Single-pass scan with decoupled look-back (Merrill & Garland, 2016).
// Each block takes the next tile of 8192 items from a ticket counter (so
// every predecessor tile is already running or done), publishes its
// aggregate, then walks back over its predecessors' status words 32 at a
// time until it meets an inclusive prefix.  Status word: bits 63-62 flag
// (1 = aggregate, 2 = inclusive prefix), bits 61-0 value.  Sums are 64-bit
// so that an overflow of the 32-bit offsets is detected, not wrapped.
namespace {
constexpr int kScanThreads = 256;
constexpr int kScanItems = kScanTileItems / kScanThreads;  // 32
constexpr uint64_t kFlagA = 1ull << 62;
constexpr uint64_t kFlagP = 2ull << 62;
constexpr uint64_t kValMask = (1ull << 62) - 1;

__host__ __device__ constexpr uint32_t spad(uint32_t p) { return p + (p >> 5); }

__device__ __forceinline__ uint64_t warp_incl_scan64(uint64_t v) {
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint64_t o = __shfl_up_sync(0xffffffffu, v, d);
    if (lane_id() >= static_cast<uint32_t>(d)) v += o;
  }
  return v;
}
}  // namespace

// kMode 0: counts[i]; 1: counts computed from recs[i]; 2: counts[gather[i]].
template <int kMode>
__global__ void __launch_bounds__(kScanThreads)
    k_scan(const uint32_t* counts, const float4* recs,
           const uint32_t* gather, FrameGeom fg, uint32_t n,
           uint32_t* __restrict__ offsets, uint64_t* status, uint32_t* ticket,
           uint32_t ticket_base, uint64_t* total64, uint32_t* total32, uint32_t* err) {
  constexpr bool kFromRecords = kMode == 1;
  __shared__ uint32_t s_items[spad(kScanTileItems) + 1];
  __shared__ uint64_t s_warp[kScanThreads / 32];
  __shared__ uint64_t s_excl;
  __shared__ uint32_t s_tile;
  begin_launch();
  const uint32_t t = threadIdx.x;
  const uint32_t lane = lane_id();
  const uint32_t warp = t >> 5;
  if (t == 0) s_tile = atomicAdd(ticket, 1u) - ticket_base;
  __syncthreads();
  const uint32_t tile = s_tile;
  const uint64_t base = static_cast<uint64_t>(tile) * kScanTileItems;

  // Coalesced (striped) load of the tile's counts, transposed through
  // shared memory to a blocked layout for the per-thread serial scan.
  bool bad = false;
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    const uint32_t p = j * kScanThreads + t;
    const uint64_t idx = base + p;
    uint32_t v = 0;
    if (idx < n) {
      if constexpr (kMode == 1) {
        const TileRect q = tile_rect(__ldca(recs + idx), fg);
        bad |= q.invalid;
        v = q.count;
      } else if constexpr (kMode == 2) {
        v = __ldca(counts + __ldca(gather + idx));
      } else {
        v = __ldca(counts + idx);
      }
    }
    s_items[spad(p)] = v;
  }
  if (kFromRecords && __any_sync(0xffffffffu, bad) && lane == 0)
    latch_error(err, TDGS_ERR_INVALID_ARGUMENT, kSiteScan);
  __syncthreads();
  uint32_t mine[kScanItems];
  uint64_t tsum = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    mine[k] = s_items[spad(t * kScanItems + k)];
    tsum += mine[k];
  }
  const uint64_t winc = warp_incl_scan64(tsum);
  if (lane == 31) s_warp[warp] = winc;
  __syncthreads();
  if (warp == 0) {
    uint64_t w = lane < kScanThreads / 32 ? s_warp[lane] : 0;
    w = warp_incl_scan64(w);
    if (lane < kScanThreads / 32) s_warp[lane] = w;  // inclusive warp totals
  }
  __syncthreads();
  const uint64_t agg = s_warp[kScanThreads / 32 - 1];
  const uint64_t texcl = winc - tsum + (warp ? s_warp[warp - 1] : 0);

  // Look-back by warp 0.
  if (warp == 0) {
    uint64_t excl = 0;
    if (tile == 0) {
      if (lane == 0) st_release(status, kFlagP | (agg & kValMask));
    } else {
      if (lane == 0) st_release(status + tile, kFlagA | (agg & kValMask));
      int64_t k = static_cast<int64_t>(tile) - 1;
      uint32_t spins = 0;
      while (true) {
        const int64_t kk = k - lane;
        uint64_t s = kk >= 0 ? ld_acquire(status + kk) : kFlagP;
        while (__any_sync(0xffffffffu, (s >> 62) == 0)) {
          if (++spins > kSpinLimit) break;
          if ((s >> 62) == 0) {
            __nanosleep(32);
            s = ld_acquire(status + kk);
          }
        }
        if (spins > kSpinLimit) {
          if (lane == 0) latch_error(err, TDGS_ERR_TIMEOUT, kSiteScanTimeout);
          break;
        }
        const uint32_t pmask = __ballot_sync(0xffffffffu, (s >> 62) == 2);
        const uint32_t stop = pmask ? __ffs(pmask) - 1 : 31;
        uint64_t v = lane <= stop ? (s & kValMask) : 0;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
        excl += v;
        if (pmask) break;
        k -= 32;
      }
      if (lane == 0) st_release(status + tile, kFlagP | ((excl + agg) & kValMask));
    }
    if (lane == 0) s_excl = excl;
  }
  __syncthreads();
  const uint64_t tile_excl = s_excl;
  const uint64_t incl_end = tile_excl + agg;
  if (incl_end > 0xffffffffull && t == 0) latch_error(err, TDGS_ERR_OVERFLOW, kSiteScan);
  uint64_t run = tile_excl + texcl;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    s_items[spad(t * kScanItems + k)] = static_cast<uint32_t>(run);
    run += mine[k];
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    const uint32_t p = j * kScanThreads + t;
    const uint64_t idx = base + p;
    if (idx < n) offsets[idx] = s_items[spad(p)];
  }
  if (t == 0 && base + kScanTileItems >= n) {  // last tile writes the total
    if (total64) *total64 = incl_end;
    if (total32) *total32 = incl_end > 0xffffffffull ? 0xffffffffu : static_cast<uint32_t>(incl_end);
  }
}

cudaError_t launch_scan(const uint32_t* counts, const float4* recs, const uint32_t* gather,
                        FrameGeom fg, uint32_t n, uint32_t* offsets, uint64_t* status,
                        uint32_t* ticket, uint32_t ticket_base, uint64_t* total64,
                        uint32_t* total32, uint32_t* err, cudaStream_t s) {
  const uint32_t tiles = ceil_div(n, kScanTileItems);
  if (tiles == 0) return cudaSuccess;
  const auto fn = recs ? k_scan<1> : gather ? k_scan<2> : k_scan<0>;
  return launch_after(fn, tiles, kScanThreads, 0, s, counts, recs, gather, fg, n, offsets, status, ticket, ticket_base,
                      total64, total32, err);
}

// ------------------------------------------------------------- duplicate
// Load-balanced expansion.  A warp owns 32 consecutive Gaussians; their
// pairs occupy one contiguous output range (their offsets are consecutive
// in the scan).  The warp walks that range 32 pairs at a time, lane l taking
// pair p = step + l.  The Gaussians with pairs lie compacted in shared memory;
// those that start inside the step are one word of bits (one warp OR), so the
// owner of a pair is a population count, not a search.  (ty, tx) come from the
// local index by a float reciprocal with one exact correction step.  Every
// store is a fully coalesced 256-byte (keys) / 128-byte (values) run.
// kNorm: the paper's 32-bit key (Sec. IV-B), tile << 10 | q with q the
// depth normalised to 2^10 over the visible range norm[0..1] (float bits).
struct DupOwner {
  uint32_t start, first, w;  // first pair (relative), first tile, columns
  float rw;                  // 1 / columns
};
template <bool kNorm>
__global__ void __launch_bounds__(256)
    k_duplicate(const float4* g, const uint32_t* offsets, uint32_t n,
                FrameGeom fg, void* __restrict__ keys_raw, uint32_t* __restrict__ values,
                uint32_t cap, const uint32_t* norm, uint32_t* err) {
  __shared__ __align__(16) DupOwner s_owner[8][32];
  __shared__ uint2 s_pay[8][32];  // low key word, index
  begin_launch();
  float dmin = 0.0f, scale = 0.0f;
  if constexpr (kNorm) {
    dmin = __uint_as_float(norm[0]);
    scale = norm_scale(dmin, __uint_as_float(norm[1]));
  }
  const uint32_t lane = lane_id(), w8 = threadIdx.x >> 5;
  const uint32_t lt = lanemask_lt(), le = lt | (1u << lane);
  const uint32_t warps_total = (gridDim.x * blockDim.x) >> 5;
  const uint32_t gx = static_cast<uint32_t>(fg.gx);
  bool bad = false, over = false;
  for (uint32_t wg = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
       static_cast<uint64_t>(wg) * 32u < n; wg += warps_total) {
    const uint32_t i = wg * 32u + lane;
    TileRect q;
    q.x0 = q.y0 = q.x1 = q.y1 = 0;
    q.count = 0;
    uint64_t start = 0;
    uint32_t low = 0;
    if (i < n) {
      const float4 rec = __ldca(g + i);
      q = tile_rect(rec, fg);
      start = __ldca(offsets + i);
      bad |= q.invalid;
      low = kNorm ? norm_depth(rec.z, dmin, scale) : __float_as_uint(rec.z);
    }
    // the warp's range: from its first Gaussian with pairs to the end of its
    // last one; positions relative to it, in 32 bits, none at or beyond cap
    const uint32_t with = __ballot_sync(0xffffffffu, q.count != 0u);
    if (with == 0u) continue;
    const uint64_t begin = __shfl_sync(0xffffffffu, start, __ffs(with) - 1);
    const uint64_t end = __shfl_sync(0xffffffffu, start + q.count, 31 - __clz(with));
    if (end > cap) over = true;
    const uint64_t stop = end < cap ? end : cap;
    const uint64_t span = stop > begin ? stop - begin : 0;
    const uint32_t nrel = static_cast<uint32_t>(span);  // (cap has 32 bits)
    const uint64_t rel = start - begin;
    const bool mine = q.count != 0u && rel < nrel;
    const uint32_t mask = __ballot_sync(0xffffffffu, mine);
    const uint32_t wd = static_cast<uint32_t>(q.x1 - q.x0);
    __syncwarp();  // the last Gaussians' owners are read
    if (mine) {
      const uint32_t r = __popc(mask & lt);
      s_owner[w8][r] = DupOwner{static_cast<uint32_t>(rel),
                                static_cast<uint32_t>(q.y0) * gx + static_cast<uint32_t>(q.x0), wd,
                                __frcp_rn(static_cast<float>(wd))};
      s_pay[w8][r] = make_uint2(low, i);
    }
    __syncwarp();
    uint32_t seen = 0xffffffffu;  // owners that start before the step, less one
    for (uint64_t p64 = 0; p64 < nrel; p64 += 32) {
      const uint32_t p0 = static_cast<uint32_t>(p64);
      const uint32_t at = static_cast<uint32_t>(rel) - p0;
      const uint32_t starts = __reduce_or_sync(0xffffffffu, mine && at < 32u ? 1u << at : 0u);
      const uint32_t src = (seen + __popc(starts & le)) & 31u;
      seen += __popc(starts);
      const uint32_t p = p0 + lane;
      if (p64 + lane < nrel) {
        const DupOwner o = s_owner[w8][src];
        const uint2 pay = s_pay[w8][src];
        const uint32_t j = p - o.start;
        uint32_t ry, rx;
        if (j < (1u << 22)) {
          ry = __float2uint_rz(__fmul_rn(__uint2float_rn(j), o.rw));
          rx = j - ry * o.w;
          if (static_cast<int32_t>(rx) < 0) {
            --ry;
            rx += o.w;
          } else if (rx >= o.w) {
            ++ry;
            rx -= o.w;
          }
        } else {
          ry = j / o.w;
          rx = j - ry * o.w;
        }
        const uint32_t tile = o.first + ry * gx + rx;
        const uint64_t dst = begin + p;
        if constexpr (kNorm)
          static_cast<uint32_t*>(keys_raw)[dst] = (tile << 10) | pay.x;
        else
          static_cast<uint64_t*>(keys_raw)[dst] = (static_cast<uint64_t>(tile) << 32) | pay.x;
        values[dst] = pay.y;
      }
    }
  }
  if (__any_sync(0xffffffffu, bad) && lane == 0) latch_error(err, TDGS_ERR_INVALID_ARGUMENT, kSiteDuplicate);
  if (__any_sync(0xffffffffu, over) && lane == 0) latch_error(err, TDGS_ERR_CAPACITY, kSiteDuplicate);
}

cudaError_t launch_duplicate(const float4* g, const uint32_t* offsets, uint32_t n,
                             FrameGeom fg, uint64_t* keys, uint32_t* values, uint32_t cap,
                             uint32_t* err, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const uint32_t warps = ceil_div(n, 32);
  const uint32_t blocks = ceil_div(warps, 8);
  const uint32_t grid = blocks < 152u * 32u ? blocks : 152u * 32u;
  return launch_after(k_duplicate<false>, grid, 256, 0, s, g, offsets, n, fg, keys, values, cap, nullptr, err);
}

cudaError_t launch_duplicate_norm(const float4* g, const uint32_t* offsets, uint32_t n, FrameGeom fg,
                                  uint32_t* keys, uint32_t* values, uint32_t cap, const uint32_t* norm,
                                  uint32_t* err, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const uint32_t warps = ceil_div(n, 32);
  const uint32_t blocks = ceil_div(warps, 8);
  const uint32_t grid = blocks < 152u * 32u ? blocks : 152u * 32u;
  return launch_after(k_duplicate<true>, grid, 256, 0, s, g, offsets, n, fg, keys, values, cap, norm, err);
}

// Smallest and largest depth (float bits; positive finite depths order as
// unsigned integers) of the Gaussians with pairs: norm[0] min, norm[1] max
// (all ones / zero on entry).
__global__ void __launch_bounds__(256) k_norm_range(const float4* g, const uint32_t* counts,
                                                    uint32_t n, uint32_t* norm) {
  uint32_t lo = 0xffffffffu, hi = 0u;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i = next_of(i, gridDim.x * blockDim.x, n)) {
    if (__ldca(counts + i)) {
      const uint32_t b = __float_as_uint(__ldca(&g[i].z));
      lo = min(lo, b);
      hi = max(hi, b);
    }
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (lane_id() == 0) {
    if (lo != 0xffffffffu) atomicMin(norm, lo);
    if (hi != 0u) atomicMax(norm + 1, hi);
  }
}

cudaError_t launch_norm_range(const float4* g, const uint32_t* counts, uint32_t n, uint32_t* norm, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const uint32_t blocks = ceil_div(n, 256);
  const uint32_t grid = blocks < 152u * 8u ? blocks : 152u * 8u;
  k_norm_range<<<grid, 256, 0, s>>>(g, counts, n, norm);
  return cudaGetLastError();
}

// Four keys per thread.  The normalised depths are 0 .. 1023 whatever the
// frame, so their range is constant.
__global__ void __launch_bounds__(256) k_norm_keys(uint32_t* __restrict__ keys, uint32_t n,
                                                   const uint32_t* range, uint32_t* __restrict__ out,
                                                   uint32_t* __restrict__ raw) {
  __shared__ uint32_t s_raw[kRawBins + 1];
  begin_launch();
  for (uint32_t i = threadIdx.x; i <= kRawBins; i += blockDim.x) s_raw[i] = 0;
  __syncthreads();
  const float dmin = __uint_as_float(__ldcg(range + 2));
  const float scale = norm_scale(dmin, __uint_as_float(__ldcg(range + 3)));
  const uint32_t first = (blockIdx.x * blockDim.x + threadIdx.x) * 4;
#pragma unroll
  for (uint32_t u = 0; u < 4; ++u) {
    if (first + u < n) {
      const uint32_t k = keys[first + u];
      const uint32_t q = k != 0xffffffffu ? norm_depth(__uint_as_float(k), dmin, scale) : k;
      if (k != 0xffffffffu) keys[first + u] = q;
      if (raw) atomicAdd(&s_raw[k != 0xffffffffu ? q & (kRawBins - 1) : kRawBins], 1u);
    }
  }
  if (raw) {
    __syncthreads();
    for (uint32_t i = threadIdx.x; i <= kRawBins; i += blockDim.x)
      if (s_raw[i]) atomicAdd(raw + i, s_raw[i]);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    out[2] = 0u;
    out[3] = 1023u;
  }
}

cudaError_t launch_norm_keys(uint32_t* keys, uint32_t n, const uint32_t* range, uint32_t* out, uint32_t* raw,
                             cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  return launch_after(k_norm_keys, ceil_div(n, 1024), 256, 0, s, keys, n, range, out, raw);
}

// ---------------------------------------------------------- tile ranges
// Identify Range: where a key's tile differs from the previous key's, the
// previous tile's range ends and this one's starts.  ranges is zeroed
// beforehand, so tiles without pairs stay {0, 0}.  Each key's word with the
// tile is read once; the previous one comes from the lane before (the first
// lane reads it again).
// K, kShift: 64-bit keys with the tile above bit 32, or the 32-bit
// normalised keys with the tile above bit 10.
constexpr int kRangeItems = 4;
template <typename K, int kShift>
__global__ void __launch_bounds__(256) k_tile_ranges(const K* keys, uint32_t m,
                                                     uint32_t num_tiles, uint2* ranges,
                                                     uint32_t* err) {
  begin_launch();
  const uint32_t* words = reinterpret_cast<const uint32_t*>(keys);
  constexpr uint32_t kStep = sizeof(K) / 4, kHigh = sizeof(K) == 8 ? 1 : 0;
  auto tile_of = [&](uint64_t k) { return __ldca(words + k * kStep + kHigh) >> (kShift & 31); };
  const uint32_t lane = lane_id();
  const uint64_t stride = static_cast<uint64_t>(gridDim.x) * blockDim.x * kRangeItems;
  bool bad = false;
  for (uint64_t w0 = (static_cast<uint64_t>(blockIdx.x) * blockDim.x + (threadIdx.x & ~31u)) * kRangeItems; w0 < m;
       w0 += stride) {
    uint32_t t[kRangeItems];
#pragma unroll
    for (int u = 0; u < kRangeItems; ++u) {
      const uint64_t k = w0 + u * 32 + lane;
      t[u] = k < m ? tile_of(k) : 0u;
    }
    uint32_t last = w0 > 0 && lane == 0 ? tile_of(w0 - 1) : 0u;  // the tile before lane 0's
#pragma unroll
    for (int u = 0; u < kRangeItems; ++u) {
      const uint64_t k = w0 + u * 32 + lane;
      uint32_t prev = __shfl_up_sync(0xffffffffu, t[u], 1);
      if (lane == 0) prev = last;
      last = __shfl_sync(0xffffffffu, t[u], 31);
      if (k < m) {
        bad |= t[u] >= num_tiles;
        if (k == 0 || t[u] != prev) {
          if (t[u] < num_tiles) ranges[t[u]].x = static_cast<uint32_t>(k);
          if (k > 0 && prev < num_tiles) ranges[prev].y = static_cast<uint32_t>(k);
        }
        if (k + 1 == m && t[u] < num_tiles) ranges[t[u]].y = m;
      }
    }
  }
  if (__any_sync(0xffffffffu, bad) && lane == 0) latch_error(err, TDGS_ERR_INVALID_ARGUMENT, kSiteRanges);
}

cudaError_t launch_tile_ranges(const uint64_t* keys, uint32_t m, uint32_t num_tiles,
                               uint2* ranges, uint32_t* err, cudaStream_t s) {
  if (m == 0) return cudaSuccess;
  const uint32_t blocks = m / (256 * kRangeItems) + 1;
  const uint32_t grid = blocks < 152u * 16u ? blocks : 152u * 16u;
  return launch_after(k_tile_ranges<uint64_t, 32>, grid, 256, 0, s, keys, m, num_tiles, ranges, err);
}

cudaError_t launch_tile_ranges_norm(const uint32_t* keys, uint32_t m, uint32_t num_tiles, uint2* ranges,
                                    uint32_t* err, cudaStream_t s) {
  if (m == 0) return cudaSuccess;
  const uint32_t blocks = m / (256 * kRangeItems) + 1;
  const uint32_t grid = blocks < 152u * 16u ? blocks : 152u * 16u;
  return launch_after(k_tile_ranges<uint32_t, 10>, grid, 256, 0, s, keys, m, num_tiles, ranges, err);
}

}  // namespace tdgs
