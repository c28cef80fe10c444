// Rendering (Sec. II-A "Rendering"; Sec. IV-C "Efficient Tile-Based
// Rendering"): one thread block per 16x16 tile blends the tile's sorted
// Gaussians front to back into every pixel, one pixel per thread, with the
// three colour channels unrolled.  The paper gives each thread four pixels so
// one Gaussian fetch serves four SIMD lanes; on this GPU one pixel per thread
// (256 threads per tile) measured fastest -- 0.44 / 0.36 / 0.34 ms for 4 / 2 /
// 1 pixels per thread on the 1280x720 frame of the 500k scene -- because tiles
// with many Gaussians set the kernel's end and more threads per tile finish
// them sooner.
//
// Further measures:
//  * tiles run heaviest first when they take more than one wave of
//    resident blocks.  A one-block kernel buckets the tiles by their
//    Gaussian count (64 buckets, descending) and block b renders the b-th
//    tile of that order, so the long tiles start in the first wave instead
//    of setting the end of the last one (longest-processing-time list
//    scheduling).  The order inside a bucket comes from shared-memory
//    atomics and may differ between calls; no pixel depends on it.  Images
//    whose tiles all fit in one wave render in raster order without it.
//  * the staged conic is stored as (-a/2, -b, -c/2), so the exponent is
//    dx (A dx + B dy) + C dy^2 in five operations; each staged Gaussian is
//    two 16-byte shared-memory words, read with two loads per step; the
//    blend loop is unrolled eight times (242 -> 231 us against four; two
//    pixels per thread measured 243-265 us).  A finished pixel keeps
//    testing its flag each step: letting it run on with T = 0 instead made
//    whole finished warps do every step's arithmetic (361 against 241 us).
//  * culling per warp: a Gaussian reaches a pixel only inside the ellipse
//    where power >= cut, so when it is staged, its thread marks the warps the
//    ellipse can reach, with a margin; each warp then blends only the list of
//    staged Gaussians that reach it, kept in front-to-back order by one ballot
//    per 32.  What a warp skips is what its pixels' own cut test would have
//    skipped, so the image is unchanged.  A warp's pixels are 8 x 4: an
//    ellipse of w x h pixels meets (w + 8)(h + 4) / 32 warps on average,
//    against (w + 16)(h + 2) / 32 for rows of 16 x 2.  With the list holding
//    byte offsets, the colour one 16-byte word and stopped warps leaving the
//    batch, a render call went 266 -> 222 us (500k Gaussians, 1280x720), 135 ->
//    112 (300k, 640x360) and 517 -> 441 (700k, 3840x2160).  The bound of 6
//    blocks per SM holds the kernel at 40 registers (64 without it: 242, 122
//    and 524 us); 8 blocks spill and measure the same.
//  * the order kernel keeps its tiles' counts in registers.
//
// Per pixel (sample point = the pixel's integer coordinate), in float32
// with CUDA's fast exponential and multiply-adds (the result is compared
// with the oracle's blend within a tolerance):
//   d = mean - pixel; power = -0.5 (a dx^2 + c dy^2) - b dx dy
//   skip if power > 0; alpha = min(0.99, opacity exp(power));
//   skip if alpha < 1/255; T' = T (1 - alpha); stop if T' < 1e-4;
//   C += rgb alpha T; T = T'
// and the pixel is C + T background.  The block stops fetching when all
// its pixels have stopped.
#include "render.cuh"
#include "tdgs_internal.cuh"

namespace tdgs {

namespace {

constexpr int kRenderThreads = 256;             // one 16x16 tile per block, one pixel per thread
constexpr int kOrderThreads = 1024;             // the tile-order kernel's one block
constexpr uint32_t kOrderBuckets = 64;          // Gaussian-count buckets, heaviest first
static_assert(kOrderBuckets == 64, "the bucket scan takes two counts per lane of one warp");

constexpr int kRenderWarps = kRenderThreads / 32;
static_assert(kRenderWarps <= 8, "one bit per warp in an 8-bit mask");

__device__ __forceinline__ uint32_t tile_len(uint2 r) { return r.y > r.x ? r.y - r.x : 0u; }

// Pixels of a warp: 8 x 4, two warps across the tile and four down.
constexpr int kWarpW = 8, kWarpH = 4;
static_assert(kWarpW * kWarpH == 32 && 2 * kWarpW == 16 && 4 * kWarpH == 16, "eight warps cover the tile");

// Warps of the tile a staged Gaussian can reach (bit w: warp w, whose pixels
// are columns 8 (w & 1) .. + 7 and rows 4 (w >> 1) .. + 3 of the tile).  A
// pixel passes the cut test only inside the ellipse d^T Q d <= K, K = -2 cut,
// where Q = [[a, b], [b, c]] is the conic; its squared half-extents are
// K a / det in y and K c / det in x (det = ac - b^2).  A warp is left out
// when all its rows, or all its columns, lie farther from the mean than 1.01
// half-extents plus a quarter pixel (tested on squares).  det comes from one
// fused multiply-add (relative error below 6e-5 when det > 1e-3 ac, inside
// the 1 %); with |cut| <= ln 255 and the terms of the exponent below
// sqrt(ac / det) K, float rounding moves the cut boundary by about 1e-3 pixel
// at most, inside the quarter pixel.  With `ellipse`, a warp is also left out
// when the ellipse d^T Q d <= 1.0201 K misses its rectangle grown by a quarter
// pixel: the least d^T Q d over the rectangle lies on the edges that face the
// mean, at the edge's own minimum or its nearer corner.  That costs the
// staging thread 110 instructions, so only tiles of more than one batch take
// it (render of 700k Gaussians: 400x300 88 -> 84 us, 20k at 320x180 29 -> 27,
// but 4K with 86 Gaussians a tile 455 -> 467).  Flatter conics, Q not positive
// definite or not finite, and means that are no number reach every warp (the
// exponent of such a mean is no number either, which no test of a pixel
// leaves out; the clamps here would take it for a coordinate).  K < 0: no
// pixel passes the cut test (no warp).
__device__ __forceinline__ uint32_t warp_mask(float mx, float my, float4 c, float cut, float tx0, float ty0,
                                              bool ellipse) {
  const float K = -2.0f * cut;
  if (K < 0.0f) return 0u;
  const uint32_t all = (1u << kRenderWarps) - 1u;
  const float ac = c.x * c.z;
  const float det = fmaf(-c.y, c.y, ac);
  if (!(c.x > 0.0f && c.z > 0.0f && det > 1e-3f * ac && K < 1e30f)) return all;
  if (isnan(mx) || isnan(my)) return all;
  const float hy2 = __fdividef(K * c.x, det) * 1.0201f;
  const float hx2 = __fdividef(K * c.z, det) * 1.0201f;
  if (!(hy2 < 1e30f && hx2 < 1e30f)) return all;
  const float xr = mx - tx0, yr = my - ty0;  // the mean inside the tile
  uint32_t columns = 0, m = 0;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const float c0 = static_cast<float>(kWarpW * h);
    const float ex = fmaxf(fmaxf(c0 - xr, xr - (c0 + (kWarpW - 1.0f))) - 0.25f, 0.0f);
    if (ex * ex <= hx2) columns |= 1u << h;
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float r0 = static_cast<float>(kWarpH * q);
    const float ey = fmaxf(fmaxf(r0 - yr, yr - (r0 + (kWarpH - 1.0f))) - 0.25f, 0.0f);
    if (ey * ey <= hy2) m |= columns << (2 * q);
  }
  if (!ellipse) return m;
  const float bc = __fdividef(-c.y, c.z), ba = __fdividef(-c.y, c.x), K2 = K * 1.0201f;
#pragma unroll
  for (int w = 0; w < kRenderWarps; ++w) {
    const float x0 = static_cast<float>(kWarpW * (w & 1)) - 0.25f - xr, x1 = x0 + (kWarpW - 1.0f) + 0.5f;
    const float y0 = static_cast<float>(kWarpH * (w >> 1)) - 0.25f - yr, y1 = y0 + (kWarpH - 1.0f) + 0.5f;
    const float xe = fminf(fmaxf(0.0f, x0), x1), ye = fminf(fmaxf(0.0f, y0), y1);
    const float ys = fminf(fmaxf(bc * xe, y0), y1), xs = fminf(fmaxf(ba * ye, x0), x1);
    const float q1 = fmaf(xe, fmaf(c.x, xe, 2.0f * c.y * ys), c.z * ys * ys);
    const float q2 = fmaf(xs, fmaf(c.x, xs, 2.0f * c.y * ye), c.z * ye * ye);
    if (fminf(q1, q2) > K2) m &= ~(1u << w);
  }
  return m;
}

// order[0 .. tiles) = every tile once, by descending bucket of its
// Gaussian count: bucket = (max - len) * 63 / max in float (0 when every tile
// is empty).  Positions come from the exclusive bucket scan, so they are a
// permutation of 0 .. tiles-1.
__global__ void __launch_bounds__(kOrderThreads)
    k_render_order(const uint2* ranges, uint32_t tiles, uint32_t* __restrict__ order) {
  begin_launch();
  __shared__ uint32_t s_max[kOrderThreads / 32];
  __shared__ uint32_t s_cnt[kOrderBuckets];
  const uint32_t t = threadIdx.x;
  // the first tiles of each thread stay in registers; images above 8192
  // tiles read the rest again
  constexpr uint32_t kHeld = 8;
  uint32_t held[kHeld];
  uint32_t mx = 0;
#pragma unroll
  for (uint32_t k = 0; k < kHeld; ++k) {
    const uint32_t i = t + k * kOrderThreads;
    held[k] = i < tiles ? tile_len(ranges[i]) : 0u;
    mx = max(mx, held[k]);
  }
  for (uint32_t i = t + kHeld * kOrderThreads; i < tiles; i += kOrderThreads) mx = max(mx, tile_len(ranges[i]));
  mx = __reduce_max_sync(0xffffffffu, mx);
  if ((t & 31) == 0) s_max[t >> 5] = mx;
  if (t < kOrderBuckets) s_cnt[t] = 0;
  __syncthreads();
  mx = 0;
#pragma unroll
  for (int w = 0; w < kOrderThreads / 32; ++w) mx = max(mx, s_max[w]);
  const float scale = mx ? static_cast<float>(kOrderBuckets - 1) / static_cast<float>(mx) : 0.0f;
  auto bucket = [mx, scale](uint32_t len) -> uint32_t {
    return min(static_cast<uint32_t>(static_cast<float>(mx - len) * scale), kOrderBuckets - 1);
  };
#pragma unroll
  for (uint32_t k = 0; k < kHeld; ++k)
    if (t + k * kOrderThreads < tiles) atomicAdd(&s_cnt[bucket(held[k])], 1u);
  for (uint32_t i = t + kHeld * kOrderThreads; i < tiles; i += kOrderThreads)
    atomicAdd(&s_cnt[bucket(tile_len(ranges[i]))], 1u);
  __syncthreads();
  if (t < 32) {  // exclusive scan of the 64 bucket counts: two per lane
    const uint32_t c0 = s_cnt[2 * t], c1 = s_cnt[2 * t + 1];
    uint32_t incl = c0 + c1;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t o = __shfl_up_sync(0xffffffffu, incl, d);
      if (static_cast<int>(t) >= d) incl += o;
    }
    const uint32_t excl = incl - c0 - c1;
    s_cnt[2 * t] = excl;
    s_cnt[2 * t + 1] = excl + c0;
  }
  __syncthreads();
#pragma unroll
  for (uint32_t k = 0; k < kHeld; ++k)
    if (t + k * kOrderThreads < tiles) order[atomicAdd(&s_cnt[bucket(held[k])], 1u)] = t + k * kOrderThreads;
  for (uint32_t i = t + kHeld * kOrderThreads; i < tiles; i += kOrderThreads)
    order[atomicAdd(&s_cnt[bucket(tile_len(ranges[i]))], 1u)] = i;
}


__global__ void __launch_bounds__(kRenderThreads, 6)
    k_render(const float4* rec, const float4* conic, const float* rgb,
             const uint32_t* values, const uint2* ranges,
             const uint32_t* order, uint32_t gx, uint32_t width,
             uint32_t height, float3 bg, uint32_t n, float* __restrict__ image, uint32_t* err) {
  // staged Gaussians, two 16-byte loads per step: (x, y, cut, -c/2) and
  // (-a/2, -b, opacity, -); cut = the exponent below which alpha < 1/255; a
  // third one, the colour, for the pixels that blend it
  __shared__ float4 s_g0[kRenderThreads];
  __shared__ float4 s_g1[kRenderThreads];
  __shared__ float4 s_rgb[kRenderThreads];
  __shared__ uint8_t s_mask[kRenderThreads];                 // warps each staged Gaussian reaches
  __shared__ uint16_t s_list[kRenderWarps][kRenderThreads];  // per warp: staged Gaussians to blend, as byte offsets
  begin_launch();
  const uint32_t tile = order ? order[blockIdx.x] : blockIdx.x, t = threadIdx.x;
  const uint32_t warp = t >> 5, lane = t & 31;
  const uint32_t tx = (tile % gx) * 16, ty = (tile / gx) * 16;
  const uint32_t px = tx + (warp & 1) * kWarpW + (lane % kWarpW);
  const uint32_t py = ty + (warp >> 1) * kWarpH + lane / kWarpW;
  const float fx = __uint2float_rn(px), fy = __uint2float_rn(py);
  float T = 1.0f, C[3] = {0.0f, 0.0f, 0.0f};
  bool done = !(px < width && py < height);
  const uint2 r = ranges[tile];
  bool bad = false;
  const bool ellipse = tile_len(r) > kRenderThreads;
  for (uint32_t b = r.x; b < r.y; b += kRenderThreads) {
    if (__syncthreads_count(done) == kRenderThreads) break;
    const uint32_t idx = b + t;
    if (idx < r.y) {
      uint32_t g = values[idx];
      if (g >= n) {  // not an index of this frame: skipped and reported
        bad = true;
        s_g0[t] = make_float4(0.f, 0.f, __int_as_float(0x7f800000), 0.f);
        s_g1[t] = make_float4(0.f, 0.f, 0.f, 0.f);
        s_mask[t] = 0;
        s_rgb[t] = make_float4(0.f, 0.f, 0.f, 0.f);
      } else {
        const float4 q = __ldca(rec + g);
        const float4 c = __ldca(conic + g);
        // opacity * exp(power) < 1/255 exactly when power < -ln(255 opacity):
        // far pixels skip the exponential (the 1/255 test below stays)
        const float cut = c.w > 0.0f ? -__logf(255.0f * c.w) : __int_as_float(0x7f800000);
        s_g0[t] = make_float4(q.x, q.y, cut, -0.5f * c.z);
        s_g1[t] = make_float4(-0.5f * c.x, -c.y, c.w, 0.f);
        s_mask[t] = static_cast<uint8_t>(warp_mask(q.x, q.y, c, cut, __uint2float_rn(tx), __uint2float_rn(ty),
                                                 ellipse));
        s_rgb[t] = make_float4(__ldca(rgb + 3 * static_cast<size_t>(g)), __ldca(rgb + 3 * static_cast<size_t>(g) + 1),
                               __ldca(rgb + 3 * static_cast<size_t>(g) + 2), 0.f);
      }
    }
    __syncthreads();
    if (__all_sync(0xffffffffu, done)) continue;  // this warp's pixels have stopped
    const uint32_t cnt = min(static_cast<uint32_t>(kRenderThreads), r.y - b);
    // this warp's list of the staged Gaussians that can reach its pixels
    uint32_t nw = 0;
#pragma unroll
    for (uint32_t k = 0; k < kRenderThreads / 32; ++k) {
      const uint32_t e = k * 32 + lane;
      const bool hit = e < cnt && ((s_mask[e] >> warp) & 1u);
      const uint32_t bal = __ballot_sync(0xffffffffu, hit);
      if (hit) s_list[warp][nw + __popc(bal & ((1u << lane) - 1u))] = static_cast<uint16_t>(e * sizeof(float4));
      nw += __popc(bal);
    }
    __syncwarp();
    const char* g0p = reinterpret_cast<const char*>(s_g0);
    const char* g1p = reinterpret_cast<const char*>(s_g1);
    const char* cp = reinterpret_cast<const char*>(s_rgb);
#pragma unroll 8
    for (uint32_t jj = 0; jj < nw; ++jj) {
      const uint32_t at = s_list[warp][jj];
      const float4 g0 = *reinterpret_cast<const float4*>(g0p + at);
      const float4 g1 = *reinterpret_cast<const float4*>(g1p + at);
      if (done) continue;
      const float dx = g0.x - fx, dy = g0.y - fy;
      const float power = fmaf(dx, fmaf(g1.x, dx, g1.y * dy), g0.w * dy * dy);
      if (power > 0.0f || power < g0.z) continue;
      const float alpha = fminf(0.99f, g1.z * __expf(power));
      if (alpha < 1.0f / 255.0f) continue;
      const float test_t = T * (1.0f - alpha);
      if (test_t < 0.0001f) {
        done = true;
        continue;
      }
      const float w = alpha * T;
      const float4 col = *reinterpret_cast<const float4*>(cp + at);
      C[0] += col.x * w;
      C[1] += col.y * w;
      C[2] += col.z * w;
      T = test_t;
    }
  }
  if (__any_sync(0xffffffffu, bad) && lane == 0) latch_error(err, TDGS_ERR_INVALID_ARGUMENT, kSiteRender);
  if (px < width && py < height) {
    float* o = image + 3 * (static_cast<size_t>(py) * width + px);
    o[0] = C[0] + T * bg.x;
    o[1] = C[1] + T * bg.y;
    o[2] = C[2] + T * bg.z;
  }
}

}  // namespace

cudaError_t launch_render_order(const uint2* ranges, uint32_t tiles, uint32_t* order, cudaStream_t s) {
  if (tiles == 0) return cudaSuccess;
  return launch_after(k_render_order, 1, kOrderThreads, 0, s, ranges, tiles, order);
}

cudaError_t launch_render_ordered(const float4* rec, const float4* conic, const float* rgb, const uint32_t* values,
                                  const uint2* ranges, const uint32_t* order, uint32_t width, uint32_t height,
                                  const float* bg, uint32_t n, float* image, uint32_t* err, cudaStream_t s) {
  const uint32_t gx = (width + 15) / 16, gy = (height + 15) / 16;
  const uint32_t tiles = gx * gy;
  if (tiles == 0) return cudaSuccess;
  return launch_after(k_render, tiles, kRenderThreads, 0, s, rec, conic, rgb, values, ranges, order, gx, width, height,
                      make_float3(bg[0], bg[1], bg[2]), n, image, err);
}

cudaError_t launch_render(const float4* rec, const float4* conic, const float* rgb, const uint32_t* values,
                          const uint2* ranges, uint32_t width, uint32_t height, const float* bg, uint32_t n,
                          float* image, uint32_t* err, cudaStream_t s) {
  return launch_render_ordered(rec, conic, rgb, values, ranges, nullptr, width, height, bg, n, image, err, s);
}

uint32_t render_wave_blocks(int device) {
  int sms = 0, per_sm = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) return 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_render, kRenderThreads, 0) != cudaSuccess) return 0;
  return static_cast<uint32_t>(sms) * static_cast<uint32_t>(per_sm);
}

}  // namespace tdgs
