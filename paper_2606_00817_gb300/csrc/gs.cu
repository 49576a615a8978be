// gs.cu -- depth rendered from 3D Gaussians, the cheap supervision source the
// paper compares with clean distances (Sec. 3.2; the study of Sec. 4.2), as a
// tile rasteriser: project every Gaussian (EWA: screen covariance J V C V^T
// J^T plus a 0.3-pixel low-pass), bin it into the 16 x 16-pixel tiles its
// alpha >= 1/255 ellipse touches, then per tile sort the list by depth in
// shared memory and composite front to back, one pixel per thread:
//   alpha = min(0.99, o exp(-q / 2)),  q = dp^T S^-1 dp,
//   D += T alpha z,  A += T alpha,  T *= 1 - alpha  (stop once T < 1e-4),
// giving per pixel the expected distance t = (D / A) / (d . f) along the
// pixel ray and the hit flag A > 0.5. Many views render in one launch each.
//
// Lists: per (view, tile) counts by atomics, one exclusive scan, then a fill
// pass that writes 64-bit keys (depth bits << 32 | Gaussian index) at atomic
// cursors. The order inside a list is arbitrary; the sort by key makes the
// result independent of it (equal depths: lower index first).
#include <cstdint>
#include <cuda_fp16.h>

#include "kernels.h"

namespace ddf {

namespace {

constexpr int kTile = 16;
constexpr int kTilePx = kTile * kTile;  // threads per render block, one pixel each
constexpr int kWin = 2048;              // keys sorted and composited at a time
constexpr int kBuckets = 1024;          // buckets of a tile's list
constexpr int kBucketSort = 128;        // largest bucket sorted by counting
constexpr int kBinThreads = 512;        // (view, Gaussian) pairs per binning block
constexpr int kBinTiles = 4096;         // largest image, in tiles, whose counts fit a block
constexpr float kLowPass = 0.3f;
constexpr float kAlphaMin = 1.f / 255.f;
constexpr float kAlphaMax = 0.99f;
constexpr float kTMin = 1e-4f;
constexpr float kNear = 0.05f;

__device__ __forceinline__ float dot3(const float* a, const float* b) {
  return a[0] * b[0] + a[1] * b[1] + a[2] * b[2];
}

// The screen record of Gaussian g in view v (rec of v n + g) and the rectangle
// of tiles it touches (z < x: none).
__device__ __forceinline__ int4 gs_project_one(const float* __restrict__ means,
                                               const float* __restrict__ covs,
                                               const float* __restrict__ opac, int64_t n,
                                               const GiCamera& c, int v, int64_t g,
                                               float4* __restrict__ rec) {
  const int4 none = make_int4(0, 0, -1, -1);
  const int64_t j = static_cast<int64_t>(v) * n + g;
  const float m[3] = {means[3 * g] - c.eye[0], means[3 * g + 1] - c.eye[1],
                      means[3 * g + 2] - c.eye[2]};
  const float x = dot3(m, c.r), y = dot3(m, c.u), z = dot3(m, c.f);
  const float o = opac[g];
  if (!(z > kNear) || !(o >= kAlphaMin)) return none;
  // square pixels: the focal length in pixels is height / (2 tan(fov_y / 2))
  const float fp = static_cast<float>(c.height) / (2.f * c.tan_half);
  const float iz = 1.f / z;
  const float px = x * iz * fp + 0.5f * static_cast<float>(c.width - 1);
  const float py = -y * iz * fp + 0.5f * static_cast<float>(c.height - 1);
  // rows of J V: d(px)/d(world) and d(py)/d(world)
  float a[3], b[3];
  for (int k = 0; k < 3; ++k) {
    a[k] = fp * iz * (c.r[k] - x * iz * c.f[k]);
    b[k] = -fp * iz * (c.u[k] - y * iz * c.f[k]);
  }
  const float* C = covs + 6 * g;  // xx, xy, xz, yy, yz, zz
  float ca[3], cb[3];
  ca[0] = C[0] * a[0] + C[1] * a[1] + C[2] * a[2];
  ca[1] = C[1] * a[0] + C[3] * a[1] + C[4] * a[2];
  ca[2] = C[2] * a[0] + C[4] * a[1] + C[5] * a[2];
  cb[0] = C[0] * b[0] + C[1] * b[1] + C[2] * b[2];
  cb[1] = C[1] * b[0] + C[3] * b[1] + C[4] * b[2];
  cb[2] = C[2] * b[0] + C[4] * b[1] + C[5] * b[2];
  const float sxx = dot3(a, ca) + kLowPass;
  const float sxy = dot3(a, cb);
  const float syy = dot3(b, cb) + kLowPass;
  const float det = sxx * syy - sxy * sxy;
  if (!(det > 0.f)) return none;
  const float id = 1.f / det;
  // alpha >= 1/255 needs q <= 2 ln(255 o): the ellipse's bounding box, one
  // pixel wider on each side for rounding
  const float kq = 2.f * logf(255.f * o);
  const float hx = sqrtf(fmaxf(kq, 0.f) * sxx) + 1.f;
  const float hy = sqrtf(fmaxf(kq, 0.f) * syy) + 1.f;
  const float fx0 = fmaxf(ceilf(px - hx), 0.f), fx1 = fminf(floorf(px + hx), c.width - 1.f);
  const float fy0 = fmaxf(ceilf(py - hy), 0.f), fy1 = fminf(floorf(py + hy), c.height - 1.f);
  if (!(fx0 <= fx1) || !(fy0 <= fy1)) return none;
  const int tx0 = static_cast<int>(fx0) / kTile, tx1 = static_cast<int>(fx1) / kTile;
  const int ty0 = static_cast<int>(fy0) / kTile, ty1 = static_cast<int>(fy1) / kTile;
  rec[2 * j] = make_float4(px, py, z, o);
  // the box's half sides, rounded up to half precision, for the renderer's
  // warps. Where the rounding of q (about 1e-6 / (1 - correlation^2) of it)
  // could reach past the box's spare pixel, no box: every warp looks.
  const bool sharp = det >= 1e-3f * sxx * syy && hx < 2000.f && hy < 2000.f;
  const float inf = __int_as_float(0x7f800000);
  const __half2 box = __halves2half2(__float2half_ru(sharp ? hx : inf),
                                     __float2half_ru(sharp ? hy : inf));
  rec[2 * j + 1] = make_float4(syy * id, -sxy * id, sxx * id,
                               __int_as_float(*reinterpret_cast<const int*>(&box)));
  return make_int4(tx0, ty0, tx1, ty1);
}

// The view and Gaussian of this thread of a binning block: blocks do not
// straddle views.
struct BinBlock {
  int v;
  int64_t g;  // >= n: none
  __device__ explicit BinBlock(int64_t n) {
    const int64_t per_view = (n + kBinThreads - 1) / kBinThreads;
    v = static_cast<int>(blockIdx.x / per_view);
    g = (blockIdx.x - v * per_view) * kBinThreads + threadIdx.x;
  }
};

// Per (view, Gaussian): the screen record and the rectangle of tiles it
// touches; adds 1 to the count of every tile in it. A block takes kBinThreads
// Gaussians of one view. Neighbours in the list land on the same few dozen
// tiles of the object, so the block counts in shared memory and adds each of
// its tiles to the global count once (LOCAL; 60,000 Gaussians x 32 views of 64
// tiles: 390 us with a global atomic per Gaussian and tile, 34 us so).
template <bool LOCAL>
__global__ void __launch_bounds__(kBinThreads)
gs_project_kernel(const float* __restrict__ means, const float* __restrict__ covs,
                  const float* __restrict__ opac, int64_t n, const GiCamera* __restrict__ cams,
                  int ntx, int nty, float4* __restrict__ rec, int4* __restrict__ rect,
                  unsigned* __restrict__ count) {
  extern __shared__ unsigned s_count[];
  const int ntiles = ntx * nty;
  const BinBlock bb(n);
  const int v = bb.v;
  unsigned* cv = count + static_cast<int64_t>(v) * ntiles;
  if constexpr (LOCAL) {
    for (int i = threadIdx.x; i < ntiles; i += kBinThreads) s_count[i] = 0;
    __syncthreads();
  }
  const int4 rc = bb.g < n ? gs_project_one(means, covs, opac, n, cams[v], v, bb.g, rec)
                           : make_int4(0, 0, -1, -1);
  if (bb.g < n) rect[static_cast<int64_t>(v) * n + bb.g] = rc;
  for (int ty = rc.y; ty <= rc.w; ++ty)
    for (int tx = rc.x; tx <= rc.z; ++tx)
      atomicAdd((LOCAL ? s_count : cv) + ty * ntx + tx, 1u);
  if constexpr (LOCAL) {
    __syncthreads();
    for (int i = threadIdx.x; i < ntiles; i += kBinThreads)
      if (s_count[i] != 0) atomicAdd(cv + i, s_count[i]);
  }
}
// Exclusive scan of the tile counts (one block): off[i] = sum of count[< i],
// off[n] the total.
__global__ void gs_scan_kernel(const unsigned* __restrict__ count, int64_t n,
                               int64_t* __restrict__ off) {
  __shared__ int64_t part[1024];
  int64_t carry = 0;
  for (int64_t base = 0; base < n; base += 1024) {
    const int64_t i = base + threadIdx.x;
    const int64_t c = i < n ? static_cast<int64_t>(count[i]) : 0;
    part[threadIdx.x] = c;
    __syncthreads();
    for (int d = 1; d < 1024; d <<= 1) {  // Hillis-Steele inclusive scan
      const int64_t add = threadIdx.x >= d ? part[threadIdx.x - d] : 0;
      __syncthreads();
      part[threadIdx.x] += add;
      __syncthreads();
    }
    if (i < n) off[i] = carry + part[threadIdx.x] - c;
    carry += part[1023];
    __syncthreads();
  }
  if (threadIdx.x == 0) off[n] = carry;
}

// Writes each (view, Gaussian)'s key into the lists of its tiles. LOCAL: a
// block counts its keys per tile in shared memory, takes that many places of
// each tile's cursor at once and then places its keys (380 us with a global
// atomic per key on the lists of gs_project_kernel's comment, 34 us so).
template <bool LOCAL>
__global__ void __launch_bounds__(kBinThreads)
gs_fill_kernel(const float4* __restrict__ rec, const int4* __restrict__ rect, int64_t n, int ntx,
               int nty, const int64_t* __restrict__ off, unsigned* __restrict__ cursor,
               unsigned long long* __restrict__ keys) {
  extern __shared__ unsigned s_count[];
  const int ntiles = ntx * nty;
  const BinBlock bb(n);
  const int64_t tb = static_cast<int64_t>(bb.v) * ntiles;
  int4 rc = make_int4(0, 0, -1, -1);
  unsigned long long key = 0;
  if (bb.g < n) {
    const int64_t j = static_cast<int64_t>(bb.v) * n + bb.g;
    rc = rect[j];
    if (rc.z >= rc.x)
      key = (static_cast<unsigned long long>(__float_as_uint(rec[2 * j].z)) << 32) |
            static_cast<unsigned long long>(bb.g);
  }
  if constexpr (LOCAL) {
    for (int i = threadIdx.x; i < ntiles; i += kBinThreads) s_count[i] = 0;
    __syncthreads();
    for (int ty = rc.y; ty <= rc.w; ++ty)
      for (int tx = rc.x; tx <= rc.z; ++tx) atomicAdd(s_count + ty * ntx + tx, 1u);
    __syncthreads();
    for (int i = threadIdx.x; i < ntiles; i += kBinThreads)
      if (s_count[i] != 0) s_count[i] = atomicAdd(cursor + tb + i, s_count[i]);
    __syncthreads();
  }
  for (int ty = rc.y; ty <= rc.w; ++ty)
    for (int tx = rc.x; tx <= rc.z; ++tx) {
      const int t = ty * ntx + tx;
      keys[off[tb + t] + atomicAdd(LOCAL ? s_count + t : cursor + tb + t, 1u)] = key;
    }
}

// Ascending bitonic sort of s[0, p2), p2 a power of two; all threads call it.
__device__ void bitonic_sort(unsigned long long* s, int p2) {
  for (int k = 2; k <= p2; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = threadIdx.x; i < p2; i += blockDim.x) {
        const int l = i ^ j;
        if (l > i) {
          const unsigned long long a = s[i], b = s[l];
          if ((a > b) == ((i & k) == 0)) {
            s[i] = b;
            s[l] = a;
          }
        }
      }
      __syncthreads();
    }
}

// A pixel's composite so far.
struct Pixel {
  float fx, fy;
  float T = 1.f, D = 0.f, A = 0.f;
  bool done;
};

__device__ __forceinline__ float alpha_of(const float4& a, const float4& b, const Pixel& p) {
  const float dx = p.fx - a.x, dy = p.fy - a.y;
  const float q = b.x * dx * dx + 2.f * b.y * dx * dy + b.z * dy * dy;
  return fminf(kAlphaMax, a.w * expf(-0.5f * q));
}

__device__ __forceinline__ void add_alpha(float alpha, float z, Pixel& p) {
  const float w = p.T * alpha;
  p.D += w * z;
  p.A += w;
  p.T *= 1.f - alpha;
  p.done = p.T < kTMin;
}

// Composites the wn sorted keys of s_key front to back; true once every pixel
// of the block is opaque. Each warp owns 8 x 4 pixels and walks only the
// Gaussians whose box (outside of which alpha < 1/255) touches them: first the
// block marks for each key the warps it concerns, then every warp goes at its
// own pace, 32 keys at a time (their records through its own corner of shared
// memory, the next ones loaded meanwhile). With a block barrier every 256 keys
// the warps spent 10 of 17 cycles per instruction waiting for one another.
__device__ bool gs_composite(const unsigned long long* s_key, int wn, const float4* rv,
                             float4 (*s_rec)[2][32], uint8_t* s_warps, float tile_x, float tile_y,
                             Pixel& p) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int i = threadIdx.x; i < wn; i += kTilePx) {
    const int64_t g = static_cast<int64_t>(s_key[i] & 0xffffffffull);
    const float4 a = rv[2 * g];
    const int bits = __float_as_int(rv[2 * g + 1].w);
    const float2 h = __half22float2(*reinterpret_cast<const __half2*>(&bits));
    const float x = a.x - tile_x, y = a.y - tile_y;
    unsigned warps = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
      const float x0 = (w & 1) * 8.f, y0 = (w >> 1) * 4.f;
      if (x + h.x >= x0 && x - h.x <= x0 + 7.f && y + h.y >= y0 && y - h.y <= y0 + 3.f)
        warps |= 1u << w;
    }
    s_warps[i] = static_cast<uint8_t>(warps);
  }
  __syncthreads();
  float4(*rec)[32] = s_rec[warp];
  float4 na = make_float4(0.f, 0.f, 0.f, 0.f), nb = na;
  auto fetch = [&](int j0) {  // this lane's record of keys [j0, j0 + 32), if it concerns the warp
    const int i = j0 + lane;
    const bool mine = i < wn && ((s_warps[i] >> warp) & 1u) != 0;
    if (mine) {
      const int64_t g = static_cast<int64_t>(s_key[i] & 0xffffffffull);
      na = rv[2 * g];
      nb = rv[2 * g + 1];
    }
    return __ballot_sync(0xffffffffu, mine);
  };
  unsigned next = fetch(0);
  for (int j0 = 0; j0 < wn; j0 += 32) {
    if (__all_sync(0xffffffffu, p.done)) break;
    unsigned m = next;
    rec[0][lane] = na;
    rec[1][lane] = nb;
    __syncwarp();
    if (j0 + 32 < wn) next = fetch(j0 + 32);
    // Two alphas at a time, independent of one another and added in order: one
    // at a time the pixel's serial chain took 835 us where this takes 535.
    while (m != 0) {
      const int j1 = __ffs(m) - 1;
      m &= m - 1;
      const bool two = m != 0;
      const int j2 = two ? __ffs(m) - 1 : j1;
      m &= m - 1;
      const float4 a1 = rec[0][j1], a2 = rec[0][j2];
      const float al1 = alpha_of(a1, rec[1][j1], p);
      const float al2 = alpha_of(a2, rec[1][j2], p);
      if (!p.done && al1 >= kAlphaMin) add_alpha(al1, a1.z, p);
      if (two && !p.done && al2 >= kAlphaMin) add_alpha(al2, a2.z, p);
    }
    __syncwarp();  // the records are read before the next ones replace them
  }
  return __syncthreads_count(!p.done) == 0;  // also: the keys and marks are read
}

// One block per (view, tile), one thread per pixel. The keys not yet
// composited are split into kBuckets buckets (a linear map of the key, so the
// order of buckets is the order of keys) and taken in windows of whole
// buckets, at most kWin keys: the window's keys are dropped into their
// buckets' places in shared memory, each bucket is sorted, and the window
// composited; most pixels are opaque long before the last one. A bucket of
// more than kWin keys (a crowd at one depth) is split again by itself. Every
// split and every window reads the list once, so a list of c keys costs about
// c^2 / kWin reads where nothing turns opaque. Sorting the whole list for each
// 2,048 keys took 2,840 us on 32 views of 128 x 128 (60,000 Gaussians, some
// ten thousand keys in the fullest tiles); this takes 535 us (3 blocks an SM:
// with 4 or 5 the fullest tiles run slower, 575 us).
__global__ void __launch_bounds__(kTilePx, 3)
gs_render_kernel(const float4* __restrict__ rec, int64_t n, const GiCamera* __restrict__ cams,
                 int ntx, int nty, const int64_t* __restrict__ off,
                 const unsigned long long* __restrict__ keys, float* __restrict__ out_t,
                 uint8_t* __restrict__ out_hit) {
  __shared__ unsigned long long s_key[kWin];
  __shared__ float4 s_rec[kTilePx / 32][2][32];
  __shared__ unsigned s_off[kBuckets + 1];  // exclusive offsets of the buckets
  __shared__ unsigned s_cur[kBuckets];
  __shared__ unsigned long long s_red[16];
  __shared__ unsigned s_wsum[8];
  __shared__ uint8_t s_warps[kWin];
  const int ntiles = ntx * nty;
  const int tile = blockIdx.x;
  const int v = tile / ntiles;
  const int tt = tile - v * ntiles;
  const int tx = tt % ntx, ty = tt / ntx;
  const GiCamera& c = cams[v];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // warp w: the 8 x 4 pixels from (8 (w & 1), 4 (w / 2)) of the tile
  const int px = tx * kTile + (warp & 1) * 8 + (lane & 7);
  const int py = ty * kTile + (warp >> 1) * 4 + (lane >> 3);
  const bool inside = px < c.width && py < c.height;
  const int64_t beg = off[tile];
  const int64_t cnt = off[tile + 1] - beg;  // at most n <= 2^31
  const float4* rv = rec + 2 * static_cast<int64_t>(v) * n;
  const float tile_x = static_cast<float>(tx * kTile), tile_y = static_cast<float>(ty * kTile);
  constexpr unsigned long long kEnd = ~0ull;
  Pixel p;
  p.fx = static_cast<float>(px);
  p.fy = static_cast<float>(py);
  p.done = !inside;
  const unsigned long long* list = keys + beg;

  unsigned long long lo = 0;  // keys below are composited
  bool more = cnt > 0;
  while (more) {
    unsigned long long hi = kEnd;  // the range split here is [lo, hi)
    unsigned long long kmin, kmax;
    int sh;
    for (;;) {
      kmin = kEnd;
      kmax = 0;
      for (int64_t i = threadIdx.x; i < cnt; i += kTilePx) {
        const unsigned long long k = list[i];
        if (k >= lo && k < hi) {
          kmin = min(kmin, k);
          kmax = max(kmax, k);
        }
      }
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) {
        kmin = min(kmin, __shfl_xor_sync(0xffffffffu, kmin, d));
        kmax = max(kmax, __shfl_xor_sync(0xffffffffu, kmax, d));
      }
      if (lane == 0) {
        s_red[warp] = kmin;
        s_red[8 + warp] = kmax;
      }
      for (int i = threadIdx.x; i < kBuckets; i += kTilePx) s_cur[i] = 0;
      __syncthreads();
      for (int w = 0; w < 8; ++w) {
        kmin = min(kmin, s_red[w]);
        kmax = max(kmax, s_red[8 + w]);
      }
      more = kmin != kEnd;
      if (!more) break;
      sh = max(0, 54 - __clzll(kmax - kmin));  // (kmax - kmin) >> sh < kBuckets
      for (int64_t i = threadIdx.x; i < cnt; i += kTilePx) {
        const unsigned long long k = list[i];
        if (k >= lo && k < hi) atomicAdd(&s_cur[(k - kmin) >> sh], 1u);
      }
      __syncthreads();
      // exclusive scan, 4 buckets a thread; the counters become cursors
      static_assert(kBuckets == 4 * kTilePx && kBuckets == 1 << 10, "4 buckets a thread, 10 bits");
      unsigned k[4], sum = 0;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        k[e] = s_cur[4 * threadIdx.x + e];
        s_cur[4 * threadIdx.x + e] = 0;
        sum += k[e];
      }
      unsigned inc = sum;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const unsigned o = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += o;
      }
      if (lane == 31) s_wsum[warp] = inc;
      __syncthreads();
      unsigned base = inc - sum;
      for (int w = 0; w < warp; ++w) base += s_wsum[w];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        s_off[4 * threadIdx.x + e] = base;
        base += k[e];
      }
      if (threadIdx.x == kTilePx - 1) s_off[kBuckets] = base;
      __syncthreads();
      if (s_off[1] <= kWin) break;
      // the first bucket alone is too full: split it (keys differ, so sh > 0)
      lo = kmin;
      hi = kmin + (1ull << sh);
      __syncthreads();
    }
    if (!more) break;

    const unsigned total = s_off[kBuckets];
    int b0 = 0;
    while (more && b0 < kBuckets && s_off[b0] < total) {
      const unsigned base = s_off[b0];
      int b1 = b0, top = kBuckets;  // the largest b1 with at most kWin keys in [b0, b1)
      while (b1 < top) {
        const int mid = (b1 + top + 1) >> 1;
        if (s_off[mid] - base <= kWin) b1 = mid;
        else top = mid - 1;
      }
      if (b1 == b0) break;  // bucket b0 is too full: split from its start on
      const int wn = static_cast<int>(s_off[b1] - base);
      for (int64_t i = threadIdx.x; i < cnt; i += kTilePx) {
        const unsigned long long k = list[i];
        if (k < lo || k >= hi) continue;
        const int b = static_cast<int>((k - kmin) >> sh);
        if (b >= b0 && b < b1) s_key[s_off[b] - base + atomicAdd(&s_cur[b], 1u)] = k;
      }
      __syncthreads();
      // sort each bucket by counting the smaller keys in it, 8 keys a thread
      unsigned long long mine[kWin / kTilePx];
      int place[kWin / kTilePx];
      bool big = false;
#pragma unroll
      for (int e = 0; e < kWin / kTilePx; ++e) {
        const int i = e * kTilePx + threadIdx.x;
        place[e] = -1;
        if (i >= wn) continue;
        mine[e] = s_key[i];
        const int b = static_cast<int>((mine[e] - kmin) >> sh);
        const int first = static_cast<int>(s_off[b] - base);
        const int end = static_cast<int>(s_off[b + 1] - base);
        place[e] = first;
        if (end - first > kBucketSort) {
          big = true;
          continue;
        }
        for (int j = first; j < end; ++j) place[e] += s_key[j] < mine[e] ? 1 : 0;
      }
      if (__syncthreads_or(big)) {
        int p2 = 1;
        while (p2 < wn) p2 <<= 1;
        for (int i = wn + threadIdx.x; i < p2; i += kTilePx) s_key[i] = kEnd;
        __syncthreads();
        bitonic_sort(s_key, p2);
      } else {
#pragma unroll
        for (int e = 0; e < kWin / kTilePx; ++e)
          if (place[e] >= 0) s_key[place[e]] = mine[e];
        __syncthreads();
      }
      more = !gs_composite(s_key, wn, rv, s_rec, s_warps, tile_x, tile_y, p);
      b0 = b1;
    }
    if (b0 < kBuckets && s_off[b0] < total)
      lo = kmin + (static_cast<unsigned long long>(b0) << sh);
    else if (hi != kEnd)
      lo = hi;
    else
      more = false;
    __syncthreads();  // everyone has read the offsets
  }
  if (!inside) return;
  const float fx = p.fx, fy = p.fy, D = p.D, A = p.A;
  const float sx = (2.f * (fx + 0.5f) / c.width - 1.f) * c.tan_half *
                   (static_cast<float>(c.width) / c.height);
  const float sy = (1.f - 2.f * (fy + 0.5f) / c.height) * c.tan_half;
  const int64_t o = static_cast<int64_t>(v) * c.width * c.height +
                    static_cast<int64_t>(py) * c.width + px;
  out_t[o] = A > 0.f ? D / A * sqrtf(1.f + sx * sx + sy * sy) : __int_as_float(0x7f800000);
  out_hit[o] = A > 0.5f ? 1 : 0;
}

// Pixel-centre rays of each view (same model as the shadow / AO images).
__global__ void camera_rays_kernel(const GiCamera* __restrict__ cams, int nv, int64_t npx,
                                   RayOut r) {
  const int64_t j = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (j >= npx * nv) return;
  const int v = static_cast<int>(j / npx);
  const GiCamera& c = cams[v];
  const int64_t i = j - static_cast<int64_t>(v) * npx;
  const int x = static_cast<int>(i % c.width), y = static_cast<int>(i / c.width);
  const float sx = (2.f * (static_cast<float>(x) + 0.5f) / c.width - 1.f) * c.tan_half *
                   (static_cast<float>(c.width) / c.height);
  const float sy = (1.f - 2.f * (static_cast<float>(y) + 0.5f) / c.height) * c.tan_half;
  float d[3];
  for (int k = 0; k < 3; ++k) d[k] = c.f[k] + sx * c.r[k] + sy * c.u[k];
  const float inv = rsqrtf(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
  for (int k = 0; k < 3; ++k) {
    r.p[k][j] = c.eye[k];
    r.p[3 + k][j] = d[k] * inv;
  }
}

}  // namespace

int gs_tiles(int extent) { return (extent + kTile - 1) / kTile; }

cudaError_t launch_gs_project(const float* means, const float* covs, const float* opac, int64_t n,
                              const GiCamera* cams, int nv, int ntx, int nty, float4* rec,
                              int4* rect, unsigned* count, cudaStream_t s) {
  const int64_t blocks = (n + kBinThreads - 1) / kBinThreads * nv;
  if (blocks <= 0) return cudaSuccess;
  // an image of more tiles than a block's counts (1,024 x 1,024 pixels) counts globally
  if (ntx * nty <= kBinTiles)
    gs_project_kernel<true><<<static_cast<unsigned>(blocks), kBinThreads, ntx * nty * 4, s>>>(
        means, covs, opac, n, cams, ntx, nty, rec, rect, count);
  else
    gs_project_kernel<false><<<static_cast<unsigned>(blocks), kBinThreads, 0, s>>>(
        means, covs, opac, n, cams, ntx, nty, rec, rect, count);
  return cudaGetLastError();
}

cudaError_t launch_gs_scan(const unsigned* count, int64_t n, int64_t* off, cudaStream_t s) {
  gs_scan_kernel<<<1, 1024, 0, s>>>(count, n, off);
  return cudaGetLastError();
}

cudaError_t launch_gs_fill(const float4* rec, const int4* rect, int64_t n, int nv, int ntx,
                           int nty, const int64_t* off, unsigned* cursor,
                           unsigned long long* keys, cudaStream_t s) {
  const int64_t blocks = (n + kBinThreads - 1) / kBinThreads * nv;
  if (blocks <= 0) return cudaSuccess;
  if (ntx * nty <= kBinTiles)
    gs_fill_kernel<true><<<static_cast<unsigned>(blocks), kBinThreads, ntx * nty * 4, s>>>(
        rec, rect, n, ntx, nty, off, cursor, keys);
  else
    gs_fill_kernel<false><<<static_cast<unsigned>(blocks), kBinThreads, 0, s>>>(
        rec, rect, n, ntx, nty, off, cursor, keys);
  return cudaGetLastError();
}

cudaError_t launch_gs_render(const float4* rec, int64_t n, const GiCamera* cams, int nv, int ntx,
                             int nty, const int64_t* off, const unsigned long long* keys,
                             float* out_t, uint8_t* out_hit, cudaStream_t s) {
  const int64_t blocks = static_cast<int64_t>(nv) * ntx * nty;
  if (blocks <= 0) return cudaSuccess;
  gs_render_kernel<<<static_cast<unsigned>(blocks), kTilePx, 0, s>>>(rec, n, cams, ntx, nty, off,
                                                                     keys, out_t, out_hit);
  return cudaGetLastError();
}

cudaError_t launch_camera_rays(const GiCamera* cams, int nv, int64_t npx, RayOut r,
                               cudaStream_t s) {
  const int64_t m = npx * nv;
  if (m <= 0) return cudaSuccess;
  camera_rays_kernel<<<static_cast<unsigned>((m + 255) / 256), 256, 0, s>>>(cams, nv, npx, r);
  return cudaGetLastError();
}

}  // namespace ddf
