// Area-coverage rasterisation of rectangle masks: m[i][j] = area of the union
// of the rectangles [x0, x1) x [y0, y1) inside pixel [j, j+1) x [i, i+1)
// (pixel units, periodic with period N, overlaps counted once).  The grey-
// level mask is the object of Eq. (1) for shapes off the pixel grid.
//
// Five launches per batch: every rectangle is split at the period into at
// most four pieces and each piece counted into the 16 x 16-pixel tiles it
// touches (atomics), one CTA per clip scans the tile counts, one thread
// places the clips' lists one after another, the pieces are filed into their
// tiles' lists, and one CTA per tile computes its 256 pixels.  The lists fit
// the workspace by construction: a rectangle with sides of at most S pixels
// reaches at most (ceil(S/16) + 5)^2 tiles; a larger or empty rectangle
// marks its clip, whose mask is then written as NaN.  A pixel's value is
// exact up to FP32 rounding: empty and fully covered pixels are recognised
// directly, pixels of one or two pieces measured in closed form; otherwise the
// pixel is swept in x between consecutive piece edges, and in each slab the
// union length in y of the pieces spanning it is measured by walking up
// through their intervals.
// The result does not depend on the order of a tile's list.
#include <cstdint>

#include "fft_common.cuh"
#include "litho_internal.h"

namespace litho {

namespace {

constexpr int kTile = 16;
constexpr int kScanThreads = 1024, kScanRun = 4;  // tiles a thread of the scan takes in a row
// tile kernel: a warp per tile with a 64-piece cache (larger lists are read from global memory); four
// tiles a CTA, since a CTA waits for its slowest tile (eight: 783 us against 718)
constexpr int kRastWarps = 4, kTileCache = 64, kTilePix = kTile * kTile;

// Pieces of rectangle r (x0, y0, x1, y1) after the shift into [0, n) and the
// split at n; calls f(piece) for each nonempty one.
template <class F>
__device__ __forceinline__ void for_pieces(float4 r, int n, F&& f) {
  const float fn = float(n);
  const float sx = floorf(r.x / fn) * fn, sy = floorf(r.y / fn) * fn;
  const float x0 = r.x - sx, x1 = r.z - sx, y0 = r.y - sy, y1 = r.w - sy;
  const float xa[2] = {x0, 0.f}, xb[2] = {fminf(x1, fn), x1 - fn};
  const float ya[2] = {y0, 0.f}, yb[2] = {fminf(y1, fn), y1 - fn};
  for (int a = 0; a < 2; ++a)
    for (int b = 0; b < 2; ++b)
      if (xb[a] > xa[a] && yb[b] > ya[b]) f(make_float4(xa[a], ya[b], xb[a], yb[b]));
}

template <bool FILL>
__global__ void k_rast_bin(const float4* __restrict__ rects, const long long* __restrict__ rect_start, int n,
                           long long max_rects, float max_side, int* __restrict__ count, const int* __restrict__ tile_start,
                           const long long* __restrict__ clip_base, int* __restrict__ cursor,
                           float4* __restrict__ list, int* __restrict__ bad) {
  pdl_start();
  pdl_wait(rects, rect_start, tile_start, clip_base);
  const int c = blockIdx.y, tiles = n / kTile;
  if (!FILL && blockIdx.x == 0 && threadIdx.x == 0 && rect_start[c + 1] - rect_start[c] > max_rects) bad[c] = 1;
  const long long r = rect_start[c] + (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= rect_start[c + 1]) return;
  const float4 rc = rects[r];
  // NaN-safe: anything but 0 < side <= max_side marks the clip
  if (!(rc.z - rc.x > 0.f && rc.z - rc.x <= max_side && rc.w - rc.y > 0.f && rc.w - rc.y <= max_side)) {
    if (!FILL) bad[c] = 1;
    return;
  }
  for_pieces(rc, n, [&](float4 p) {
    // tiles of the first and last pixel the piece reaches (p.x, p.y in [0, n))
    const int tx0 = int(p.x) / kTile, tx1 = min(n - 1, int(ceilf(p.z)) - 1) / kTile;
    const int ty0 = int(p.y) / kTile, ty1 = min(n - 1, int(ceilf(p.w)) - 1) / kTile;
    for (int ty = ty0; ty <= ty1; ++ty)
      for (int tx = tx0; tx <= tx1; ++tx) {
        const size_t t = (size_t)c * tiles * tiles + (size_t)ty * tiles + tx;
        if (!FILL) {
          atomicAdd(count + t, 1);
        } else {
          list[clip_base[c] + tile_start[t] + atomicAdd(cursor + t, 1)] = p;
        }
      }
  });
}

// One CTA per clip: exclusive scan of its tile counts (cursor cleared), kScanRun tiles per thread and
// round (256 threads with one tile each took 50 us for 64 clips of 16384 tiles: 64 rounds of two block
// barriers; now 14).
__global__ void __launch_bounds__(kScanThreads) k_rast_scan(const int* __restrict__ count, int tiles2, int* __restrict__ tile_start,
                                                            int* __restrict__ cursor, int* __restrict__ total) {
  __shared__ int warp_sums[kScanThreads / 32];
  pdl_start();
  pdl_wait(count);
  const int c = blockIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const size_t base = (size_t)c * tiles2;
  int run = 0;
  for (int t0 = 0; t0 < tiles2; t0 += kScanThreads * kScanRun) {
    const int t = t0 + threadIdx.x * kScanRun;
    int v[kScanRun], sum = 0;
#pragma unroll
    for (int k = 0; k < kScanRun; ++k) {
      v[k] = t + k < tiles2 ? count[base + t + k] : 0;
      sum += v[k];
    }
    int x = sum;
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[w] = x;
    __syncthreads();
    if (w == 0) {
      int s = warp_sums[lane];
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += y;
      }
      warp_sums[lane] = s;
    }
    __syncthreads();
    int at = run + (w > 0 ? warp_sums[w - 1] : 0) + x - sum;
#pragma unroll
    for (int k = 0; k < kScanRun; ++k)
      if (t + k < tiles2) {
        tile_start[base + t + k] = at;
        cursor[base + t + k] = 0;
        at += v[k];
      }
    run += warp_sums[kScanThreads / 32 - 1];
    __syncthreads();
  }
  if (threadIdx.x == 0) total[c] = run;
}

// Offsets of the clips' lists: clip_base[c] = sum of the totals before c.
__global__ void k_rast_base(const int* __restrict__ total, int b, long long* __restrict__ clip_base) {
  pdl_start();
  pdl_wait(total);
  long long run = 0;
  for (int c = 0; c < b; ++c) {
    clip_base[c] = run;
    run += total[c];
  }
  clip_base[b] = run;
}

// Union area of the pieces within the unit pixel at (px, py).
__device__ float pixel_area(const float4* pcs, int np, float px, float py) {
  const float X1 = px + 1.f, Y1 = py + 1.f;
  float area = 0.f, xa = px;
  while (xa < X1) {
    float xb = X1;  // next piece edge above xa
    for (int k = 0; k < np; ++k) {
      const float4 p = pcs[k];
      if (p.y >= Y1 || p.w <= py) continue;
      if (p.x > xa && p.x < xb) xb = p.x;
      if (p.z > xa && p.z < xb) xb = p.z;
    }
    // union length in y of the pieces spanning [xa, xb)
    float len = 0.f, y = py;
    while (y < Y1) {
      float top = -1.f, next = Y1;
      for (int k = 0; k < np; ++k) {
        const float4 p = pcs[k];
        if (p.x > xa || p.z < xb) continue;
        if (p.y <= y && p.w > y) top = fmaxf(top, fminf(p.w, Y1));
        else if (p.y > y && p.y < next) next = p.y;
      }
      if (top > y) {
        len += top - y;
        y = top;
      } else {
        y = next;
      }
    }
    area += (xb - xa) * len;
    xa = xb;
  }
  return area;
}

// Area of a piece within the unit pixel at (px, py), which it reaches.
__device__ __forceinline__ float overlap(const float4& p, float px, float py) {
  return (fminf(p.z, px + 1.f) - fmaxf(p.x, px)) * (fminf(p.w, py + 1.f) - fmaxf(p.y, py));
}

// A warp per 16 x 16 tile.  A lane takes a column of 8 pixels: the rows a piece covers or reaches are
// bit masks from its rounded edges, tested once per piece instead of once per pixel.  Pixels that no
// piece reaches are 0, those that one covers 1; the grey ones are gathered, so that whole warps
// measure them: one or two pieces in closed form (A + B - A B), the rest, pooled over the CTA's
// tiles, by the sweep of pixel_area.  The tile is put together in shared memory and written by rows.
// 64 clips of 2048^2, 18 k rectangles each:
// 2062 -> 718 us (a CTA of 64 threads per tile that tested every pixel against every piece and
// swept every grey pixel).
template <bool VEC>
__global__ void __launch_bounds__(32 * kRastWarps) k_rast_tiles(const float4* __restrict__ list,
                                                                const int* __restrict__ count,
                                                                const int* __restrict__ tile_start,
                                                                const long long* __restrict__ clip_base,
                                                                const int* __restrict__ bad, int n,
                                                                float* __restrict__ mask) {
  __shared__ float4 cache[kRastWarps][kTileCache];
  __shared__ __align__(16) float value[kRastWarps][kTilePix];
  __shared__ unsigned char grey[kRastWarps][kTilePix];
  __shared__ unsigned short pool[kRastWarps * kTilePix];  // warp << 8 | pixel
  __shared__ const float4* pieces[kRastWarps];
  __shared__ int n_pieces[kRastWarps], n_pool;
  pdl_start();
  pdl_wait(list, count, tile_start, clip_base, bad);
  const int tiles = n / kTile, c = blockIdx.y, lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const int t0 = blockIdx.x * kRastWarps, t = t0 + wp;
  const bool live = t < tiles * tiles;
  const size_t ti = (size_t)c * tiles * tiles + t;
  const int flagged = bad[c], np = live && !flagged ? count[ti] : 0;
  const float4* pcs = list + clip_base[c] + (np > 0 ? tile_start[ti] : 0);
  if (threadIdx.x == 0) n_pool = 0;
  const int ty = t / tiles, tx = t - ty * tiles;
  const float bx = float(tx * kTile), by = float(ty * kTile);  // the tile's corner
  if (np <= kTileCache) {
    for (int k = lane; k < np; k += 32) cache[wp][k] = pcs[k];
    pcs = cache[wp];
  }
  if (lane == 0) {
    pieces[wp] = pcs;
    n_pieces[wp] = np;
  }
  __syncthreads();  // n_pool and the caches
  // rows 8 (lane / 16) ... + 7 of column lane % 16
  const int col = lane % kTile, row0 = lane / kTile * 8;
  const float px = bx + float(col), py0 = by + float(row0);
  unsigned full = 0, touch = 0;
  for (int k = 0; k < np; ++k) {
    const float4 p = pcs[k];
    // rows r with p.y <= y and p.w >= y + 1, and with p.y < y + 1 and p.w > y (y = py0 + r)
    const int f0 = max(0, int(ceilf(p.y - py0))), f1 = min(8, int(floorf(p.w - py0)));
    const int g0 = max(0, int(floorf(p.y - py0))), g1 = min(8, int(ceilf(p.w - py0)));
    const unsigned mf = f1 > f0 ? (1u << f1) - (1u << f0) : 0u, mg = g1 > g0 ? (1u << g1) - (1u << g0) : 0u;
    if (p.x <= px && p.z >= px + 1.f) full |= mf;
    if (p.x < px + 1.f && p.z > px) touch |= mg;
  }
  const unsigned g = touch & ~full;
#pragma unroll
  for (int r = 0; r < 8; ++r) value[wp][(row0 + r) * kTile + col] = full >> r & 1u ? 1.f : 0.f;
  int x = __popc(g);  // inclusive warp scan of the grey counts
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  const int n_grey = __shfl_sync(0xffffffffu, x, 31);
  int at = x - __popc(g);
  for (unsigned m = g; m; m &= m - 1) grey[wp][at++] = (unsigned char)((row0 + __ffs(m) - 1) * kTile + col);
  __syncwarp();
  for (int i = lane; i < n_grey; i += 32) {
    const int q = grey[wp][i];
    const float qx = bx + float(q % kTile), qy = by + float(q / kTile);
    int hits = 0;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
    for (int k = 0; k < np; ++k) {
      const float4 p = pcs[k];
      if (p.x < qx + 1.f && p.z > qx && p.y < qy + 1.f && p.w > qy) {
        if (hits == 0)
          a = p;
        else
          b = p;
        ++hits;
      }
    }
    if (hits <= 2) {
      float area = overlap(a, qx, qy);
      if (hits == 2) {
        area += overlap(b, qx, qy);
        const float4 i2 = make_float4(fmaxf(a.x, b.x), fmaxf(a.y, b.y), fminf(a.z, b.z), fminf(a.w, b.w));
        const float w = fminf(i2.z, qx + 1.f) - fmaxf(i2.x, qx), h = fminf(i2.w, qy + 1.f) - fmaxf(i2.y, qy);
        if (w > 0.f && h > 0.f) area -= w * h;
      }
      value[wp][q] = area;
    } else {
      pool[atomicAdd(&n_pool, 1)] = (unsigned short)(wp << 8 | q);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n_pool; i += blockDim.x) {
    const int w = pool[i] >> 8, q = pool[i] & 255, tt = t0 + w, wy = tt / tiles, wx = tt - wy * tiles;
    value[w][q] = pixel_area(pieces[w], n_pieces[w], float(wx * kTile + q % kTile), float(wy * kTile + q / kTile));
  }
  __syncthreads();
  if (!live) return;
  float* dst = mask + ((size_t)c * n + ty * kTile) * n + tx * kTile;
#pragma unroll
  for (int k = 0; k < 2; ++k) {  // four pixels of row 8 k + lane / 4
    const int row = 8 * k + lane / 4, cx = lane % 4 * 4;
    float4 v = *reinterpret_cast<const float4*>(&value[wp][row * kTile + cx]);
    if (flagged) v.x = v.y = v.z = v.w = __int_as_float(0x7fc00000);
    float* o = dst + (size_t)row * n + cx;
    if constexpr (VEC) {
      *reinterpret_cast<float4*>(o) = v;
    } else {
      o[0] = v.x;
      o[1] = v.y;
      o[2] = v.z;
      o[3] = v.w;
    }
  }
}

// Workspace: per-tile counts, starts and cursors, the clips' flags, totals and
// list offsets, then the piece lists.
struct RasterLayout {
  int *count, *tile_start, *cursor, *bad, *total;
  long long* clip_base;
  float4* list;
  size_t bytes;
};

size_t up256(size_t x) { return (x + 255) / 256 * 256; }

RasterLayout raster_layout(int b, int n, long long max_rects, int max_side, void* ws) {
  char* p = static_cast<char*>(ws);
  const size_t tiles2 = size_t(n / kTile) * (n / kTile) * b;
  const long long per_rect = raster_tiles_per_rect(max_side);
  RasterLayout L;
  size_t o = 0;
  auto take = [&](size_t bytes) {
    void* q = p ? p + o : nullptr;
    o += up256(bytes);
    return q;
  };
  L.count = static_cast<int*>(take(tiles2 * sizeof(int)));
  L.tile_start = static_cast<int*>(take(tiles2 * sizeof(int)));
  L.cursor = static_cast<int*>(take(tiles2 * sizeof(int)));
  L.bad = static_cast<int*>(take(size_t(b) * sizeof(int)));
  L.total = static_cast<int*>(take(size_t(b) * sizeof(int)));
  L.clip_base = static_cast<long long*>(take(size_t(b + 1) * sizeof(long long)));
  L.list = static_cast<float4*>(take(size_t(b) * size_t(max_rects) * size_t(per_rect) * sizeof(float4)));
  L.bytes = o;
  return L;
}

}  // namespace

// Tiles one rectangle with sides of at most s pixels can reach once split at
// the period: at most ceil(s/16) + 5 per axis.
long long raster_tiles_per_rect(int s) {
  const long long a = (s + kTile - 1) / kTile + 5;
  return a * a;
}

size_t raster_workspace_bytes(int b, int n, long long max_rects, int max_side) {
  return raster_layout(b, n, max_rects, max_side, nullptr).bytes;
}

cudaError_t launch_raster(const float4* rects, const long long* rect_start, int b, long long max_rects,
                          int max_side, int n, float* mask, void* ws, cudaStream_t st) {
  const RasterLayout L = raster_layout(b, n, max_rects, max_side, ws);
  const int tiles = n / kTile;
  const size_t tiles2 = size_t(tiles) * tiles;
  cudaError_t e = cudaMemsetAsync(L.count, 0, tiles2 * b * sizeof(int), st);
  if (e == cudaSuccess) e = cudaMemsetAsync(L.bad, 0, size_t(b) * sizeof(int), st);
  if (e != cudaSuccess) return e;
  if (max_rects > 0) {
    const dim3 grid(unsigned((max_rects + 255) / 256), b);
    e = launch_pdl(k_rast_bin<false>, grid, 256, 0, st, rects, rect_start, n, max_rects, float(max_side), L.count,
                   nullptr, nullptr, nullptr, nullptr, L.bad);
  }
  if (e == cudaSuccess)
    e = launch_pdl(k_rast_scan, b, kScanThreads, 0, st, L.count, int(tiles2), L.tile_start, L.cursor, L.total);
  if (e == cudaSuccess) e = launch_pdl(k_rast_base, 1, 1, 0, st, L.total, b, L.clip_base);
  if (e == cudaSuccess && max_rects > 0) {
    const dim3 grid(unsigned((max_rects + 255) / 256), b);
    e = launch_pdl(k_rast_bin<true>, grid, 256, 0, st, rects, rect_start, n, max_rects, float(max_side), L.count,
                   L.tile_start, L.clip_base, L.cursor, L.list, L.bad);
  }
  auto kern = (reinterpret_cast<uintptr_t>(mask) & 15) == 0 ? k_rast_tiles<true> : k_rast_tiles<false>;
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, dim3(unsigned((tiles2 + kRastWarps - 1) / kRastWarps), b), 32 * kRastWarps, 0, st, L.list,
                    L.count, L.tile_start, L.clip_base, L.bad, n, mask);
}

}  // namespace litho
