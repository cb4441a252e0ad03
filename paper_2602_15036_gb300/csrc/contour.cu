// Contours of the resist image and the edge-placement error (paper section
// II.D and Eqs. (6)-(8)).
//
// Marching squares: cell (i, j) has the corners TL = I[i][j], TR = I[i][j+1],
// BR = I[i+1][j+1], BL = I[i+1][j] (periodic); a corner is inside when
// I >= T.  Edges 0 top (TL-TR), 1 right (TR-BR), 2 bottom (BL-BR), 3 left
// (TL-BL) are crossed where their corners differ, at the point of linear
// interpolation of I - T from the edge's first corner to its second.  Each
// segment is oriented with the corner it cuts off on its left when that
// corner is inside and on its right when outside, and, between opposite
// edges, with the inside pair on its left (left of p0 -> p1: cross(p1 - p0,
// q - p0) > 0).  A saddle (only TL and BR, or only TR and BL, inside) joins
// its inside corners when ((TL + TR) + (BR + BL)) / 4 >= T and separates them
// otherwise.  The segment table below is that rule worked out per case.
//
// Five launches, all deterministic: the inside bits of every pixel, from them
// the number of segments per row of cells, one CTA per plane scanning its
// rows' counts, one warp placing the planes one after another, and the
// segments written at those offsets in row-major cell order (saddle segments
// ordered by their start edge).
#include <algorithm>
#include <cstdint>

#include "litho_internal.h"

namespace litho {

namespace {

// Segment table: for each case (inside bits TL = 1, TR = 2, BR = 4, BL = 8)
// up to two (start edge, end edge) pairs packed as s0 | e0 << 2 | s1 << 4 | e1 << 6,
// with the count in bits 8-9.  Saddles 5 and 10 have a second entry for the
// separated variant (index 16 + case).
__constant__ uint16_t kSegTable[32] = {
    // 0: none
    0,
    // 1 TL in: top -> left
    (1 << 8) | (0 | 3 << 2),
    // 2 TR in: right -> top
    (1 << 8) | (1 | 0 << 2),
    // 3 TL, TR in: right -> left
    (1 << 8) | (1 | 3 << 2),
    // 4 BR in: bottom -> right
    (1 << 8) | (2 | 1 << 2),
    // 5 TL, BR in, joined: top -> right (cuts TR), bottom -> left (cuts BL)
    (2 << 8) | (0 | 1 << 2) | ((2 | 3 << 2) << 4),
    // 6 TR, BR in: bottom -> top
    (1 << 8) | (2 | 0 << 2),
    // 7 BL out: bottom -> left
    (1 << 8) | (2 | 3 << 2),
    // 8 BL in: left -> bottom
    (1 << 8) | (3 | 2 << 2),
    // 9 TL, BL in: top -> bottom
    (1 << 8) | (0 | 2 << 2),
    // 10 TR, BL in, joined: right -> bottom (cuts BR), left -> top (cuts TL)
    (2 << 8) | (1 | 2 << 2) | ((3 | 0 << 2) << 4),
    // 11 BR out: right -> bottom
    (1 << 8) | (1 | 2 << 2),
    // 12 BR, BL in: left -> right
    (1 << 8) | (3 | 1 << 2),
    // 13 TR out: top -> right
    (1 << 8) | (0 | 1 << 2),
    // 14 TL out: left -> top
    (1 << 8) | (3 | 0 << 2),
    // 15: none
    0,
    // 16..31: separated saddles (only 21 and 26 used)
    0, 0, 0, 0, 0,
    // 21 = 16 + 5, TL and BR cut off: top -> left, bottom -> right
    (2 << 8) | (0 | 3 << 2) | ((2 | 1 << 2) << 4),
    0, 0, 0, 0,
    // 26 = 16 + 10, TR and BL cut off: right -> top, left -> bottom
    (2 << 8) | (1 | 0 << 2) | ((3 | 2 << 2) << 4),
    0, 0, 0, 0, 0};

struct Cell {
  float tl, tr, br, bl;
};

// Index into the segment table (case, or 16 + case for a separated saddle).
__device__ __forceinline__ int cell_case(const Cell& c, float thr) {
  const int cs = (c.tl >= thr) | (c.tr >= thr) << 1 | (c.br >= thr) << 2 | (c.bl >= thr) << 3;
  if (cs == 5 || cs == 10) {
    const float centre = ((c.tl + c.tr) + (c.br + c.bl)) * 0.25f;
    if (!(centre >= thr)) return 16 + cs;
  }
  return cs;
}

// Crossing point of edge e (0 top, 1 right, 2 bottom, 3 left) in cell-local coordinates (x, y), without branches.
__device__ __forceinline__ float2 edge_point(const Cell& c, int e, float thr) {
  const float va = e == 1 ? c.tr : e == 2 ? c.bl : c.tl;
  const float vb = e == 0 ? c.tr : e == 3 ? c.bl : c.br;
  const float da = va - thr, db = vb - thr;
  const float t = da / (da - db);
  const float ax = e == 1 ? 1.f : 0.f, ay = e == 2 ? 1.f : 0.f;
  const bool horiz = (e & 1) == 0;
  return make_float2(ax + (horiz ? t : 0.f), ay + (horiz ? 0.f : t));
}

// Exclusive block scan of one int per thread (blockDim.x a multiple of 32, at
// most 1024); returns the thread's offset, *total the sum.
__device__ __forceinline__ int block_exclusive_scan(int v, int* total) {
  __shared__ int warp_sums[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_sums[w] = x;
  __syncthreads();
  if (w == 0) {
    int s = lane < nw ? warp_sums[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += y;
    }
    if (lane < nw) warp_sums[lane] = s;  // inclusive
  }
  __syncthreads();
  const int before = (w > 0 ? warp_sums[w - 1] : 0) + x - v;
  *total = warp_sums[nw - 1];
  __syncthreads();  // warp_sums reusable
  return before;
}

// One CTA per plane: exclusive scan of the plane's row counts into
// row_start (offsets within the plane) and the plane's total.  Chunks of one
// row per thread (contiguous loads and stores), the running total carried.
__global__ void __launch_bounds__(1024) k_ms_scan(const int* __restrict__ row_count, int n,
                                                         long long* __restrict__ row_start,
                                                         long long* __restrict__ plane_total) {
  const size_t base = (size_t)blockIdx.x * n;
  long long run = 0;
  for (int r0 = 0; r0 < n; r0 += blockDim.x) {
    const int r = r0 + threadIdx.x;
    const int c = r < n ? row_count[base + r] : 0;
    int chunk;
    const int before = block_exclusive_scan(c, &chunk);
    if (r < n) row_start[base + r] = run + before;
    run += chunk;
  }
  if (threadIdx.x == 0) plane_total[blockIdx.x] = run;
}

// plane_start[p] = sum of the totals of the planes before p; [planes] = all.  One warp.
__global__ void __launch_bounds__(32) k_ms_planes(const long long* __restrict__ plane_total, int planes,
                                                  long long* __restrict__ plane_start) {
  long long run = 0;
  for (int p0 = 0; p0 < planes; p0 += 32) {
    const int p = p0 + threadIdx.x;
    const long long v = p < planes ? plane_total[p] : 0;
    long long x = v;
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(0xffffffffu, x, o);
      if (int(threadIdx.x) >= o) x += y;
    }
    if (p < planes) plane_start[p] = run + x - v;
    run += __shfl_sync(0xffffffffu, x, 31);
  }
  if (threadIdx.x == 0) plane_start[planes] = run;
}

// The planes' inside bits, row by row: bit k of word w of a row is [pixel 32 w + k >= T].  Everything that
// depends only on which pixels are inside (the number of segments of a cell: half its crossed edges) is
// then worked out 32 cells at a time, and the pixels themselves are read once here and once more only
// at the cells that hold a segment.  A warp takes kBitWords words (independent loads, HBM-bound).
constexpr int kBitWords = 16;

// WHOLE: rows are whole words (n % 32 == 0), so words follow pixels and only the last warp can run out.
template <bool WHOLE>
__global__ void __launch_bounds__(256) k_ms_bits(const float* __restrict__ img, int n, int words, float thr,
                                                 long long total, unsigned* __restrict__ bits) {
  const int lane = threadIdx.x & 31;
  const long long w0 = ((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5) * kBitWords;
  if (w0 >= total) return;  // uniform across the warp
  float v[kBitWords];
  if (WHOLE && w0 + kBitWords <= total) {
    const float* src = img + w0 * 32 + lane;
#pragma unroll
    for (int k = 0; k < kBitWords; ++k) v[k] = __ldg(src + 32 * k);
  } else {
    long long row = w0 / words;
    int w = int(w0 - row * words);
#pragma unroll
    for (int k = 0; k < kBitWords; ++k) {
      const int j = 32 * w + lane;
      // a pixel past the row or the planes is outside
      v[k] = w0 + k < total && j < n ? __ldg(img + row * n + j) : __int_as_float(0x7fc00000);
      if (++w == words) {
        w = 0;
        ++row;
      }
    }
  }
  unsigned b[kBitWords];
#pragma unroll
  for (int k = 0; k < kBitWords; ++k) b[k] = __ballot_sync(0xffffffffu, v[k] >= thr);
  if (lane == 0) {
    if (w0 + kBitWords <= total) {  // w0 is a multiple of 16 words: 64-byte aligned
#pragma unroll
      for (int k = 0; k < kBitWords; k += 4)
        *reinterpret_cast<uint4*>(bits + w0 + k) = make_uint4(b[k], b[k + 1], b[k + 2], b[k + 3]);
    } else {
#pragma unroll
      for (int k = 0; k < kBitWords; ++k)
        if (w0 + k < total) bits[w0 + k] = b[k];
    }
  }
}

// Cells 32 w .. 32 w + 31 of a row, from the inside bits of its pixel rows (r0 above, r1 below): `some`, the
// cells that hold a segment, and `two`, those that hold two (all four edges crossed).
struct CellBits {
  unsigned some, two;
};

// Word w of a row, its first pixel repeated after its last, and the word shifted by one pixel.
__device__ __forceinline__ void row_word(const unsigned* __restrict__ r, int w, int words, int n, unsigned* a,
                                         unsigned* next) {
  unsigned x = __ldg(r + w);
  const unsigned first = __ldg(r) & 1u;
  unsigned up;  // bit 0 of the following word
  if (w + 1 < words) {
    up = __ldg(r + w + 1) & 1u;
  } else {
    up = first;
    if (n % 32) x |= first << (n % 32);
  }
  *a = x;
  *next = x >> 1 | up << 31;
}

__device__ __forceinline__ CellBits cell_bits(const unsigned* __restrict__ r0, const unsigned* __restrict__ r1, int w,
                                              int words, int n) {
  if (w >= words) return CellBits{0u, 0u};
  unsigned t, tn, b, bn;
  row_word(r0, w, words, n, &t, &tn);
  row_word(r1, w, words, n, &b, &bn);
  const unsigned h = t ^ tn, g = b ^ bn, v = t ^ b, vn = tn ^ bn;
  const unsigned valid = w == words - 1 && n % 32 ? (1u << (n % 32)) - 1u : 0xffffffffu;
  return CellBits{(h | g | v | vn) & valid, h & g & v & vn & valid};
}

// Segments of every row of cells: a warp per row.
__global__ void __launch_bounds__(256) k_ms_count(const unsigned* __restrict__ bits, int n, int words, int planes,
                                                  int* __restrict__ row_count) {
  const int lane = threadIdx.x & 31, i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, p = blockIdx.y;
  if (i >= n) return;
  const unsigned* plane = bits + (size_t)p * n * words;
  const unsigned *r0 = plane + (size_t)i * words, *r1 = plane + (size_t)(i + 1 == n ? 0 : i + 1) * words;
  int cnt = 0;
  for (int w = lane; w < words; w += 32) {
    const CellBits c = cell_bits(r0, r1, w, words, n);
    cnt += __popc(c.some) + __popc(c.two);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) cnt += __shfl_down_sync(0xffffffffu, cnt, o);
  if (lane == 0) row_count[(size_t)p * n + i] = cnt;
}

// Emit: a warp per row of cells.  Each of 16 lanes puts the segments of a word's 32 cells, as (column,
// segment of the cell), into the warp's queue at the place a warp scan gives it; the queue holds them
// in output order, and whenever it has 32 the lanes compute one each from the cell's corner pixels.
// So the crossing arithmetic runs on full warps, and finding the segments costs a few instructions per
// 32 cells.  48 planes of 2048^2 (15 M segments), all launches of the contours: 868 -> 425 us (pixel
// rows walked twice in 128-cell chunks, rounds of 32 segments per chunk, a third full).
constexpr int kEmitWarps = 8, kEmitWords = 16, kEmitQueue = 32 + kEmitWords * 64;

__global__ void __launch_bounds__(32 * kEmitWarps) k_ms_emit(const float* __restrict__ img,
                                                             const unsigned* __restrict__ bits, int n, int words,
                                                             float thr, const long long* __restrict__ row_start,
                                                             const long long* __restrict__ plane_start,
                                                             long long capacity, float4* __restrict__ seg,
                                                             int* __restrict__ cell_id) {
  __shared__ uint16_t tab[32];
  __shared__ unsigned queue[kEmitWarps][kEmitQueue];  // column | segment << 31
  if (threadIdx.x < 32) tab[threadIdx.x] = kSegTable[threadIdx.x];
  __syncthreads();
  const int p = blockIdx.y, lane = threadIdx.x & 31, i = blockIdx.x * kEmitWarps + (threadIdx.x >> 5);
  if (i >= n) return;  // no block barrier below
  unsigned* mine = queue[threadIdx.x >> 5];
  const int i1 = i + 1 == n ? 0 : i + 1;
  const float *ra = img + ((size_t)p * n + i) * n, *rb = img + ((size_t)p * n + i1) * n;
  const unsigned *r0 = bits + ((size_t)p * n + i) * words, *r1 = bits + ((size_t)p * n + i1) * words;
  long long o = plane_start[p] + row_start[(size_t)p * n + i];  // output index of the queue's head
  int len = 0;
  // the queue's entries [at, at + 32) below `len`, one per lane
  auto emit = [&](int at) {
    if (at + lane < len) {
      const unsigned e = mine[at + lane];
      const int j = int(e & 0x7fffffffu), q = int(e >> 31), j1 = j + 1 == n ? 0 : j + 1;
      const Cell cl{__ldg(ra + j), __ldg(ra + j1), __ldg(rb + j1), __ldg(rb + j)};
      const uint16_t ent = tab[cell_case(cl, thr)];
      const int s_e = (ent >> (4 * q)) & 3, e_e = (ent >> (4 * q + 2)) & 3;
      const float2 pa = edge_point(cl, s_e, thr);
      const float2 pb = edge_point(cl, e_e, thr);
      if (o + lane < capacity) {
        seg[o + lane] = make_float4(j + pa.x, i + pa.y, j + pb.x, i + pb.y);
        if (cell_id) cell_id[o + lane] = i * n + j;
      }
    }
  };
  for (int w0 = 0; w0 < words; w0 += kEmitWords) {
    const CellBits c = lane < kEmitWords ? cell_bits(r0, r1, w0 + lane, words, n) : CellBits{0u, 0u};
    const int cnt = __popc(c.some) + __popc(c.two);
    int x = cnt;  // inclusive warp scan
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, s);
      if (lane >= s) x += y;
    }
    const int total = __shfl_sync(0xffffffffu, x, 31);
    if (total == 0) continue;
    int at = len + x - cnt;
    for (unsigned m = c.some; m; m &= m - 1) {
      const int k = __ffs(m) - 1;
      const unsigned col = unsigned(32 * (w0 + lane) + k);
      mine[at++] = col;
      if (c.two >> k & 1u) mine[at++] = col | 1u << 31;
    }
    len += total;
    __syncwarp();
    int done = 0;
    for (; len - done >= 32; done += 32, o += 32) emit(done);
    if (done > 0) {  // the rest moves to the front
      const unsigned e = done + lane < len ? mine[done + lane] : 0u;
      __syncwarp();
      mine[lane] = e;
      len -= done;
      __syncwarp();
    }
  }
  emit(0);
}

// ---- Eq. (6) at control points ----------------------------------------------------------------
__device__ __forceinline__ float bilin(float a, float b, float c, float d, float fx, float fy) {
  return (1.f - fy) * ((1.f - fx) * a + fx * b) + fy * ((1.f - fx) * c + fx * d);
}

// Offsets of a point's 4 x 4 neighbourhood (rows and columns floor - 1 .. floor + 2, periodic) and its
// fractions: the same for every plane, so formed once per point.
struct EpeSite {
  size_t row[4];
  int col[4];
  float fx, fy;
};

__device__ __forceinline__ EpeSite epe_site(float2 r, int n) {
  EpeSite s;
  const float fj = floorf(r.x), fi = floorf(r.y);
  s.fx = r.x - fj;
  s.fy = r.y - fi;
  auto wrap = [&](int v) { return v >= 0 && v < n ? v : ((v % n) + n) % n; };
  int j = wrap(int(fj) - 1), i = wrap(int(fi) - 1);
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    s.row[a] = (size_t)i * n;
    s.col[a] = j;
    i = i + 1 == n ? 0 : i + 1;
    j = j + 1 == n ? 0 : j + 1;
  }
  return s;
}

// Eq. (6) at a site of plane I.
__device__ __forceinline__ float epe_at(const float* __restrict__ I, const EpeSite& s, float inv_pixel, float thr) {
  float v[4][4];  // rows i0-1 .. i0+2, columns j0-1 .. j0+2
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b)
      v[a][b] = ((a == 0 || a == 3) && (b == 0 || b == 3)) ? 0.f : __ldg(I + s.row[a] + s.col[b]);
  const float fx = s.fx, fy = s.fy;
  const float e = bilin(v[1][1], v[1][2], v[2][1], v[2][2], fx, fy);
  // central differences at the four corners (per pixel)
  const float gx = bilin(0.5f * (v[1][2] - v[1][0]), 0.5f * (v[1][3] - v[1][1]), 0.5f * (v[2][2] - v[2][0]),
                         0.5f * (v[2][3] - v[2][1]), fx, fy);
  const float gy = bilin(0.5f * (v[2][1] - v[0][1]), 0.5f * (v[2][2] - v[0][2]), 0.5f * (v[3][1] - v[1][1]),
                         0.5f * (v[3][2] - v[1][2]), fx, fy);
  const float g = sqrtf(gx * gx + gy * gy) * inv_pixel;
  return g > 0.f ? -(e - thr) / g : __int_as_float(0x7fc00000);
}

// One thread per control point, every plane in turn.
__global__ void k_epe(const float* __restrict__ img, int planes, int n, int m, float inv_pixel, float thr,
                      const float2* __restrict__ pts, float* __restrict__ epe) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= m) return;
  const EpeSite s = epe_site(pts[k], n);
  for (int p = 0; p < planes; ++p) epe[(size_t)p * m + k] = epe_at(img + (size_t)p * n * n, s, inv_pixel, thr);
}

// All clips' points in one launch: point k belongs to the last clip c with
// start[c] <= k (empty clips are passed over), whose planes follow one another
// in img.  Whatever start holds, c stays in [0, clips).  With the sites' offsets
// formed once per point (two integer divisions per row and column and plane
// before) 6.7 M points x 3 planes of 2048^2: 231 -> 201 us.
__global__ void k_epe_batch(const float* __restrict__ img, int clips, int planes, int n, long long m, float inv_pixel,
                            float thr, const float2* __restrict__ pts, const long long* __restrict__ start,
                            float* __restrict__ epe) {
  const long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (k >= m) return;
  int lo = 0, hi = clips - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(start + mid) <= k)
      lo = mid;
    else
      hi = mid - 1;
  }
  const EpeSite s = epe_site(pts[k], n);
  const float* I = img + (size_t)lo * planes * n * n;
  for (int p = 0; p < planes; ++p) epe[(size_t)p * m + k] = epe_at(I + (size_t)p * n * n, s, inv_pixel, thr);
}

__global__ void k_epe_focus(const float* __restrict__ epe, int m, int f0, int fp, int fn, float tol_neg,
                            float tol_pos, float* __restrict__ avg, float* __restrict__ eff) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= m) return;
  const float e0 = epe[(size_t)f0 * m + k];
  const float a = (e0 + epe[(size_t)fp * m + k] + epe[(size_t)fn * m + k]) / 3.f;
  if (avg) avg[k] = a;
  if (eff) eff[k] = e0 > tol_pos ? e0 - tol_pos : e0 < tol_neg ? e0 - tol_neg : a;
}

}  // namespace

// The workspace: segments and first segment of every row, segments of every plane, the inside bits.
struct ContourLayout {
  int* count;
  long long *start, *plane_total;
  unsigned* bits;
  int words;  // per row
  size_t bytes;
};

static ContourLayout contour_layout(int planes, int n, void* ws) {
  const size_t rows = size_t(planes) * n;
  char* p = static_cast<char*>(ws);
  size_t o = 0;
  auto take = [&](size_t bytes) {
    void* q = p ? p + o : nullptr;
    o += (bytes + 255) / 256 * 256;
    return q;
  };
  ContourLayout L;
  L.words = (n + 31) / 32;
  L.count = static_cast<int*>(take(rows * sizeof(int)));
  L.start = static_cast<long long*>(take(rows * sizeof(long long)));
  L.plane_total = static_cast<long long*>(take(size_t(planes) * sizeof(long long)));
  L.bits = static_cast<unsigned*>(take(rows * L.words * sizeof(unsigned)));
  L.bytes = o;
  return L;
}

size_t contour_workspace_bytes(int planes, int n) { return contour_layout(planes, n, nullptr).bytes; }

cudaError_t launch_contours(const float* img, int planes, int n, float thr, float4* seg, int* cell_id,
                            long long capacity, long long* plane_start, void* ws, cudaStream_t st) {
  const ContourLayout L = contour_layout(planes, n, ws);
  const long long total = (long long)planes * n * L.words, warps = (total + kBitWords - 1) / kBitWords;
  auto bits = n % 32 == 0 ? k_ms_bits<true> : k_ms_bits<false>;
  bits<<<unsigned((warps + 7) / 8), 256, 0, st>>>(img, n, L.words, thr, total, L.bits);
  k_ms_count<<<dim3((n + 7) / 8, planes), 256, 0, st>>>(L.bits, n, L.words, planes, L.count);
  k_ms_scan<<<planes, 1024, 0, st>>>(L.count, n, L.start, L.plane_total);
  k_ms_planes<<<1, 32, 0, st>>>(L.plane_total, planes, plane_start);
  if (capacity > 0)
    k_ms_emit<<<dim3((n + kEmitWarps - 1) / kEmitWarps, planes), 32 * kEmitWarps, 0, st>>>(
        img, L.bits, n, L.words, thr, L.start, plane_start, capacity, seg, cell_id);
  return cudaGetLastError();
}

cudaError_t launch_epe(const float* img, int planes, int n, float pixel_nm, float thr, const float2* pts, int m,
                       float* epe, cudaStream_t st) {
  k_epe<<<(m + 255) / 256, 256, 0, st>>>(img, planes, n, m, 1.0f / pixel_nm, thr, pts, epe);
  return cudaGetLastError();
}

cudaError_t launch_epe_batch(const float* img, int clips, int planes, int n, float pixel_nm, float thr,
                             const float2* pts, const long long* start, long long m, float* epe, cudaStream_t st) {
  k_epe_batch<<<unsigned((m + 255) / 256), 256, 0, st>>>(img, clips, planes, n, m, 1.0f / pixel_nm, thr, pts, start,
                                                        epe);
  return cudaGetLastError();
}

cudaError_t launch_epe_focus(const float* epe, int m, int f0, int fp, int fn, float tol_neg, float tol_pos,
                             float* avg, float* eff, cudaStream_t st) {
  k_epe_focus<<<(m + 255) / 256, 256, 0, st>>>(epe, m, f0, fp, fn, tol_neg, tol_pos, avg, eff);
  return cudaGetLastError();
}

}  // namespace litho
