// Resist model (paper Eq. (5)): I_blur = g (x) I with a periodic, separable,
// normalised Gaussian g[j] ~ exp(-(j p)^2 / (2 s^2)), |j| <= R = ceil(4 s / p),
// then printed = [I_blur >= T] (ties print, as the ">=" of Eqs. (16)-(17)).
//
// One pass over HBM, by tiles.  Radii up to 12 (k_resist): a CTA takes TW x
// SH pixels.  Rows first, straight from global memory (the periodic halo is
// read through L1): a thread blurs 8 adjacent pixels from a window of 8 + 2R
// values in registers, so an output costs (8 + 2R)/8 loaded values instead of
// 2R + 1, and leaves them in a shared strip of SH + 2R rows; then a thread
// blurs two adjacent columns over a register window of PER + 2R rows with the
// packed two-lane FMA and writes I_blur (f32) and printed (u8).  Both sums run
// over the taps in the same order as the loop version (k_resist_any, larger
// radii), so a pixel's value does not depend on the tile.  Bound by the FMA
// pipe for R = 10 (2 (2R + 1) FMAs a pixel), by HBM for small radii.
// Measured: 16 planes of 2048^2, R = 10, 503 -> 168 us; 24 planes, R = 5, 471 -> 192 us
// (32 x 128 strips that loaded 2R + 1 shared values per pixel and row).
#include <cmath>

#include "fft_common.cuh"
#include "litho_internal.h"

namespace litho {

namespace {

constexpr int kThreads = 256;

// ALIGNED: 16-byte loads and paired stores; n a multiple of TW and SH.
template <int R, int TW, int SH, bool ALIGNED>
__global__ void __launch_bounds__(kThreads, R > 10 ? 2 : 3) k_resist(const float* __restrict__ img, int n,
                                                        const __grid_constant__ ResistTaps taps, float thr,
                                                     float* __restrict__ iblur, uint8_t* __restrict__ printed) {
  constexpr int ROWS = SH + 2 * R, SEG = TW / 8, HR = (R + 3) / 4 * 4, WIN = 8 + 2 * HR;
  constexpr int PAIRS = TW / 2, GROUPS = kThreads / PAIRS, PER = SH / GROUPS;
  static_assert(SH % GROUPS == 0, "whole row groups");
  __shared__ __align__(16) float hb[ROWS * TW];  // horizontally blurred rows
  const int x0 = blockIdx.x * TW, y0 = blockIdx.y * SH;
  pdl_start();
  pdl_wait(img);
  const size_t plane = (size_t)blockIdx.z * n * n;
  const float* src = img + plane;
  // rows: hb[ry][x] = sum_a g[a] I[y0 + ry - R][x0 + x - a]
  for (int i = threadIdx.x; i < ROWS * SEG; i += kThreads) {
    const int ry = i / SEG, xs = x0 + (i % SEG) * 8;
    int gy = y0 + ry - R;
    gy += gy < 0 ? n : gy >= n ? -n : 0;
    const float* row = src + (size_t)gy * n;
    float w[WIN];
#pragma unroll
    for (int q = 0; q < WIN / 4; ++q) {
      int gx = xs - HR + 4 * q;
      gx += gx < 0 ? n : gx >= n ? -n : 0;
      if constexpr (ALIGNED) {
        const float4 v = ld_dep(reinterpret_cast<const float4*>(row + gx));
        w[4 * q] = v.x;
        w[4 * q + 1] = v.y;
        w[4 * q + 2] = v.z;
        w[4 * q + 3] = v.w;
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) w[4 * q + e] = ld_dep(row + gx + e);
      }
    }
    float o[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      o[j] = 0.f;
#pragma unroll
      for (int a = -R; a <= R; ++a) o[j] = fmaf(taps.g[a + R], w[j + HR - a], o[j]);
    }
    float4* d = reinterpret_cast<float4*>(hb + ry * TW + (i % SEG) * 8);
    d[0] = make_float4(o[0], o[1], o[2], o[3]);
    d[1] = make_float4(o[4], o[5], o[6], o[7]);
  }
  __syncthreads();
  // columns: rows y0 + grp PER ... of columns x0 + 2 cp, x0 + 2 cp + 1
  const int cp = threadIdx.x % PAIRS;
  constexpr int STEP = R > 6 && PER > 8 ? 8 : PER;  // rows per window: three CTAs per SM without spills
#pragma unroll 1
  for (int yy = (threadIdx.x / PAIRS) * PER, y1 = yy + PER; yy < y1; yy += STEP) {
    float2 win[STEP + 2 * R];
#pragma unroll
    for (int j = 0; j < STEP + 2 * R; ++j) win[j] = *reinterpret_cast<const float2*>(hb + (yy + j) * TW + 2 * cp);
#pragma unroll
    for (int i = 0; i < STEP; ++i) {
      float2 acc = make_float2(0.f, 0.f);
#pragma unroll
      for (int a = -R; a <= R; ++a) acc = __ffma2_rn(make_float2(taps.g[a + R], taps.g[a + R]), win[i + R - a], acc);
      const size_t o = plane + (size_t)(y0 + yy + i) * n + x0 + 2 * cp;
      const uint8_t pa = acc.x >= thr ? 1 : 0, pb = acc.y >= thr ? 1 : 0;
      if constexpr (ALIGNED) {
        *reinterpret_cast<float2*>(iblur + o) = acc;
        if (printed) *reinterpret_cast<uchar2*>(printed + o) = make_uchar2(pa, pb);
      } else {
        iblur[o] = acc.x;
        iblur[o + 1] = acc.y;
        if (printed) {
          printed[o] = pa;
          printed[o + 1] = pb;
        }
      }
    }
  }
}

// Any radius.  A CTA takes W x SH pixels; the tile and its periodic halo go to shared memory, rows at an odd
// pitch, so that lanes on different rows, and lanes on different columns, read different banks.  Each
// thread forms eight neighbouring outputs (of a row, then of a column) from a window of 15 values that
// moves by eight taps at a time: one shared-memory load per eight FMAs, taps in the order of the fixed radii.
// 265 planes of 1024^2: 28.3 -> 4.46 ms at R = 40, 6.33 -> 2.85 ms at R = 20 (a load for every FMA); bound by
// the FP32 pipe and the shared-memory loads of the halo rows.

// o[j] = sum over t of taps.g[t] s[(j + 2 r - t) stride], t = 0 .. 2 r.
__device__ __forceinline__ void blur8(const float* s, int stride, const ResistTaps& taps, float (&o)[8]) {
  const int last = 2 * taps.radius;
  float w[15];  // w[m] = s[last - 8 c - 7 + m] in chunk c
#pragma unroll
  for (int m = 0; m < 15; ++m) w[m] = last - 7 + m >= 0 ? s[(last - 7 + m) * stride] : 0.f;
#pragma unroll
  for (int j = 0; j < 8; ++j) o[j] = 0.f;
  int t0 = 0;
  for (; t0 + 15 <= last; t0 += 8) {  // whole chunks, and the next one's eight values exist
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float g = taps.g[t0 + i];
#pragma unroll
      for (int j = 0; j < 8; ++j) o[j] = fmaf(g, w[j - i + 7], o[j]);
    }
#pragma unroll
    for (int m = 14; m >= 8; --m) w[m] = w[m - 8];
#pragma unroll
    for (int m = 0; m < 8; ++m) w[m] = s[(last - t0 - 15 + m) * stride];
  }
  for (; t0 <= last; t0 += 8) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (t0 + i > last) break;
      const float g = taps.g[t0 + i];
#pragma unroll
      for (int j = 0; j < 8; ++j) o[j] = fmaf(g, w[j - i + 7], o[j]);
    }
#pragma unroll
    for (int m = 14; m >= 8; --m) w[m] = w[m - 8];
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const int k = last - t0 - 15 + m;
      w[m] = k >= 0 ? s[k * stride] : 0.f;
    }
  }
}

template <int W, int SH, int NT>
__global__ void __launch_bounds__(NT) k_resist_any(const float* __restrict__ img, int n,
                                                   const __grid_constant__ ResistTaps taps, float thr,
                                                   float* __restrict__ iblur, uint8_t* __restrict__ printed) {
  extern __shared__ float sm[];
  const int r = taps.radius, rows = SH + 2 * r, wi = W + 2 * r, pitch = wi | 1, hp = W + 1;
  float* tile = sm;                // [rows][pitch]
  float* hb = sm + rows * pitch;   // [rows][hp] horizontally blurred rows
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int x0 = blockIdx.x * W, y0 = blockIdx.y * SH;
  pdl_start();
  pdl_wait(img);
  const size_t plane = (size_t)blockIdx.z * n * n;
  const float* src = img + plane;
  for (int ry = warp; ry < rows; ry += NT / 32) {  // r < n/2: one wrap at most
    int gy = y0 + ry - r;
    gy += gy < 0 ? n : gy >= n ? -n : 0;
    for (int rx = lane; rx < wi; rx += 32) {
      int gx = x0 + rx - r;
      gx += gx < 0 ? n : gx >= n ? -n : 0;
      tile[ry * pitch + rx] = ld_dep(src + (size_t)gy * n + gx);
    }
  }
  __syncthreads();
  float o[8];
  for (int i = threadIdx.x; i < rows * (W / 8); i += NT) {  // lanes on rows
    const int seg = i / rows, ry = i - seg * rows;
    blur8(tile + ry * pitch + 8 * seg, 1, taps, o);
#pragma unroll
    for (int j = 0; j < 8; ++j) hb[ry * hp + 8 * seg + j] = o[j];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < W * (SH / 8); i += NT) {  // lanes on columns
    const int x = i % W, y = i / W * 8;
    blur8(hb + y * hp + x, hp, taps, o);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const size_t at = plane + (size_t)(y0 + y + j) * n + x0 + x;
      iblur[at] = o[j];
      if (printed) printed[at] = o[j] >= thr ? 1 : 0;
    }
  }
}

size_t any_bytes(int r, int w, int sh) { return sizeof(float) * (sh + 2 * r) * (((w + 2 * r) | 1) + w + 1); }

template <int W, int SH, int NT>
cudaError_t launch_any(const float* img, int planes, int n, const ResistTaps& taps, float thr, float* iblur,
                       uint8_t* printed, cudaStream_t st) {
  const size_t sm = any_bytes(taps.radius, W, SH);  // 199 KB at radius 64 for 32 x 128
  cudaError_t e = cudaFuncSetAttribute(k_resist_any<W, SH, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_resist_any<W, SH, NT>, dim3(n / W, n / SH, planes), NT, sm, st, img, n, taps, thr, iblur,
                    printed);
}

template <int R>
cudaError_t launch_r(const float* img, int planes, int n, const ResistTaps& taps, float thr, float* iblur,
                     uint8_t* printed, cudaStream_t st) {
  const bool aligned = (reinterpret_cast<uintptr_t>(img) & 15) == 0 && (reinterpret_cast<uintptr_t>(iblur) & 7) == 0 &&
                       (reinterpret_cast<uintptr_t>(printed) & 1) == 0;
#define RUN(TW, SH, A)                                                                                            \
  return launch_pdl(k_resist<R, TW, SH, A>, dim3(n / TW, n / SH, planes), kThreads, 0, st, img, n, taps, thr, iblur, \
                    printed)
  // 128-row tiles read (128 + 2R)/128 of the rows; with fewer than two of them per SM, 32-row tiles
  // fill the chip instead
  if (!aligned) RUN(32, 32, false);
  if (n % 128 == 0 && (long long)planes * (n / 64) * (n / 128) >= 304) RUN(64, 128, true);
  if (n % 64 == 0) RUN(64, 32, true);
  RUN(32, 32, true);
#undef RUN
}

}  // namespace

bool resist_taps(double sigma_nm, double pixel_nm, ResistTaps* t, std::string* why) {
  if (!(sigma_nm > 0.0) || !(pixel_nm > 0.0)) {
    *why = "sigma_nm and pixel_nm must be > 0";
    return false;
  }
  const int r = int(std::ceil(4.0 * sigma_nm / pixel_nm));
  if (r > kMaxResistRadius) {
    *why = "resist blur radius ceil(4 sigma / pixel) above 64 pixels";
    return false;
  }
  double g[2 * kMaxResistRadius + 1], sum = 0.0;
  for (int j = -r; j <= r; ++j) {
    g[j + r] = std::exp(-(j * pixel_nm) * (j * pixel_nm) / (2.0 * sigma_nm * sigma_nm));
    sum += g[j + r];
  }
  t->radius = r;
  for (int j = 0; j < 2 * r + 1; ++j) t->g[j] = float(g[j] / sum);
  return true;
}

cudaError_t launch_resist(const float* img, int planes, int n, const ResistTaps& taps, float threshold, float* iblur,
                          uint8_t* printed, cudaStream_t st) {
  if (n % 32 != 0 || 2 * taps.radius >= n) return cudaErrorInvalidValue;
  switch (taps.radius) {
#define R_CASE(R) \
  case R: return launch_r<R>(img, planes, n, taps, threshold, iblur, printed, st);
    R_CASE(1) R_CASE(2) R_CASE(3) R_CASE(4) R_CASE(5) R_CASE(6) R_CASE(7) R_CASE(8) R_CASE(9) R_CASE(10)
    R_CASE(11) R_CASE(12)
#undef R_CASE
    default:
      if (n % 128 != 0) return launch_any<32, 32, 512>(img, planes, n, taps, threshold, iblur, printed, st);
      // two tiles per SM while they fit (radius 37); then one, by twice the threads, and wide enough
      // for less of a halo where that fits (radius 56) and fills the chip.  265 planes of 1024^2, 32 and 64 wide:
      // 2840 and 3251 us at R = 20, 8627 (by 512 threads) and 4455 at R = 40; 64 of 2048^2 at R = 64, by 512 and
      // 1024 threads: 9.98 and 8.12 ms
      if (2 * any_bytes(taps.radius, 32, 128) <= 226 * 1024)
        return launch_any<32, 128, 512>(img, planes, n, taps, threshold, iblur, printed, st);
      if (any_bytes(taps.radius, 64, 128) <= 227 * 1024 && (long long)planes * (n / 64) * (n / 128) >= 152)
        return launch_any<64, 128, 1024>(img, planes, n, taps, threshold, iblur, printed, st);
      return launch_any<32, 128, 1024>(img, planes, n, taps, threshold, iblur, printed, st);
  }
}

}  // namespace litho
