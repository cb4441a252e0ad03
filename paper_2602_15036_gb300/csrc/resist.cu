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
        const float4 v = __ldg(reinterpret_cast<const float4*>(row + gx));
        w[4 * q] = v.x;
        w[4 * q + 1] = v.y;
        w[4 * q + 2] = v.z;
        w[4 * q + 3] = v.w;
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) w[4 * q + e] = __ldg(row + gx + e);
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

// Any radius, taps in a loop: a 32 x SH strip and its halo in shared memory, a warp per row for the
// horizontal sums, a thread per column for the vertical ones.
template <int SH>
__global__ void __launch_bounds__(kThreads) k_resist_any(const float* __restrict__ img, int n,
                                                         const __grid_constant__ ResistTaps taps, float thr,
                                                         float* __restrict__ iblur, uint8_t* __restrict__ printed) {
  constexpr int SW = 32, WARPS = kThreads / 32, PER = SH / WARPS;
  extern __shared__ float sm[];
  const int r = taps.radius, rows_in = SH + 2 * r, wi = SW + 2 * r;
  float* tile = sm;               // [rows_in][wi] the strip and its periodic halo
  float* hb = sm + rows_in * wi;  // [rows_in][SW] horizontally blurred rows
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int plane = blockIdx.z, x0 = blockIdx.x * SW, y0 = blockIdx.y * SH;
  const float* src = img + (size_t)plane * n * n;
  for (int ry = warp; ry < rows_in; ry += WARPS) {  // r < n/2: one wrap at most
    int gy = y0 + ry - r;
    gy += gy < 0 ? n : gy >= n ? -n : 0;
    for (int rx = lane; rx < wi; rx += 32) {
      int gx = x0 + rx - r;
      gx += gx < 0 ? n : gx >= n ? -n : 0;
      tile[ry * wi + rx] = __ldg(src + (size_t)gy * n + gx);
    }
  }
  __syncthreads();
  for (int ry = warp; ry < rows_in; ry += WARPS) {
    const float* t = tile + ry * wi + lane + r;
    float acc = 0.f;
    for (int a = -r; a <= r; ++a) acc = fmaf(taps.g[a + r], t[-a], acc);
    hb[ry * SW + lane] = acc;
  }
  __syncthreads();
  const int yy = warp * PER;
  float* dst = iblur + (size_t)plane * n * n;
  uint8_t* pr = printed ? printed + (size_t)plane * n * n : nullptr;
  for (int i = 0; i < PER; ++i) {
    const float* c = hb + (yy + i + r) * SW + lane;
    float acc = 0.f;
    for (int a = -r; a <= r; ++a) acc = fmaf(taps.g[a + r], c[-a * SW], acc);
    const size_t o = (size_t)(y0 + yy + i) * n + x0 + lane;
    dst[o] = acc;
    if (pr) pr[o] = acc >= thr ? 1 : 0;
  }
}

template <int SH>
cudaError_t launch_any(const float* img, int planes, int n, const ResistTaps& taps, float thr, float* iblur,
                       uint8_t* printed, cudaStream_t st) {
  const int r = taps.radius;
  const size_t sm = sizeof(float) * ((SH + 2 * r) * (32 + 2 * r) + (SH + 2 * r) * 32);
  cudaError_t e = cudaFuncSetAttribute(k_resist_any<SH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  k_resist_any<SH><<<dim3(n / 32, n / SH, planes), kThreads, sm, st>>>(img, n, taps, thr, iblur, printed);
  return cudaGetLastError();
}

template <int R>
cudaError_t launch_r(const float* img, int planes, int n, const ResistTaps& taps, float thr, float* iblur,
                     uint8_t* printed, cudaStream_t st) {
  const bool aligned = (reinterpret_cast<uintptr_t>(img) & 15) == 0 && (reinterpret_cast<uintptr_t>(iblur) & 7) == 0 &&
                       (reinterpret_cast<uintptr_t>(printed) & 1) == 0;
#define RUN(TW, SH, A) \
  k_resist<R, TW, SH, A><<<dim3(n / TW, n / SH, planes), kThreads, 0, st>>>(img, n, taps, thr, iblur, printed)
  // 128-row tiles read (128 + 2R)/128 of the rows; with fewer than two of them per SM, 32-row tiles
  // fill the chip instead
  if (!aligned)
    RUN(32, 32, false);
  else if (n % 128 == 0 && (long long)planes * (n / 64) * (n / 128) >= 304)
    RUN(64, 128, true);
  else if (n % 64 == 0)
    RUN(64, 32, true);
  else
    RUN(32, 32, true);
#undef RUN
  return cudaGetLastError();
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
      return n % 128 == 0 ? launch_any<128>(img, planes, n, taps, threshold, iblur, printed, st)
                          : launch_any<32>(img, planes, n, taps, threshold, iblur, printed, st);
  }
}

}  // namespace litho
