// FFT-based kernels: mask spectrum (crop), stage 1 (band multiply + inverse
// transform over v), and stage 2 of the FP32 path (inverse transform over u
// fused with the |E_k|^2 accumulation over all kernels).
//
// Paper Section III.A: the object spectrum O(f) of Eq. (1) (thin-mask reading:
// the mask's DFT), and the SOCS image of Eq. (4), I = sum_k lam_k |O (x) phi_k|^2,
// evaluated as E_j = IDFT(M . Psi_j) restricted to the C x C band crop (Psi: kernelset.cu).
//
// Data layout (all row-major, x fastest):
//   mask    [b][N][N] f32
//   rowbuf  [b][N][C/2 + 8] c64   row DFT of the mask, the columns 0 <= u <= C/2 (the mask is real)
//   mhat    [b][C][C] c64   N^-2 DFT(m) on the crop, [v][u]
//   t1      [j][N][C] c64   stage-1 field T_j[y][u] = sum_v mhat[v][u] Psi_j[v][u] e^{2 pi i v y/N}
//   q       [plane][N][..] c64  half band rows of a real plane (0 <= u < h; with a blur, the image's then the blur's)
//   img     [plane][N][N] f32
#include <algorithm>
#include <cfloat>

#include "fft_common.cuh"
#include "litho_internal.h"
#include "stage1.cuh"

namespace litho {

namespace {

__device__ __forceinline__ int freq_of(int idx, int n) { return idx < n / 2 ? idx : idx - n; }

// Spectra of real planes are kept for u >= 0 only ("half"): S(-v, -u) = conj S(v, u), so the column
// transforms run on half the columns.  A half row holds k = u in [0, crop/2); the mask spectrum, whose
// crop has u = -crop/2 but not u = crop/2, keeps k = crop/2 as well (stride crop/2 + 8).

// ---- mask spectrum, pass 1: two real rows per complex transform ----------------------------
// z = m[y0] + i m[y1]; Z = DFT(z); X(u) = (Z(u) + conj Z(-u))/2, Y(u) = (Z(u) - conj Z(-u))/(2i),
// written for u in [0, cols) with row stride ld.  Mask: m; Sigmoid: sigmoid(alpha m) (the ILT's theta); Copy:
// m, which is also written to copy + b copy_stride on the way (the AI input's first channel).
enum class RowInput { Mask, Sigmoid, Copy };
template <int N, RowInput IN>
__global__ void __launch_bounds__(Plan<N>::NT) k_mask_rows(const float* __restrict__ m, float alpha, int crop,
                                                            const float2* __restrict__ tw_g,
                                                            float2* __restrict__ rowbuf, int cols, int ld,
                                                            int pairs_per_cta, float* __restrict__ copy,
                                                            size_t copy_stride) {
  extern __shared__ float2 smem[];
  float2* tw = smem;
  float2* buf = smem + N;
  float2* zc = smem + N + PadLen<N>::value;  // Z(u) for u in [-C/2, C/2], index u + C/2 (crop + 1 <= N + 1 entries)
  pdl_start();
  load_twiddles<N>(tw, tw_g);
  pdl_wait(m);
  __syncthreads();
  const int b = blockIdx.y, t = threadIdx.x, half = crop / 2;
  constexpr int R0 = Plan<N>::R[0], NB0 = N / R0;
  static_assert(PassShape<N, Plan<N>::NT, R0>::PER == 1, "one first-pass butterfly per thread");
  // this thread's first-pass inputs (columns t + r N/R0 of both rows) of a pair, loaded one pair ahead
  float2 nxt[R0];
  auto prefetch = [&](int pr) {
    const float* r0 = m + ((size_t)b * N + 2 * pr) * N;
#pragma unroll
    for (int r = 0; r < R0; ++r)
      nxt[r] = t < NB0 ? make_float2(ld_dep(r0 + t + r * NB0), ld_dep(r0 + N + t + r * NB0)) : make_float2(0.f, 0.f);
  };
  auto value = [&](float2 v) {
    return IN == RowInput::Sigmoid ? make_float2(sigmoidf(alpha * v.x), sigmoidf(alpha * v.y)) : v;
  };
  const int pr0 = blockIdx.x * pairs_per_cta, pr1 = min(N / 2, (blockIdx.x + 1) * pairs_per_cta);
  if (pr0 < pr1) prefetch(pr0);
  // pairs [pr0, pr1): the next pair's first pass writes buf only after a
  // barrier that follows this pair's reads of zc
  for (int pr = pr0; pr < pr1; ++pr) {
    const int y0 = 2 * pr;
    float2 cur[R0];
#pragma unroll
    for (int r = 0; r < R0; ++r) cur[r] = nxt[r];
    if (IN == RowInput::Copy && t < NB0) {
      float* c0 = copy + b * copy_stride + (size_t)y0 * N + t;
#pragma unroll
      for (int r = 0; r < R0; ++r) {
        c0[r * NB0] = cur[r].x;
        c0[N + r * NB0] = cur[r].y;
      }
    }
    auto load = [&](int, int r, int) { return value(cur[r]); };
    auto use = [&](int, int, int idx, float2 v) {
      const int u = freq_of(idx, N);
      if (u >= -half && u <= half) zc[u + half] = v;
      if (u == -N / 2 && half == N / 2) zc[crop] = v;  // crop == N: Z(N/2) is Z(-N/2)
    };
    // once the first pass has consumed this pair, the next pair's loads go out
    auto after_first = [&]() {
      if (pr + 1 < pr1) prefetch(pr + 1);
    };
    fft_load_use<N, -1, decltype(load), decltype(use), false>(buf, tw, t, load, use, after_first);
    __syncthreads();
    float2* o0 = rowbuf + ((size_t)b * N + y0) * ld;
    float2* o1 = o0 + ld;
    for (int k = t; k < cols; k += blockDim.x) {
      const float2 zp = zc[half + k], zm = zc[half - k];
      o0[k] = make_float2(0.5f * (zp.x + zm.x), 0.5f * (zp.y - zm.y));
      o1[k] = make_float2(0.5f * (zp.y + zm.y), -0.5f * (zp.x - zm.x));
    }
  }
}


// ---- mask spectrum, pass 2: column DFTs of the columns u >= 0, crop rows kept ------------------
// Columns u = k for k in [0, cols) of half rows with stride ld.  MIRROR (the mask spectrum on its whole
// crop): a column u also gives the column -u, S(-v, -u) = conj S(v, u).  Without it only the columns
// u >= 0 are written (index u + crop/2), times gain[v] gain[u] when gain is given: the spectrum of the
// plane's blur, |v| < crop/2.  W columns per CTA with the lanes interleaved over them: the first pass reads from global
// memory and the last one writes there, 8 W bytes of a row at a time, with no copy through shared memory.
// 64 masks of 2048^2: 330 -> 182 us (every column transformed, and staged in shared memory).
template <int N, int W, bool MIRROR>
__global__ void __launch_bounds__(Plan<N>::NT * W) k_mask_cols(const float2* __restrict__ rowbuf, int crop, int cols,
                                                               int ld, const float2* __restrict__ tw_g,
                                                               const float* __restrict__ gain,
                                                               float2* __restrict__ mhat) {
  constexpr int NT = Plan<N>::NT, LD = (PadLen<N>::value + 15) / 16 * 16 + 16 / W;
  extern __shared__ float2 smem[];
  float2* tw = smem;
  float2* buf = smem + N;
  pdl_start();
  load_twiddles<N>(tw, tw_g);
  pdl_wait(rowbuf, gain);
  __syncthreads();
  const int b = blockIdx.y, tid = threadIdx.x, g = tid % W, t = tid / W, k = blockIdx.x * W + g, half = crop / 2;
  const bool live = k < cols;
  const float2* src = rowbuf + (size_t)b * N * ld + k;
  auto load = [&](int, int, int y) { return ld_dep_if(src + (size_t)y * ld, live); };
  const float scale = 1.0f / (float(N) * float(N));
  const float gu = gain && live ? scale * ld_dep(gain + half + k) : scale;
  float2* dst = mhat + (size_t)b * crop * crop;
  auto use = [&](int, int, int idx, float2 v) {
    const int f = freq_of(idx, N), cv = half + f, cm = half - f;
    if (!live) return;
    if (MIRROR) {
      v = make_float2(v.x * scale, v.y * scale);
      if (k < half && cv >= 0 && cv < crop) dst[(size_t)cv * crop + half + k] = v;
      if (k > 0 && cm >= 0 && cm < crop) dst[(size_t)cm * crop + half - k] = make_float2(v.x, -v.y);
      // crop == N: v = -N/2 is its own mirror
      if (k > 0 && f == -N / 2 && crop == N) dst[half - k] = make_float2(v.x, -v.y);
    } else if (cv >= 0 && cv < crop) {
      // v = -crop/2 has no mirror on the crop: without it the plane stays real (no consumer reads it)
      const float s = cv == 0 ? 0.f : gain ? gu * ld_dep(gain + cv) : gu;
      dst[(size_t)cv * crop + half + k] = make_float2(s * v.x, s * v.y);
    }
  };
  fft_load_use<N, -1, decltype(load), decltype(use), false>(buf + g * LD, tw, t, load, use);
}

// Transfer function of the periodic separable blur on an n-point grid:
// gain[i] = sum_a g[a] cos(2 pi f a / n) for the crop frequency f = i - crop/2
// (the taps are even, so the transform is real).  The angle is reduced
// exactly in integers before cospi.
__global__ void k_blur_gain(ResistTaps taps, int n, int crop, float* __restrict__ gain) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  pdl_start();  // the sum needs nothing from the kernel before: only the store waits for it
  const int f = i - crop / 2, r = taps.radius;
  float acc = taps.g[r];
  for (int a = 1; a <= r; ++a) {
    const long long e = ((long long)f * a % n + n) % n;  // f a mod n, in [0, n)
    acc = fmaf(2.0f * taps.g[r + a], cospif(2.0f * float(e) / float(n)), acc);
  }
  pdl_wait();
  if (i < crop) gain[i] = acc;
}

// ---- stage 1: band multiply + inverse transform over v (stage1.cuh), FP32 output ------------------
struct OutC64 {
  static constexpr bool kRowWise = false;
  float2* t1;
  int n, crop;
  __device__ __forceinline__ int first() const { return 0; }  // first crop column, and the rows' stride
  __device__ __forceinline__ int ld(int c) const { return c; }
  __device__ __forceinline__ float2* column(int j, int c) const { return t1 + (size_t)j * n * crop + c; }
  __device__ float scale(int) const { return 1.f; }
  template <int W>
  __device__ void store_row(int, int, int, float, const float2 (&)[W]) const {}
};

// The columns u >= 0 alone, as half rows of stride `stride` (any spectra, no kernels).
struct OutHalf {
  static constexpr bool kRowWise = false;
  float2* q;
  int n, half, stride;
  __device__ __forceinline__ int first() const { return half; }
  __device__ __forceinline__ int ld(int) const { return stride; }
  __device__ __forceinline__ float2* column(int j, int c) const { return q + (size_t)j * n * stride + (c - half); }
  __device__ float scale(int) const { return 1.f; }
  template <int W>
  __device__ void store_row(int, int, int, float, const float2 (&)[W]) const {}
};

// ---- stage 2 (FP32 path): one image row per CTA, all kernels of the plane ------------------------
// Rows of up to 256 points are one warp's: two warps share the plane's kernels (G = 2, half of them each), where a
// chain of many kernels is what an SM of few rows waits for.  256^2 images of one plane and 12 fields, one and
// two warps a row: 2 clips 19.2 and 18.9 us, 4 28.6 and 20.9, 8 30.3 and 28.5, 12 40.1 and 38.8, 20 59.4 and
// 59.1; two planes of 5: 1 clip 16.3 and 19.1 us, 20 51.2 and 61.6.  Whole calls by rows, 12 fields: 256 points
// 1024 rows 28.5 and 20.8, 2048 30.0 and 28.3, 3072 39.7 and 38.8, 4096 47.4 and 48.8; 128 points 20.1 and 17.8,
// 21.9 and 20.8, 28.0 and 27.8, 32.6 and 34.6; 64 points 2048 rows 20.1 and 18.1, 3072 24.2 and 24.1, 4096 27.8
// and 28.7; 8 fields of 128 points 2048 rows 17.4 and 17.2, 3072 21.7 and 22.2.  Below 768 rows the launches take
// longer than the chain.
// How many warps there are depends on the clips of the launch, a clip's bits must not: these rows' sums are
// always those of the first half of the fields and of the rest, whether two warps form them or one after the other.
template <int N>
struct Stage2Halves {
  static constexpr bool value = Plan<N>::NT == 32;
};

template <int N, bool BANDED, int G>
__global__ void __launch_bounds__(Plan<N>::NT * G, 512 / Plan<N>::NT / G)
    k_stage2(const float2* __restrict__ t1, const __grid_constant__ FieldSet fs, int crop, float dose,
             const float2* __restrict__ tw_g, float* __restrict__ img, const __grid_constant__ PlaneOut po) {
  using PL = Plan<N>;
  constexpr int NT = PL::NT;
  constexpr int RL = PL::R[PL::P - 1];
  constexpr int PERL = PassShape<N, NT, RL>::PER;
  __shared__ float2 bufs[G][PadLen<N>::value];
  __shared__ float2 tw[N];
  __shared__ float part[G > 1 ? N : 1];
  pdl_start();
  load_twiddles<N>(tw, tw_g);
  pdl_wait(t1);
  __syncthreads();
  const int y = blockIdx.x, plane = blockIdx.y, t = threadIdx.x % NT, grp = threadIdx.x / NT, half = crop / 2;
  float2* buf = bufs[grp];
  const int clip = plane / fs.planes, pl = plane - clip * fs.planes, nk = fs.start[pl + 1] - fs.start[pl];
  const float2* base = t1 + ((size_t)(clip * fs.fields() + fs.start[pl]) * N + y) * crop;
  static_assert(G == 1 || (G == 2 && Stage2Halves<N>::value), "two warps take the halves of the fields");
  constexpr bool kFold = Stage2Halves<N>::value && G == 1;  // this warp forms both halves' sums
  const int nh = (nk + 1) / 2, j0 = grp * nh, rounds = G == 2 ? nh : nk;
  float acc[PERL][RL], first[PERL][RL];
#pragma unroll
  for (int p = 0; p < PERL; ++p)
#pragma unroll
    for (int q = 0; q < RL; ++q) acc[p][q] = first[p][q] = 0.f;
  // middle-pass twiddles in registers: measured faster for 2048-point rows,
  // slower for 1024 (where the registers they take cost more than the
  // shared-memory reads they save)
  constexpr bool kMid = MidTwiddles<N, +1>::kUsable && N >= 2048;
  MidTwiddles<N, +1> mid;
  if constexpr (kMid) mid.load(tw, t);
  // this thread's first-pass inputs of a kernel's band row, loaded one kernel ahead: while the later
  // passes of the one before run (8 planes of 2048^2: 925 -> 882 us)
  constexpr int R0 = PL::R[0], NB0 = N / R0;
  static_assert(PassShape<N, NT, R0>::PER == 1, "one first-pass butterfly per thread");
  float2 nxt[R0];
  auto prefetch = [&](int j) {
    const float2* row = base + (size_t)j * N * crop;
#pragma unroll
    for (int r = 0; r < R0; ++r) {
      const int c = t + r * NB0 - (r < R0 / 2 ? 0 : N) + half;  // index t + r N/R0 < N/2 exactly when r < R0/2
      const bool zero = (BANDED && r >= R0 / 4 && r < 3 * R0 / 4) || t >= NB0 || j >= nk || c < 0 || c >= crop;
      nxt[r] = ld_dep_if(row + c, !zero);
    }
  };
  prefetch(j0);
  for (int i = 0; i < rounds; ++i) {  // every warp runs every round (block barriers)
    if constexpr (kFold) {
      if (i == nh) {
#pragma unroll
        for (int p = 0; p < PERL; ++p)
#pragma unroll
          for (int q = 0; q < RL; ++q) {
            first[p][q] = acc[p][q];
            acc[p][q] = 0.f;
          }
      }
    }
    float2 cur[R0];
#pragma unroll
    for (int r = 0; r < R0; ++r) cur[r] = nxt[r];
    auto load = [&](int, int r, int) { return cur[r]; };
    auto after_first = [&]() {
      if (i + 1 < rounds) prefetch(j0 + i + 1);
    };
    auto use = [&](int p, int q, int, float2 v) { acc[p][q] = fmaf(v.x, v.x, fmaf(v.y, v.y, acc[p][q])); };
    if constexpr (kMid)
      fft_load_use_mid<N, +1, decltype(load), decltype(use), BANDED>(buf, tw, t, load, use, mid, after_first);
    else
      fft_load_use<N, +1, decltype(load), decltype(use), BANDED>(buf, tw, t, load, use, after_first);
  }
  if constexpr (kFold) {
#pragma unroll
    for (int p = 0; p < PERL; ++p)
#pragma unroll
      for (int q = 0; q < RL; ++q) acc[p][q] = first[p][q] + acc[p][q];
  }
  if constexpr (G > 1) {
#pragma unroll
    for (int p = 0; p < PERL; ++p)
#pragma unroll
      for (int q = 0; q < RL; ++q)
        if (grp > 0 && t + p * NT < N / RL) part[t + p * NT + q * (N / RL)] = acc[p][q];
    __syncthreads();
    if (grp > 0) return;
#pragma unroll
    for (int p = 0; p < PERL; ++p)
#pragma unroll
      for (int q = 0; q < RL; ++q)
        if (t + p * NT < N / RL) acc[p][q] += part[t + p * NT + q * (N / RL)];
  }
  for (int d = po.first[pl]; d < po.first[pl + 1]; ++d) {
    float* out = img + ((size_t)(clip * po.out_planes + po.list[d]) * N + y) * N;
#pragma unroll
    for (int p = 0; p < PERL; ++p) {
      const int jj = t + p * NT;
      if (jj < N / RL) {
#pragma unroll
        for (int q = 0; q < RL; ++q) out[jj + q * (N / RL)] = dose * acc[p][q];
      }
    }
  }
}

// ---- band rows to image rows: the inverse transform along x ----------------------------------------------
// Second half of the exact Fourier interpolation from the coarse grid, from half rows: with the spectra
// A(u) and B(u) of two real rows, one transform of A + i B (A(-u) = conj A(u)) gives both as its real and
// imaginary parts.

// Element u of A + i B from the half rows a, b of `h` columns.
__device__ __forceinline__ float2 two_rows(const float2* __restrict__ a, const float2* __restrict__ b, int h, int u) {
  const int k = u < 0 ? -u : u;
  const float2 x = ld_dep_if(a + k, k < h), y = ld_dep_if(b + k, k < h);
  return u < 0 ? make_float2(x.x + y.y, y.x - x.y) : make_float2(x.x - y.y, x.y + y.x);
}

// Band rows q of h columns two by two (unit i: rows 2 i and 2 i + 1 of q).  RESIST: the two are a row's image
// and its blur: img = Re (skipped when NULL), iblur = Im, printed = [Im >= threshold] (skipped when NULL).
// Otherwise they are two rows of the image: img rows 2 i and 2 i + 1, times scale.  Plane p of `planes`
// per clip goes to its planes of `po`.  With ext (image rows only) the extremes of what is written are
// folded into ext = (min, max) as ordered integers.  Bound by HBM (the rows written).
template <int N, bool BANDED, bool RESIST>
__global__ void __launch_bounds__(Plan<N>::NT) k_band_rows(const float2* __restrict__ q, int h, float scale,
                                                           const float2* __restrict__ tw_g, float thr,
                                                           float* __restrict__ img, float* __restrict__ iblur,
                                                           uint8_t* __restrict__ printed, int planes,
                                                           const __grid_constant__ PlaneOut po, int units_per_cta,
                                                           uint2* __restrict__ ext) {
  constexpr int NT = Plan<N>::NT, RL = Plan<N>::R[Plan<N>::P - 1], PERL = PassShape<N, NT, RL>::PER;
  constexpr int UNITS = RESIST ? N : N / 2;
  __shared__ float2 buf[PadLen<N>::value];
  __shared__ float2 tw[N];
  pdl_start();
  load_twiddles<N>(tw, tw_g);
  pdl_wait(q);
  __syncthreads();
  const int p = blockIdx.y, t = threadIdx.x, clip = p / planes, pl = p - clip * planes;
  const int d0 = po.first[pl], d1 = po.first[pl + 1];
  float lo = FLT_MAX, hi = -FLT_MAX;
  for (int i = blockIdx.x * units_per_cta; i < min(UNITS, (blockIdx.x + 1) * units_per_cta); ++i) {
    const float2* row = q + ((size_t)p * UNITS + i) * 2 * h;
    auto load = [&](int, int r, int idx) {  // first pass: idx < N/2 exactly when r < R/2
      return two_rows(row, row + h, h, r < Plan<N>::R[0] / 2 ? idx : idx - N);
    };
    float2 res[PERL][RL];
    auto use = [&](int pp, int qq, int, float2 v) { res[pp][qq] = v; };
    fft_load_use<N, +1, decltype(load), decltype(use), BANDED>(buf, tw, t, load, use);
    for (int d = d0; d < d1; ++d) {
      const size_t o = ((size_t)(clip * po.out_planes + po.list[d]) * N + (RESIST ? i : 2 * i)) * N + t;
#pragma unroll
      for (int pp = 0; pp < PERL; ++pp)
        if (t + pp * NT < N / RL) {
#pragma unroll
          for (int qq = 0; qq < RL; ++qq) {
            const size_t at = o + pp * NT + qq * (N / RL);
            if (RESIST) {
              if (img) img[at] = res[pp][qq].x;
              iblur[at] = res[pp][qq].y;
              if (printed) printed[at] = res[pp][qq].y >= thr ? 1 : 0;
            } else {
              const float a = scale * res[pp][qq].x, b = scale * res[pp][qq].y;
              img[at] = a;
              img[at + N] = b;
              lo = fminf(lo, fminf(a, b));
              hi = fmaxf(hi, fmaxf(a, b));
            }
          }
        }
    }
  }
  if (!RESIST && ext) {
    for (int o = 16; o > 0; o >>= 1) {
      lo = fminf(lo, __shfl_down_sync(0xffffffffu, lo, o));
      hi = fmaxf(hi, __shfl_down_sync(0xffffffffu, hi, o));
    }
    __shared__ float2 warp_ext[(NT + 31) / 32];
    if (t % 32 == 0) warp_ext[t / 32] = make_float2(lo, hi);
    __syncthreads();
    if (t == 0) {
      for (int w = 1; w < (NT + 31) / 32; ++w) {
        lo = fminf(lo, warp_ext[w].x);
        hi = fmaxf(hi, warp_ext[w].y);
      }
      atomicMin(&ext->x, ordered(lo));
      atomicMax(&ext->y, ordered(hi));
    }
  }
}

// ILT forward end on the coarse grid, for a pair of rows (y0, y0 + 1) of a
// full-grid plane from the half band rows of its blur: one inverse transform
// of Bl_y0 + i Bl_y1 gives both blurred rows as its real and imaginary parts.
// The sigmoid resist z = 1 / (1 + e^{-beta (blur - thr)}) (a smooth Eq. (5)),
// the residual d = z - target of the squared-residual ILT loss and
// dL/dI = 2 d beta z (1 - z) follow on the spot; the two dL/dI rows go forward as one complex row
// q[y0] + i q[y1] and leave as their two half spectra, as k_mask_rows writes
// them.  The pair's sum of d^2 goes to partial[plane][pair] in FP64: one
// partial per row pair, whatever the launch shape, so the loss does not
// depend on how clips are grouped.  Plane p belongs to clip
// p / planes_per_clip of `target`.
template <int N>
struct GradRowsShape {
  using PL = Plan<N>;
  static constexpr int NT = PL::NT, R0 = PL::R[0], RL = PL::R[PL::P - 1];
  static constexpr int PERL = (N / RL + NT - 1) / NT;
  // the inverse transform's last pass hands thread t the elements t + NT r,
  // r = p + PERL q, which are the forward first pass's inputs of thread t
  static constexpr bool kRegs = N / R0 == NT && N / RL == PERL * NT && R0 == PERL * RL;
};

template <int N, bool BANDED>
__global__ void __launch_bounds__(Plan<N>::NT, N >= 512 ? 640 / Plan<N>::NT : 1) k_resist_grad_rows(const float2* __restrict__ band, int crop,
                                                                   const float2* __restrict__ tw_g,
                                                                   const float* __restrict__ target,
                                                                   int planes_per_clip,
                                                                   const __grid_constant__ PlaneWeight weight,
                                                                   float beta, float thr,
                                                                   float2* __restrict__ rowbuf,
                                                                   double* __restrict__ partial, int pairs_per_cta) {
  using SH = GradRowsShape<N>;
  constexpr int NT = SH::NT, NW = (NT + 31) / 32, PERL = SH::PERL, RL = SH::RL;
  extern __shared__ float2 smem[];
  float2* tw = smem;
  float2* buf = smem + N;
  // Z(u) on the crop, index u + C/2 (crop + 1 entries); without kRegs, first
  // the pair's dL/dI rows (N entries: x row y0, y row y0 + 1)
  float2* zq = smem + N + PadLen<N>::value;
  __shared__ double wsum[NW];
  pdl_start();
  load_twiddles<N>(tw, tw_g);
  pdl_wait(band, target);
  __syncthreads();
  const int p = blockIdx.y, t = threadIdx.x, half = crop / 2;
  const float* tg = target + (size_t)(p / planes_per_clip) * N * N;
  const float wgt = weight.w[p % planes_per_clip], beta2 = 2.0f * wgt * beta;
  for (int pr = blockIdx.x * pairs_per_cta; pr < min(N / 2, (blockIdx.x + 1) * pairs_per_cta); ++pr) {
    const int y0 = 2 * pr;
    const float2* r0 = band + ((size_t)p * N + y0) * half;
    const float* t0 = tg + (size_t)y0 * N;
    const float* t1 = t0 + N;
    auto load = [&](int, int r, int idx) {  // first pass: idx < N/2 exactly when r < R/2
      return two_rows(r0, r0 + half, half, r < Plan<N>::R[0] / 2 ? idx : idx - N);
    };
    float racc = 0.f;  // this thread's residuals of the pair, summed in FP32 before the FP64 sum
    float2 want[PERL][RL];  // the targets at this thread's outputs, loaded while the later passes run
    auto after_first = [&]() {
#pragma unroll
      for (int pp = 0; pp < PERL; ++pp)
#pragma unroll
        for (int qq = 0; qq < RL; ++qq) {
          const int x = t + pp * NT + qq * (N / RL);
          want[pp][qq] = t + pp * NT < N / RL ? make_float2(ld_dep(t0 + x), ld_dep(t1 + x)) : make_float2(0.f, 0.f);
        }
    };
    float2 qreg[SH::kRegs ? SH::R0 : 1];
    auto use = [&](int pp, int qq, int x, float2 v) {
      const float z0 = 1.0f / (1.0f + expf(-beta * (v.x - thr)));
      const float z1 = 1.0f / (1.0f + expf(-beta * (v.y - thr)));
      const float d0 = z0 - want[pp][qq].x, d1 = z1 - want[pp][qq].y;
      racc = fmaf(d0, d0, fmaf(d1, d1, racc));
      const float2 q = make_float2(beta2 * d0 * z0 * (1.0f - z0), beta2 * d1 * z1 * (1.0f - z1));
      if constexpr (SH::kRegs)
        qreg[pp + PERL * qq] = q;
      else
        zq[x] = q;
    };
    fft_load_use<N, +1, decltype(load), decltype(use), BANDED>(buf, tw, t, load, use, after_first);
    double acc = double(racc);
    auto usez = [&](int, int, int idx, float2 v) {
      const int u = freq_of(idx, N);
      if (u >= -half && u <= half) zq[u + half] = v;
      if (u == -N / 2 && half == N / 2) zq[crop] = v;  // crop == N: Z(N/2) is Z(-N/2)
    };
    if constexpr (SH::kRegs) {
      auto loadq = [&](int, int r, int) { return qreg[r]; };
      fft_load_use<N, -1, decltype(loadq), decltype(usez), false>(buf, tw, t, loadq, usez);
    } else {
      __syncthreads();  // both dL/dI rows in zq
      auto loadz = [&](int, int, int idx) { return zq[idx]; };
      fft_load_use<N, -1, decltype(loadz), decltype(usez), false>(buf, tw, t, loadz, usez);
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (t % 32 == 0) wsum[t / 32] = acc;
    __syncthreads();  // Z on the crop and the warps' sums
    if (t == 0) {
      double sum = 0.0;
      for (int w = 0; w < NW; ++w) sum += wsum[w];
      partial[(size_t)p * (N / 2) + pr] = wgt * sum;
    }
    float2* o0 = rowbuf + ((size_t)p * N + y0) * half;
    float2* o1 = o0 + half;
    for (int k = t; k < half; k += NT) {
      const float2 zp = zq[half + k], zm = zq[half - k];
      o0[k] = make_float2(0.5f * (zp.x + zm.x), 0.5f * (zp.y - zm.y));
      o1[k] = make_float2(0.5f * (zp.y + zm.y), -0.5f * (zp.x - zm.x));
    }
  }
}

template <int N, bool RESIST>
cudaError_t band_rows_n(const float2* q, int clips, int planes, int h, float scale, const float2* tw, float thr,
                        float* img, float* iblur, uint8_t* printed, const PlaneOut& po, cudaStream_t st,
                        uint2* ext = nullptr) {
  const int units = RESIST ? N : N / 2;
  const int per = rows_per_cta(units, clips * planes, Plan<N>::NT, 8 * (N + PadLen<N>::value)), grid = (units + per - 1) / per;
  auto kern = 4 * h <= N ? k_band_rows<N, true, RESIST> : k_band_rows<N, false, RESIST>;
  return launch_pdl(kern, dim3(grid, clips * planes), Plan<N>::NT, 0, st, q, h, scale, tw, thr, img, iblur, printed,
                    planes, po, per, ext);
}

template <int N>
cudaError_t resist_grad_rows_n(const float2* band, int planes, int crop, const float2* tw, const float* target,
                               int planes_per_clip, const PlaneWeight& weight, float beta, float thr, float2* rowbuf,
                               double* partial, cudaStream_t st) {
  static_assert(Plan<N>::NT % 32 == 0, "whole warps");
  const size_t sm = sizeof(float2) * (N + PadLen<N>::value + (GradRowsShape<N>::kRegs ? crop + 1 : N + 1));
  const int ppc = rows_per_cta(N / 2, planes, Plan<N>::NT, sm), grid = (N / 2 + ppc - 1) / ppc;
  auto kern = 2 * crop <= N ? k_resist_grad_rows<N, true> : k_resist_grad_rows<N, false>;
  cudaError_t e = smem_attrs(kern, sm);
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, dim3(grid, planes), Plan<N>::NT, sm, st, band, crop, tw, target, planes_per_clip, weight,
                    beta, thr, rowbuf, partial, ppc);
}

template <int N, int W, bool MIRROR>
cudaError_t mask_cols_w(const float2* rowbuf, int b, int crop, int cols, int ld, const float2* tw, const float* gain,
                        float2* mhat, cudaStream_t st) {
  const size_t sm = sizeof(float2) * (N + size_t(W) * ((PadLen<N>::value + 15) / 16 * 16 + 16 / W));
  cudaError_t e = smem_attrs(k_mask_cols<N, W, MIRROR>, sm);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_mask_cols<N, W, MIRROR>, dim3((cols + W - 1) / W, b), Plan<N>::NT * W, sm, st, rowbuf, crop,
                    cols, ld, tw, gain, mhat);
}

template <int N>
cudaError_t load_mask_cols_n() {
  cudaError_t e = load_kernel(k_mask_cols<N, 4, true>);
  if (e == cudaSuccess) e = load_kernel(k_mask_cols<N, 8, true>);
  if (e == cudaSuccess) e = load_kernel(k_mask_cols<N, 4, false>);
  return e != cudaSuccess ? e : load_kernel(k_mask_cols<N, 8, false>);
}

// Half rows of the mask spectrum (whole: with k = crop/2) or of any real plane.
inline int half_cols(int crop, bool whole) { return crop / 2 + (whole ? 1 : 0); }
inline int half_ld(int crop, bool whole) { return crop / 2 + (whole ? 8 : 0); }

template <int N>
cudaError_t mask_cols_n(const float2* rowbuf, int b, int crop, const float2* tw, float2* mhat, const float* gain,
                        bool whole, cudaStream_t st) {
  const int cols = half_cols(crop, whole), ld = half_ld(crop, whole);
  // 8 columns a CTA (64-byte pieces of a row); 4 (whole 32-byte sectors) while that leaves SMs without a CTA
  const bool few = (long long)b * ((cols + 7) / 8) < 152;
  if (whole)
    return few ? mask_cols_w<N, 4, true>(rowbuf, b, crop, cols, ld, tw, gain, mhat, st)
               : mask_cols_w<N, 8, true>(rowbuf, b, crop, cols, ld, tw, gain, mhat, st);
  return few ? mask_cols_w<N, 4, false>(rowbuf, b, crop, cols, ld, tw, gain, mhat, st)
             : mask_cols_w<N, 8, false>(rowbuf, b, crop, cols, ld, tw, gain, mhat, st);
}

template <int N>
cudaError_t mask_rows_n(const float* m, RowInput in, float alpha, int b, int crop, const float2* tw, float2* rowbuf,
                        bool whole, cudaStream_t st, float* copy = nullptr, size_t copy_stride = 0) {
  const size_t smr = sizeof(float2) * (2 * N + PadLen<N>::value + 1);
  auto kern = in == RowInput::Sigmoid ? k_mask_rows<N, RowInput::Sigmoid>
              : in == RowInput::Copy  ? k_mask_rows<N, RowInput::Copy>
                                      : k_mask_rows<N, RowInput::Mask>;
  cudaError_t e = smem_attrs(kern, smr);
  if (e != cudaSuccess) return e;
  const int ppc = rows_per_cta(N / 2, b, Plan<N>::NT, smr);
  return launch_pdl(kern, dim3((N / 2 + ppc - 1) / ppc, b), Plan<N>::NT, smr, st, m, alpha, crop, tw, rowbuf,
                    half_cols(crop, whole), half_ld(crop, whole), ppc, copy, copy_stride);
}

template <int N>
cudaError_t stage1_n(const float2* mhat, const float2* phi, int nk, int crop, const float2* tw, float2* t1,
                     cudaStream_t st, int clips) {
  return launch_stage1_cols<N, Stage1W<N>::W>(mhat, phi, nk, crop, tw, OutC64{t1, N, crop}, st, clips);
}

// Only the columns u >= 0 of nk spectra (index u + crop/2), written as half rows.
template <int N>
cudaError_t stage1_half_n(const float2* spec, int nk, int crop, const float2* tw, float2* q, int ld,
                          cudaStream_t st) {
  return launch_stage1_cols<N, Stage1W<N>::W>(spec, nullptr, nk, crop, tw, OutHalf{q, N, crop / 2, ld}, st, 1,
                                              crop / 2);
}

template <int N>
cudaError_t stage2_n(const float2* t1, const FieldSet& fs, int clips, int crop, float dose, const float2* tw,
                     float* img, const PlaneOut& po, cudaStream_t st) {
  const dim3 grid(N, clips * fs.planes);
  constexpr int G = Stage2Halves<N>::value ? 2 : 1;
  const int rows = N * clips * fs.planes;
  if (G > 1 && fs.fields() >= 8 * fs.planes && rows >= 768 && rows <= 3072) {
    auto kern = 2 * crop <= N ? k_stage2<N, true, G> : k_stage2<N, false, G>;
    return launch_pdl(kern, grid, Plan<N>::NT * G, 0, st, t1, fs, crop, dose, tw, img, po);
  }
  auto kern = 2 * crop <= N ? k_stage2<N, true, 1> : k_stage2<N, false, 1>;
  return launch_pdl(kern, grid, Plan<N>::NT, 0, st, t1, fs, crop, dose, tw, img, po);
}

template <int N>
cudaError_t load_stage2_n(int crop) {
  if constexpr (Stage2Halves<N>::value) {
    cudaError_t e = load_kernel(2 * crop <= N ? k_stage2<N, true, 1> : k_stage2<N, false, 1>);
    return e != cudaSuccess ? e : load_kernel(2 * crop <= N ? k_stage2<N, true, 2> : k_stage2<N, false, 2>);
  }
  return cudaSuccess;  // one shape
}

// Transform sizes of the full grid (powers of two) ...
#define LITHO_DISPATCH_N(n, CALL)          \
  switch (n) {                             \
    case 32: return CALL(32);              \
    case 64: return CALL(64);              \
    case 128: return CALL(128);            \
    case 256: return CALL(256);            \
    case 512: return CALL(512);            \
    case 1024: return CALL(1024);          \
    case 2048: return CALL(2048);          \
    default: return cudaErrorInvalidValue; \
  }

// ... and of the forward transforms on a coarse grid (also 896, tensor-core path)
#define LITHO_DISPATCH_NC(n, CALL)          \
  switch (n) {                             \
    case 32: return CALL(32);              \
    case 64: return CALL(64);              \
    case 128: return CALL(128);            \
    case 256: return CALL(256);            \
    case 512: return CALL(512);            \
    case 1024: return CALL(1024);          \
    case 2048: return CALL(2048);          \
    case 896: return CALL(896);            \
    default: return cudaErrorInvalidValue; \
  }

}  // namespace

bool fft_twiddle_table(int n, float2* out) {
  switch (n) {
    case 32: fill_twiddle_table<32>(out); return true;
    case 64: fill_twiddle_table<64>(out); return true;
    case 128: fill_twiddle_table<128>(out); return true;
    case 256: fill_twiddle_table<256>(out); return true;
    case 512: fill_twiddle_table<512>(out); return true;
    case 1024: fill_twiddle_table<1024>(out); return true;
    case 2048: fill_twiddle_table<2048>(out); return true;
    case 896: fill_twiddle_table<896>(out); return true;
    default: return false;
  }
}

cudaError_t launch_mask_spectrum(const float* m, int b, int n, int crop, const float2* tw, float2* rowbuf,
                                 float2* mhat, cudaStream_t st) {
  cudaError_t e = launch_mask_rows(m, b, n, crop, tw, rowbuf, true, st);
  return e != cudaSuccess ? e : launch_mask_cols(rowbuf, b, n, crop, tw, mhat, nullptr, true, st);
}

cudaError_t launch_band_rows_real(const float2* q, int clips, int planes, int n, int h, float scale, const float2* tw,
                                  float* out, const PlaneOut& po, cudaStream_t st, uint2* ext) {
#define CALL(N) band_rows_n<N, false>(q, clips, planes, h, scale, tw, 0.f, out, nullptr, nullptr, po, st, ext)
  LITHO_DISPATCH_N(n, CALL)
#undef CALL
}

cudaError_t launch_mask_rows(const float* m, int b, int n, int crop, const float2* tw, float2* rowbuf, bool whole,
                             cudaStream_t st) {
#define CALL(N) mask_rows_n<N>(m, RowInput::Mask, 0.f, b, crop, tw, rowbuf, whole, st)
  LITHO_DISPATCH_NC(n, CALL)
#undef CALL
}

cudaError_t launch_sigmoid_spectrum(const float* theta, float alpha, int b, int n, int crop, const float2* tw,
                                    float2* rowbuf, float2* mhat, cudaStream_t st) {
  auto rows = [&]() {
#define CALL(N) mask_rows_n<N>(theta, RowInput::Sigmoid, alpha, b, crop, tw, rowbuf, true, st)
    LITHO_DISPATCH_N(n, CALL)
#undef CALL
  };
  const cudaError_t e = rows();
  return e != cudaSuccess ? e : launch_mask_cols(rowbuf, b, n, crop, tw, mhat, nullptr, true, st);
}

cudaError_t launch_mask_spectrum_copy(const float* m, int b, int n, int crop, const float2* tw, float2* rowbuf,
                                      float2* mhat, float* copy, size_t copy_stride, cudaStream_t st) {
  auto rows = [&]() {
#define CALL(N) mask_rows_n<N>(m, RowInput::Copy, 0.f, b, crop, tw, rowbuf, true, st, copy, copy_stride)
    LITHO_DISPATCH_N(n, CALL)
#undef CALL
  };
  const cudaError_t e = rows();
  return e != cudaSuccess ? e : launch_mask_cols(rowbuf, b, n, crop, tw, mhat, nullptr, true, st);
}

cudaError_t launch_blur_gain(const ResistTaps& taps, int n, int crop, float* gain, cudaStream_t st) {
  if (n < 1 || crop < 1) return cudaErrorInvalidValue;
  return launch_pdl(k_blur_gain, (crop + 127) / 128, 128, 0, st, taps, n, crop, gain);
}

cudaError_t launch_resist_grad_rows(const float2* band, int planes, int n, int crop, const float2* tw,
                                    const float* target, int planes_per_clip, const PlaneWeight& weight, float beta,
                                    float thr, float2* rowbuf, double* partial, cudaStream_t st) {
#define CALL(N) \
  resist_grad_rows_n<N>(band, planes, crop, tw, target, planes_per_clip, weight, beta, thr, rowbuf, partial, st)
  LITHO_DISPATCH_N(n, CALL)
#undef CALL
}
cudaError_t launch_mask_cols(const float2* rowbuf, int b, int n, int crop, const float2* tw, float2* mhat,
                             const float* gain, bool whole, cudaStream_t st) {
#define CALL(N) mask_cols_n<N>(rowbuf, b, crop, tw, mhat, gain, whole, st)
  LITHO_DISPATCH_NC(n, CALL)
#undef CALL
}
cudaError_t launch_band_rows_resist(const float2* q, int clips, int planes, int n, int h, const float2* tw,
                                    float threshold, float* img, float* iblur, uint8_t* printed, const PlaneOut& po,
                                    cudaStream_t st) {
#define CALL(N) band_rows_n<N, true>(q, clips, planes, h, 1.0f, tw, threshold, img, iblur, printed, po, st)
  LITHO_DISPATCH_N(n, CALL)
#undef CALL
}

cudaError_t launch_stage1_half(const float2* spec, int nk, int n, int crop, const float2* tw, float2* q, int ld,
                               cudaStream_t st) {
#define CALL(N) stage1_half_n<N>(spec, nk, crop, tw, q, ld, st)
  LITHO_DISPATCH_N(n, CALL)
#undef CALL
}

cudaError_t launch_stage1_fft(const float2* mhat, const float2* phi, int nk, int n, int crop, const float2* tw,
                              float2* t1, cudaStream_t st, int clips) {
  if (nk == 0) return cudaSuccess;  // every kernel has lambda = 0: no field
#define CALL(N) stage1_n<N>(mhat, phi, nk, crop, tw, t1, st, clips)
  LITHO_DISPATCH_N(n, CALL)
#undef CALL
}

cudaError_t load_clip_shapes(int n, int nc, int crop) {
  auto cols = [&](int m) {
#define CALL(N) load_mask_cols_n<N>()
    LITHO_DISPATCH_NC(m, CALL)
#undef CALL
  };
  auto rows = [&](int m) {
    if (stage2_w32_supported(m, crop)) return load_stage2_w32(crop);
#define CALL(N) load_stage2_n<N>(crop)
    LITHO_DISPATCH_N(m, CALL)
#undef CALL
  };
  cudaError_t e = cols(n);
  if (e == cudaSuccess) e = rows(n);
  if (e == cudaSuccess && nc > 0) e = rows(nc);
  return e;
}

cudaError_t launch_stage2_fft(const float2* t1, const FieldSet& fs, int clips, int n, int crop, float dose,
                              const float2* tw, float* img, const PlaneOut& po, cudaStream_t st, const float2* tw32,
                              const float2* tw512, float2* spec, int spec_crop) {
  if (tw32 && stage2_w32_supported(n, crop))
    return launch_stage2_w32(t1, fs, clips, n, crop, dose, tw32, img, po, st, spec, spec_crop);
  if (spec) return cudaErrorInvalidValue;  // only the warp-per-row kernel writes row spectra
  if (tw512 && stage2_w512_supported(n, crop))
    return launch_stage2_w512(t1, fs, clips, n, crop, dose, tw512, img, po, st);
#define CALL(N) stage2_n<N>(t1, fs, clips, crop, dose, tw, img, po, st)
  LITHO_DISPATCH_N(n, CALL)
#undef CALL
}

}  // namespace litho
