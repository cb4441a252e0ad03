// Column pass of the exact Fourier interpolation from a coarse grid (paper
// Eq. (4) evaluated on nc x nc, then resampled to N x N): for each column u >= 0
// of the half row spectra R[p][y][u] of coarse images (y in [0, NC)),
//
//   S[v][u] = NC^-2 sum_y R[y][u] e^{-2 pi i v y/NC},   |v| < C2/2
//   A[y][u] = sum_v S[v][u] e^{+2 pi i v y/N},          y in [0, N): the image's half rows
//   B[y][u] = sum_v gain[v] gain[u] S[v][u] e^{...}:    its blur's half rows (with gain)
//
// in one kernel: the forward transform on NC, the crop and the scale, and the
// inverse transform or transforms on N, with the column staying in shared
// memory or registers in between.  The image is real, so the columns u < 0
// are the conjugates of these and are not formed.  Thread layout as in stage
// 1: column w = tid mod W, transform thread t = tid / W, so the loads of R and
// the stores cover W adjacent columns of 32/W rows per warp.
#include "fft_common.cuh"
#include "litho_internal.h"

namespace litho {

namespace {

template <int N, int W>
struct InterpShape {
  static constexpr int LD = (PadLen<N>::value + 15) / 16 * 16 + 16 / W;
};

// IMAGE, BLUR: which of A and B are formed; with both, row y holds A then B.  16 planes 1024 -> 2048 with
// both: 169 -> 140 us; 8 planes of image alone 81 -> 41 us; 24 planes 512 -> 1024 of blur alone (ILT) 56 -> 30
// us (all columns transformed, image and blur as one complex plane).  With both, four columns a CTA and
// two CTAs per SM: the inputs of the second transform stay in registers.
template <int NC, int N, int W, bool IMAGE, bool BLUR>
__global__ void __launch_bounds__(Plan<N>::NT * W, Plan<N>::NT * W <= 512 ? 2 : 1)
    k_interp_cols(const float2* __restrict__ rspec, int h, const float2* __restrict__ tw_nc_g,
                  const float2* __restrict__ tw_n_g, const float* __restrict__ gain, float2* __restrict__ q) {
  constexpr int NT = Plan<N>::NT, NTC = Plan<NC>::NT, T = NT * W, LD = InterpShape<N, W>::LD;
  constexpr bool BANDED = 2 * NC <= N;  // |v| < C2/2 <= NC/2 <= N/4
  constexpr int R0 = Plan<N>::R[0], NB0 = N / R0;
  static_assert(NTC <= NT, "the coarse transform runs on a subset of the threads");
  static_assert(PassShape<N, NT, R0>::PER == 1, "one first-pass butterfly per thread");
  extern __shared__ float4 smem_raw[];
  float2* smem = reinterpret_cast<float2*>(smem_raw);
  float2* tw_n = smem;
  float2* tw_c = smem + N;
  float2* buf = smem + N + NC;
  const int tid = threadIdx.x, g = tid % W, t = tid / W;
  const int u = blockIdx.x * W + g, p = blockIdx.y;
  pdl_start();
  for (int i = tid; i < N; i += T) tw_n[i] = tw_n_g[i];
  for (int i = tid; i < NC; i += T) tw_c[i] = tw_nc_g[i];
  pdl_wait(rspec, gain);
  __syncthreads();
  // forward transform over y on NC, shared by all NT threads of the column
  // (a pass with fewer butterflies than threads leaves the rest idle)
  const float2* src = rspec + (size_t)p * NC * h + u;
  auto load_c = [&](int y) { return ld_dep(src + (size_t)y * h); };
  fft_load_smem<NC, -1, decltype(load_c), false, NT>(buf + g * LD, tw_c, t, load_c);
  // crop and scale: this thread's inputs of the inverse transforms (v = t + r N/R0, the upper half negative)
  const float scale = 1.0f / (float(NC) * float(NC));
  const float gu = BLUR ? ld_dep(gain + h + u) : 0.f;
  float2 s[R0];
#pragma unroll
  for (int r = 0; r < R0; ++r) {
    const int v = t + r * NB0 - (r < R0 / 2 ? 0 : N);
    const bool in = t < NB0 && v > -h && v < h;
    s[r] = make_float2(0.f, 0.f);
    if ((BANDED && r >= R0 / 4 && r < 3 * R0 / 4) || !in) continue;
    const float2 x = buf[g * LD + pad16(v < 0 ? v + NC : v)];
    s[r] = make_float2(x.x * scale, x.y * scale);
  }
  const int ld = IMAGE && BLUR ? 2 * h : h;
  float2* dst = q + (size_t)p * N * ld + u;
  if (IMAGE) {  // the first pass's barrier before its stores follows every thread's reads above
    auto load = [&](int, int r, int) { return s[r]; };
    auto use = [&](int, int, int y, float2 v) { dst[(size_t)y * ld] = v; };
    fft_load_use<N, +1, decltype(load), decltype(use), BANDED>(buf + g * LD, tw_n, t, load, use);
  }
  if (BLUR) {
    if (IMAGE) dst += h;
    auto load = [&](int, int r, int idx) {
      const int v = idx - (r < R0 / 2 ? 0 : N);
      const float gg = v > -h && v < h ? ld_dep(gain + v + h) * gu : 0.f;
      return make_float2(s[r].x * gg, s[r].y * gg);
    };
    auto use = [&](int, int, int y, float2 v) { dst[(size_t)y * ld] = v; };
    fft_load_use<N, +1, decltype(load), decltype(use), BANDED>(buf + g * LD, tw_n, t, load, use);
  }
}

template <int NC, int N, bool IMAGE, bool BLUR>
cudaError_t interp_cols_t(const float2* rspec, int planes, int h, const float2* tw_nc, const float2* tw_n,
                          const float* gain, float2* q, cudaStream_t st) {
  constexpr int W = IMAGE && BLUR && N == 2048 ? 4 : 8;
  if (h % W != 0 || 2 * h > NC) return cudaErrorInvalidValue;
  const size_t sm = sizeof(float2) * (size_t(N) + NC + size_t(W) * InterpShape<N, W>::LD);
  cudaError_t e = smem_attrs(k_interp_cols<NC, N, W, IMAGE, BLUR>, sm);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_interp_cols<NC, N, W, IMAGE, BLUR>, dim3(h / W, planes), Plan<N>::NT * W, sm, st, rspec, h,
                    tw_nc, tw_n, gain, q);
}

template <int NC, int N>
cudaError_t interp_cols_n(const float2* rspec, int planes, int h, const float2* tw_nc, const float2* tw_n,
                          const float* gain, bool image, float2* q, cudaStream_t st) {
  if (!gain) return interp_cols_t<NC, N, true, false>(rspec, planes, h, tw_nc, tw_n, gain, q, st);
  return image ? interp_cols_t<NC, N, true, true>(rspec, planes, h, tw_nc, tw_n, gain, q, st)
               : interp_cols_t<NC, N, false, true>(rspec, planes, h, tw_nc, tw_n, gain, q, st);
}

}  // namespace

bool interp_cols_supported(int nc, int n) {
  if (nc == 896) return n == 1024 || n == 2048;
  return nc >= 32 && (nc == n / 2 || nc == n / 4 || nc == n / 8) && n >= 64 && n <= 2048;
}

cudaError_t launch_interp_cols(const float2* rspec, int planes, int nc, int n, int h, const float2* tw_nc,
                               const float2* tw_n, const float* gain, bool image, float2* q, cudaStream_t st) {
#define IC(NC, N) \
  if (nc == NC && n == N) return interp_cols_n<NC, N>(rspec, planes, h, tw_nc, tw_n, gain, image, q, st);
  IC(1024, 2048) IC(512, 2048) IC(256, 2048) IC(896, 2048)
  IC(512, 1024) IC(256, 1024) IC(128, 1024) IC(896, 1024)
  IC(256, 512) IC(128, 512) IC(64, 512)
  IC(128, 256) IC(64, 256) IC(32, 256)
  IC(64, 128) IC(32, 128)
  IC(32, 64)
#undef IC
  return cudaErrorInvalidValue;
}

}  // namespace litho
