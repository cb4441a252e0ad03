// Input channels of the AI initialiser (paper Eq. (9)) and its
// lithography-consistency images (Eqs. (15)-(17)).
//
// Eq. (9), as read here: X[c] = (Z_t, I0 / max I0, (dI/dM - min) / (max - min))
// with I0 the aerial image of the target at one focus plane, dI/dM the
// gradient of the plane's total intensity with respect to the mask pixels
// (the adjoint of Eq. (4) applied to ones, as litho_intensity_vjp computes
// it; both channels come from one set of stage-1 fields, see ai_channels)
// and the extremes taken over the whole batch (a constant channel maps to 0).
// Eqs. (15)-(17): Z_round = [G (x) Z_t >= tau_round] with the resist's
// periodic Gaussian, Z_print = [I >= tau_print], L_litho = sum |Z_print -
// Z_round| per clip (an integer count, reduced in a fixed order).
#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstdint>

#include "fft_common.cuh"
#include "litho_internal.h"

namespace litho {

namespace {

constexpr int kReduceThreads = 256;

// Blocks per clip of a pass over b clips: about eight CTAs of kReduceThreads per SM in all.
unsigned blocks_per_clip(int b, size_t items) {
  const size_t want = std::max<size_t>(1, size_t(8) * 152 / b);
  return unsigned(std::max<size_t>(1, std::min(want, (items + kReduceThreads - 1) / kReduceThreads)));
}

// Extremes of one channel of X[b][3][nn] (clip blockIdx.y; x at the channel) into *ext = (min, max), as
// ordered integers: (~0, 0) on entry.  nn is a multiple of 4.  For the channels whose rows are not written
// by k_band_rows, which folds them in as it goes.
__global__ void __launch_bounds__(kReduceThreads) k_minmax(const float4* __restrict__ x, size_t nn4,
                                                           uint2* __restrict__ ext) {
  __shared__ float smin[kReduceThreads / 32], smax[kReduceThreads / 32];
  float lo = FLT_MAX, hi = -FLT_MAX;
  const float4* src = x + size_t(blockIdx.y) * 3 * nn4;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nn4; i += (size_t)gridDim.x * blockDim.x) {
    const float4 v = src[i];
    lo = fminf(lo, fminf(fminf(v.x, v.y), fminf(v.z, v.w)));
    hi = fmaxf(hi, fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w)));
  }
  for (int o = 16; o > 0; o >>= 1) {
    lo = fminf(lo, __shfl_down_sync(0xffffffffu, lo, o));
    hi = fmaxf(hi, __shfl_down_sync(0xffffffffu, hi, o));
  }
  if (threadIdx.x % 32 == 0) {
    smin[threadIdx.x / 32] = lo;
    smax[threadIdx.x / 32] = hi;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kReduceThreads / 32; ++w) {
      lo = fminf(lo, smin[w]);
      hi = fmaxf(hi, smax[w]);
    }
    atomicMin(&ext->x, ordered(lo));
    atomicMax(&ext->y, ordered(hi));
  }
}

// Channels 1 and 2 of every clip: v -> (v - lo) s with lo = 0, s = 1/max (channel 1) or lo = min,
// s = 1/(max - min) (channel 2); s = 0 when the range is empty.
__global__ void __launch_bounds__(kReduceThreads) k_normalize(float4* __restrict__ x, size_t nn4,
                                                              const uint2* __restrict__ ext) {
  const uint2 e = ext[blockIdx.z];
  const float lo = blockIdx.z == 0 ? 0.f : from_ordered(e.x), hi = from_ordered(e.y);
  const float s = hi > lo ? 1.0f / (hi - lo) : 0.f;
  float4* dst = x + (size_t(blockIdx.y) * 3 + 1 + blockIdx.z) * nn4;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nn4; i += (size_t)gridDim.x * blockDim.x) {
    float4 v = dst[i];
    v.x = (v.x - lo) * s;
    v.y = (v.y - lo) * s;
    v.z = (v.z - lo) * s;
    v.w = (v.w - lo) * s;
    dst[i] = v;
  }
}

// z_print = [I >= thr], 16 pixels a step and thread, and, with `out`, the number of pixels where it
// differs from z_round, per clip (grid y): the XOR of two 0/1 bytes is one bit; each block adds its
// count to the clip's total with an integer atomic (exact, so the result does not depend on the
// order).  out must be zero on entry.  VEC: I is 16-byte aligned.  HBM-bound: 5 bytes a pixel read, 1
// written (a threshold kernel and a counting one that read both prints again took 150 us for 16
// planes of 2048^2, this one 62 us).
template <bool VEC>
__global__ void __launch_bounds__(kReduceThreads) k_print(const float* __restrict__ img, float thr,
                                                          const uint4* __restrict__ z_round, size_t pieces,
                                                          uint4* __restrict__ z_print,
                                                          unsigned long long* __restrict__ out) {
  __shared__ unsigned warp_sum[kReduceThreads / 32];
  pdl_start();
  pdl_wait(img, z_round);
  const size_t base = size_t(blockIdx.y) * pieces;
  unsigned c = 0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < pieces; i += (size_t)gridDim.x * blockDim.x) {
    unsigned z[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float4 v;
      const float* s = img + (base + i) * 16 + 4 * q;
      if constexpr (VEC)
        v = ld_dep(reinterpret_cast<const float4*>(s));
      else
        v = make_float4(ld_dep(s), ld_dep(s + 1), ld_dep(s + 2), ld_dep(s + 3));
      z[q] = unsigned(v.x >= thr) | unsigned(v.y >= thr) << 8 | unsigned(v.z >= thr) << 16 | unsigned(v.w >= thr) << 24;
    }
    z_print[base + i] = make_uint4(z[0], z[1], z[2], z[3]);
    if (out) {
      const uint4 r = z_round[base + i];
      c += __popc(z[0] ^ r.x) + __popc(z[1] ^ r.y) + __popc(z[2] ^ r.z) + __popc(z[3] ^ r.w);
    }
  }
  if (!out) return;
  for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
  if (threadIdx.x % 32 == 0) warp_sum[threadIdx.x / 32] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long t = 0;
    for (int w = 0; w < kReduceThreads / 32; ++w) t += warp_sum[w];
    if (t) atomicAdd(out + blockIdx.y, t);
  }
}

size_t up256(size_t x) { return (x + 255) / 256 * 256; }

}  // namespace

}  // namespace litho

using namespace litho;

extern "C" {

litho_status litho_ai_inputs_workspace_size(const litho_kernels* h, int b, size_t* bytes) {
  if (!h || !bytes || b < 1) {
    set_error("null argument or b < 1");
    return LITHO_EINVAL;
  }
  *bytes = up256(ai_channels_bytes(h, b)) + up256(2 * sizeof(uint2));
  return LITHO_OK;
}

litho_status litho_ai_inputs(const litho_kernels* h, const float* target_dev, int b, double dose, int focus,
                             litho_precision prec, float* x_dev, void* workspace_dev, size_t workspace_bytes,
                             void* stream) {
  if (!h || !target_dev || !x_dev || !workspace_dev || b < 1 || b > 65535) {
    set_error("null argument or b outside [1, 65535]");
    return LITHO_EINVAL;
  }
  if (focus < 0 || focus >= h->n_focus || !std::isfinite(dose)) {
    set_error("focus must index a plane of the kernel set; dose finite");
    return LITHO_EINVAL;
  }
  if ((int(prec) & ~LITHO_GRID_COARSE) != LITHO_PREC_FFT32) {
    set_error("litho_ai_inputs implements the FP32 FFT path only (LITHO_PREC_FFT32, optionally | LITHO_GRID_COARSE)");
    return LITHO_EUNSUPPORTED;
  }
  size_t need = 0;
  litho_status s = litho_ai_inputs_workspace_size(h, b, &need);
  if (s != LITHO_OK) return s;
  if (workspace_bytes < need || (reinterpret_cast<uintptr_t>(workspace_dev) & 255) != 0) {
    set_error("workspace must be 256-byte aligned and hold %zu bytes (%zu given)", need, workspace_bytes);
    return workspace_bytes < need ? LITHO_ENOMEM : LITHO_EINVAL;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const size_t nn = size_t(h->n) * h->n;
  uint2* ext = reinterpret_cast<uint2*>(static_cast<char*>(workspace_dev) + up256(ai_channels_bytes(h, b)));
  for (int ch = 0; ch < 2; ++ch) {  // (~0, 0): nothing seen yet
    LITHO_TRY_CUDA(cudaMemsetAsync(&ext[ch].x, 0xff, sizeof(unsigned), st));
    LITHO_TRY_CUDA(cudaMemsetAsync(&ext[ch].y, 0, sizeof(unsigned), st));
  }
  bool found[2];
  s = ai_channels(h, target_dev, b, dose, focus, (int(prec) & LITHO_GRID_COARSE) != 0, x_dev, workspace_dev, ext, found,
                  st);
  if (s != LITHO_OK) return s;
  ProfScope ps(kStageIltReduce, st, 1);
  for (int ch = 0; ch < 2; ++ch)
    if (!found[ch])
      k_minmax<<<dim3(blocks_per_clip(b, nn / 4), b), kReduceThreads, 0, st>>>(
          reinterpret_cast<const float4*>(x_dev + (1 + ch) * nn), nn / 4, ext + ch);
  const dim3 grid(blocks_per_clip(2 * b, nn / 4), b, 2);
  k_normalize<<<grid, kReduceThreads, 0, st>>>(reinterpret_cast<float4*>(x_dev), nn / 4, ext);
  LITHO_TRY_CUDA(cudaGetLastError());
  return LITHO_OK;
}

litho_status litho_print_images(const float* target_dev, const float* intensity_dev, int b, int n, double pixel_nm,
                                double sigma_round_nm, double tau_round, double tau_print, uint8_t* z_round_dev,
                                uint8_t* z_print_dev, int64_t* loss_dev, float* blur_dev, void* stream) {
  if (!target_dev || !intensity_dev || !z_round_dev || !z_print_dev || !blur_dev || b < 1 || n < 32 || n % 32) {
    set_error("null argument, b < 1, or n not a multiple of 32");
    return LITHO_EINVAL;
  }
  if (!std::isfinite(tau_round) || !std::isfinite(tau_print)) {
    set_error("thresholds must be finite");
    return LITHO_EINVAL;
  }
  if (((reinterpret_cast<uintptr_t>(z_round_dev) | reinterpret_cast<uintptr_t>(z_print_dev)) & 15) != 0) {
    set_error("z_round_dev and z_print_dev must be 16-byte aligned");
    return LITHO_EINVAL;
  }
  ResistTaps taps;
  std::string why;
  if (!resist_taps(sigma_round_nm, pixel_nm, &taps, &why)) {
    set_error("%s", why.c_str());
    return LITHO_EINVAL;
  }
  if (2 * taps.radius >= n) {
    set_error("blur radius must be below n/2");
    return LITHO_EINVAL;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const size_t nn = size_t(n) * n;
  ProfScope ps(kStageResist, st, 2);
  if (loss_dev) LITHO_TRY_CUDA(cudaMemsetAsync(loss_dev, 0, size_t(b) * sizeof(int64_t), st));
  LITHO_TRY_CUDA(launch_resist(target_dev, b, n, taps, float(tau_round), blur_dev, z_round_dev, st));
  const size_t pieces = nn / 16;
  const dim3 grid(blocks_per_clip(b, pieces), b);
  auto kern = (reinterpret_cast<uintptr_t>(intensity_dev) & 15) == 0 ? k_print<true> : k_print<false>;
  LITHO_TRY_CUDA(launch_pdl(kern, grid, kReduceThreads, 0, st, intensity_dev, float(tau_print),
                            reinterpret_cast<const uint4*>(z_round_dev), pieces, reinterpret_cast<uint4*>(z_print_dev),
                            reinterpret_cast<unsigned long long*>(loss_dev)));
  LITHO_TRY_CUDA(cudaGetLastError());
  return LITHO_OK;
}

}  // extern "C"
