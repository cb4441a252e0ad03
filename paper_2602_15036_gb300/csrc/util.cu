// Small device utilities that belong to no stage of the imaging path.
#include <algorithm>

#include "litho_internal.h"

namespace litho {

namespace {

// One thread spinning on the SM clock for a fixed number of cycles: it always
// ends (no flag or peer is waited on).
__global__ void k_delay(long long cycles) {
  const long long t0 = clock64();
  while (clock64() - t0 < cycles) __nanosleep(1000);
}

// A copy between page-locked host memory and the device by the SMs (T: float4 when both ends allow it).
template <class T>
__global__ void __launch_bounds__(256) k_host_copy(T* __restrict__ dst, const T* __restrict__ src, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    dst[i] = src[i];
}

}  // namespace

cudaError_t launch_host_copy(float* dst, const float* src, size_t floats, cudaStream_t st) {
  const bool vec = ((reinterpret_cast<uintptr_t>(dst) | reinterpret_cast<uintptr_t>(src)) & 15) == 0 && floats % 4 == 0;
  const size_t n = vec ? floats / 4 : floats;
  const unsigned blocks = unsigned(std::min<size_t>((n + 255) / 256, 64));
  if (vec)
    k_host_copy<<<blocks, 256, 0, st>>>(reinterpret_cast<float4*>(dst), reinterpret_cast<const float4*>(src), n);
  else
    k_host_copy<<<blocks, 256, 0, st>>>(dst, src, n);
  return cudaGetLastError();
}

cudaError_t launch_delay(cudaStream_t st, double ms) {
  int dev = 0, khz = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&khz, cudaDevAttrClockRate, dev);
  if (e != cudaSuccess) return e;
  k_delay<<<1, 1, 0, st>>>((long long)(ms * double(khz > 0 ? khz : 2000000)));
  return cudaGetLastError();
}

}  // namespace litho
