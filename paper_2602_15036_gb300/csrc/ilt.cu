// ILT loss and its adjoint (mask gradient) on the FP32 FFT path.
//
// Objective (pixel-based ILT, the paper's Section I prior art; dI/dM is the
// input channel of its Eq. (9)):
//   m = sigmoid(a theta),  I_f = D sum_k lam_fk |E_fk|^2 (Eq. (4)),
//   Ib_f = g (x) I_f (Eq. (5) blur),  Z_f = sigmoid(b (Ib_f - t)),
//   L = sum_f sum_x (Z_f - target)^2.
// Adjoint by the chain rule (g symmetric, so the blur is its own adjoint):
//   q_f = 2 (Z_f - target) b Z_f (1 - Z_f),  G_f = g (x) q_f          (= dL/dI_f)
//   H_fk(u) = sum_x G_f(x) E_fk(x) e^{-2 pi i u.x/N}    on the crop
//   S(u) = sum_f sum_k lam_fk conj(Phi_fk(u)) H_fk(u)
// with sqrt(lam) Phi replaced by the kernel set's Psi, which give the same I (kernelset.cu).
//   dL/dm(x) = 2 D N^-2 Re sum_u S(u) e^{+2 pi i u.x/N},  dL/dtheta = dL/dm a m (1 - m).
//
// Kernels (per clip, for a group of P focus planes at a time):
//   (mask spectrum of sigmoid(a theta), stage 1, stage 2, resist blur: shared with the forward path)
//   k_resist_grad    Z, q and per-block FP64 partial sums of (Z - target)^2
//                    (coarse grid: k_resist_grad_rows, per row pair, with the
//                    forward row spectra of q)
//   k_adj_rows       per image row: E_fk from the stage-1 field (inverse FFT),
//                    times G_f, forward FFT, crop columns -> U_fk[y][c]
//   k_adj_cols       per crop column block and run of a clip's fields: forward
//                    FFT over y, crop rows, times conj(Psi), summed over
//                    the run in registers -> one partial S per run
//   k_sum_planes     S = sum of a clip's runs in fixed order, and the fixed-order
//                    FP64 sum of its loss partials (deterministic)
//   k_grad_rows      band-to-full inverse of S along x (after stage 1 along y),
//                    real part, chain factor -> dL/dtheta
// The fields E are never stored: each backward row recomputes E_fk from the
// stage-1 field T_fk (C values per row) that the forward pass kept.
#include <algorithm>
#include <cmath>

#include "fft_common.cuh"
#include "litho_internal.h"

namespace litho {

namespace {

constexpr int kPartials = 1024;  // blocks of k_resist_grad, fixed for a deterministic reduction

__device__ __forceinline__ int freq_of_idx(int idx, int n) { return idx < n / 2 ? idx : idx - n; }

// Clip blockIdx.y: its `planes` planes of ib and q, its target, its
// kPartials partial sums (the same partition for every group size).
__global__ void __launch_bounds__(256) k_resist_grad(const float* __restrict__ ib, const float* __restrict__ target,
                                                     size_t nn, int planes, const __grid_constant__ PlaneWeight weight,
                                                     float beta, float thr, float* __restrict__ q,
                                                     double* __restrict__ partial) {
  pdl_start();
  pdl_wait(ib, target);
  const size_t clip = blockIdx.y;
  ib += clip * planes * nn;
  q += clip * planes * nn;
  target += clip * nn;
  partial += clip * gridDim.x;
  double acc = 0.0;
  const size_t total = nn * planes, stride = (size_t)gridDim.x * blockDim.x;
  size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  int pl = int(i / nn);
  size_t pix = i - pl * nn;  // i mod nn and i div nn, carried along instead of recomputed
  for (; i < total; i += stride) {
    const float z = 1.0f / (1.0f + expf(-beta * (ld_dep(ib + i) - thr)));
    const float d = z - ld_dep(target + pix), w = weight.w[pl];
    acc += double(w) * double(d) * double(d);
    q[i] = 2.0f * w * d * beta * z * (1.0f - z);
    pix += stride;
    while (pix >= nn) {
      pix -= nn;
      ++pl;
    }
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  __shared__ double ws[8];
  if (threadIdx.x % 32 == 0) ws[threadIdx.x / 32] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < 8; ++w) s += ws[w];
    partial[blockIdx.x] = s;
  }
}

// Backward rows: for every kernel of the plane, E = inverse FFT of the band row
// T[y][:], P = G[y][:] E, U[y][c] = forward FFT of P on the crop columns.
// Planes of a clip and their fields as in `fs`; plane pl of clip i takes G at plane i g_planes + pl of g.
// BANDED (2 crop <= N): the band row's zero half is skipped in the first pass.
// CTA z of gridDim.z takes every gridDim.z-th field of its plane (the fields are independent).
template <int N, bool BANDED>
__global__ void __launch_bounds__(Plan<N>::NT) k_adj_rows(const float2* __restrict__ t1,
                                                          const __grid_constant__ FieldSet fs, int crop,
                                                          const float* __restrict__ g, int g_planes,
                                                          const float2* __restrict__ tw_g, float2* __restrict__ u) {
  using PL = Plan<N>;
  constexpr int NT = PL::NT, RL = PL::R[PL::P - 1];
  constexpr int PERL = PassShape<N, NT, RL>::PER;
  extern __shared__ float2 sm[];
  float2* tw = sm;
  float2* bufa = sm + N;
  float2* bufb = sm + N + PadLen<N>::value;
  pdl_start();
  load_twiddles<N>(tw, tw_g);
  pdl_wait(t1, g);
  const int y = blockIdx.x, plane = blockIdx.y, t = threadIdx.x, half = crop / 2;
  const int clip = plane / fs.planes, pl = plane - clip * fs.planes;
  float gv[PERL][RL];
  const float* grow = g + ((size_t)(clip * g_planes + pl) * N + y) * N;
#pragma unroll
  for (int p = 0; p < PERL; ++p)
#pragma unroll
    for (int q = 0; q < RL; ++q) {
      const int jj = t + p * NT;
      gv[p][q] = jj < N / RL ? ld_dep(grow + jj + q * (N / RL)) : 0.f;
    }
  __syncthreads();
  for (int k = fs.start[pl] + blockIdx.z; k < fs.start[pl + 1]; k += gridDim.z) {
    const size_t rowoff = ((size_t)(clip * fs.fields() + k) * N + y) * crop;
    const float2* row = t1 + rowoff;
    auto load_band = [&](int, int r, int idx) {
      const int c = (r < PL::R[0] / 2 ? idx : idx - N) + half;  // first pass: idx < N/2 exactly when r < R/2
      return ld_dep_if(row + c, c >= 0 && c < crop);
    };
    auto times_g = [&](int p, int q, int idx, float2 v) {
      bufb[pad16(idx)] = make_float2(v.x * gv[p][q], v.y * gv[p][q]);
    };
    fft_load_use<N, +1, decltype(load_band), decltype(times_g), BANDED>(bufa, tw, t, load_band, times_g);
    __syncthreads();
    auto load_prod = [&](int idx) { return bufb[pad16(idx)]; };
    float2* urow = u + rowoff;
    auto store_crop = [&](int, int, int idx, float2 v) {
      const int c = freq_of_idx(idx, N) + half;
      if (c >= 0 && c < crop) urow[c] = v;
    };
    fft_load_use<N, -1>(bufa, tw, t, load_prod, store_crop);
  }
}

// Backward rows for 512-point rows, two rows per warp (same result as
// k_adj_rows<512>): per kernel, E = inverse transform of the band row, P = G E,
// U = forward transform of P on the crop columns.  512 = 16 x 32 in Stockham
// order:
//   inverse pass 1 (radix 16): lane l takes x[l + 32 r] of both rows -> 16 l + q;
//   inverse pass 2 (radix 32): lanes 0-15 take row A, lanes 16-31 row B; lane j
//     takes position j + 16 r, applies w^(r j) (w = e^{+2 pi i/512}) and forms a
//     32-point DFT whose output q is E(x) at x = j + 16 q;
//   forward pass 1 (radix 32): the forward transform's first butterfly j needs
//     P(j + 16 r), r < 32 -- exactly what lane j holds, so P = G E and this
//     pass stay in registers (output q at 32 j + q);
//   forward pass 2 (radix 16): lane l takes position l + 32 r of both rows,
//     applies conj(w)^(r l) and forms a 16-point DFT whose output q is U(u) at
//     u = l + 32 q; the crop columns are stored.
// Two shared-memory exchanges per row and kernel (padded i + i/16 and
// i + i/32, conflict-free), no block barrier inside the kernel loop; the next
// kernel's band rows are staged with cp.async while the current ones are
// transformed.  BANDED: crop / 2 <= 128, so inputs r in [4, 12) of the first
// pass are zero.
constexpr int kAdjWarps = 8;
constexpr int kAdjTw1 = 31 * 16, kAdjTw2 = 15 * 32;  // w^(r j), r < 32, j < 16; conj(w)^(r l), r < 16, l < 32
constexpr int kAdjBuf = 512 + 32;                     // one row, either padding

__device__ __forceinline__ void adj_cp16(void* smem_dst, const void* gmem_src) {
  const unsigned sa = static_cast<unsigned>(__cvta_generic_to_shared(smem_dst));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gmem_src) : "memory");
}

template <bool BANDED>
__global__ void __launch_bounds__(32 * kAdjWarps, 2)
    k_adj_rows_w512(const float2* __restrict__ t1, const __grid_constant__ FieldSet fs, int crop,
                    const float* __restrict__ g, int g_planes, const float2* __restrict__ tw_g,
                    float2* __restrict__ u) {
  constexpr int N = 512;
  extern __shared__ float4 smem_raw[];
  float2* tw1 = reinterpret_cast<float2*>(smem_raw);  // inverse pass 2: (r - 1) 16 + j
  float2* tw2 = tw1 + kAdjTw1;                        // forward pass 2: (r - 1) 32 + l
  float2* bufs = tw2 + kAdjTw2;                       // [warp][2 rows][kAdjBuf]
  float2* stage0 = bufs + kAdjWarps * 2 * kAdjBuf;    // [warp][2 rows][crop]
  pdl_start();
  for (int i = threadIdx.x; i < kAdjTw1 + kAdjTw2; i += blockDim.x) tw1[i] = tw_g[i];
  pdl_wait(g);
  __syncthreads();
  const int lane = threadIdx.x % 32, wp = threadIdx.x / 32, half = crop / 2;
  const int y0 = (blockIdx.x * kAdjWarps + wp) * 2, plane = blockIdx.y;
  if (y0 >= N) return;  // no block barrier below
  float2* buf = bufs + wp * 2 * kAdjBuf;
  float2* stage = stage0 + (size_t)wp * 2 * crop;
  const int clip = plane / fs.planes, pl = plane - clip * fs.planes, nk = fs.start[pl + 1] - fs.start[pl];
  const size_t field = (size_t)N * crop, first = (size_t)(clip * fs.fields() + fs.start[pl]) * field;
  const float2* t1p = t1 + first;
  float2* up = u + first;
  // this lane's row in passes 2 and 3 (inverse pass 2, forward pass 1) and its butterfly
  const int rsel = lane / 16, jj = lane % 16;
  float gv[32];  // G(y, jj + 16 q) of the lane's row
  {
    const float* grow = g + ((size_t)(clip * g_planes + pl) * N + y0 + rsel) * N;
#pragma unroll
    for (int q = 0; q < 32; ++q) gv[q] = ld_dep(grow + jj + 16 * q);
  }
  auto fetch = [&](int k) {  // band rows y0, y0 + 1 of kernel k: 2 x crop/2 pieces of 16 bytes
    const float2* src = t1p + (size_t)k * field + (size_t)y0 * crop;
    for (int i = lane; i < crop; i += 32) adj_cp16(stage + 2 * i, src + 2 * i);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int kz = gridDim.z;
  if (int(blockIdx.z) < nk) fetch(blockIdx.z);
  for (int k = blockIdx.z; k < nk; k += kz) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncwarp();
    // inverse pass 1 for both rows (lane l: x[l + 32 r])
    float2 a[2][16];
#pragma unroll
    for (int row = 0; row < 2; ++row) {
      const float2* band = stage + row * crop;
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        if (BANDED && r >= 4 && r < 12) {
          a[row][r] = make_float2(0.f, 0.f);
        } else {
          const int idx = lane + 32 * r;
          const int c = (r < 8 ? idx : idx - N) + half;
          a[row][r] = (c >= 0 && c < crop) ? band[c] : make_float2(0.f, 0.f);
        }
      }
    }
    __syncwarp();  // both band rows are in registers: the staging buffer takes the next kernel
    if (k + kz < nk) fetch(k + kz);
#pragma unroll
    for (int row = 0; row < 2; ++row) {
      dft_reg<16, +1, BANDED>(a[row]);
#pragma unroll
      for (int q = 0; q < 16; ++q) buf[row * kAdjBuf + pad16(16 * lane + q)] = a[row][q];
    }
    __syncwarp();
    // inverse pass 2: lane j = jj of row rsel, positions j + 16 r
    float2 v[32];
    const float2* rb = buf + rsel * kAdjBuf;
#pragma unroll
    for (int r = 0; r < 32; ++r) {
      v[r] = rb[pad16(jj + 16 * r)];
      if (r > 0) v[r] = cmul(v[r], tw1[(r - 1) * 16 + jj]);
    }
    __syncwarp();  // the row buffers are read; the forward pass writes them next
    dft32<+1, false>(v);  // v[q] = E(jj + 16 q)
    // P = G E, then forward pass 1 over the same 32 values
#pragma unroll
    for (int q = 0; q < 32; ++q) v[q] = make_float2(v[q].x * gv[q], v[q].y * gv[q]);
    dft32<-1, false>(v);  // output q at 32 jj + q
    float2* wb = buf + rsel * kAdjBuf;
#pragma unroll
    for (int q = 0; q < 32; ++q) wb[32 * jj + q + jj] = v[q];  // padded i + i/32 (i = 32 jj + q)
    __syncwarp();
    // forward pass 2 for both rows: lane l, positions l + 32 r
#pragma unroll
    for (int row = 0; row < 2; ++row) {
      const float2* fb = buf + row * kAdjBuf;
      float2 b[16];
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        const int i = lane + 32 * r;
        b[r] = fb[i + i / 32];
        if (r > 0) b[r] = cmul(b[r], tw2[(r - 1) * 32 + lane]);
      }
      dft_reg<16, -1, false>(b);  // b[q] = U(lane + 32 q)
      float2* urow = up + (size_t)k * field + (size_t)(y0 + row) * crop;
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const int idx = lane + 32 * q;
        const int c = (q < 8 ? idx : idx - N) + half;
        if (c >= 0 && c < crop) urow[c] = b[q];
      }
    }
    __syncwarp();  // the row buffers are free for the next kernel
  }
}

// Backward columns: forward FFT over y of U_j[:, c], crop rows, times conj(Psi_j);
// field j uses kernel j mod period.  W columns per CTA with the lanes of a
// warp interleaved over them (as in stage 1): the first pass reads U straight
// from global memory (W adjacent columns of 32/W rows per warp load: whole
// sectors), the last pass hands each thread the same output positions for
// every field, and a CTA runs a run of fields in turn so that its twiddle
// table is loaded once.
template <int N> struct AdjW { static constexpr int W = Plan<N>::NT <= 64 ? 8 : 4; };

// Where the adjoint columns keep their sums: in registers they cost the
// 512-point kernel its second CTA per SM (or spills), in shared memory they
// cost the 1024-point one (twice the slots); so shared memory up to 512.
template <int N> struct AdjAccInSmem { static constexpr bool value = N <= 512; };

// Runs of fields per clip in the adjoint columns: one field each for up to 16
// fields (a small call's chain of transforms is then one long: 12 fields of 256^2 13.6 -> 10.0 us), else at most
// 8 runs of equal length but for the last.  A function of the clip's field
// count alone, so a clip's sums do not depend on how many clips a launch holds.
int adj_col_splits(int period) {
  const int per = period <= 16 ? 1 : (period + 7) / 8;
  return std::max(1, (period + per - 1) / per);
}

// Per crop column block and run of fields j in [j0, j1) of one clip (the
// clip's `period` fields split into `splits` runs): the forward transform over
// y of each field's column, the crop, conj(Psi) times it, summed over the run (in registers, or up to 512 points in shared
// memory, one slot per thread and output position) and written once, to
// part[clip splits + split][cv][c].  k_sum_planes then adds a clip's runs in
// order, so the sum's order depends on the clip's own field count only.
template <int N>
__global__ void __launch_bounds__(Plan<N>::NT * AdjW<N>::W, AdjAccInSmem<N>::value ? 2 : 1) k_adj_cols(const float2* __restrict__ u,
                                                                        const float2* __restrict__ phi,
                                                                        int crop, const float2* __restrict__ tw_g,
                                                                        float2* __restrict__ part, int period,
                                                                        int splits) {
  constexpr int W = AdjW<N>::W, NT = Plan<N>::NT, LD = (PadLen<N>::value + 15) / 16 * 16 + 16 / W;
  constexpr int RL = Plan<N>::R[Plan<N>::P - 1], PERL = PassShape<N, NT, RL>::PER;
  constexpr int T = NT * W;
  constexpr bool kSmem = AdjAccInSmem<N>::value;
  extern __shared__ float2 sm[];
  float2* tw = sm;
  float2* buf = sm + N;
  constexpr int R0 = Plan<N>::R[0], NB0 = N / R0;
  static_assert(PassShape<N, NT, R0>::PER == 1, "one first-pass butterfly per thread");
  const int tid = threadIdx.x, g = tid % W, t = tid / W, c0 = blockIdx.x * W, half = crop / 2;
  const int clip = blockIdx.y / splits, split = blockIdx.y % splits, jb = (period + splits - 1) / splits;
  float2* acc_s = buf + W * LD;  // kSmem: this thread's PERL x RL sums at (pp RL + q) T + tid
  float2 acc_r[kSmem ? 1 : PERL * RL];
  auto acc = [&](int i) -> float2& {
    if constexpr (kSmem)
      return acc_s[i * T + tid];  // read and written by tid alone
    else
      return acc_r[i];
  };
  const int j0 = clip * period + split * jb, j1 = min(j0 + jb, (clip + 1) * period);
  pdl_start();
  load_twiddles<N>(tw, tw_g);
  pdl_wait(u);
  // this thread's first-pass inputs (rows t + r N/R0) of a field, loaded one field ahead
  float2 nxt[R0];
  auto prefetch = [&](int j) {
    const float2* src = u + (size_t)j * N * crop + c0 + g;  // row y at src[y crop]
#pragma unroll
    for (int r = 0; r < R0; ++r) nxt[r] = t < NB0 ? ld_dep(src + (size_t)(t + r * NB0) * crop) : make_float2(0.f, 0.f);
  };
  if (j0 < j1) prefetch(j0);
  __syncthreads();
#pragma unroll
  for (int i = 0; i < PERL * RL; ++i) acc(i) = make_float2(0.f, 0.f);
  for (int j = j0; j < j1; ++j) {
    const int jk = j % period;
    const float2* ph = phi + (size_t)jk * crop * crop + c0 + g;
    float2 cur[R0];
#pragma unroll
    for (int r = 0; r < R0; ++r) cur[r] = nxt[r];
    auto load = [&](int, int r, int) { return cur[r]; };
    // once the first pass has consumed this field's inputs, the next field's loads go out
    auto after_first = [&]() {
      if (j + 1 < j1) prefetch(j + 1);
    };
    auto use = [&](int pp, int q, int idx, float2 h) {
      const int cv = freq_of_idx(idx, N) + half;
      if (cv >= 0 && cv < crop) {
        const float2 p = __ldg(ph + (size_t)cv * crop);
        // += conj(p) h
        float2& a = acc(pp * RL + q);
        a = make_float2(fmaf(p.x, h.x, fmaf(p.y, h.y, a.x)), fmaf(p.x, h.y, fmaf(-p.y, h.x, a.y)));
      }
    };
    fft_load_use<N, -1, decltype(load), decltype(use), false>(buf + g * LD, tw, t, load, use, after_first);
  }
  // the last pass's output positions of this thread: idx = jj + q N/RL, jj = t + pp NT
  float2* dst = part + (size_t)blockIdx.y * crop * crop + c0 + g;  // crop row cv at dst[cv crop]
#pragma unroll
  for (int pp = 0; pp < PERL; ++pp) {
    const int jj = t + pp * NT;
    if (jj < N / RL) {
#pragma unroll
      for (int q = 0; q < RL; ++q) {
        const int cv = freq_of_idx(jj + q * (N / RL), N) + half;
        if (cv >= 0 && cv < crop) dst[(size_t)cv * crop] = acc(pp * RL + q);
      }
    }
  }
}

// The adjoint for dL/dI = 1 on every pixel (the AI input's gradient channel,
// Eq. (9), and the intensity VJP without an upstream).  By Parseval,
// sum_x |E_k(x)|^2 = N^2 sum_v |mhat(v) Phi_k(v)|^2, so the sum the adjoint
// rows and columns form for G = 1 collapses to
//   S(v,u) = N^2 sum_k lam_k |Phi_k(v,u)|^2 mhat(v,u),
// exactly (on the coarse grid too: there G is the constant (N/nc)^2 and the
// transforms are on nc).  No field is transformed.  The sum over a plane's
// kernels does not depend on the mask: the kernel set keeps it (`power`, per
// set, rounded once from FP64; even in the frequency unless the set has an edge,
// since only the real part of the result's transform is taken).  Clip blockIdx.y; the planes' sets are listed
// in `sets`.
__global__ void k_ones_adjoint(const float2* __restrict__ mhat, const float* __restrict__ power,
                               const __grid_constant__ PlaneOut sets, size_t cc, float n2, float2* __restrict__ s) {
  pdl_start();
  pdl_wait(mhat);
  mhat += (size_t)blockIdx.y * cc;
  s += (size_t)blockIdx.y * cc;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < cc; i += (size_t)gridDim.x * blockDim.x) {
    float d = 0.f;
    for (int f = 0; f < sets.out_planes; ++f) d += __ldg(power + sets.list[f] * cc + i);
    const float2 m = ld_dep(mhat + i);
    s[i] = make_float2(n2 * d * m.x, n2 * d * m.y);
  }
}

// The sets of focus planes [f0, f0 + count), for k_ones_adjoint.
PlaneOut sets_of(const litho_kernels* h, int f0, int count) {
  PlaneOut o{};
  o.out_planes = count;
  for (int i = 0; i < count; ++i) o.list[i] = h->set_of[f0 + i];
  return o;
}

// out[i nu + u] = the sum of clip i's upstream planes list[first[u]] ... (blockIdx.y = i nu + u).
__global__ void k_sum_upstream(const float* __restrict__ up, size_t nn, int nu, const __grid_constant__ PlaneOut planes,
                               float* __restrict__ out) {
  pdl_start();
  pdl_wait(up);
  const int clip = blockIdx.y / nu, u = blockIdx.y - clip * nu;
  up += (size_t)clip * planes.out_planes * nn;
  out += (size_t)blockIdx.y * nn;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nn; i += (size_t)gridDim.x * blockDim.x) {
    float a = ld_dep(up + planes.list[planes.first[u]] * nn + i);
    for (int d = planes.first[u] + 1; d < planes.first[u + 1]; ++d) a += ld_dep(up + planes.list[d] * nn + i);
    out[i] = a;
  }
}

// s[clip] (+)= sum over the clip's `planes` planes of sk, in order (clip = blockIdx.y).  With `partial`, the
// last block of a clip forms its loss instead: loss[clip] (+)= the fixed-order FP64 sum of its `count`
// partials (a kernel of its own took a launch's 6 us of every small step).
__global__ void __launch_bounds__(256) k_sum_planes(const float2* __restrict__ sk, int planes, size_t cc,
                                                    float2* __restrict__ s, int accumulate,
                                                    const double* __restrict__ partial, int count,
                                                    double* __restrict__ loss) {
  pdl_start();
  pdl_wait(sk, partial);
  const int blocks = gridDim.x - (partial ? 1 : 0);
  if (int(blockIdx.x) == blocks) {
    __shared__ double w[8];
    partial += (size_t)blockIdx.y * count;
    double a = 0.0;
    for (int i = threadIdx.x; i < count; i += blockDim.x) a += ld_dep(partial + i);
    for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
    if (threadIdx.x % 32 == 0) w[threadIdx.x / 32] = a;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = accumulate ? loss[blockIdx.y] : 0.0;
      for (int i = 0; i < 8; ++i) t += w[i];
      loss[blockIdx.y] = t;
    }
    return;
  }
  sk += (size_t)blockIdx.y * planes * cc;
  s += (size_t)blockIdx.y * cc;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < cc; i += (size_t)blocks * blockDim.x) {
    float2 a = accumulate ? s[i] : make_float2(0.f, 0.f);
    for (int j = 0; j < planes; ++j) {
      const float2 v = ld_dep(sk + (size_t)j * cc + i);
      a.x += v.x;
      a.y += v.y;
    }
    s[i] = a;
  }
}

// The adjoint columns' runs of g clips into s; with partial, the clips' losses too.
cudaError_t launch_sum_planes(const float2* sk, int runs, size_t cc, float2* s, int accumulate, int g,
                              const double* partial, int count, double* loss, cudaStream_t st) {
  const unsigned blocks = unsigned(std::min<size_t>(256, (cc + 255) / 256)) + (partial ? 1 : 0);
  return launch_pdl(k_sum_planes, dim3(blocks, g), 256, 0, st, sk, runs, cc, s, accumulate, partial, count, loss);
}

// Final rows: grad[y][x] = scale Re(sum_c Q[y][c] e^{2 pi i u_c x/N}), times a m (1 - m) with theta (m =
// sigmoid(a theta)).  rows_per_cta rows per CTA share its twiddle table.  BANDED: 2 crop <= N.
template <int N, bool BANDED>
__global__ void __launch_bounds__(Plan<N>::NT) k_grad_rows(const float2* __restrict__ qf, int crop, float scale,
                                                           const float* __restrict__ theta, float alpha,
                                                           const float2* __restrict__ tw_g, float* __restrict__ grad,
                                                           long long grad_stride, int rows_per_cta) {
  extern __shared__ float2 sm[];
  float2* tw = sm;
  float2* buf = sm + N;
  pdl_start();
  load_twiddles<N>(tw, tw_g);
  pdl_wait(qf, theta);
  __syncthreads();
  const int t = threadIdx.x, half = crop / 2;
  const size_t clip = blockIdx.y;  // clip of the group: its band rows, theta and gradient
  constexpr int NT = Plan<N>::NT, RL = Plan<N>::R[Plan<N>::P - 1], PERL = PassShape<N, NT, RL>::PER;
  for (int y = blockIdx.x * rows_per_cta; y < min(N, int(blockIdx.x + 1) * rows_per_cta); ++y) {
    const float2* row = qf + (clip * N + y) * crop;
    const float* th = theta ? theta + (clip * N + y) * N : nullptr;
    auto load = [&](int, int r, int idx) {
      const int c = (r < Plan<N>::R[0] / 2 ? idx : idx - N) + half;  // first pass: idx < N/2 exactly when r < R/2
      return ld_dep_if(row + c, c >= 0 && c < crop);
    };
    float tv[PERL][RL];  // theta at this thread's outputs, loaded while the later passes run
    auto after_first = [&]() {
#pragma unroll
      for (int p = 0; p < PERL; ++p)
#pragma unroll
        for (int q = 0; q < RL; ++q)
          tv[p][q] = th && t + p * NT < N / RL ? ld_dep(th + t + p * NT + q * (N / RL)) : 0.f;
    };
    float* gr = grad + clip * grad_stride + (size_t)y * N;
    auto use = [&](int p, int q, int x, float2 v) {
      if (theta) {
        const float m = sigmoidf(alpha * tv[p][q]);
        gr[x] = scale * v.x * alpha * m * (1.0f - m);
      } else {
        gr[x] = scale * v.x;  // the gradient with respect to the mask itself
      }
    };
    fft_load_use<N, +1, decltype(load), decltype(use), BANDED>(buf, tw, t, load, use, after_first);
  }
}

template <int N>
cudaError_t adj_rows_n(const float2* t1, const FieldSet& fs, int clips, int crop, const float* g, int g_planes,
                       const float2* tw, float2* u, cudaStream_t st, const float2* tw512) {
  const int planes = clips * fs.planes;
  // fields per CTA: all of a plane's (its G row stays in registers), or with fewer than four waves of CTAs
  // the plane's fields dealt out to up to 8, at least two to each (12 planes of 512^2 151 -> 126 us, 2 of
  // 256^2 17.6 -> 10.8 us)
  int most = 1;
  for (int p = 0; p < fs.planes; ++p) most = std::max(most, fs.start[p + 1] - fs.start[p]);
  auto runs = [&](int ctas, int slots) {
    int z = 1;
    while (z < 8 && 2 * z <= most && (long long)ctas * z < 4LL * slots) z *= 2;
    return z;
  };
  if (N == 512 && tw512 && crop % 2 == 0 && crop / 2 <= 128) {  // two rows per warp
    const size_t sm = sizeof(float2) * (kAdjTw1 + kAdjTw2 + kAdjWarps * 2 * (size_t(kAdjBuf) + crop));
    cudaError_t e = smem_attrs(k_adj_rows_w512<true>, sm);
    if (e != cudaSuccess) return e;
    const int ctas = N / (2 * kAdjWarps) * planes;
    return launch_pdl(k_adj_rows_w512<true>, dim3(N / (2 * kAdjWarps), planes, runs(ctas, 2 * 152)), 32 * kAdjWarps, sm, st, t1, fs, crop,
                      g, g_planes, tw512, u);
  }
  const size_t sm = sizeof(float2) * (N + 2 * PadLen<N>::value);
  auto kern = 2 * crop <= N ? k_adj_rows<N, true> : k_adj_rows<N, false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, dim3(N, planes, runs(N * planes, 152 * 512 / Plan<N>::NT)), Plan<N>::NT, sm, st, t1, fs, crop,
                    g, g_planes, tw, u);
}

template <int N>
cudaError_t adj_cols_n(const float2* u, const float2* phi, int crop, const float2* tw, float2* part, int clips,
                       int period, cudaStream_t st) {
  constexpr int W = AdjW<N>::W;
  if (crop % W != 0) return cudaErrorInvalidValue;
  constexpr int LD = (PadLen<N>::value + 15) / 16 * 16 + 16 / W;
  constexpr int RL = Plan<N>::R[Plan<N>::P - 1], PERL = PassShape<N, Plan<N>::NT, RL>::PER;
  const size_t sm = sizeof(float2) * (N + W * LD + (AdjAccInSmem<N>::value ? size_t(PERL) * RL * Plan<N>::NT * W : 0));
  cudaError_t e = smem_attrs(k_adj_cols<N>, sm);
  if (e != cudaSuccess) return e;
  // runs of all clips on one grid axis, which holds 65535: thousands of clips take more than one launch
  // (clips on an axis of their own: VJP of 4 clips of 1024^2 358.0 -> 360.1 us, of 2 of 2048^2 766 -> 773)
  const int splits = adj_col_splits(period), most = 65535 / splits;
  for (int c = 0; c < clips && e == cudaSuccess; c += most)
    e = launch_pdl(k_adj_cols<N>, dim3(crop / W, std::min(most, clips - c) * splits), Plan<N>::NT * W, sm, st,
                   u + size_t(c) * period * N * crop, phi, crop, tw, part + size_t(c) * splits * crop * crop, period,
                   splits);
  return e;
}

template <int N>
cudaError_t grad_rows_n(const float2* qf, int crop, float scale, const float* theta, float alpha, const float2* tw,
                        float* grad, int clips, long long grad_stride, cudaStream_t st) {
  const size_t sm = sizeof(float2) * (N + PadLen<N>::value);
  auto kern = 2 * crop <= N ? k_grad_rows<N, true> : k_grad_rows<N, false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  const int per = rows_per_cta(N, clips, Plan<N>::NT, sm);
  return launch_pdl(kern, dim3((N + per - 1) / per, clips), Plan<N>::NT, sm, st, qf, crop, scale, theta, alpha, tw,
                    grad, grad_stride, per);
}

#define ILT_DISPATCH(n, CALL)              \
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

cudaError_t launch_adj_rows(int n, const float2* t1, const FieldSet& fs, int clips, int crop, const float* g,
                            int g_planes, const float2* tw, float2* u, cudaStream_t st, const float2* tw512) {
#define CALL(N) adj_rows_n<N>(t1, fs, clips, crop, g, g_planes, tw, u, st, tw512)
  ILT_DISPATCH(n, CALL)
#undef CALL
}
// part receives clips x adj_col_splits(period) crop x crop sums.
cudaError_t launch_adj_cols(int n, const float2* u, const float2* phi, int crop, const float2* tw, float2* part,
                            int clips, int period, cudaStream_t st) {
#define CALL(N) adj_cols_n<N>(u, phi, crop, tw, part, clips, period, st)
  ILT_DISPATCH(n, CALL)
#undef CALL
}
// Clip i of `clips` writes grad + i grad_stride.
cudaError_t launch_grad_rows(int n, const float2* qf, int crop, float scale, const float* theta, float alpha,
                             const float2* tw, float* grad, int clips, long long grad_stride, cudaStream_t st) {
#define CALL(N) grad_rows_n<N>(qf, crop, scale, theta, alpha, tw, grad, clips, grad_stride, st)
  ILT_DISPATCH(n, CALL)
#undef CALL
}

size_t up256(size_t x) { return (x + 255) / 256 * 256; }

struct IltLayout {
  float2 *rowbuf, *mhat, *t1, *u, *sk, *s, *qf;
  float *img, *blur;
  double *partial, *loss;
  // coarse grid (nc x nc, band 2C of the image): coarse images and the coarse
  // samples of the low-passed dL/dI (ic), row spectra on nc (mid), band rows
  // on N (big), image spectra (spec)
  float* ic;
  float2 *mid, *big, *spec;
  float* gain;  // the resist blur's transfer function on the 2C band
  size_t bytes;
};

// Clips per group: the group's stage-1 fields at the full grid within 2 GiB,
// and groups of equal size.
int ilt_group(const litho_kernels* h, int b) {
  const size_t per_clip = size_t(h->n_focus) * h->k * h->n * h->crop * sizeof(float2);
  const size_t cap = std::max<size_t>(1, std::min<size_t>(size_t(b), (size_t(2) << 30) / per_clip));
  const size_t groups = (size_t(b) + cap - 1) / cap;
  return int((size_t(b) + groups - 1) / groups);
}

// Carves the workspace for groups of G clips and P focus planes at a time
// (P = all planes with G = ilt_group, or P = 1 with G = 1).  The b FP64
// losses come first, so their address does not depend on P or G.
IltLayout ilt_layout(const litho_kernels* h, int b, int P, int G, void* base) {
  const size_t N = h->n, C = h->crop, K = h->k, g = size_t(G), PG = size_t(P) * G;
  IltLayout L{};
  size_t off = 0;
  char* p = static_cast<char*>(base);
  auto take = [&](size_t bytes) -> char* {
    char* r = p ? p + off : nullptr;
    off += up256(bytes);
    return r;
  };
  L.loss = reinterpret_cast<double*>(take(size_t(b) * 8));
  L.rowbuf = reinterpret_cast<float2*>(take(g * N * C * 8));
  L.mhat = reinterpret_cast<float2*>(take(g * C * C * 8));
  L.t1 = reinterpret_cast<float2*>(take(PG * K * N * C * 8));
  L.u = reinterpret_cast<float2*>(take(PG * K * N * C * 8));
  L.sk = reinterpret_cast<float2*>(take(PG * K * C * C * 8));
  L.s = reinterpret_cast<float2*>(take(g * C * C * 8));
  L.qf = reinterpret_cast<float2*>(take(g * N * C * 8));
  L.img = reinterpret_cast<float*>(take(PG * N * N * 4));
  L.blur = reinterpret_cast<float*>(take(PG * N * N * 4));
  // k_resist_grad: kPartials per clip; the coarse grid's fused rows: one per row pair of each plane
  L.partial = reinterpret_cast<double*>(take(g * std::max<size_t>(kPartials, size_t(P) * N / 2) * 8));
  const size_t NC = h->nc, C2 = 2 * C;
  if (NC > 0) {
    L.ic = reinterpret_cast<float*>(take(PG * NC * NC * 4));
    L.mid = reinterpret_cast<float2*>(take(PG * NC * C2 * 8));
    L.big = reinterpret_cast<float2*>(take(PG * N * C2 * 8));
    L.spec = reinterpret_cast<float2*>(take(PG * C2 * C2 * 8));
    L.gain = reinterpret_cast<float*>(take(C2 * 4));
  }
  L.bytes = off;
  return L;
}

// Planes and clips per pass for a workspace of `bytes` (false: below the minimum).
bool ilt_plan(const litho_kernels* h, int b, int planes, size_t bytes, int* P, int* G) {
  const int g = ilt_group(h, b);
  if (bytes >= ilt_layout(h, b, planes, g, nullptr).bytes) {
    *P = planes;
    *G = g;
    return true;
  }
  *P = 1;  // one focus plane of one clip at a time: its stage-1 fields are rebuilt per plane
  *G = 1;
  return bytes >= ilt_layout(h, b, 1, 1, nullptr).bytes;
}

}  // namespace

void adj512_table(float2* out) {
  const double two_pi = 2.0 * 3.14159265358979323846;
  for (int r = 1; r < 32; ++r)
    for (int j = 0; j < 16; ++j) {
      const double a = two_pi * double(r * j) / 512.0;
      out[(r - 1) * 16 + j] = make_float2(float(std::cos(a)), float(std::sin(a)));
    }
  for (int r = 1; r < 16; ++r)
    for (int l = 0; l < 32; ++l) {
      const double a = two_pi * double(r * l) / 512.0;
      out[kAdjTw1 + (r - 1) * 32 + l] = make_float2(float(std::cos(a)), float(-std::sin(a)));
    }
}

double* ilt_loss_device(const litho_kernels* h, int b, void* workspace, size_t workspace_bytes) {
  (void)h;
  (void)b;
  (void)workspace_bytes;
  return static_cast<double*>(workspace);  // the losses lead every layout
}

size_t ai_channels_bytes(const litho_kernels* h, int b) { return ilt_layout(h, b, 1, ilt_group(h, b), nullptr).bytes; }

litho_status ai_channels(const litho_kernels* h, const float* target, int b, double dose, int focus, bool coarse,
                         float* x, void* workspace, uint2* ext, bool found[2], cudaStream_t st) {
  const int G = ilt_group(h, b), N = h->n, C = h->crop;
  IltLayout L = ilt_layout(h, b, 1, G, workspace);
  const size_t nn = size_t(N) * N;
  coarse = coarse && h->nc > 0 && interp_cols_supported(h->nc, N);
  const int NE = coarse ? h->nc : N, C2 = 2 * C;
  const float2* twe = coarse ? h->d_twc : h->d_tw;
  const int set = h->set_of[focus];
  const FieldSet fs = field_set(h, set, 1);
  const PlaneOut one = plane_out_identity(1);
  PlaneOut channel1 = one;  // straight into x[.][1], a clip's second of three planes
  channel1.out_planes = 3;
  channel1.list[0] = 1;
  const float2* psi = h->d_psi + h->set_start[set] * (size_t(C) * C);
  const float scale = float(2.0 * dose / (double(N) * double(N)));
  // a 1024-point coarse grid: the warp-per-row stage 2 writes the coarse image's row spectra itself
  const bool rows2 = coarse && h->d_tw32 && stage2_w32_supported(NE, C);
  found[0] = coarse;
  found[1] = !h->edge;
  for (int c0 = 0; c0 < b; c0 += G) {
    const int g = std::min(G, b - c0);
    float* dst = x + size_t(c0) * 3 * nn;
    {  // channel 1: the aerial image of the targets (interpolated from the coarse grid)
      ProfScope ps(kStageIltForward, st, coarse ? (rows2 ? 6 : 7) : 4);
      LITHO_TRY_CUDA(launch_mask_spectrum_copy(target + c0 * nn, g, N, C, h->d_tw, L.rowbuf, L.mhat, dst, 3 * nn, st));
      LITHO_TRY_CUDA(launch_stage1_fft(L.mhat, psi, fs.fields(), NE, C, twe, L.t1, st, g));
      LITHO_TRY_CUDA(launch_stage2_fft(L.t1, fs, g, NE, C, float(dose), twe, coarse ? L.ic : dst,
                                       coarse ? one : channel1, st, h->d_tw32, h->d_tw512, rows2 ? L.mid : nullptr, C2));
      if (coarse) {
        if (!rows2) LITHO_TRY_CUDA(launch_mask_rows(L.ic, g, NE, C2, twe, L.mid, false, st));
        LITHO_TRY_CUDA(launch_interp_cols(L.mid, g, NE, N, C, twe, h->d_tw, nullptr, true, L.big, st));
        LITHO_TRY_CUDA(launch_band_rows_real(L.big, g, 1, N, C, 1.0f, h->d_tw, dst, channel1, st, ext));
      }
    }
    {  // channel 2: the adjoint applied to dL/dI = 1, in closed form (k_ones_adjoint)
      PlaneOut channel2 = channel1;
      channel2.list[0] = 2;
      ProfScope ps(kStageIltBackward, st, 3);
      LITHO_TRY_CUDA(launch_pdl(k_ones_adjoint, dim3(128, g), 256, 0, st, L.mhat, h->d_power, sets_of(h, focus, 1),
                                size_t(C) * C, float(double(N) * double(N)), L.s));
      if (h->edge) {
        LITHO_TRY_CUDA(launch_stage1_fft(L.s, nullptr, g, N, C, h->d_tw, L.qf, st));
        LITHO_TRY_CUDA(launch_grad_rows(N, L.qf, C, scale, nullptr, 0.f, h->d_tw, x + (size_t(c0) * 3 + 2) * nn, g,
                                        (long long)3 * nn, st));
      } else {  // S(-u) = conj S(u): half the columns, two rows to a transform
        LITHO_TRY_CUDA(launch_stage1_half(L.s, g, N, C, h->d_tw, L.qf, C / 2, st));
        LITHO_TRY_CUDA(launch_band_rows_real(L.qf, g, 1, N, C / 2, scale, h->d_tw, dst, channel2, st, ext + 1));
      }
    }
  }
  return LITHO_OK;
}

}  // namespace litho

using namespace litho;

extern "C" {

litho_status litho_ilt_workspace_size(const litho_kernels* h, int b, size_t* full_bytes, size_t* min_bytes) {
  if (!h || b < 1) {
    set_error("null handle or b < 1");
    return LITHO_EINVAL;
  }
  if (full_bytes) *full_bytes = ilt_layout(h, b, h->n_focus, ilt_group(h, b), nullptr).bytes;
  if (min_bytes) *min_bytes = ilt_layout(h, b, 1, 1, nullptr).bytes;
  return LITHO_OK;
}

litho_status litho_ilt_grad(const litho_kernels* h, const float* theta_dev, const float* target_dev, int b,
                            double dose, double mask_steep, double resist_steep, double threshold, double sigma_nm,
                            litho_precision prec, float* grad_dev, double* loss_host, void* workspace_dev,
                            size_t workspace_bytes, void* stream) {
  if (!h || !theta_dev || !target_dev || !grad_dev || !workspace_dev || b < 1) {
    set_error("null argument or b < 1");
    return LITHO_EINVAL;
  }
  if ((int(prec) & ~LITHO_GRID_COARSE) != LITHO_PREC_FFT32) {
    set_error("litho_ilt_grad implements the FP32 FFT path only (LITHO_PREC_FFT32, optionally | LITHO_GRID_COARSE)");
    return LITHO_EUNSUPPORTED;
  }
  if (!std::isfinite(dose) || !std::isfinite(mask_steep) || !std::isfinite(resist_steep) ||
      !std::isfinite(threshold)) {
    set_error("non-finite parameter");
    return LITHO_EINVAL;
  }
  if ((reinterpret_cast<uintptr_t>(workspace_dev) & 255) != 0) {
    set_error("workspace must be 256-byte aligned");
    return LITHO_EINVAL;
  }
  if ((reinterpret_cast<uintptr_t>(theta_dev) & 15) != 0) {
    set_error("theta must be 16-byte aligned");
    return LITHO_EINVAL;
  }
  ResistTaps taps;
  std::string why;
  if (!resist_taps(sigma_nm, h->pixel_nm, &taps, &why)) {
    set_error("%s", why.c_str());
    return LITHO_EINVAL;
  }
  if (2 * taps.radius >= h->n) {
    set_error("blur radius must be below n/2");
    return LITHO_EINVAL;
  }
  const int F = h->n_focus, N = h->n, C = h->crop;
  int P, G;
  if (!ilt_plan(h, b, F, workspace_bytes, &P, &G)) {
    set_error("workspace too small: %zu bytes given, at least %zu needed", workspace_bytes,
              ilt_layout(h, b, 1, 1, nullptr).bytes);
    return LITHO_ENOMEM;
  }
  IltLayout L = ilt_layout(h, b, P, G, workspace_dev);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const size_t nn = size_t(N) * N;
  const float scale = float(2.0 * dose / (double(N) * double(N)));
  // Coarse grid: the fields, the image and the adjoint transforms run on
  // nc >= 2C.  The image is interpolated exactly to N for the resist and the
  // loss; dL/dI enters the adjoint only through its frequencies below C in
  // magnitude (the products with the fields are cropped to the field band),
  // so it is low-passed to the 2C band and sampled on nc, times (N/nc)^2 for
  // the sums over nc^2 instead of N^2 points.  No product frequency aliases
  // into the field band on nc >= 2C, so the result is the full-grid one.
  const bool coarse = (int(prec) & LITHO_GRID_COARSE) && h->nc > 0 && interp_cols_supported(h->nc, N);
  const int NE = coarse ? h->nc : N, C2 = 2 * C;
  const float2* twe = coarse ? h->d_twc : h->d_tw;
  const float lp_scale = float((double(N) / NE) * (double(N) / NE));
  if (coarse) LITHO_TRY_CUDA(launch_blur_gain(taps, N, C2, L.gain, st));
  // a 1024-point coarse grid: the warp-per-row stage 2 writes the coarse image's row spectra itself
  const bool rows2 = coarse && h->d_tw32 && stage2_w32_supported(NE, C);
  // coarse grid: the row spectra of dL/dI on the 2C band, gp x N x 2C, in the image buffer (gp x N x N floats)
  // (the coarse grid is a power of two nc <= N/2 with 2C <= nc, so 2 x 2C floats fit in a row of N)
  if (coarse && 2 * C2 > N) {
    set_error("coarse grid band 2C = %d wider than half the grid (%d)", C2, N);
    return LITHO_EINVAL;
  }
  float2* qrows = reinterpret_cast<float2*>(L.img);
  // Focus planes that share an image are evaluated once and counted as often as they occur (their
  // q = dL/dI adds up): with the full workspace all kernel sets at a time, else one.
  const int U = h->n_sets, PU = P == F ? U : 1;
  const PlaneOut each = plane_out_identity(PU);
  // Groups of g clips: every launch covers the group's g x PU planes (plane
  // i PU + p is set u0 + p of clip c0 + i).
  for (int c0 = 0; c0 < b; c0 += G) {
    const int g = std::min(G, b - c0), gp = g * PU;
    {
      ProfScope ps(kStageIltForward, st, 2);
      LITHO_TRY_CUDA(launch_sigmoid_spectrum(theta_dev + c0 * nn, float(mask_steep), g, N, C, h->d_tw, L.rowbuf, L.mhat,
                                             st));
    }
    for (int u0 = 0; u0 < U; u0 += PU) {
      const FieldSet fs = field_set(h, u0, PU);
      const float2* psi = h->d_psi + h->set_start[u0] * (size_t(C) * C);
      PlaneWeight weight{};
      for (int f = 0; f < F; ++f)
        if (h->set_of[f] >= u0 && h->set_of[f] < u0 + PU) ++weight.w[h->set_of[f] - u0];
      {
        ProfScope ps(kStageIltForward, st, coarse ? (rows2 ? 4 : 5) : 4);
        LITHO_TRY_CUDA(launch_stage1_fft(L.mhat, psi, fs.fields(), NE, C, twe, L.t1, st, g));
        LITHO_TRY_CUDA(launch_stage2_fft(L.t1, fs, g, NE, C, float(dose), twe, coarse ? L.ic : L.img, each, st,
                                         h->d_tw32, h->d_tw512, rows2 ? L.mid : nullptr, C2));
        if (coarse) {  // the blurred image straight from the interpolation (blur applied to the spectrum)
          if (!rows2) LITHO_TRY_CUDA(launch_mask_rows(L.ic, gp, NE, C2, twe, L.mid, false, st));
          LITHO_TRY_CUDA(launch_interp_cols(L.mid, gp, NE, N, C, twe, h->d_tw, L.gain, false, L.big, st));
          // blurred rows, resist, dL/dI and its row spectra on the 2C band (into the free image
          // buffer), partial losses per row pair
          LITHO_TRY_CUDA(launch_resist_grad_rows(L.big, gp, N, C2, h->d_tw, target_dev + c0 * nn, PU, weight,
                                                 float(resist_steep), float(threshold), qrows, L.partial, st));
        } else {
          LITHO_TRY_CUDA(launch_resist(L.img, gp, N, taps, float(threshold), L.blur, nullptr, st));
          LITHO_TRY_CUDA(launch_pdl(k_resist_grad, dim3(kPartials, g), 256, 0, st, L.blur, target_dev + c0 * nn, nn,
                                    PU, weight, float(resist_steep), float(threshold), L.img, L.partial));
        }
        LITHO_TRY_CUDA(cudaGetLastError());
      }
      {
        ProfScope ps(kStageIltBackward, st, coarse ? 6 : 4);
        const float* gsrc = L.blur;
        if (coarse) {  // low-pass of g (x) q: the spectrum of q on the 2C band times the blur's transfer function
          LITHO_TRY_CUDA(launch_mask_cols(qrows, gp, N, C2, h->d_tw, L.spec, L.gain, false, st));
          LITHO_TRY_CUDA(launch_stage1_half(L.spec, gp, NE, C2, twe, L.mid, C, st));
          LITHO_TRY_CUDA(launch_band_rows_real(L.mid, g, PU, NE, C, lp_scale, twe, L.ic, each, st));
          gsrc = L.ic;
        } else {
          LITHO_TRY_CUDA(launch_resist(L.img, gp, N, taps, float(threshold), L.blur, nullptr, st));
        }
        LITHO_TRY_CUDA(launch_adj_rows(NE, L.t1, fs, g, C, gsrc, PU, twe, L.u, st, h->d_tw512));
        LITHO_TRY_CUDA(launch_adj_cols(NE, L.u, psi, C, twe, L.sk, g, fs.fields(), st));
        LITHO_TRY_CUDA(launch_sum_planes(L.sk, adj_col_splits(fs.fields()), size_t(C) * C, L.s, u0 > 0 ? 1 : 0, g,
                                         L.partial, coarse ? PU * N / 2 : kPartials, L.loss + c0, st));
      }
    }
    ProfScope ps(kStageIltBackward, st, 2);
    LITHO_TRY_CUDA(launch_stage1_fft(L.s, nullptr, g, N, C, h->d_tw, L.qf, st));
    LITHO_TRY_CUDA(launch_grad_rows(N, L.qf, C, scale, theta_dev + c0 * nn, float(mask_steep), h->d_tw,
                                    grad_dev + c0 * nn, g, (long long)nn, st));
  }
  if (loss_host) {
    LITHO_TRY_CUDA(cudaMemcpyAsync(loss_host, L.loss, size_t(b) * sizeof(double), cudaMemcpyDeviceToHost, st));
    LITHO_TRY_CUDA(cudaStreamSynchronize(st));
  }
  return LITHO_OK;
}

litho_status litho_intensity_vjp_workspace_size(const litho_kernels* h, int b, size_t* full_bytes, size_t* min_bytes) {
  return litho_ilt_workspace_size(h, b, full_bytes, min_bytes);
}

litho_status litho_intensity_vjp(const litho_kernels* h, const float* mask_dev, int b, double dose,
                                 litho_precision prec, int f_first, int f_count, const float* upstream_dev,
                                 float* dm_dev, void* workspace_dev, size_t workspace_bytes, void* stream) {
  if (!h || !mask_dev || !dm_dev || !workspace_dev || b < 1) {
    set_error("null argument or b < 1");
    return LITHO_EINVAL;
  }
  if (f_first < 0 || f_count < 1 || f_first + f_count > h->n_focus || !std::isfinite(dose)) {
    set_error("focus planes [f_first, f_first + f_count) must lie in [0, n_focus); dose finite");
    return LITHO_EINVAL;
  }
  if ((int(prec) & ~LITHO_GRID_COARSE) != LITHO_PREC_FFT32) {
    set_error("litho_intensity_vjp implements the FP32 FFT path only (LITHO_PREC_FFT32, optionally | "
              "LITHO_GRID_COARSE)");
    return LITHO_EUNSUPPORTED;
  }
  if ((reinterpret_cast<uintptr_t>(workspace_dev) & 255) != 0) {
    set_error("workspace must be 256-byte aligned");
    return LITHO_EINVAL;
  }
  const int F = h->n_focus, N = h->n, C = h->crop;
  int P, G;
  if (!ilt_plan(h, b, f_count, workspace_bytes, &P, &G)) {
    set_error("workspace too small: %zu bytes given, at least %zu needed", workspace_bytes,
              ilt_layout(h, b, 1, 1, nullptr).bytes);
    return LITHO_ENOMEM;
  }
  // clips are grouped when their upstream planes follow one another: all
  // focus planes of each clip, or no upstream (ones)
  if (upstream_dev && !(P == F && f_first == 0)) G = 1;
  IltLayout L = ilt_layout(h, b, P, G, workspace_dev);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const size_t nn = size_t(N) * N;
  const float scale = float(2.0 * dose / (double(N) * double(N)));
  // coarse grid as in litho_ilt_grad: the upstream low-passed to the 2C band
  // and sampled on nc (no upstream: the closed form, on no grid)
  const bool coarse = (int(prec) & LITHO_GRID_COARSE) && h->nc > 0 && interp_cols_supported(h->nc, N);
  const int NE = coarse ? h->nc : N, C2 = 2 * C;
  const float2* twe = coarse ? h->d_twc : h->d_tw;
  const float lp_scale = float((double(N) / NE) * (double(N) / NE));
  ProfScope ps(kStageIltBackward, st, 1);
  for (int c0 = 0; c0 < b; c0 += G) {
    const int g = std::min(G, b - c0);
    LITHO_TRY_CUDA(launch_mask_spectrum(mask_dev + c0 * nn, g, N, C, h->d_tw, L.rowbuf, L.mhat, st));
    if (!upstream_dev) {  // dL/dI = 1 on every pixel of the selected planes: the closed form
      LITHO_TRY_CUDA(launch_pdl(k_ones_adjoint, dim3(128, g), 256, 0, st, L.mhat, h->d_power,
                                sets_of(h, f_first, f_count), size_t(C) * C, float(double(N) * double(N)), L.s));
    }
    for (int f0 = f_first; upstream_dev && f0 < f_first + f_count; f0 += P) {
      int p = std::min(P, f_first + f_count - f0);
      const float* up = upstream_dev + (size_t(c0) * F + f0) * nn;
      // the kernel sets of these planes in order, and the planes of each
      int sets[kMaxPlanes], nu = 0;
      for (int f = 0; f < p; ++f) sets[f] = h->set_of[f0 + f];
      std::sort(sets, sets + p);
      nu = int(std::unique(sets, sets + p) - sets);
      PlaneOut planes{};
      planes.out_planes = p;
      bool in_order = nu == p;
      for (int i = 0, at = 0; i < nu; ++i) {
        for (int f = 0; f < p; ++f)
          if (h->set_of[f0 + f] == sets[i]) {
            in_order = in_order && f == i;
            planes.list[at++] = (unsigned char)f;
          }
        planes.first[i + 1] = (unsigned char)at;
      }
      if (!in_order) {  // planes with the same fields: their upstreams add up
        LITHO_TRY_CUDA(launch_pdl(k_sum_upstream, dim3(unsigned(std::min<size_t>((nn + 255) / 256, 1024)), g * nu),
                                  256, 0, st, up, nn, nu, planes, L.img));
        up = L.img;
        p = nu;
      }
      if (coarse) {
        LITHO_TRY_CUDA(launch_mask_rows(up, g * p, N, C2, h->d_tw, L.big, false, st));
        LITHO_TRY_CUDA(launch_mask_cols(L.big, g * p, N, C2, h->d_tw, L.spec, nullptr, false, st));
        LITHO_TRY_CUDA(launch_stage1_half(L.spec, g * p, NE, C2, twe, L.mid, C, st));
        LITHO_TRY_CUDA(launch_band_rows_real(L.mid, g, p, NE, C, lp_scale, twe, L.ic, plane_out_identity(p), st));
        up = L.ic;
      }
      // sets that follow one another in the kernel set share their launches
      for (int r0 = 0, r1; r0 < p; r0 = r1) {
        for (r1 = r0 + 1; r1 < p && sets[r1] == sets[r0] + (r1 - r0);) ++r1;
        const FieldSet fs = field_set(h, sets[r0], r1 - r0);
        const float2* psi = h->d_psi + h->set_start[sets[r0]] * (size_t(C) * C);
        LITHO_TRY_CUDA(launch_stage1_fft(L.mhat, psi, fs.fields(), NE, C, twe, L.t1, st, g));
        LITHO_TRY_CUDA(
            launch_adj_rows(NE, L.t1, fs, g, C, up + size_t(r0) * NE * NE, p, twe, L.u, st, h->d_tw512));
        LITHO_TRY_CUDA(launch_adj_cols(NE, L.u, psi, C, twe, L.sk, g, fs.fields(), st));
        LITHO_TRY_CUDA(launch_sum_planes(L.sk, adj_col_splits(fs.fields()), size_t(C) * C, L.s,
                                         f0 > f_first || r0 > 0 ? 1 : 0, g, nullptr, 0, nullptr, st));
      }
    }
    if (!upstream_dev && !h->edge) {  // the closed form's S(-u) = conj S(u)
      LITHO_TRY_CUDA(launch_stage1_half(L.s, g, N, C, h->d_tw, L.qf, C / 2, st));
      LITHO_TRY_CUDA(launch_band_rows_real(L.qf, g, 1, N, C / 2, scale, h->d_tw, dm_dev + c0 * nn,
                                           plane_out_identity(1), st));
      continue;
    }
    LITHO_TRY_CUDA(launch_stage1_fft(L.s, nullptr, g, N, C, h->d_tw, L.qf, st));
    LITHO_TRY_CUDA(launch_grad_rows(N, L.qf, C, scale, nullptr, 0.f, h->d_tw, dm_dev + c0 * nn, g, (long long)nn,
                                    st));
  }
  return LITHO_OK;
}

}  // extern "C"
