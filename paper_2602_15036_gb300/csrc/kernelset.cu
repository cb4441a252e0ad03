// The SOCS kernels as the device evaluates them: for every focus plane the
// smallest set of fields that gives the plane's image, with sqrt(lambda)
// folded in, so that I = dose sum_p |IDFT(M Psi_p)|^2.
//
// The object is a real mask, so M(-u) = conj M(u), and a kernel with
// Psi(-u) = conj Psi(u) gives a real field.  Every kernel is
// sqrt(lam) Phi = h + i h' with h, h' of that form, and its |E|^2 is the sum
// of the squares of the two real fields of h and h'.  The plane's image is
// thus the quadratic form Q = sum h h^T of 2 K real fields, and any set of
// fields with the same Q gives the same image (Eq. (4)) and the same
// gradient.  Where Q has rank r < 2 K, its r eigenvectors, scaled by the roots
// of their eigenvalues and taken two to a complex kernel (|e + i e'|^2 =
// e^2 + e'^2), are ceil(r/2) < K kernels.  That is the case in focus: with an
// unaberrated pupil and a centrosymmetric source the TCC is real and even,
// each h or h' is zero up to a phase, and half the transforms suffice.  Planes
// whose Q agree (+z and -z of such a system) share one set.  Nothing is
// assumed about the optics: the Gram matrices of the h decide, in FP64, once
// per kernel set, and relative to each kernel's own weight; a plane that does not reduce keeps sqrt(lam) Phi.
//
// Measured when it was added (K = 24, planes at -50/0/+50 nm: 36 fields a clip instead of 72):
// 64 clips of 2048^2 with resist 15.50 -> 9.78 ms, 8 clips on the full grid
// 5.96 -> 3.27 ms, on the tensor cores 5.18 -> 3.12 ms; ILT step of 16 clips
// of 1024^2, K = 16, 5 planes 3.62 -> 2.16 ms; one 2048^2 clip in focus 149 ->
// 117 us.  Fewer and larger fields average their rounding over fewer terms: error against 64 bits (relative, four
// sets of inputs, with the half spectra that came later) 3.6e-7 and 3.6e-7, 2.6e-7 -> 2.7e-7, 3.1e-6 -> 3.0e-6,
// 1.15e-6 -> 1.18e-6, 3.75e-7 -> 3.8e-7.
#include <algorithm>
#include <cmath>
#include <new>

#include "litho_internal.h"

namespace litho {

namespace {

constexpr int kMaxReduceK = 64;                       // kernels per plane the reduction considers (2 K-square Jacobi)
constexpr size_t kMaxReduceBytes = size_t(2) << 30;   // FP64 kernels held on the device at once while the set is built
// A field is left out, and two planes share a set, only where no kernel's own image misses it, however little the
// kernel weighs beside the others: a mask whose spectrum the strong kernels do not pass is imaged by the weak one alone.
constexpr double kRankTol = 1e-12;   // eigenvalues of Q below this share of the largest may be left out ...
constexpr double kOwnTol = 0x1p-26;  // ... when that takes no more than this share from any kernel's own weight,
constexpr double kNoise = 1e-14;     // or they are rounding (and below what FP32 fields of the largest leave)
constexpr int kSpanBlocks = 64;      // partial sums per kernel in k_span

// Crop index of -u: entry 0 is u = -C/2, its own mirror on a full-width crop
// (C = N) and required to be zero otherwise.
__device__ __forceinline__ int mirror(int i, int crop) {
  const int v = i / crop, u = i - v * crop;
  return (v ? crop - v : 0) * crop + (u ? crop - u : 0);
}

// out[k][l] = (Re, Im) of sum_u A_k(u) conj B_l(u), then of sum_u A_k(u) B_l(-u); block (l, k).
__global__ void __launch_bounds__(256) k_gram(const double2* __restrict__ a, const double2* __restrict__ b, int crop,
                                              double4* __restrict__ out) {
  const int cc = crop * crop;
  a += (size_t)blockIdx.y * cc;
  b += (size_t)blockIdx.x * cc;
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  for (int i = threadIdx.x; i < cc; i += blockDim.x) {
    const double2 x = a[i], y = b[i], z = b[mirror(i, crop)];
    s[0] += x.x * y.x + x.y * y.y;
    s[1] += x.y * y.x - x.x * y.y;
    s[2] += x.x * z.x - x.y * z.y;
    s[3] += x.x * z.y + x.y * z.x;
  }
  __shared__ double w[8][4];
  for (int q = 0; q < 4; ++q) {
    for (int o = 16; o > 0; o >>= 1) s[q] += __shfl_down_sync(0xffffffffu, s[q], o);
    if (threadIdx.x % 32 == 0) w[threadIdx.x / 32][q] = s[q];
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    double t = 0.0;
    for (int i = 0; i < 8; ++i) t += w[i][threadIdx.x];
    reinterpret_cast<double*>(out + (size_t)blockIdx.y * gridDim.x + blockIdx.x)[threadIdx.x] = t;
  }
}

// flag[f] = 1 when a kernel of plane f is nonzero at u = -C/2 (no mirror on the crop); block per kernel.
__global__ void k_edge(const double2* __restrict__ phi, int crop, int nk, int* __restrict__ flag) {
  const double2* p = phi + (size_t)blockIdx.x * crop * crop;
  bool any = false;
  for (int i = threadIdx.x; i < crop; i += blockDim.x) {
    const double2 x = p[i], y = p[(size_t)i * crop];
    any = any || x.x != 0.0 || x.y != 0.0 || y.x != 0.0 || y.y != 0.0;
  }
  if (any) flag[blockIdx.x / nk] = 1;
}

// psi_p(u) = sum_k alpha[p][k] Phi_k(u) + beta[p][k] conj Phi_k(-u); blockIdx.y = p.
__global__ void __launch_bounds__(256) k_combine(const double2* __restrict__ phi, int nk, int crop,
                                                 const double2* __restrict__ alpha, const double2* __restrict__ beta,
                                                 float2* __restrict__ psi) {
  const int cc = crop * crop, p = blockIdx.y, i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= cc) return;
  const int m = mirror(i, crop);
  double re = 0.0, im = 0.0;
  for (int k = 0; k < nk; ++k) {
    const double2 x = phi[(size_t)k * cc + i], y = phi[(size_t)k * cc + m];
    const double2 a = alpha[p * nk + k], b = beta[p * nk + k];
    re += a.x * x.x - a.y * x.y + b.x * y.x + b.y * y.y;
    im += a.x * x.y + a.y * x.x + b.y * y.x - b.x * y.y;
  }
  psi[(size_t)p * cc + i] = make_float2(float(re), float(im));
}

// part[k][block] = its share of sum_u |root_k Phi_k(u) - sum_l alpha[k][l] Psi_l(u) + beta[k][l] conj Psi_l(-u)|^2:
// what of kernel k (of phi) the kernels psi do not span.  blockIdx.y = k.
__global__ void __launch_bounds__(256) k_span(const double2* __restrict__ phi, const double2* __restrict__ psi, int nk,
                                              int crop, const double2* __restrict__ alpha,
                                              const double2* __restrict__ beta, const double2* __restrict__ root,
                                              double* __restrict__ part) {
  const int cc = crop * crop, k = blockIdx.y;
  const double r = root[k].x;
  double sum = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < cc; i += gridDim.x * blockDim.x) {
    const int m = mirror(i, crop);
    double re = r * phi[(size_t)k * cc + i].x, im = r * phi[(size_t)k * cc + i].y;
    for (int l = 0; l < nk; ++l) {
      const double2 x = psi[(size_t)l * cc + i], y = psi[(size_t)l * cc + m];
      const double2 a = alpha[k * nk + l], b = beta[k * nk + l];
      re -= a.x * x.x - a.y * x.y + b.x * y.x + b.y * y.y;
      im -= a.x * x.y + a.y * x.x + b.y * y.x - b.x * y.y;
    }
    sum += re * re + im * im;
  }
  __shared__ double w[8];
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o);
  if (threadIdx.x % 32 == 0) w[threadIdx.x / 32] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < 8; ++i) t += w[i];
    part[(size_t)k * gridDim.x + blockIdx.x] = t;
  }
}

// One kernel that is kept: psi = root Phi.
__global__ void __launch_bounds__(256) k_scale(const double2* __restrict__ phi, double root, size_t cc,
                                               float2* __restrict__ psi) {
  const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (i < cc) psi[i] = make_float2(float(root * phi[i].x), float(root * phi[i].y));
}
// power += lam |Phi|^2 (the closed-form adjoint of ones, see k_ones_adjoint).
__global__ void __launch_bounds__(256) k_add_power(const double2* __restrict__ phi, double lam, size_t cc,
                                                   double* __restrict__ dsum) {
  const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (i < cc) dsum[i] += lam * (phi[i].x * phi[i].x + phi[i].y * phi[i].y);
}
// y = x rounded, or with `even` (x(u) + x(-u))/2.
__global__ void __launch_bounds__(256) k_round(const double* __restrict__ x, int crop, int even,
                                               float* __restrict__ y) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < crop * crop) y[i] = float(even ? 0.5 * (x[i] + x[mirror(i, crop)]) : x[i]);
}

// Eigenvalues (descending) and eigenvectors (columns of v) of a real symmetric
// matrix by cyclic Jacobi rotations; false when it does not settle.
bool jacobi(std::vector<double>& a, int n, std::vector<double>& ev, std::vector<double>& v) {
  v.assign(size_t(n) * n, 0.0);
  for (int i = 0; i < n; ++i) v[size_t(i) * n + i] = 1.0;
  double norm = 0.0;
  for (double x : a) norm += x * x;
  bool done = false;
  for (int sweep = 0; sweep < 60 && !done; ++sweep) {
    double off = 0.0;
    for (int p = 0; p < n; ++p)
      for (int q = p + 1; q < n; ++q) off += a[size_t(p) * n + q] * a[size_t(p) * n + q];
    done = off <= 1e-34 * norm;
    for (int p = 0; p < n && !done; ++p)
      for (int q = p + 1; q < n; ++q) {
        const double g = a[size_t(p) * n + q];
        if (g == 0.0) continue;
        const double th = (a[size_t(q) * n + q] - a[size_t(p) * n + p]) / (2.0 * g);
        const double t = (th >= 0 ? 1.0 : -1.0) / (std::fabs(th) + std::sqrt(th * th + 1.0));
        const double c = 1.0 / std::sqrt(t * t + 1.0), s = t * c;
        for (int i = 0; i < n; ++i) {
          const double x = a[size_t(i) * n + p], y = a[size_t(i) * n + q];
          a[size_t(i) * n + p] = c * x - s * y;
          a[size_t(i) * n + q] = s * x + c * y;
        }
        for (int i = 0; i < n; ++i) {
          const double x = a[size_t(p) * n + i], y = a[size_t(q) * n + i];
          a[size_t(p) * n + i] = c * x - s * y;
          a[size_t(q) * n + i] = s * x + c * y;
        }
        for (int i = 0; i < n; ++i) {
          const double x = v[size_t(i) * n + p], y = v[size_t(i) * n + q];
          v[size_t(i) * n + p] = c * x - s * y;
          v[size_t(i) * n + q] = s * x + c * y;
        }
      }
  }
  std::vector<int> order(n);
  for (int i = 0; i < n; ++i) order[i] = i;
  std::sort(order.begin(), order.end(), [&](int x, int y) { return a[size_t(x) * n + x] > a[size_t(y) * n + y]; });
  ev.resize(n);
  std::vector<double> w(size_t(n) * n);
  for (int j = 0; j < n; ++j) {
    ev[j] = a[size_t(order[j]) * n + order[j]];
    for (int i = 0; i < n; ++i) w[size_t(i) * n + j] = v[size_t(i) * n + order[j]];
  }
  v.swap(w);
  return done;
}

// Inner products of the real fields' kernels h_2k + i h_2k+1 = root_k Phi_k of
// two planes, from k_gram's sums P = sum A conj B and R = sum A B(-u):
// <h, h> = Re(P + R)/2, <h', h'> = Re(P - R)/2, <h, h'> = Im(R - P)/2,
// <h', h> = Im(R + P)/2.
std::vector<double> real_gram(const std::vector<double4>& g, const double* root_a, int ka, const double* root_b,
                              int kb) {
  std::vector<double> out(size_t(4) * ka * kb);
  for (int k = 0; k < ka; ++k)
    for (int l = 0; l < kb; ++l) {
      const double4 e = g[size_t(k) * kb + l];
      const double r = 0.5 * root_a[k] * root_b[l];
      double* o = &out[size_t(2 * k) * (2 * kb) + 2 * l];
      o[0] = r * (e.x + e.z);
      o[1] = r * (e.w - e.y);
      o[2 * kb] = r * (e.w + e.y);
      o[2 * kb + 1] = r * (e.x - e.z);
    }
  return out;
}

double sum_sq(const std::vector<double>& a) {
  double s = 0.0;
  for (double x : a) s += x * x;
  return s;
}

// The two real fields' share of kernel k in Q: |h_2k|^2 + |h_2k+1|^2.
double own_weight(const std::vector<double>& g, int nk, int k) {
  return g[size_t(2 * k) * (2 * nk) + 2 * k] + g[size_t(2 * k + 1) * (2 * nk) + 2 * k + 1];
}

// How many eigenvectors of Q (ev descending, columns of v) its image needs.
int kept_rank(const std::vector<double>& g, int nk, const std::vector<double>& ev, const std::vector<double>& v) {
  const int n = 2 * nk;
  std::vector<double> taken(nk, 0.0);  // from each kernel's weight by the eigenvectors left out
  int r = n;
  for (; r > 0 && ev[r - 1] <= kRankTol * ev[0]; --r) {
    if (ev[r - 1] <= kNoise * ev[0]) continue;
    bool missed = false;
    for (int k = 0; k < nk; ++k) {
      const double a = v[size_t(2 * k) * n + r - 1], b = v[size_t(2 * k + 1) * n + r - 1];
      taken[k] += ev[r - 1] * (a * a + b * b);
      missed = missed || taken[k] > kOwnTol * own_weight(g, nk, k);
    }
    if (missed) break;
  }
  return r;
}

// Device memory while a set is built, and the stream it is built on: a set may be built beside running work (the
// server's builder thread), for which neither cudaFree nor a copy on the default stream should wait.  The pool is
// its own, so that nothing of it stays reserved.
class Scratch {
 public:
  cudaStream_t st = nullptr;
  Scratch() = default;
  Scratch(const Scratch&) = delete;
  Scratch& operator=(const Scratch&) = delete;
  ~Scratch() {
    if (base_) cudaFreeAsync(base_, st);
    if (st) cudaStreamSynchronize(st);
    if (pool_) cudaMemPoolDestroy(pool_);
    if (st) cudaStreamDestroy(st);
  }
  cudaError_t open(int device, size_t bytes) {
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = device;
    cudaError_t e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaMemPoolCreate(&pool_, &props);
    return e != cudaSuccess ? e : cudaMallocFromPoolAsync(&base_, bytes, pool_, st);
  }
  template <class T>
  T* at(size_t offset) const {
    return reinterpret_cast<T*>(static_cast<char*>(base_) + offset);
  }
  // Copies that the host waits for: the other end is pageable.
  cudaError_t up(void* dst, const void* src, size_t bytes) { return copy(dst, src, bytes, cudaMemcpyHostToDevice); }
  cudaError_t down(void* dst, const void* src, size_t bytes) { return copy(dst, src, bytes, cudaMemcpyDeviceToHost); }

 private:
  cudaError_t copy(void* dst, const void* src, size_t bytes, cudaMemcpyKind kind) {
    const cudaError_t e = cudaMemcpyAsync(dst, src, bytes, kind, st);
    return e != cudaSuccess ? e : cudaStreamSynchronize(st);
  }
  cudaMemPool_t pool_ = nullptr;
  void* base_ = nullptr;
};

// whole: all FP64 kernels on the device at once, so that planes can be reduced and shared; otherwise one kernel
// at a time.  *no_memory tells whether a failure was for want of device memory.
litho_status build(litho_kernels* h, bool whole, bool* no_memory) {
  const int F = h->n_focus, K = h->k, C = h->crop;
  const size_t cc = size_t(C) * C, plane_len = size_t(K) * cc;
  const double2* host = reinterpret_cast<const double2*>(h->phi_host.data());
  std::vector<double> root(size_t(F) * K);  // sqrt(lambda); 0 for the kernels the FP32 path leaves out
  for (size_t i = 0; i < root.size(); ++i) root[i] = float(h->lambda[i]) > 0.f ? std::sqrt(h->lambda[i]) : 0.0;

  struct Set {
    int plane;                         // its first focus plane
    bool reduced = false;
    std::vector<double> gram;          // 2K x 2K, when the plane can be reduced or shared
    std::vector<double> ev, v;         // its eigenvalues (descending) and eigenvectors, the first `rank` of them needed
    int rank = 0;
    std::vector<double2> alpha, beta;  // [kernels][K] when reduced
    int kernels = 0;
  };
  std::vector<Set> sets;
  size_t bytes = 0;
  auto place = [&](size_t b) {
    const size_t at = bytes;
    bytes += (b + 255) / 256 * 256;
    return at;
  };
  const size_t kk = size_t(K) * K, o_phi = place((whole ? F * plane_len : cc) * sizeof(double2)),
               o_power = place(cc * sizeof(double)), o_gram = place(whole ? kk * sizeof(double4) : 0),
               o_coef = place(whole ? (2 * kk + K) * sizeof(double2) : 0),
               o_span = place(whole ? size_t(K) * kSpanBlocks * sizeof(double) : 0), o_flag = place(F * sizeof(int));
  Scratch sc;
  // an allocation's status
  auto memory = [&](cudaError_t e) -> litho_status {
    *no_memory = e == cudaErrorMemoryAllocation;
    LITHO_TRY_CUDA(e);
    return LITHO_OK;
  };
  litho_status st = memory(sc.open(h->device, bytes));
  if (st != LITHO_OK) return st;
  double2 *phi64 = sc.at<double2>(o_phi), *coef = sc.at<double2>(o_coef);  // coef: alpha, beta, roots (see upload_coef)
  double4* gram_d = sc.at<double4>(o_gram);
  double *power = sc.at<double>(o_power), *span_d = sc.at<double>(o_span);
  int* flag_d = sc.at<int>(o_flag);
  std::vector<int> edge(F, 1);
  if (whole) {
    LITHO_TRY_CUDA(sc.up(phi64, host, F * plane_len * sizeof(double2)));
    if (C < h->n) {
      LITHO_TRY_CUDA(cudaMemsetAsync(flag_d, 0, F * sizeof(int), sc.st));
      k_edge<<<F * K, 128, 0, sc.st>>>(phi64, C, K, flag_d);
      LITHO_TRY_CUDA(cudaGetLastError());
      LITHO_TRY_CUDA(sc.down(edge.data(), flag_d, F * sizeof(int)));
    } else {
      edge.assign(F, 0);
    }
  }
  // C = n: every frequency has its mirror, but u = -C/2 is left out of half spectra
  h->edge = C == h->n || std::find(edge.begin(), edge.end(), 1) != edge.end();
  auto gram = [&](int fa, int fb, std::vector<double>* out) -> litho_status {
    std::vector<double4> g(size_t(K) * K);
    k_gram<<<dim3(K, K), 256, 0, sc.st>>>(phi64 + fa * plane_len, phi64 + fb * plane_len, C, gram_d);
    LITHO_TRY_CUDA(cudaGetLastError());
    LITHO_TRY_CUDA(sc.down(g.data(), gram_d, g.size() * sizeof(double4)));
    *out = real_gram(g, &root[size_t(fa) * K], K, &root[size_t(fb) * K], K);
    return LITHO_OK;
  };
  // a h_2k + b h_2k+1 = root ((a - i b) Phi + (a + i b) conj Phi(-u))/2 for complex a, b: alpha from coef[0],
  // beta from coef[K^2], and plane f's roots from coef[2 K^2].
  std::vector<double2> ab(whole ? 2 * kk + K : 0);
  auto upload_coef = [&](const std::vector<double2>& alpha, const std::vector<double2>& beta, int f) -> litho_status {
    std::copy(alpha.begin(), alpha.end(), ab.begin());
    std::copy(beta.begin(), beta.end(), ab.begin() + kk);
    for (int k = 0; k < K; ++k) ab[2 * kk + k] = make_double2(root[size_t(f) * K + k], 0.0);
    LITHO_TRY_CUDA(sc.up(coef, ab.data(), ab.size() * sizeof(double2)));
    return LITHO_OK;
  };
  // Whether plane f (its Gram matrix g) has the image of set e: in the basis of e's needed eigenvectors E_j =
  // sum_i v_ij h_i / sqrt(ev_j), plane f's form is diag(ev), entry by entry relative to the entry's own
  // eigenvalues, and every kernel of f lies in their span (formed point by point: the difference of two
  // norms would leave rounding the size of the bound).
  auto same = [&](const Set& e, int f, const std::vector<double>& g, bool* out) -> litho_status {
    *out = false;
    const int n = 2 * K, r = e.rank;
    std::vector<double> x;
    litho_status s = gram(e.plane, f, &x);
    if (s != LITHO_OK) return s;
    std::vector<double> c(size_t(r) * n, 0.0);  // c[j][l] = <E_j, h'_l>
    for (int j = 0; j < r; ++j) {
      for (int i = 0; i < n; ++i) {
        const double w = e.v[size_t(i) * n + j] / std::sqrt(e.ev[j]);
        for (int l = 0; l < n; ++l) c[size_t(j) * n + l] += w * x[size_t(i) * n + l];
      }
      for (int q = 0; q <= j; ++q) {
        double d = q == j ? -e.ev[j] : 0.0;
        for (int l = 0; l < n; ++l) d += c[size_t(j) * n + l] * c[size_t(q) * n + l];
        if (!(std::fabs(d) <= kOwnTol * std::sqrt(e.ev[j] * e.ev[q]))) return LITHO_OK;
      }
    }
    std::vector<double2> alpha(size_t(K) * K), beta(size_t(K) * K);
    std::vector<double> d(size_t(n) * 2);  // kernel k of f = sum_i (d[i][0] + i d[i][1]) h_i of e
    for (int k = 0; k < K; ++k) {
      std::fill(d.begin(), d.end(), 0.0);
      for (int j = 0; j < r; ++j)
        for (int i = 0; i < n; ++i) {
          const double w = e.v[size_t(i) * n + j] / std::sqrt(e.ev[j]);
          d[2 * i] += w * c[size_t(j) * n + 2 * k];
          d[2 * i + 1] += w * c[size_t(j) * n + 2 * k + 1];
        }
      for (int l = 0; l < K; ++l) {
        const double *a = &d[4 * l], *b = &d[4 * l + 2], w = 0.5 * root[size_t(e.plane) * K + l];
        alpha[size_t(k) * K + l] = make_double2(w * (a[0] + b[1]), w * (a[1] - b[0]));
        beta[size_t(k) * K + l] = make_double2(w * (a[0] - b[1]), w * (a[1] + b[0]));
      }
    }
    if ((s = upload_coef(alpha, beta, f)) != LITHO_OK) return s;
    k_span<<<dim3(kSpanBlocks, K), 256, 0, sc.st>>>(phi64 + f * plane_len, phi64 + e.plane * plane_len, K, C, coef,
                                                    coef + kk, coef + 2 * kk, span_d);
    LITHO_TRY_CUDA(cudaGetLastError());
    std::vector<double> part(size_t(K) * kSpanBlocks);
    LITHO_TRY_CUDA(sc.down(part.data(), span_d, part.size() * sizeof(double)));
    for (int k = 0; k < K; ++k) {
      double left = 0.0;
      for (int i = 0; i < kSpanBlocks; ++i) left += part[size_t(k) * kSpanBlocks + i];
      if (!(left <= kOwnTol * kOwnTol * own_weight(g, K, k))) return LITHO_OK;
    }
    *out = true;
    return LITHO_OK;
  };
  for (int f = 0; f < F; ++f) {
    Set t;
    t.plane = f;
    int nonzero = 0;
    for (int k = 0; k < K; ++k) nonzero += root[size_t(f) * K + k] > 0.0;
    t.kernels = nonzero;
    int shared = -1;
    for (size_t e = 0; e < sets.size() && shared < 0; ++e)
      if (nonzero == 0 && sets[e].kernels == 0) shared = int(e);  // dark planes
    if (shared < 0 && !edge[f]) {
      litho_status s = gram(f, f, &t.gram);
      if (s != LITHO_OK) return s;
      const double na = sum_sq(t.gram);
      if (!std::isfinite(na)) t.gram.clear();
      for (size_t e = 0; e < sets.size() && shared < 0 && !t.gram.empty(); ++e) {
        if (sets[e].rank == 0) continue;
        const double nb = sum_sq(sets[e].gram);
        if (std::fabs(na - nb) > 1e-6 * std::max(na, nb)) continue;
        bool equal;
        if ((s = same(sets[e], f, t.gram, &equal)) != LITHO_OK) return s;
        if (equal) shared = int(e);
      }
    }
    if (shared >= 0) {
      h->set_of[f] = (unsigned char)shared;
      continue;
    }
    h->set_of[f] = (unsigned char)sets.size();
    std::vector<double> a = t.gram;
    if (!a.empty() && jacobi(a, 2 * K, t.ev, t.v) && t.ev[0] > 0.0) {
      const int r = t.rank = kept_rank(t.gram, K, t.ev, t.v);
      if ((r + 1) / 2 < nonzero) {
        t.reduced = true;
        t.kernels = (r + 1) / 2;
        t.alpha.resize(size_t(t.kernels) * K);
        t.beta.resize(size_t(t.kernels) * K);
        auto at = [&](int row, int col) { return col < r ? t.v[size_t(row) * (2 * K) + col] : 0.0; };
        for (int q = 0; q < t.kernels; ++q)
          for (int k = 0; k < K; ++k) {
            // eigenvectors (a1, b1) and (a2, b2) on h_2k, h_2k+1, the second times i
            const double a1 = at(2 * k, 2 * q), b1 = at(2 * k + 1, 2 * q);
            const double a2 = at(2 * k, 2 * q + 1), b2 = at(2 * k + 1, 2 * q + 1), w = 0.5 * root[size_t(f) * K + k];
            t.alpha[size_t(q) * K + k] = make_double2(w * (a1 + b2), w * (a2 - b1));
            t.beta[size_t(q) * K + k] = make_double2(w * (a1 - b2), w * (a2 + b1));
          }
      }
    }
    sets.push_back(std::move(t));
  }

  h->n_sets = int(sets.size());
  h->set_start[0] = 0;
  for (int u = 0; u < h->n_sets; ++u) h->set_start[u + 1] = h->set_start[u] + sets[u].kernels;
  const size_t total = std::max(1, h->set_start[h->n_sets]);
  if ((st = memory(cudaMalloc(&h->d_psi, total * cc * sizeof(float2)))) != LITHO_OK) return st;
  if ((st = memory(cudaMalloc(&h->d_power, h->n_sets * cc * sizeof(float)))) != LITHO_OK) return st;
  const unsigned blocks = unsigned((cc + 255) / 256);
  for (int u = 0; u < h->n_sets; ++u) {
    const Set& t = sets[u];
    float2* psi = h->d_psi + h->set_start[u] * cc;
    LITHO_TRY_CUDA(cudaMemsetAsync(power, 0, cc * sizeof(double), sc.st));
    int at = 0;
    for (int k = 0; k < K; ++k) {
      const double r = root[size_t(t.plane) * K + k];
      if (r == 0.0) continue;
      const double2* src = phi64 + (whole ? t.plane * plane_len + k * cc : 0);
      if (!whole) LITHO_TRY_CUDA(sc.up(phi64, host + t.plane * plane_len + k * cc, cc * sizeof(double2)));
      if (!t.reduced) k_scale<<<blocks, 256, 0, sc.st>>>(src, r, cc, psi + (at++) * cc);
      k_add_power<<<blocks, 256, 0, sc.st>>>(src, h->lambda[size_t(t.plane) * K + k], cc, power);
    }
    if (t.reduced) {
      if ((st = upload_coef(t.alpha, t.beta, t.plane)) != LITHO_OK) return st;
      k_combine<<<dim3(blocks, t.kernels), 256, 0, sc.st>>>(phi64 + t.plane * plane_len, K, C, coef,
                                                            coef + kk, psi);
    }
    k_round<<<blocks, 256, 0, sc.st>>>(power, C, h->edge ? 0 : 1, h->d_power + u * cc);
    LITHO_TRY_CUDA(cudaGetLastError());
  }
  LITHO_TRY_CUDA(cudaStreamSynchronize(sc.st));  // the set is read from any stream afterwards
  return LITHO_OK;
}

}  // namespace

litho_status build_kernel_set(litho_kernels* h) {
  try {
    const size_t bytes = h->phi_host.size() * sizeof(double);
    const bool whole = h->k <= kMaxReduceK && bytes <= kMaxReduceBytes;
    bool no_memory;
    litho_status s = build(h, whole, &no_memory);
    if (s != LITHO_OK && whole && no_memory) {  // beside a nearly full device: the set as given, no scratch of its size
      cudaFree(h->d_psi);
      cudaFree(h->d_power);
      h->d_psi = nullptr;
      h->d_power = nullptr;
      s = build(h, false, &no_memory);
    }
    return s;
  } catch (const std::bad_alloc&) {
    set_error("host allocation failed while building the kernel set");
    return LITHO_ENOMEM;
  }
}

// Planes [0, count) of the sets [first, first + count): their fields in order.
FieldSet field_set(const litho_kernels* h, int first, int count) {
  FieldSet s{};
  s.planes = count;
  for (int p = 0; p <= count; ++p) s.start[p] = h->set_start[first + p] - h->set_start[first];
  return s;
}

PlaneOut plane_out(const litho_kernels* h) {
  PlaneOut o{};
  o.out_planes = h->n_focus;
  int at = 0;
  for (int u = 0; u < h->n_sets; ++u) {
    o.first[u] = (unsigned char)at;
    for (int f = 0; f < h->n_focus; ++f)
      if (h->set_of[f] == u) o.list[at++] = (unsigned char)f;
  }
  o.first[h->n_sets] = (unsigned char)at;
  return o;
}

PlaneOut plane_out_identity(int planes) {
  PlaneOut o{};
  o.out_planes = planes;
  for (int u = 0; u < planes; ++u) o.first[u] = o.list[u] = (unsigned char)u;
  o.first[planes] = (unsigned char)planes;
  return o;
}

}  // namespace litho
