// Internal declarations shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <complex>
#include <mutex>
#include <string>
#include <vector>

#include "../../include/litho.h"

namespace litho {

// thread-local error message behind litho_last_error()
void set_error(const char* fmt, ...);

// The runtime keeps a failed call's error until it is read: it is read here, so that the next call's check
// (ours, or that of another library on this thread) does not report it again.
#define LITHO_TRY_CUDA(expr)                                                                   \
  do {                                                                                         \
    cudaError_t e_ = (expr);                                                                   \
    if (e_ != cudaSuccess) {                                                                   \
      cudaGetLastError();                                                                      \
      ::litho::set_error("%s failed: %s (%s:%d)", #expr, cudaGetErrorString(e_), __FILE__, __LINE__); \
      return LITHO_ECUDA;                                                                      \
    }                                                                                          \
  } while (0)

using cd = std::complex<double>;

constexpr int kMaxPlanes = 64;  // focus planes of a kernel set

// The planes a launch evaluates per clip and the fields of each: plane p of
// clip i sums the fields [start[p], start[p + 1]) of the clip's start[planes].
struct FieldSet {
  int planes;
  int start[kMaxPlanes + 1];
  __host__ __device__ int fields() const { return start[planes]; }
};
// Where a launch's planes go: plane p of clip i is written to the output
// planes list[first[p]] ... of the clip's out_planes.
struct PlaneOut {
  int out_planes;
  unsigned char first[kMaxPlanes + 1], list[kMaxPlanes];
};

// ---- per-stage device timing (prof.cpp) ------------------------------------------------------
enum Stage {
  kStageMaskSpectrum = 0,
  kStageStage1Fft,
  kStageStage2Fft,
  kStageGemmOperands,
  kStageStage2Gemm,
  kStageResist,
  kStageIltForward,
  kStageIltBackward,
  kStageIltReduce,
  kStageUpsample,
  kStageUpsampleResist,
  kStageContours,
  kStageEpe,
  kStageRaster,
  kStageCount
};
// Records a CUDA event pair around its lifetime on `st` when profiling is on.
class ProfScope {
 public:
  ProfScope(int stage, cudaStream_t st, int launches);
  ~ProfScope();
  ProfScope(const ProfScope&) = delete;
  ProfScope& operator=(const ProfScope&) = delete;

 private:
  int stage_;
  cudaStream_t st_;
  int launches_;
  void* a_ = nullptr;
};

// ---- host optics builder (optics.cpp) -------------------------------------------------------
struct SourcePoints {
  std::vector<double> sx, sy, w;  // units of NA/wavelength; sum w = 1
};
bool sample_source(const litho_optics& o, SourcePoints* out, std::string* why);
int band_crop(const litho_optics& o, const SourcePoints& s, int n, double pixel_nm);

struct FocusKernels {
  std::vector<double> lambda;  // [k], descending, 0 beyond rank
  std::vector<cd> phi;         // [k][C][C]
  int rank = 0;
  double trace = 0.0, gap = 0.0;
};
// Eigen-kernels of the TCC of one focus plane (Eqs. (2)-(3)).
bool build_focus_kernels(const litho_optics& o, const SourcePoints& s, int n, double pixel_nm, double z_nm, int k,
                         int crop, FocusKernels* out, std::string* why);
// Cyclic Jacobi for a Hermitian matrix (row-major, n x n, destroyed). Eigenvalues
// ascending in `ev` are not guaranteed: the caller sorts.  V columns = eigenvectors.
void hermitian_jacobi(std::vector<cd>& a, int n, std::vector<double>& ev, std::vector<cd>& v);

// ---- device data for the GEMM path --------------------------------------------------------
struct GemmOperands;  // gemm.cu

}  // namespace litho

struct litho_kernels {
  int n = 0, crop = 0, n_focus = 0, k = 0;
  double pixel_nm = 0.0;
  std::vector<int> rank;
  std::vector<double> lambda, trace, gap;  // [F*K], [F], [F]
  std::vector<double> phi_host;            // [F][K][C][C][2]
  // The fields the device evaluates (kernelset.cu): n_sets sets of kernels Psi with
  // sqrt(lambda) folded in, set u at d_psi + set_start[u] C^2; plane f is the image of set set_of[f].
  int n_sets = 0, set_start[litho::kMaxPlanes + 1] = {};
  unsigned char set_of[litho::kMaxPlanes] = {};
  float2* d_psi = nullptr;                 // [set_start[n_sets]][C][C]
  float* d_power = nullptr;                // [n_sets][C][C]: sum_k lam_k |Phi_k|^2 (without edge: made even in u)
  bool edge = true;                        // a kernel may be nonzero at u = -C/2, whose mirror is off the crop
  float2* d_tw = nullptr;                  // FFT twiddle table for N
  int nc = 0;                              // FP32 FFT coarse grid: smallest power of two >= 2 crop (0: not below N)
  float2* d_twc = nullptr;                 // FFT twiddle table for nc
  int nc_tc = 0;                           // tensor-core coarse grid: as nc, or 896 when 2 crop <= 896 < nc
  float2* d_twc_tc = nullptr;              // FFT twiddle table for nc_tc (d_twc when nc_tc == nc)
  float2* d_tw32 = nullptr;                // second-pass twiddles of the warp-per-row 1024-point stage 2
                                           // (when N or nc is 1024, else NULL)
  float2* d_tw512 = nullptr;               // twiddles of the 512-point adjoint rows, two rows per warp
                                           // (when N or nc is 512, else NULL)
  litho::GemmOperands* gemm = nullptr;     // lazily built per precision
  int device = 0;
  // streams and events of the pipelined host-buffer path (created on first use)
  std::mutex host_mu;
  cudaStream_t host_streams[3] = {nullptr, nullptr, nullptr};  // input copies, kernels, output copies
  cudaEvent_t host_events[3] = {nullptr, nullptr, nullptr};
  // timing events of the host-buffer path (one start, three per chunk), grown on demand
  std::vector<cudaEvent_t> host_timing;
  std::vector<cudaEvent_t> host_sync;  // ordering events of the host-buffer path, three per chunk
};

namespace litho {

// Coarse grid for a band of C columns on an N grid (api.cpp): smallest power
// of two >= 2C, or with allow896 also 896; 0 when not below N.
int coarse_grid(int C, int N, bool allow896);

// Coarse evaluation grid of a precision's path (0 when it does not apply) and its twiddle table.
inline int coarse_n(const litho_kernels* h, litho_precision p) { return p == LITHO_PREC_FFT32 ? h->nc : h->nc_tc; }
inline const float2* coarse_tw(const litho_kernels* h, litho_precision p) {
  return p == LITHO_PREC_FFT32 ? h->d_twc : h->d_twc_tc;
}

// ---- the device's kernel sets (kernelset.cu) --------------------------------------------------
// Fills n_sets, set_start, set_of, d_psi and d_power from lambda and phi_host.
litho_status build_kernel_set(litho_kernels* h);
// The planes of sets [first, first + count) as a launch's planes.
FieldSet field_set(const litho_kernels* h, int first, int count);
// Set u of a launch over all sets goes to every focus plane it is the image of.
PlaneOut plane_out(const litho_kernels* h);
// Plane p goes to output plane p (library intermediates).
PlaneOut plane_out_identity(int planes);

// ---- launchers (fft.cu) ---------------------------------------------------------------------
// The N-entry per-pass twiddle table the FFT kernels expect (false if n unsupported).
bool fft_twiddle_table(int n, float2* out);
// Mask spectrum: m[b][n][n] -> mhat[b][C][C] = N^-2 DFT(m) on the crop.  rowbuf: [b][n][C/2 + 8].
cudaError_t launch_mask_spectrum(const float* m, int b, int n, int crop, const float2* tw, float2* rowbuf,
                                 float2* mhat, cudaStream_t st);
// The same of the mask sigmoid(alpha theta).
cudaError_t launch_sigmoid_spectrum(const float* theta, float alpha, int b, int n, int crop, const float2* tw,
                                    float2* rowbuf, float2* mhat, cudaStream_t st);
// The mask spectrum, the masks also copied to copy + i copy_stride.
cudaError_t launch_mask_spectrum_copy(const float* m, int b, int n, int crop, const float2* tw, float2* rowbuf,
                                      float2* mhat, float* copy, size_t copy_stride, cudaStream_t st);
// Its two passes.  Row DFTs of real planes, the frequencies u >= 0: rowbuf[b][n][C/2], index u, or (whole:
// with u = C/2) [b][n][C/2 + 8].
cudaError_t launch_mask_rows(const float* m, int b, int n, int crop, const float2* tw, float2* rowbuf, bool whole,
                             cudaStream_t st);
// Column DFTs times n^-2 on the crop.  whole: mhat[b][C][C]; else only its columns u >= 0 (index u + C/2),
// times gain[v] gain[u] with gain [C].
cudaError_t launch_mask_cols(const float2* rowbuf, int b, int n, int crop, const float2* tw, float2* mhat,
                             const float* gain, bool whole, cudaStream_t st);
// Column pass of the interpolation from an nc grid to an n grid (interp.cu), for half rows of h columns
// rspec[p][nc][h]: q[p][n][h] = the inverse transform on n of the crop 2h of nc^-2 x the forward transform
// on nc; with gain [2h] the same times gain[v] gain[u] (the blur's half rows), or with `image` too both,
// q[p][n][2][h].
bool interp_cols_supported(int nc, int n);
cudaError_t launch_interp_cols(const float2* rspec, int planes, int nc, int n, int h, const float2* tw_nc,
                               const float2* tw_n, const float* gain, bool image, float2* q, cudaStream_t st);
// Inverse column transform of the columns u >= 0 of spectra spec[nk][C][C]: half rows q[nk][n][ld] (ld >= C/2).
cudaError_t launch_stage1_half(const float2* spec, int nk, int n, int crop, const float2* tw, float2* q, int ld,
                               cudaStream_t st);
// Stage 1 (band multiply + inverse DFT over v): for kernels psi[nk][C][C],
// t1[j][y][c] = sum_v mhat[v][c] psi_j[v][c] e^{+2 pi i v y/N}, j in [0, nk).
// psi == NULL transforms nk spectra mhat[j][C][C] themselves.  With kernels,
// `clips` spectra mhat[clips][C][C] are imaged in one launch; clip i writes
// t1[j + i nk].
cudaError_t launch_stage1_fft(const float2* mhat, const float2* psi, int nk, int n, int crop, const float2* tw,
                              float2* t1, cudaStream_t st, int clips = 1);
// Stage 2 FFT path: I[y][x] = dose * sum_j |sum_c t1[j][y][c] e^{+2 pi i u_c x/N}|^2
// over the fields of each plane of `fs`, for `clips` clips whose fields follow
// one another in t1; the image of a plane goes to its planes of `po` in img
// (planes of n^2).  With tw32 (the kernel set's d_tw32) a 1024-point row takes
// the warp-per-row radix-32 kernel, with tw512 (d_tw512) 512-point rows the
// two-rows-per-warp kernel.  spec (with tw32 only): instead of the image, each
// image row's forward transform on the frequencies u in [0, spec_crop/2), laid
// out as launch_mask_rows writes them ([clips][planes][n][spec_crop/2]); img
// is not written.
cudaError_t launch_stage2_fft(const float2* t1, const FieldSet& fs, int clips, int n, int crop, float dose,
                              const float2* tw, float* img, const PlaneOut& po, cudaStream_t st,
                              const float2* tw32 = nullptr, const float2* tw512 = nullptr, float2* spec = nullptr,
                              int spec_crop = 0);
// The warp-per-row stage 2 for 1024-point rows (stage2_w32.cu) and its
// second-pass twiddle table (31 x 32 entries w^(r l), r in [1, 32), l in [0, 32)).
bool stage2_w32_supported(int n, int crop);
// The two-rows-per-warp stage 2 for 512-point rows (twiddles: the kernel set's d_tw512).
bool stage2_w512_supported(int n, int crop);
cudaError_t launch_stage2_w512(const float2* t1, const FieldSet& fs, int clips, int n, int crop, float dose,
                               const float2* tw512, float* img, const PlaneOut& po, cudaStream_t st);
void stage2_w32_table(float2* out);
constexpr int kStage2W32TableLen = 31 * 32;
cudaError_t launch_stage2_w32(const float2* t1, const FieldSet& fs, int clips, int n, int crop, float dose,
                              const float2* tw2, float* img, const PlaneOut& po, cudaStream_t st,
                              float2* spec = nullptr, int c2 = 0);

// Loads the kernels that the FP32 calls of an n-point set with a crop and a coarse grid nc (0: none) choose
// between by the number of their clips (the mask spectrum's columns, stage 2 and the spectra of the ILT's dL/dI).
cudaError_t load_clip_shapes(int n, int nc, int crop);
cudaError_t load_stage2_w32(int crop);

// A device-side delay of about `ms` milliseconds on `st` (util.cu): one
// thread spinning on the SM clock for a fixed number of cycles, which always
// ends.  The slow request of the serving tests.
cudaError_t launch_delay(cudaStream_t st, double ms);

// dst[i] = src[i] by a kernel, one end page-locked host memory that the device can address: a copy that
// does not wait in a copy engine's queue behind the copies of other streams.
cudaError_t launch_host_copy(float* dst, const float* src, size_t floats, cudaStream_t st);

// Twiddle table of the 512-point adjoint-rows kernel (ilt.cu): kAdj512TableLen entries.
constexpr int kAdj512TableLen = 31 * 16 + 15 * 32;
void adj512_table(float2* out);

// Device address of the per-clip FP64 losses inside an ILT workspace (ilt.cu).
double* ilt_loss_device(const litho_kernels* h, int b, void* workspace, size_t workspace_bytes);

// The channels of Eq. (9) before normalisation (ilt.cu): for b targets at focus plane `focus`, x[c][0] = the
// target, x[c][1] = the aerial image and x[c][2] = the gradient of the plane's total intensity with
// respect to the mask pixels (x: [b][3][n][n]), in groups of clips; `coarse` evaluates the fields and the
// adjoint on the coarse grid.  The extremes of channels 1 and 2 are folded into ext[0] and ext[1] (ordered
// integers, (~0, 0) on entry) where a kernel writes the channel by rows; found[i] tells.  Workspace:
// ai_channels_bytes(h, b).
size_t ai_channels_bytes(const litho_kernels* h, int b);
litho_status ai_channels(const litho_kernels* h, const float* target, int b, double dose, int focus, bool coarse,
                         float* x, void* workspace, uint2* ext, bool found[2], cudaStream_t st);

// Image rows from half band rows q[p][n][h] of `clips` x `planes` planes p, times scale; plane p of a clip
// goes to its planes of `po` in out.  ext: its (min, max) are updated as ordered integers.
cudaError_t launch_band_rows_real(const float2* q, int clips, int planes, int n, int h, float scale, const float2* tw,
                                  float* out, const PlaneOut& po, cudaStream_t st, uint2* ext = nullptr);

struct ResistTaps;
// gain[i] = sum_a g[a] cos(2 pi (i - crop/2) a / n): the blur's transfer function on the crop.
cudaError_t launch_blur_gain(const ResistTaps& taps, int n, int crop, float* gain, cudaStream_t st);
// Image and blur rows from their half band rows q[p][n][2][h]: img (skipped when NULL), iblur, printed =
// [iblur >= threshold] (skipped when NULL).
cudaError_t launch_band_rows_resist(const float2* q, int clips, int planes, int n, int h, const float2* tw,
                                    float threshold, float* img, float* iblur, uint8_t* printed, const PlaneOut& po,
                                    cudaStream_t st);
// ILT forward end on the coarse grid, per pair of full-grid rows: blurred rows from the
// blur's half band rows, sigmoid resist, dL/dI and its half row spectra (rowbuf, as
// launch_mask_rows), and one FP64 partial loss per row pair at partial[plane][pair]
// (planes x n/2 doubles).  Plane p uses target clip p / planes_per_clip and counts weight.w[p mod planes_per_clip]
// times (the focus planes that share its image).
struct PlaneWeight {
  unsigned char w[kMaxPlanes];
};
cudaError_t launch_resist_grad_rows(const float2* band, int planes, int n, int crop, const float2* tw,
                                    const float* target, int planes_per_clip, const PlaneWeight& weight, float beta,
                                    float thr, float2* rowbuf, double* partial, cudaStream_t st);

// ---- rectangle rasterisation (raster.cu) -----------------------------------------------------
long long raster_tiles_per_rect(int max_side);
size_t raster_workspace_bytes(int b, int n, long long max_rects, int max_side);
cudaError_t launch_raster(const float4* rects, const long long* rect_start, int b, long long max_rects,
                          int max_side, int n, float* mask, void* ws, cudaStream_t st);

// ---- contours and edge placement (contour.cu) -----------------------------------------------
size_t contour_workspace_bytes(int planes, int n);
cudaError_t launch_contours(const float* img, int planes, int n, float thr, float4* seg, int* cell_id,
                            long long capacity, long long* plane_start, void* ws, cudaStream_t st);
cudaError_t launch_epe(const float* img, int planes, int n, float pixel_nm, float thr, const float2* pts, int m,
                       float* epe, cudaStream_t st);
// Eq. (6) for all clips' points in one launch (points of clip c at [start[c], start[c+1])).
cudaError_t launch_epe_batch(const float* img, int clips, int planes, int n, float pixel_nm, float thr,
                             const float2* pts, const long long* start, long long m, float* epe, cudaStream_t st);
cudaError_t launch_epe_focus(const float* epe, int m, int f0, int fp, int fn, float tol_neg, float tol_pos,
                             float* avg, float* eff, cudaStream_t st);

// ---- resist (resist.cu) ---------------------------------------------------------------------
constexpr int kMaxResistRadius = 64;
struct ResistTaps {
  int radius;
  float g[2 * kMaxResistRadius + 1];
};
bool resist_taps(double sigma_nm, double pixel_nm, ResistTaps* t, std::string* why);
cudaError_t launch_resist(const float* img, int planes, int n, const ResistTaps& taps, float threshold, float* iblur,
                          uint8_t* printed, cudaStream_t st);

}  // namespace litho
