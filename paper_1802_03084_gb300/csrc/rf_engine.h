// rf_engine.h -- internal interface between the host orchestration
// (rf_api.cpp) and the CUDA kernels.  Plain C++ types only.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "realfast_gb300.h"

namespace rf {

// Gridding entry flags (low bits of GridEntry.cflags).
constexpr int ENT_CONJ = 1;  // contribute conj(R) (folded into the half plane)
constexpr int ENT_NEG = 2;   // checkerboard sign (-1)^(iu + iv) is -1

// One contribution of a (baseline, channel) visibility to a half-plane cell.
// bc = row c * nbl + b of the Stokes-I time series; cflags = (c << 2) | flags;
// row = the cell's v index iv mod N in its column; cell = the cell's global
// index (cells numbered by column, then row).
struct GridEntry {
  int32_t bc;
  int32_t cflags;
  int32_t row;
  int32_t cell;
};

// Device tables of a plan (all device pointers).
struct DevTables {
  const int32_t* delays;        // [ndm][nchan] integrations
  const int32_t* dt_list;       // [ndt]
  const int2* ranges;           // [nranges] cell-aligned entry ranges, one per gridding warp
  const int32_t* col_cell_ptr;  // [ncol + 1] first cell of each column
  const int32_t* cell_row;      // [ncells] row (iv mod N) of each cell
  const GridEntry* ent;         // [nent] sorted by (column, row)
  const int32_t* ongrid_chan;   // [nchan] on-grid baselines per channel
  const float2* twiddle;        // length-N FFT table (fft_twiddle_table(N)): [0, N) exp(+2 pi i m / N)
  // twiddle table of the column pass's sub-transforms, fft_twiddle_table(L)
  // with L = N / col_split(N) (the same table as `twiddle` when N <= 1024)
  const float2* twiddle_col;
  // runs of every imaged column: the column's cells at rows v1 + L v2 for one
  // v1 (cells sort by (v1 mod TL, v1 div TL, v2) within a column, so a run is
  // consecutive); col_runs[col_run_ptr[col] + j] = (first cell << 4) | cells,
  // the first cell counted within the column
  const int32_t* col_run_ptr;   // [ncol + 1]
  const int32_t* col_runs;
  // per column and lane t of the TL lanes of a column sub-transform (E = L / TL
  // values a lane): x = bits r for which row t + r TL is occupied (any v2), y =
  // the lane's first run within the column; runs sort by (lane, r)
  const int2* col_lane;         // [ncol][TL]
  // per run j and sub-transform p = 1 .. R-1 (R = col_split(N) > 1): the
  // decimation-in-frequency twiddle w_N^(v1 p) of the run's row v1, at
  // col_run_tw[j (R - 1) + p - 1] (computed in FP64, rounded once)
  const float2* col_run_tw;
  // boxcar-resampled Stokes I per dt index s, phase-split: element (row, p, i)
  // at sdt_ptr[s] + row * dt * sdt_lp[s] + p * sdt_lp[s] + i holds
  // sum_{j < dt, i dt + p + j < nint} S[row][i dt + p + j]
  const unsigned long long* sdt_ptr;  // [ndt] device addresses (dt = 1: S itself)
  const int32_t* sdt_lp;              // [ndt] phase length ceil(nint_pad / dt)
};

// Group of consecutive output integrations of one (DM, dt) trial imaged
// together by the gridding/column-FFT kernel, and the images derived from
// them.  The transforms of an image are linear in the visibilities, and a
// boxcar of 2^L dt integrations is the sum of 2^L consecutive ones of dt, so
// image t' of the trial of width 2^L dt is the sum of images 2^L t' ..
// 2^L t' + 2^L - 1 of the same DM: it takes no transform of its own.  t0 is a
// multiple of 32 wherever a sum is searched.
struct Group {
  int32_t d;
  int32_t s;
  int32_t t0;
  int32_t nimg;
  int32_t img0;  // index of the group's first image in the image list
  int32_t base0;  // index of its first image among the transformed images
  // sums of 2, 4, 8 and 16: how many are searched, the first one's index in
  // the image list
  int32_t nsum[4], isum[4];
  int32_t pad[2];
};

// Up to unit_images(pairs) consecutive transformed images of a group, for the
// row pass: the transformed-image index of the first, how many there are, and
// the image list's indices of the first one and of the first sum of 2, 4, 8
// and 16 of them (-1: not searched).
struct Unit {
  int32_t base, n, img[5], pad;
};
// Sums of 8 and 16 images take the row pass that transforms images in pairs
// (k_rowfft_duo: four levels of sums), which goes up to 2048^2.  Plans without
// them, or above that size, take k_rowfft_tree (two rows of one image a
// transform, two levels): per transform it is the faster one (2048^2, widths
// 1 .. 16: 3.90 us an image against 4.13; 512^2 with clipped noise, widths 1,
// 2, 4: 4.05 ms against 4.41), but each width more that is a sum saves the
// gridding, column pass and row transforms of its images (2048^2, widths 1 ..
// 16: 291 ms against 262).
constexpr bool pairs_possible(int npix) { return npix <= 2048; }
constexpr int unit_images(bool pairs) { return pairs ? 16 : 4; }
// Position of image row r of column u within its block of XB rows in the
// column-FFT output that k_rowfft_duo reads: r ^ duo_swizzle(npix, u), so that
// the 16 lanes which read 8-byte values of consecutive columns from shared
// memory at once (or of several rows, where a transform has fewer lanes)
// meet 16 different bank pairs.
__host__ __device__ constexpr int duo_swizzle(int npix, int u) {
  return npix >= 512 ? (u / (npix / 512)) & (npix >= 1024 ? 8192 / npix - 1 : 15) : (u * (512 / npix)) & 15;
}

// Tensor map of a column-FFT output buffer T[slot][u][N] (as FP32 pairs) for
// the row pass's tile copies: nbox boxes of `rows` u rows each cover ncol.
struct TileMap {
  CUtensorMap map;
  int nbox;
  int rows;
};

// Launch options of the column and row passes when the waves of a search
// are overlapped (wave w + 1's column pass beside wave w's row pass, on two
// streams).  one_per_sm: the column pass asks for enough shared memory that
// a second column block no longer fits an SM, while a row block still does;
// items_per_block > 0: the row pass runs blocks of that many work items
// instead of one persistent block per slot, so that blocks of the two passes
// can take turns on an SM; priority (if set_priority): the launch's
// scheduling priority (lower values first).
struct PassLaunch {
  bool one_per_sm = false;
  int items_per_block = 0;
  bool set_priority = false;
  int priority = 0;
};

// Boxes of at most 256 rows (a multiple of 8) covering ncol rows.
inline void tile_boxes(int ncol, int* nbox, int* rows) {
  const int n0 = (ncol + 255) / 256;
  *rows = ((ncol + n0 - 1) / n0 + 7) / 8 * 8;  // whole swizzle atoms per box
  *nbox = (ncol + *rows - 1) / *rows;
}

// Statistics of one periodicity pair (DM trial d, fluctuation frequency k).
struct DevPeriodic {
  int32_t d, k, x, y;
  float amplitude, sigma, snr;
  int32_t pad;
};

// A candidate whose products are computed: trial (d, s, t') and pixel (x, y).
struct CandRef {
  int32_t d, s, t, x, y;
  int32_t pad[3];
};

// Twiddle table of a length-n FFT (n a power of two, 16..8192): entries
// [0, n) hold exp(+2 pi i m / n); when the transform has a second pass
// (n >= 64) entries n + (r / 2) 64 + 2 k + (r mod 2), r < P2, k < 32, hold
// that pass's twiddles exp(+2 pi i k r / (32 P2)), P2 = fft_pass2_radix(n)
// (the two r of a pair side by side, for 16-byte loads).  For n = 2048 a
// third section of the same layout, at n + 1024, holds
// exp(+2 pi i r (2k + 1) / 2048): the second-pass twiddles of the odd-pixel
// half of a row transform split into two length-1024 transforms, with the
// split's twiddle exp(+2 pi i r / 2048) folded in.  All are computed in FP64
// and rounded to FP32.
constexpr int fft_ilog2(int n) { return n <= 1 ? 0 : 1 + fft_ilog2(n >> 1); }
constexpr int fft_pass2_radix(int n) {
  // radix-E passes (E = 32, 16 for n = 16), the last of radix n / E^k
  return n < 64 ? 0 : (fft_ilog2(n) < 10 ? (1 << (fft_ilog2(n) - 5)) : 32);
}
constexpr int fft_twiddle_len(int n) { return n + 32 * fft_pass2_radix(n) + (n == 2048 ? 1024 : 0); }
// Fills out[0 .. fft_twiddle_len(n)).
void fft_twiddle_table(int n, float2* out);

// Cell of an off-grid (baseline, channel) in the per-row cell table.
constexpr int kOffGrid = -2147483647 - 1;

// Largest pixel of a part of one image (raw pixel units).
struct StatPartial {
  float max;
  int32_t idx;  // y * N + x of max (lowest on ties)
};

// With the clipped noise, of the same part: the sums of d = J - mean0 and d^2
// over its `kept` pixels J with |d| <= clip sigmas.
struct ClipPartial {
  float sum;
  float sumsq;
  int32_t kept;
  int32_t pad;
};

// Mean and noise of one image over all its pixels, from the Parseval sums.
struct ImgNoise {
  double mean;
  double sigma;
};

// Statistics of the row pass, per slot of a wave: the maximum of every part of
// an image (partials), with the clipped noise also the kept-pixel sums (clip
// and cparts are set together); or, where only candidates are wanted (best and
// gate are set together), each image's largest pixel if it is not below its
// gate: best[slot] starts at 0 and ends as the largest best_key of such pixels.
// rms[slot] (plans with sums): how bright an image is, raw units (see may_pair).
struct PassStats {
  StatPartial* partials = nullptr;  // [slot][partials per image]
  const float2* clip = nullptr;
  ClipPartial* cparts = nullptr;    // [slot][partials per image]
  unsigned long long* best = nullptr;
  const float* gate = nullptr;
  const float* rms = nullptr;
};

// Whether two images, of RMS a and b, may share transforms (k_rowfft_duo): a
// transform's FP32 rounding is relative to both, and one pixel that is not
// finite spoils both.  At most 1.5 times apart (two images of noise are within
// some percent), either's error is at most 1.3 times that of two rows of its
// own; unlimited, a saturated integration put 0.2 sigma into its neighbour at
// 10^6 times its brightness, and one NaN took the neighbour's candidate.
constexpr float kPairContrast = 1.5f;
// A sum of images carries the FP32 rounding of its parts' transforms.  Noise adds
// up to the sum's own power; where the parts' power is more than kSumCancel times
// that (mean-subtracted samples of a whole segment, interference that changes
// sign), the rounding is more than twice that of a transform of the sum's own, in
// the end all there is: a width as long as a mean-subtracted segment came out at
// 10 to 16 sigma where its own transform gives the 4 to 5 of noise.
constexpr double kSumCancel = 4.0;
#ifdef __CUDACC__
__device__ __forceinline__ bool may_pair(float a, float b) {
  return a <= kPairContrast * b && b <= kPairContrast * a && a + b < INFINITY;  // false for NaN
}
#endif

// A pixel as a key: of two pixels the larger value has the larger key, of two
// equal ones the lower index.  Never 0 (the value is not NaN).
#ifdef __CUDACC__
__device__ __forceinline__ unsigned best_order(float v) {
  const unsigned b = __float_as_uint(v);
  return b & 0x80000000u ? ~b : b | 0x80000000u;
}
__device__ __forceinline__ unsigned long long best_key(float v, int pixel) {
  return (unsigned long long)best_order(v) << 32 | (0xffffffffu - (unsigned)pixel);
}
__device__ __forceinline__ float best_max(unsigned long long key) {
  const unsigned b = (unsigned)(key >> 32);
  return __uint_as_float(b & 0x80000000u ? b & 0x7fffffffu : ~b);
}
__device__ __forceinline__ int best_pixel(unsigned long long key) { return (int)(0xffffffffu - (unsigned)key); }
#endif

// Clipping radius of the optional one-pass clipped noise, in units of the
// noise over all pixels.
constexpr double kClipSigmas = 5.0;

// Candidate record written on the device.
struct DevCand {
  int32_t d, s, t, x, y;
  float snr, peak, sigma;
};

// Per-image statistics written on the device (verification path).
struct DevStat {
  float peak, sigma, snr;
  int32_t x, y;
  int32_t pad;
  double mean;
  double weight;
};

struct SegmentGeom {
  int nint;       // integrations in this segment
  int nint_pad;   // row pitch of the Stokes-I buffer (elements)
  int nbl;
  int nchan;
  int npix;
  int ncol;       // half-plane columns imaged: 0 .. iu_max
  int ndm;
  int max_cells;  // largest number of occupied cells in one column
  int ncells;     // occupied cells of the half plane
  int nranges;    // gridding ranges
  bool partial;   // PARTIAL edge rule: a sample at or past nint is absent
  bool idx32;     // every sample index of every resampled series fits in 32 bits
  bool fp16;      // Stokes-I stored as half2
  // Row order of the column-FFT output T[slot][u][i]: with tsplit = R > 1,
  // index i = p L + k (L = N / R) holds image row y = R k + p (the column
  // pass's R sub-transforms of length L, one per residue p of y mod R, are
  // stored one after the other); tsplit <= 1: i = y.
  int tsplit;
};

// Sub-transforms per column in the batched column pass: N <= 1024 is one
// length-N transform; larger N are split R = N / 1024 ways along v (one
// radix-R decimation-in-frequency step folded into the gather of the
// column's cells), leaving R transforms of length 1024.
constexpr int col_split(int n) { return n >= 2048 ? n / 1024 : 1; }

// ---------------------------------------------------------------- launchers
// All launchers return cudaSuccess or the launch error.

// Stokes-I ingest of integrations [t_begin, t_begin + nt) from `vis`
// ([nt][nbl][nchan][npol] complex64, already offset to t_begin) into the
// time-major buffer S[c * nbl + b][t].
cudaError_t launch_ingest(const float2* vis, int nt, int t_begin, int npol, const SegmentGeom& g, void* S,
                          cudaStream_t st);

// Subtract from every row of S its mean over the first nint integrations.
cudaError_t launch_mean_subtract(const SegmentGeom& g, void* S, cudaStream_t st);

// Boxcar resampling of S into the phase-split series of width dt (see
// DevTables::sdt_ptr) for the first nint integrations.
cudaError_t launch_resample(const SegmentGeom& g, const void* S, void* Sdt, int dt, int lp, cudaStream_t st);

// W of each listed image (img_info[i] = {d, s, t, 0}); n_on = on-grid
// (baseline, channel) pairs.
cudaError_t launch_weights(const int4* img_info, int nimg, bool partial, const SegmentGeom& g,
                           const DevTables& tb, double n_on, double* weight, cudaStream_t st);

// Gridding (pass A1) of groups [g_begin, g_begin + ngroups): the cell sums
// of every image, cellbuf[group - g_begin][cell][32 images].
cudaError_t launch_grid_cells(const SegmentGeom& g, const DevTables& tb, const Group* groups, int g_begin,
                              int ngroups, float2* cellbuf, cudaStream_t st);

// The same for groups of one image each, of any trials: from the series
// resampled to each one's width, or, with `direct`, from S (bitwise the same).
cudaError_t launch_grid_single(const SegmentGeom& g, const DevTables& tb, const Group* groups, int g_begin,
                               int ngroups, const void* S, bool direct, float2* cellbuf, cudaStream_t st);

// Column FFTs (pass A2) of the same groups from cellbuf; writes
// Tbuf[b][col][y], b = transformed-image index - base_base, and for every
// image of the groups, sums of others included, the Parseval sums
// colsq[slot][col] (weighted sum of |H|^2 over the column) and
// mean0[slot] = Re H(u = 0, v = 0), slot = image index - img_base.  `duo`: in
// the row order of k_rowfft_duo (duo_swizzle).
cudaError_t launch_colfft(const SegmentGeom& g, const DevTables& tb, const Group* groups, int g_begin,
                          int ngroups, int img_base, int base_base, const float2* cellbuf, float2* Tbuf,
                          float* colsq, float* mean0, bool duo, cudaStream_t st, const PassLaunch* pl = nullptr);

// Noise of each of `nimg` slots (first image img_base) from the Parseval sums
// colsq, before the row pass.  gate[i] and best[i] (if not null): the raw pixel
// value below which a maximum cannot make image i a candidate, and 0.  clip[i] (if not null): the
// clipping window of the clipped noise in raw pixel units (the image times
// 2W), {mean0[i], kClipSigmas * sigma over all pixels}.  rms[i] (if not null):
// the raw image's RMS over all pixels.
cudaError_t launch_image_noise(const SegmentGeom& g, const float* colsq, const float* mean0, const double* weight,
                               int nimg, int img_base, double threshold, ImgNoise* noise, float* gate,
                               unsigned long long* best, float2* clip, float* rms, cudaStream_t st);

// After it, where images are sums of others: sums of the units whose images cancel
// (see kSumCancel) are listed in redo, *nredo of them (indices in the image list),
// and lose their weight, so that the finalisation passes them over.
cudaError_t launch_check_sums(const Unit* units, int nunits, int img_base, const float* rms, double* weight,
                              int* nredo, int* redo, cudaStream_t st);

// Row C2R (pass B) + statistics of `nimg` images in slots [0, nimg) whose
// first image index is img_base.  Optionally writes the scaled images.
// `ps` names the per-slot inputs and outputs of the statistics.
cudaError_t launch_rowfft_stats(const SegmentGeom& g, const DevTables& tb, const float2* Tbuf, int nimg,
                                int img_base, const double* weight, const PassStats& ps, float* images,
                                const TileMap* tm, int* err, cudaStream_t st, const PassLaunch* pl = nullptr);

// The same for the transformed images of nunits units (T slots relative to
// base_base, statistics slots to img_base) and the images derived from them,
// npix >= kTreeMinNpix.  With `pairs` (npix <= 2048) T is in duo order and tm
// maps boxes of one image's XB rows; unit_partials(shape, pairs) partials per
// image.
cudaError_t launch_rowfft_tree(const SegmentGeom& g, const DevTables& tb, const float2* Tbuf, const Unit* units,
                               int nunits, bool pairs, int img_base, int base_base, const PassStats& ps,
                               const TileMap* tm, int* err, cudaStream_t st, const PassLaunch* pl = nullptr);
constexpr int kTreeMinNpix = 64;  // below, a row-pass block is less than a warp

// Reduce nparts partials per image (or take ps.best), compute sigma / snr, append candidates and
// (optionally) per-image stats for images [img_base, img_base + nimg).
// Under ps.clip the mean and sigma are those of the kept pixels, from the
// partials' sums around mean0.
cudaError_t launch_finalize(const SegmentGeom& g, const PassStats& ps, int nparts, const ImgNoise* noise,
                            const float* mean0, const int4* img_info, const double* weight, int nimg, int img_base, double threshold,
                            DevCand* cands, int* ncand, int cand_cap, DevStat* stats, cudaStream_t st);

// Buffers of the plain per-trial form (chunks of up to `cap` images).
struct PlainBuffers {
  const void* S;          // Stokes-I time series (as for the batched form)
  float2* R;              // [nbl * nchan][cap] dedispersed, resampled
  float2* grid;           // [cap][N][N/2 + 1] dense half planes
  float2* T;              // [cap][N/2][N] column-FFT output
  float* images;          // [cap][N][N]
  StatPartial* partials;  // [cap][partials per image] (row pass output, unused)
  const int4* ent;        // [nent] {bc, col, row, flags}
  int nent;
  int cap;
};

// One unfused launch set for images [img0, img0 + nk) = t' t0 .. t0+nk-1 of
// trial (d, s): dedisperse, grid (atomics), column FFTs, row FFTs writing the
// images, image statistics read back from HBM (a second read for the
// clipped noise with `clip`).
cudaError_t launch_plain_chunk(const SegmentGeom& g, const DevTables& tb, const PlainBuffers& pb, int d, int s,
                               int t0, int nk, int img0, const int4* img_info, const double* weight,
                               double threshold, DevCand* cands, int* ncand, int cand_cap, DevStat* stats,
                               cudaStream_t st, bool clip = false);

// Compile-time layout facts per image size, for host-side sizing.
struct ImageKernelShape {
  int images_per_group;   // B
  int cols_per_cta;       // C
  int threads_a;
  int smem_a;
  int warps_per_col;      // WPC: warps sharing one column's gridding (pass A)
  int rows_per_cta;       // RB (pass B)
  int partials_per_image; // partials written by pass B per image: N/2 row pairs x warps per transform
  int threads_b;
  int smem_b;
  int smem_a_per_cell;  // column pass: shared bytes per occupied cell of the largest column
  int smem_b_per_row;   // row pass: shared bytes per tile row (one per column imaged)
  bool tile_tma;        // row-pass tiles arrive by tensor copies (boxes, 1 KB alignment)
};
bool image_kernel_shape(int npix, ImageKernelShape* out);
// Partials per image of launch_rowfft_tree: one per row where images are
// transformed in pairs, else as launch_rowfft_stats, one per row pair.
inline int unit_partials(const ImageKernelShape& s, bool pairs) { return s.partials_per_image * (pairs ? 2 : 1); }

// Streaming multiprocessors of the current device (cached per device: launch
// shapes are sized from it, and another GPU of the process may differ).
int sm_count();

// Lanes of one column sub-transform of length l, and values each takes.
constexpr int col_lanes(int l) { return l >= 32 ? l / 32 : 1; }

// Sets the thread-local message returned by rf_last_error().
void set_last_error(const char* msg);

// Candidate products.  cellbc[c * nbl + b] = (iu, iv) or (kOffGrid, 0).
// spec/wch: [n][nchan] FP64 spectrum and w_c; spec_out: FP32 copy or NULL;
// spec_mom: [n][6] {mean, std, skew, excess kurtosis, w-mean, channels}.
cudaError_t launch_cand_spectrum(const SegmentGeom& g, const DevTables& tb, const int2* cellbc, const CandRef* refs,
                                 int n, double2* spec, double* wch, float2* spec_out, double* spec_mom,
                                 cudaStream_t st);
// out: [n][4] {mean, std, skew, excess kurtosis} of each image's npx pixels,
// in nslices slices per image (image_moment_slices); part: [n][nslices][4]
// scratch.
int image_moment_slices(int n, size_t npx);
cudaError_t launch_image_moments(const float* images, int n, size_t npx, int nslices, double* part, double* out,
                                 cudaStream_t st);

// Periodicity search.  Time transform of the dedispersed windows of nb DM
// trials (dms[j] indexes delays) into out[(2 j + q) nrows + row][kk].
cudaError_t launch_period_dft(const SegmentGeom& g, const void* S, const int* delays, const int* dms, int nb,
                              int L, const float2* twl, int kmin, int K, int kpad, float2* out, cudaStream_t st);
// Row pass over npairs (U, Q) image pairs: partials[j * N + y] = row maxima of I_U^2 + I_Q^2.
// tm (may be null): tensor map of Tbuf with boxes of one image's XB rows, for
// the tensor-copy tiles at N = 1024 (T is then in duo order); err: set when a bounded tile wait gives up.
cudaError_t launch_rowfft_power(const SegmentGeom& g, const DevTables& tb, const float2* Tbuf, const int4* pairs,
                                int npairs, StatPartial* partials, const TileMap* tm, int* err, cudaStream_t st);
// Per pair: amplitude, sigma, snr, pixel; stats[pair_base + j]; candidates appended.
cudaError_t launch_finalize_power(const SegmentGeom& g, const StatPartial* partials, const float* colsq,
                                  const float* mean0, const int4* pairs, int npairs, int pair_base, double W,
                                  double threshold, DevPeriodic* stats, DevPeriodic* cands, int* ncand, int cand_cap,
                                  cudaStream_t st);

// One block waits, at most `polls` polls, on an mbarrier that nothing
// arrives at; *status = 1 when the wait gave up (it always should).
cudaError_t launch_wait_selftest(int polls, int* status, cudaStream_t st);

// ---------------------------------------------------------- host helpers --
// For the stream runtime (host code only).
struct PlanGeometry {
  int nbl, nchan, npol, max_nint, max_delay, device;
  bool host_only;
  std::vector<int> dt;
};
rf_status plan_geometry(const struct ::rf_plan* p, PlanGeometry* g);
// One search of nint integrations in which every (DM, dt) is limited to
// t' < span / dt besides the plan's edge rule (span 0: no limit).  Returns
// the candidates and, if stats is not NULL, every image's statistics.
rf_status search_span(struct ::rf_plan* p, const void* vis, int nint, int span, void* stream,
                      std::vector<rf_candidate>* cands, std::vector<rf_image_stat>* stats);

}  // namespace rf
