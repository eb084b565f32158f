// rf_noalloc.cu -- rf_image_stats_noalloc: image one caller-supplied uv
// half-plane and measure its peak, noise and S/N without allocating any
// memory.
//
// Who needs it: code that must not call cudaMalloc -- a caller recording
// work into a CUDA graph (cudaMalloc cannot be captured), a real-time loop
// that cannot take the latency or the failure modes of the allocator, or a
// host framework that owns the device memory pool and forbids allocations by
// libraries it hosts.  Such a caller passes device pointers for the input
// and the output; the column-FFT intermediate and the row-block partials this
// imaging needs live in one file-scope __device__ array, sized for images up
// to RF_NOALLOC_MAX_NPIX pixels a side, which every GPU that loads this
// library holds until the process exits.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <mutex>
#include <vector>

#include "realfast_gb300.h"
#include "rf_engine.h"
#include "rf_image.cuh"

namespace rf {
namespace {

constexpr int kMaxN = RF_NOALLOC_MAX_NPIX;
constexpr int kMaxDevices = 64;

// Scratch: column-FFT output T[u][y] (u < N/2), the row-pair partials of
// the statistics kernel, the per-column Parseval sums and the (0, 0) term.  Every byte a call reads is written by
// the same call first, so nothing has to start at zero.
constexpr size_t kTBytes = (size_t)kMaxN * (kMaxN / 2) * sizeof(float2);
constexpr size_t kPartialBytes = (size_t)ImgCfg<kMaxN>::PARTIALS * sizeof(StatPartial);
constexpr size_t kColsqBytes = (kMaxN / 2 + 64) * sizeof(float);  // Parseval column sums, mean term, block count
static __device__ __align__(256) unsigned char g_noalloc_scratch[kTBytes + kPartialBytes + kColsqBytes];

// Twiddle tables of the length-N transforms (fft_twiddle_table) for N = 16,
// 32, ..., kMaxN, back to back (constants written once per device at
// set-up, not scratch).
constexpr int twiddle_offset(int n) { return n <= 16 ? 0 : twiddle_offset(n >> 1) + fft_twiddle_len(n >> 1); }
constexpr int kTwiddleElems = twiddle_offset(kMaxN) + fft_twiddle_len(kMaxN);
static __device__ __align__(256) float2 g_noalloc_twiddle[kTwiddleElems];

struct DeviceSetup {
  bool ready = false;
  unsigned char* scratch = nullptr;
  float2* twiddle = nullptr;
};
DeviceSetup g_setup[kMaxDevices];
std::mutex g_setup_mu;

rf_status setup_error(rf_status s, const char* what, cudaError_t e) {
  char buf[256];
  snprintf(buf, sizeof(buf), "rf_image_stats_noalloc set-up: %s: %s", what, cudaGetErrorString(e));
  set_last_error(buf);
  return s;
}

// Once per device, with that device current: resolve the device addresses
// of the two arrays (host code cannot use the symbols themselves) and write
// the twiddle tables.
rf_status ensure_setup(int dev, DeviceSetup** out) {
  std::lock_guard<std::mutex> lk(g_setup_mu);
  DeviceSetup& d = g_setup[dev];
  if (!d.ready) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return setup_error(RF_ERR_CUDA, "cudaGetSymbolAddress(scratch)", e);
    d.scratch = static_cast<unsigned char*>(p);
    e = cudaGetSymbolAddress(&p, g_noalloc_twiddle);
    if (e != cudaSuccess) return setup_error(RF_ERR_CUDA, "cudaGetSymbolAddress(twiddle)", e);
    d.twiddle = static_cast<float2*>(p);
    std::vector<float2> tw(kTwiddleElems);
    for (int n = 16; n <= kMaxN; n <<= 1) fft_twiddle_table(n, tw.data() + twiddle_offset(n));
    e = cudaMemcpy(d.twiddle, tw.data(), tw.size() * sizeof(float2), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return setup_error(RF_ERR_CUDA, "twiddle upload", e);
    d.ready = true;
  }
  *out = &d;
  return RF_OK;
}

// Column pass of the imaging kernels, reading a dense half-plane grid
// H[v][u] (row length N/2 + 1) instead of gathering visibilities: each of the
// XA transforms of a CTA takes one column u < N/2, applies the
// (-1)^(u + v) phase-centre shift and inverse-FFTs it along v.
template <int N>
__global__ void __launch_bounds__(ImgCfg<N>::T * ImgCfg<N>::XA)
    k_colfft_dense(const float2* __restrict__ grid, float2* __restrict__ T, const float2* __restrict__ tw,
                   float* __restrict__ colsq, float* __restrict__ mean0) {
  using K = ImgCfg<N>;
  constexpr int W = N / 2 + 1;
  constexpr int NC = N / 2;
  extern __shared__ float2 sm[];
  const int tid = threadIdx.x;
  const int col0 = blockIdx.x * K::XA;
  constexpr int THREADS = K::T * K::XA;
  for (int i = tid; i < N * K::XA; i += THREADS) {
    const int c = i % K::XA;
    const int v = i / K::XA;
    const int u = col0 + c;
    float2 h = make_float2(0.f, 0.f);
    if (u < NC) {
      h = __ldg(grid + (size_t)v * W + u);
      if ((u + v) & 1) h = make_float2(-h.x, -h.y);
    }
    sm[c * K::STRIDE + padx(v)] = h;
  }
  __syncthreads();
  const int xf = tid / K::T;
  const int t = tid - xf * K::T;
  const int u = col0 + xf;
  {
    // Parseval: weighted sum of |H|^2 down the column (twice for u > 0)
    float acc = 0.f;
    for (int v = t; v < N; v += K::T) {
      const float2 h = sm[xf * K::STRIDE + padx(v)];
      acc = fmaf(h.x, h.x, fmaf(h.y, h.y, acc));
    }
    constexpr int WL = K::T < 32 ? K::T : 32;
#pragma unroll
    for (int off = WL / 2; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if (t == 0 && u < NC) {
      colsq[u] = (u == 0 ? 1.f : 2.f) * acc;
      if (u == 0) *mean0 = sm[xf * K::STRIDE].x;
    }
  }
  float2 v[K::E];
  fft_inverse_to_regs<N>(v, sm + xf * K::STRIDE, tw, t, xf);
  if (u < NC) {
    float2* dst = T + (size_t)u * N;
    constexpr int LP = FftShape<N>::LAST_P;
#pragma unroll
    for (int m = 0; m < K::E / LP; ++m)
#pragma unroll
      for (int q = 0; q < LP; ++q) dst[fft_out_index<N>(t, m, q)] = v[m * LP + dft_perm<LP>(q)];
  }
}

// Reduce the row partials and the Parseval column sums of one image into an
// rf_image_stat by the THREADS threads of one block: strided over both, then a
// fixed tree of the lanes and of the warps.  (One thread walking them in turn
// waits for a load after a load: a call at 1024^2 took 73.7 us so, 41.0 this
// way.)
template <int THREADS>
__device__ __forceinline__ void noalloc_finalize(const StatPartial* __restrict__ partials, int nparts,
                                                 const float* __restrict__ colsq, const float* __restrict__ mean0,
                                                 int npix, double weight, rf_image_stat* __restrict__ out) {
  constexpr int NW = THREADS / 32;
  __shared__ double w_sq[NW];
  __shared__ float w_max[NW];
  __shared__ int w_idx[NW];
  const int tid = threadIdx.x;
  double sq = 0.0;
  float mx = -FLT_MAX;
  int mi = INT_MAX;
  // read past the first level cache: other blocks of the same launch wrote them
#pragma unroll 8
  for (int r = tid; r < nparts; r += THREADS) {
    const float2 p = __ldcg(reinterpret_cast<const float2*>(partials) + r);
    max_merge(mx, mi, p.x, __float_as_int(p.y));
  }
#pragma unroll 8
  for (int c = tid; c < npix / 2; c += THREADS) sq += (double)__ldcg(colsq + c);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    sq += __shfl_xor_sync(0xffffffffu, sq, off);
    const float om = __shfl_xor_sync(0xffffffffu, mx, off);
    const int oi = __shfl_xor_sync(0xffffffffu, mi, off);
    max_merge(mx, mi, om, oi);
  }
  if ((tid & 31) == 0) {
    w_sq[tid >> 5] = sq;
    w_max[tid >> 5] = mx;
    w_idx[tid >> 5] = mi;
  }
  __syncthreads();
  if (tid != 0) return;
  for (int w = 1; w < NW; ++w) {
    sq += w_sq[w];
    max_merge(mx, mi, w_max[w], w_idx[w]);
  }
  // mean = G(0,0) / 2W; mean of I^2 = sum_full |G|^2 / 4W^2 (Parseval)
  const double inv = 0.5 / weight;
  const double mean = (double)__ldcg(mean0) * inv;
  double var = sq * inv * inv - mean * mean;
  var = var > 0.0 ? var : 0.0;
  const double sigma = sqrt(var);
  const double peak = (double)mx * inv;
  rf_image_stat o;
  o.dm_idx = 0;
  o.dt_idx = 0;
  o.t_idx = 0;
  o.y = mi / npix;
  o.x = mi - o.y * npix;
  o.peak = (float)peak;
  o.sigma = (float)sigma;
  o.snr = (float)(sigma > 0.0 ? peak / sigma : 0.0);
  o.mean = mean;
  o.weight = weight;
  *out = o;
}


__global__ void __launch_bounds__(256)
    k_noalloc_finalize(const StatPartial* __restrict__ partials, int nparts, const float* __restrict__ colsq,
                       const float* __restrict__ mean0, int npix, double weight, rf_image_stat* __restrict__ out) {
  noalloc_finalize<256>(partials, nparts, colsq, mean0, npix, weight, out);
}

// N >= 64: two launches, shaped for one image.  The imaging kernels' blocks
// (32 columns or row pairs at 256^2, a tile in shared memory) suit thousands
// of images; one image then runs on four SMs and waits for its staging loops.
// Here a block is a few transforms, which load their inputs straight into
// registers (every load in flight at once; the other half of a sector is its
// neighbour's), and the last row block to finish reduces the image.
// 256^2: 34.3 to 27.9 us a call, 1024^2: 41.0 to 35.5, most of it host time now.
template <int N>
struct SingleCfg {
  static constexpr int T = ImgCfg<N>::T, E = ImgCfg<N>::E;
  static constexpr int XC = cmax(4, 32 / T);   // columns per block: 32-byte sectors
  static constexpr int XR = cmax(2, 32 / T);   // row pairs per block
  static constexpr int NC = N / 2;
  static_assert(T >= 2 && T <= 32 && E == 32 && NC % XC == 0 && NC % XR == 0, "whole warps, whole blocks");
};

// Column u of the half plane: the (-1)^(u + v) phase-centre shift, the Parseval
// sum and the inverse FFT along v into T[u][.].  Also zeroes the row launch's
// count of finished blocks.
template <int N>
__global__ void __launch_bounds__(SingleCfg<N>::T * SingleCfg<N>::XC)
    k_single_columns(const float2* __restrict__ grid, float2* __restrict__ T, const float2* __restrict__ tw,
                     float* __restrict__ colsq, float* __restrict__ mean0, unsigned* __restrict__ done) {
  using C = SingleCfg<N>;
  constexpr int TT = C::T, E = C::E;
  __shared__ float2 sm[C::XC * fft_stride<N>()];
  const int xf = threadIdx.x / TT, t = threadIdx.x % TT;
  const int u = blockIdx.x * C::XC + xf;
  if (blockIdx.x == 0 && threadIdx.x == 0) *done = 0;
  float2 v[E];
  const float2* src = grid + (size_t)t * (N / 2 + 1) + u;
#pragma unroll
  for (int r = 0; r < E; ++r) v[r] = __ldg(src + (size_t)r * TT * (N / 2 + 1));
  if ((u + t) & 1)  // rows t + r TT, TT even
#pragma unroll
    for (int r = 0; r < E; ++r) v[r] = make_float2(-v[r].x, -v[r].y);
  float acc = 0.f;
#pragma unroll
  for (int r = 0; r < E; ++r) acc = fmaf(v[r].x, v[r].x, fmaf(v[r].y, v[r].y, acc));
#pragma unroll
  for (int off = TT / 2; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
  if (t == 0) {
    colsq[u] = (u == 0 ? 1.f : 2.f) * acc;  // twice for u > 0
    if (u == 0) *mean0 = v[0].x;
  }
  fft_inverse_from_regs<N>(v, sm + xf * fft_stride<N>(), tw, t, xf);
  float2* dst = T + (size_t)u * N;
  constexpr int LP = FftShape<N>::LAST_P;
#pragma unroll
  for (int m = 0; m < E / LP; ++m)
#pragma unroll
    for (int q = 0; q < LP; ++q) dst[fft_out_index<N>(t, m, q)] = v[m * LP + dft_perm<LP>(q)];
}

// Rows y, y + 1 from T (as row_zbuild), their maximum into partials[y / 2], and
// the image's record by the block that finishes last.
template <int N>
__global__ void __launch_bounds__(SingleCfg<N>::T * SingleCfg<N>::XR)
    k_single_rows(const float2* __restrict__ T, const float2* __restrict__ tw, StatPartial* __restrict__ partials,
                  const float* __restrict__ colsq, const float* __restrict__ mean0, unsigned* __restrict__ done,
                  double weight, rf_image_stat* __restrict__ out) {
  using C = SingleCfg<N>;
  constexpr int TT = C::T, E = C::E;
  __shared__ float2 sm[C::XR * fft_stride<N>()];
  __shared__ bool last;
  const int xf = threadIdx.x / TT, t = threadIdx.x % TT;
  const int pair = blockIdx.x * C::XR + xf;
  float2 v[E];
  // rows 2 pair, 2 pair + 1 of column u: one 16-byte load
  const float4* col = reinterpret_cast<const float4*>(T) + pair;
#pragma unroll
  for (int r = 0; r < E / 2; ++r) {
    const float4 ab = col[(size_t)(t + r * TT) * (N / 2)];
    v[r] = (r == 0 && t == 0) ? make_float2(ab.x, ab.z) : make_float2(ab.x - ab.w, ab.y + ab.z);
  }
#pragma unroll
  for (int r = E / 2; r < E; ++r) {
    // column N - u; u = N / 2 has none
    float4 ab = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r > E / 2 || t > 0) ab = col[(size_t)(N - t - r * TT) * (N / 2)];
    v[r] = make_float2(ab.x + ab.w, ab.z - ab.y);
  }
  fft_inverse_from_regs<N>(v, sm + xf * fft_stride<N>(), tw, t, xf);
  PassStats ps;
  ps.partials = partials;
  row_stats<N, kParts>(v, t, pair, 0, 0, 1, 0, 0.f, ps);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(done, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  noalloc_finalize<SingleCfg<N>::T * SingleCfg<N>::XR>(partials, N / 2, colsq, mean0, N, weight, out);
}

template <int N>
cudaError_t run_noalloc(const float2* grid, double weight, const DeviceSetup& d, cudaStream_t st,
                        rf_image_stat* out) {
  using K = ImgCfg<N>;
  // The column-FFT scratch holds one image of at most kMaxN, the partials
  // area ImgCfg<kMaxN>::PARTIALS records; the Parseval sum of a column is
  // reduced within a warp, in k_single_columns as in k_colfft_dense (below
  // 64^2), which holds while a transform fits one.
  static_assert(N <= kMaxN, "image larger than the static scratch");
  static_assert(K::PARTIALS <= ImgCfg<kMaxN>::PARTIALS, "partials area too small");
  static_assert(K::T <= 32, "the Parseval reduction of a column spans one warp");
  float2* T = reinterpret_cast<float2*>(d.scratch);
  StatPartial* partials = reinterpret_cast<StatPartial*>(d.scratch + kTBytes);
  float* colsq = reinterpret_cast<float*>(d.scratch + kTBytes + kPartialBytes);
  float* mean0 = colsq + kMaxN / 2;
  const float2* tw = d.twiddle + twiddle_offset(N);
  constexpr int NC = N / 2;
  if constexpr (N >= 64) {
    using C = SingleCfg<N>;
    unsigned* done = reinterpret_cast<unsigned*>(mean0 + 1);
    k_single_columns<N><<<NC / C::XC, C::T * C::XC, 0, st>>>(grid, T, tw, colsq, mean0, done);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_single_rows<N><<<NC / C::XR, C::T * C::XR, 0, st>>>(T, tw, partials, colsq, mean0, done, weight, out);
    return cudaGetLastError();
  } else {
    // set on every call: the attribute belongs to the current device's context
    const cudaError_t attr =
        cudaFuncSetAttribute(k_colfft_dense<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, K::SMEM_A_FIXED);
    if (attr != cudaSuccess) return attr;
    k_colfft_dense<N><<<(NC + K::XA - 1) / K::XA, K::T * K::XA, K::SMEM_A_FIXED, st>>>(grid, T, tw, colsq, mean0);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    SegmentGeom g{};
    g.npix = N;
    g.ncol = NC;
    g.tsplit = 1;  // k_colfft_dense stores T in natural row order
    DevTables tb{};
    tb.twiddle = tw;
    tb.twiddle_col = tw;
    PassStats ps;
    ps.partials = partials;
    e = launch_rowfft_stats(g, tb, T, 1, 0, nullptr, ps, nullptr, nullptr, nullptr, st);
    if (e != cudaSuccess) return e;
    k_noalloc_finalize<<<1, 256, 0, st>>>(partials, K::PARTIALS, colsq, mean0, N, weight, out);
    return cudaGetLastError();
  }
}


}  // namespace
}  // namespace rf

extern "C" rf_status rf_image_stats_noalloc(const void* half_plane, int32_t npix, double weight, void* stream,
                                            rf_image_stat* stat) {
  using namespace rf;
  char buf[256];
  if (!half_plane || !stat) {
    set_last_error("rf_image_stats_noalloc: half_plane and stat must be device pointers");
    return RF_ERR_INVALID_ARG;
  }
  if (npix < 16 || (npix & (npix - 1)) || npix > RF_NOALLOC_MAX_NPIX) {
    snprintf(buf, sizeof(buf),
             "rf_image_stats_noalloc: npix %d must be a power of two in [16, %d] (the size of its static scratch)",
             npix, RF_NOALLOC_MAX_NPIX);
    set_last_error(buf);
    return RF_ERR_INVALID_ARG;
  }
  if (!(weight > 0.0) || !std::isfinite(weight)) {
    set_last_error("rf_image_stats_noalloc: weight must be > 0");
    return RF_ERR_INVALID_ARG;
  }
  if ((uintptr_t)half_plane % 8 != 0 || (uintptr_t)stat % alignof(rf_image_stat) != 0) {
    snprintf(buf, sizeof(buf), "rf_image_stats_noalloc: half_plane must be 8-byte and stat %zu-byte aligned",
             alignof(rf_image_stat));
    set_last_error(buf);
    return RF_ERR_INVALID_ARG;
  }
  // Both pointers must be device memory of the current device: a kernel
  // given host memory would fault (or, where the device can reach host
  // memory, silently read and write it).  The query allocates nothing.
  int dev = -1;
  const bool have_dev = cudaGetDevice(&dev) == cudaSuccess && dev >= 0;
  for (const void* ptr : {half_plane, static_cast<const void*>(stat)}) {
    cudaPointerAttributes attr;
    const bool ok = have_dev && cudaPointerGetAttributes(&attr, ptr) == cudaSuccess &&
                    (attr.type == cudaMemoryTypeDevice || attr.type == cudaMemoryTypeManaged) && attr.device == dev;
    if (!ok) {
      cudaGetLastError();
      set_last_error("rf_image_stats_noalloc: half_plane and stat must be device memory of the current device");
      return RF_ERR_INVALID_ARG;
    }
  }
  cudaError_t e = cudaSuccess;
  if (dev >= kMaxDevices) {
    set_last_error("rf_image_stats_noalloc: device ordinal beyond the set-up table");
    return RF_ERR_NO_DEVICE;
  }
  DeviceSetup* d = nullptr;
  rf_status s = ensure_setup(dev, &d);
  if (s != RF_OK) return s;
  const float2* grid = static_cast<const float2*>(half_plane);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  switch (npix) {
    case 16: e = run_noalloc<16>(grid, weight, *d, st, stat); break;
    case 32: e = run_noalloc<32>(grid, weight, *d, st, stat); break;
    case 64: e = run_noalloc<64>(grid, weight, *d, st, stat); break;
    case 128: e = run_noalloc<128>(grid, weight, *d, st, stat); break;
    case 256: e = run_noalloc<256>(grid, weight, *d, st, stat); break;
    case 512: e = run_noalloc<512>(grid, weight, *d, st, stat); break;
    case 1024: e = run_noalloc<1024>(grid, weight, *d, st, stat); break;
    default: e = cudaErrorInvalidValue; break;
  }
  if (e != cudaSuccess) {
    snprintf(buf, sizeof(buf), "rf_image_stats_noalloc: launch failed: %s", cudaGetErrorString(e));
    set_last_error(buf);
    return RF_ERR_CUDA;
  }
  return RF_OK;
}
