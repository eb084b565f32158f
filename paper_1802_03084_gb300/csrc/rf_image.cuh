// rf_image.cuh -- imaging kernels of one (DM, dt, t') dirty image, Sec. 3.1:
// dedispersion + boxcar resampling + nearest-neighbour gridding + 2D inverse
// FFT + image statistics.
//
// The half-plane grid H[iv][iu] (iu = 0 .. iu_max) of an image is never
// materialised in global memory: k_grid_cells (rf_kernels.cu) writes the sums of
// its occupied cells.  Pass A (k_colfft) takes one column of them at a time, adds
// up the image's noise (Parseval) and runs the length-N inverse FFT along v;
// the result T[iu][y] goes to a global scratch, the size of a wave of images.
// Pass B (k_rowfft_stats) takes two image rows y, y+1 per transform: with Z[u] =
// T[u][y] + i T[u][y+1] on the Hermitian extension (Z[N-u] = conj T[u][y] + i conj
// T[u][y+1]), one complex inverse FFT gives row y in the real part and row y+1 in
// the imaginary part.  The maximum with its lowest index is reduced in the same
// kernel (and under the clipped noise the sums over the kept pixels); the image
// itself is written only when a caller asks for it.  k_rowfft_tree and
// k_rowfft_duo are pass B for plans with widths whose images are sums of
// another width's.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <float.h>
#include <limits.h>

#include <algorithm>
#include <cstring>
#include <type_traits>
#include <utility>

#include "rf_engine.h"
#include "rf_async.cuh"
#include "rf_fft.cuh"

namespace rf {

__host__ __device__ constexpr int cmin(int a, int b) { return a < b ? a : b; }
__host__ __device__ constexpr int cmax(int a, int b) { return a > b ? a : b; }

// Compile-time launch shape per image side N.
template <int N>
struct ImgCfg {
  static constexpr int T = FftShape<N>::T;                       // threads per transform
  static constexpr int E = FftShape<N>::E;                       // values per thread
  // pass A: 256 threads, one column; a group is up to 32 consecutive t'
  // (one lane each while gridding); column FFTs in rounds of XA transforms
  static constexpr int THREADS_A = 256;
  static constexpr int NW = THREADS_A / 32;
  static constexpr int WPC = NW;                                 // warps gridding a column
  static constexpr int B = 32;                                   // images per group
  static constexpr int XA = cmin(THREADS_A / T, B);              // transforms per round
  static constexpr int CELL_PITCH = 33;                          // cell values per cell row (32 + pad)
  static constexpr int PART_IMAGES = N >= 2048 ? 16 : 32;        // images whose cells are staged at once
  static constexpr int SMEM_A_FIXED = XA * fft_stride<N>() * 8;
  // pass B (row pass): EB values per thread, TB threads per transform, XB row
  // pairs (RB rows) per work item; the column-FFT tile of the next item is
  // prefetched while the current one is transformed.  (At 2048^2, 16 values
  // a thread and twice the warps took 48.0 ms for 35.2 a wave of 8134 images.)
  static constexpr int EB = E;
  static constexpr int TB = T;
  static constexpr int XB = cmin(256 / TB, N / 2);
  static constexpr int THREADS_B = TB * XB;
  static constexpr int RB = 2 * XB;
  static constexpr int PARTIALS = (N / 2) * (TB > 32 ? TB / 32 : 1);  // row-pass partials per image
  static constexpr int CH = XB;                                  // 16-byte chunks per tile row
  static constexpr int STRIDE = fft_stride<N>();
  // N = 2048: each row-pair transform is split by one
  // decimation-in-frequency step into two length-N/2 transforms, the even
  // and the odd pixels, one per warp of the transform (see row_zbuild)
  static constexpr int RSPLIT = N == 2048 ? 2 : 1;
  static constexpr int STRIDE_B = RSPLIT * fft_stride<N / RSPLIT>();  // float2 per row transform
  static constexpr int SMEM_B_FIXED = XB * STRIDE_B * 8;
  // N >= 1024: the row-pass tile arrives by tensor copies (TMA) whose
  // 16 CH-byte rows are swizzled by the hardware: chunk c of row u lands at
  // c ^ ((u >> SWZ_SH) & (CH - 1)) for 128-, 64- and 32-byte rows.  The same
  // pattern is used by the cp.async fallback and by every read of the tile.
  static constexpr bool TILE_TMA = N >= 1024;
  static constexpr int SWZ_SH = CH == 4 ? 1 : (CH == 2 ? 2 : 0);
  __device__ static __forceinline__ int swz(int u, int c) { return c ^ ((u >> SWZ_SH) & (CH - 1)); }
  static_assert((T <= 32 || XA <= 15) && (TB <= 32 || XB <= 15), "named barriers: at most 15 wide transforms per block");
  static_assert(FftShape<N>::P2 == fft_pass2_radix(N), "twiddle table layout and FFT passes disagree");
};

// Launch shape of the batched column pass (k_colfft) per image side N: each
// column is R = col_split(N) transforms of length L = N / R (TL threads of EL
// values each); a round runs XA columns' transforms (one image each) at once.
template <int N>
struct ColCfg {
  static constexpr int R = col_split(N);
  static constexpr int L = N / R;
  static constexpr int LOG2L = FftShape<L>::LOG2N;
  static constexpr int TL = FftShape<L>::T;
  static constexpr int EL = FftShape<L>::E;
  static constexpr int THREADS = 256;
  static constexpr int XA = cmin(THREADS / (R * TL), 32);       // images per round
  static constexpr int PI = N >= 2048 ? 16 : 32;                // images whose cells are staged at once
  static constexpr int STRIDE = fft_stride<L>();
  // FFT buffers [XA][R][STRIDE]; per cell of the busiest column: the staged
  // values (PI images), its row and (at most) one run with its R - 1 twiddles
  static constexpr int SMEM_FIXED = XA * R * STRIDE * 8;
  static constexpr int SMEM_PER_CELL = PI * 8 + 4 + 4 + (R - 1) * 8;
  // staged values per cell: one of padding for R = 1 (in the place of the row and run)
  static constexpr int CELL_PITCH = R > 1 ? PI : PI + 1;
  // the Parseval sums are reduced before the transforms, not after them
  static constexpr bool EARLY = R >= 2;
  static_assert(TL <= 32, "column sub-transforms fit one warp");
  static_assert(R <= 8, "at most eight sub-transforms per column");
  static_assert((XA * R * STRIDE * 8) % 16 == 0, "staged cells start 16-byte aligned");
};

// Tensor memory of a k_rowfft_tree block: 128 columns (two sums deep, 64
// registers each) for each set of four warps; an SM has 512.
template <int N>
struct TreeCfg {
  static constexpr int COLS = 128 * ((ImgCfg<N>::THREADS_B + 127) / 128);
  static_assert((COLS & (COLS - 1)) == 0 && COLS <= 512, "tensor-memory columns");
};

// Image row of index i of the column-FFT output (see SegmentGeom::tsplit).
__device__ __forceinline__ int t_row(int i, int tsplit, int log2l) {
  return tsplit > 1 ? ((i & ((1 << log2l) - 1)) * tsplit + (i >> log2l)) : i;
}

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }


// a times w_R^k, k < R <= 8: exact for the powers of i, the sqrt(1/2)
// constant for the odd eighths.
template <int R>
__device__ __forceinline__ float2 mul_wR(float2 a, int k) {
  const int e = k * (8 / R);  // eighths of a turn
  float2 b = a;
  if (e & 1) b = cmul(a, make_float2(RF_R2_2, RF_R2_2));  // w_8
  switch (e >> 1) {  // quarter turns
    case 1: return make_float2(-b.y, b.x);
    case 2: return make_float2(-b.x, -b.y);
    case 3: return make_float2(b.y, -b.x);
    default: return b;
  }
}

// Column pass: the first-pass inputs v[r] = Y_p[t + r TL] of sub-transform p
// (of R) of staged image kl.  A column has some 50 occupied rows of 1024, so
// its runs are sorted by the lane that takes them and then by r, and a lane
// holds a mask of its r (see DevTables::col_lane): it reads its own runs one
// after the other, and the rows that are empty cost neither a store nor a
// load.  Zeroing the sub-transform's buffer, scattering the runs into it and
// loading it took some 140 of a transform's 315 shared-memory wavefronts: column
// passes of 512^2 serving 3.64 -> 3.10 ms, 1024^2 realtime 58.5 -> 54.0, 2048^2
// batching 92.3 -> 89.2, 4096^2 stress subset 4.31 -> 4.23.
// R = 1: a run is a cell, read where it was staged.  R > 1: the lanes first put
//   Y_p[v1] = w_N^(v1 p) sum_{v2 < R} H[v1 + L v2] w_R^(v2 p)
// of every run (its cells in ascending v2, a fixed order) at the start of the
// sub-transform's own buffer.  runs[j] = (first cell << 4) | cells; cellv holds
// PI images per staged cell in rows of CELL_PITCH, for R > 1 with 16-byte chunks
// swizzled by the cell.  Only the sub-transform's lanes synchronise.
template <int N>
__device__ __forceinline__ void col_gather(float2 (&v)[ColCfg<N>::EL], float2* buf, const int* __restrict__ runs,
                                           int nruns, const float2* __restrict__ cellv, const int* __restrict__ crow,
                                           int kl, bool live, const float2* __restrict__ rtw, int t, int p, int xsub,
                                           int2 mine) {
  using C = ColCfg<N>;
  constexpr int PI = C::PI, CPC = PI / 2;
  constexpr int L = C::L, R = C::R, TL = C::TL, EL = C::EL;
  const unsigned mask = live ? (unsigned)mine.x : 0u;
  const float2* q;
  constexpr int STEP = R > 1 ? 1 : C::CELL_PITCH;
  if constexpr (R > 1) {
    if (live) {
      const int kc = kl >> 1, ko = kl & 1;
      for (int j = t; j < nruns; j += TL) {
        const int m = runs[j];
        const int c0 = m >> 4;
        float2 a = cellv[c0 * PI + 2 * (kc ^ (c0 & (CPC - 1))) + ko];
        const int n = m & 15;
        if (p > 0) a = mul_wR<R>(a, ((crow[c0] >> C::LOG2L) * p) & (R - 1));
        for (int i = 1; i < n; ++i) {
          const int c = c0 + i;
          float2 h = cellv[c * PI + 2 * (kc ^ (c & (CPC - 1))) + ko];
          if (p > 0) h = mul_wR<R>(h, ((crow[c] >> C::LOG2L) * p) & (R - 1));
          a = cadd(a, h);
        }
        if (p > 0) a = cmul(a, rtw[j * (R - 1) + p - 1]);  // w_N^(v1 p), staged per run
        buf[j] = a;
      }
    }
    static_assert(L <= C::STRIDE, "runs fit the buffer");
    fft_sync<TL>(xsub);
    q = buf + mine.y;
  } else {
    q = cellv + mine.y * STEP + kl;
  }
#pragma unroll
  for (int r = 0; r < EL; ++r) {
    v[r] = make_float2(0.f, 0.f);
    if (mask >> r & 1u) {
      v[r] = *q;
      q += STEP;
    }
  }
  if constexpr (R > 1) fft_sync<TL>(xsub);  // all runs are read before the first pass stores
}

// The length-L inverse FFT of the inputs v through `buf`
// (sub-transform xsub of the block), written to dst[0 .. L) if dst, output o at
// o ^ sw.
template <int N>
__device__ __forceinline__ void col_fft_store(float2 (&v)[ColCfg<N>::EL], float2* buf, const float2* __restrict__ twc, int t, int xsub,
                                              float2* __restrict__ dst, int sw) {
  using C = ColCfg<N>;
  constexpr int L = C::L, TL = C::TL, EL = C::EL;
  fft_inverse_from_regs<L, true>(v, buf, twc, t, xsub);  // packed style (see rf_fft.cuh)
  if (dst != nullptr) {
    constexpr int LP = FftShape<L>::LAST_P;
#pragma unroll
    for (int m = 0; m < EL / LP; ++m)
#pragma unroll
      for (int q = 0; q < LP; ++q) {
        // sw < 16, and outputs of 16 lanes or more differ from t by multiples of 16
        const int o = TL >= 16 ? fft_out_index<L>(t ^ sw, m, q) : fft_out_index<L>(t, m, q) ^ sw;
        dst[o] = v[m * LP + dft_perm<LP>(q)];
      }
  }
  fft_sync<TL>(xsub);  // the buffer is reused by the next transform
}

// Pass A2: the column FFTs of one group (up to 32 consecutive t' of a
// trial) and one half-plane column u.  The column's cell sums for the
// group's images (cellbuf row per cell, 32 images) are copied to shared
// memory with cp.async, PI images at a time.  Each column is R = col_split(N)
// sub-transforms of length L = N/R.  In rounds of XA images, each
// sub-transform takes the column's runs (col_gather), which for R > 1 folds
// in one decimation-in-frequency step: sub-transform p takes
//   Y_p[v1] = w_N^(v1 p) sum_{v2 < R} H[v1 + L v2] w_R^(v2 p),
// and its length-L inverse FFT is column output y = R k + p at k, stored at
// T[slot][u][p L + k] (see SegmentGeom::tsplit).  A sub-transform
// synchronises only its own lanes (one warp or part of one), so there is no
// third FFT pass and no barrier across warps for N >= 2048.
template <int N>
__global__ void __launch_bounds__(ColCfg<N>::THREADS, 2)
    k_colfft(SegmentGeom g, DevTables tb, const Group* __restrict__ groups, int g_begin, int img_base, int base_base,
             const float2* __restrict__ cellbuf, float2* __restrict__ Tbuf, float* __restrict__ colsq,
             float* __restrict__ mean0, int duo) {
  using C = ColCfg<N>;
  constexpr int PI = C::PI;          // images staged at a time
  constexpr int CPC = PI / 2;        // 16-byte chunks per cell row
  constexpr int L = C::L, R = C::R, TL = C::TL;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* fbuf = reinterpret_cast<float2*>(smraw);                       // [XA][R][STRIDE]
  float2* cellv = reinterpret_cast<float2*>(fbuf + C::XA * R * C::STRIDE);  // [max_cells][CELL_PITCH]
  // R > 1 only
  float2* rtw = cellv + (size_t)g.max_cells * PI;                           // [max_cells][R - 1]
  int* crow = reinterpret_cast<int*>(rtw + (size_t)g.max_cells * (R - 1));  // [max_cells]
  int* runs = crow + g.max_cells;                                           // [max_cells]
  const int tid = threadIdx.x;
  const int lane = tid & 31;
  const Group* __restrict__ gp = groups + g_begin + blockIdx.x;
  const Group gr = *gp;
  const int col = blockIdx.y;
  const int cell0 = tb.col_cell_ptr[col];
  const int ncells = tb.col_cell_ptr[col + 1] - cell0;
  const float2* __restrict__ src = cellbuf + ((size_t)blockIdx.x * g.ncells + cell0) * 32;
  // the column's cell rows and runs; visible after the first staging wait
  // and barrier below
  const int run0 = tb.col_run_ptr[col];
  const int nruns = tb.col_run_ptr[col + 1] - run0;
  if constexpr (R > 1) {
    for (int c = tid; c < ncells; c += C::THREADS) crow[c] = tb.cell_row[cell0 + c];
    for (int j = tid; j < nruns; j += C::THREADS) runs[j] = tb.col_runs[run0 + j];
    for (int i = tid; i < nruns * (R - 1); i += C::THREADS) rtw[i] = tb.col_run_tw[(size_t)run0 * (R - 1) + i];
  }
  const bool dc = col == 0 && ncells > 0 && tb.cell_row[cell0] == 0;  // row 0 sorts first
  const int xf = tid / (R * TL);          // image of the round
  const int p = (tid / TL) % R;           // sub-transform: output rows y = p mod R
  const int t = tid % TL;
  const int2 mine = tb.col_lane[(size_t)col * TL + t];
  float2* buf = fbuf + (xf * R + p) * C::STRIDE;
  const int sw = duo ? duo_swizzle(N, col) : 0;
  for (int kbase = 0; kbase < gr.nimg; kbase += PI) {
    if (kbase > 0) __syncthreads();  // the previous part's cells are consumed
    if constexpr (R > 1) {
      for (int i = tid; i < ncells * CPC; i += C::THREADS) {
        const int c = i / CPC;
        const int j = i - c * CPC;
        cp_async16(cellv + c * PI + 2 * (j ^ (c & (CPC - 1))), src + c * 32 + kbase + 2 * j);
      }
    } else {
      for (int i = tid; i < ncells * PI; i += C::THREADS) {
        const int c = i / PI;
        const int j = i - c * PI;
        cp_async8(cellv + c * C::CELL_PITCH + j, src + c * 32 + kbase + j);
      }
    }
    cp_async_commit();
    cp_async_wait_all();
    __syncthreads();  // also orders the row map before its first use
    const int nk = min(PI, gr.nimg - kbase);

    // Parseval: the image's sum of squares is N^2 / (4 W^2) times the sum
    // of |G|^2 over the full Hermitian plane, which counts this column
    // twice unless u = 0; its mean is G(0, 0) / (2 W).  Lane k is image k of
    // the part (two cells a step where the part is 16 images), so the cells of
    // a sum of 2, 4, 8 or 16 images are xor-shuffles away.  FP32: a lane adds
    // every 32nd cell, in U chains that take turns, and the chains and the
    // warps' sums, which meet in the first FFT buffer, are added as a tree:
    // after the transforms, so that no barrier stands before those, unless the
    // sums' registers would spill there (C::EARLY).
    constexpr int NL = N < kTreeMinNpix ? 0 : (pairs_possible(N) ? 4 : 2);
    constexpr int NW = C::THREADS / 32, CPS = 32 / PI, U = 32 / (NW * CPS);
    const int warp = tid >> 5, kp = lane & (PI - 1);
    auto at = [&](int c, int k) {
      return R > 1 ? c * PI + 2 * ((k >> 1) ^ (c & (CPC - 1))) + (k & 1) : c * C::CELL_PITCH + k;
    };
    float a[NL + 1] = {};
    int top = 0;
    {
      float ac[U][NL + 1] = {};
#pragma unroll
      for (int lv = 1; lv <= NL; ++lv)
        if (gp->nsum[lv - 1] > 0) top = lv;
      for (int cb = warp * CPS; cb < ncells; cb += U * NW * CPS)
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (cb + u * NW * CPS >= ncells) break;
          const int c = cb + u * NW * CPS + lane / PI;
          float2 h = make_float2(0.f, 0.f);
          if (c < ncells && kp < nk) h = cellv[at(c, kp)];
          ac[u][0] = fmaf(h.x, h.x, fmaf(h.y, h.y, ac[u][0]));
#pragma unroll
          for (int lv = 1; lv <= NL; ++lv)
            if (lv <= top) {
              h.x += __shfl_xor_sync(0xffffffffu, h.x, 1 << (lv - 1));
              h.y += __shfl_xor_sync(0xffffffffu, h.y, 1 << (lv - 1));
              ac[u][lv] = fmaf(h.x, h.x, fmaf(h.y, h.y, ac[u][lv]));
            }
        }
#pragma unroll
      for (int lv = 0; lv <= NL; ++lv) {
        a[lv] = ac[0][lv] + ac[1][lv];
        if constexpr (U == 4) a[lv] += ac[2][lv] + ac[3][lv];
      }
      static_assert(NW == 8 && (U == 2 || U == 4), "the trees");
      static_assert(CPS <= 2 && (1 << NL) <= PI && NL < NW && NW * (NL + 1) * 32 * 4 <= C::SMEM_FIXED,
                    "Parseval sums fit the FFT buffers, the sums' images one part, their levels the warps");
    }

    auto reduce = [&] {
      float* red = reinterpret_cast<float*>(fbuf);  // [level][warp][32]
#pragma unroll
      for (int lv = 0; lv <= NL; ++lv)
        if (lv <= top) {
          if constexpr (CPS == 2) a[lv] += __shfl_xor_sync(0xffffffffu, a[lv], 16);
          red[(lv * NW + warp) * 32 + lane] = a[lv];
        }
      __syncthreads();
      const int lv = warp;  // warp 0: single images, warp lv: sums of 2^lv
      if (lv <= top && lane < PI) {
        const int k = kbase + lane, j = k >> lv;
        const int lim = lv == 0 ? gr.nimg : gp->nsum[lv - 1];
        if ((lane & ((1 << lv) - 1)) == 0 && j < lim) {
          const float* __restrict__ rw = red + lv * NW * 32 + lane;
          const float acc = ((rw[0] + rw[32]) + (rw[64] + rw[96])) + ((rw[128] + rw[160]) + (rw[192] + rw[224]));
          const size_t slot = (size_t)((lv == 0 ? gr.img0 : gp->isum[lv - 1]) + j - img_base);
          colsq[slot * g.ncol + col] = (col == 0 ? 1.f : 2.f) * acc;
          if (col == 0) {
            float m = 0.f;
            if (dc)
              for (int i = 0; i < 1 << lv; ++i) m += cellv[at(0, lane + i)].x;
            mean0[slot] = m;
          }
        }
      }
    };
    if constexpr (C::EARLY) {
      reduce();
      __syncthreads();  // the FFT buffers are free again
    }

    if (xf < C::XA) {
      const int nrounds = (nk + C::XA - 1) / C::XA;
      for (int rd = 0; rd < nrounds; ++rd) {
        const int kl = rd * C::XA + xf;
        const bool live = kl < nk;
        float2* dst = live ? Tbuf + ((size_t)(gr.base0 + kbase + kl - base_base) * g.ncol + col) * N + p * L : nullptr;
        float2 v[C::EL];
        col_gather<N>(v, buf, runs, nruns, cellv, crow, kl, live, rtw, t, p, xf * R + p, mine);
        col_fft_store<N>(v, buf, tb.twiddle_col, t, xf * R + p, dst, sw);
      }
    }

    if constexpr (!C::EARLY) {
      __syncthreads();  // the FFT buffers are free
      reduce();
    }
  }
}

// Maximum and minimum over aligned groups of W lanes (every lane has its
// group's): one reduction instruction over a whole warp.
template <int W>
__device__ __forceinline__ float warp_max(float v) {
  if constexpr (W == 32) {
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
  } else {
#pragma unroll
    for (int off = W / 2; off > 0; off >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, off));
    return v;
  }
}
template <int W>
__device__ __forceinline__ int warp_min(int v) {
  if constexpr (W == 32) {
    return __reduce_min_sync(0xffffffffu, v);
  } else {
#pragma unroll
    for (int off = W / 2; off > 0; off >>= 1) v = min(v, __shfl_xor_sync(0xffffffffu, v, off));
    return v;
  }
}

__device__ __forceinline__ void max_merge(float& m, int& i, float m2, int i2) {
  if (m2 > m || (m2 == m && i2 < i)) {
    m = m2;
    i = i2;
  }
}

// Row pass: the first-pass inputs of row pair xf of the item whose tile
// (T rows y0 .. y0 + RB of every imaged column u, swizzled 16-byte chunks)
// is in shared memory.
template <int N>
__device__ __forceinline__ void row_zbuild(float2 (&v)[ImgCfg<N>::EB], const float4* __restrict__ tile, int t,
                                           int xf, int ncol) {
  using K = ImgCfg<N>;
  constexpr int EB = K::EB, TB = K::TB;
  // first-pass inputs Z[u], u = t + r T: a + i b for 0 < u < ncol, the
  // Hermitian mirror conj(a) + i conj(b) for N - u < ncol, real parts at
  // u = 0, zero elsewhere (columns beyond iu_max are empty).  N/2 = (EB/2) TB,
  // so r < EB/2 can only be a direct column and r >= EB/2 only a mirror.
  if constexpr (K::RSPLIT == 2) {
    // split transform: pixel x = 2 k + s is output k of the length-H = N/2
    // inverse DFT of Y_s[u'] = (Z[u'] + (-1)^s Z[u' + H]) exp(+2 pi i u' s / N)
    // (one decimation-in-frequency step).  Warp s of the transform builds
    // Y_s at u' = j + 32 r (lane j, r < 32): Z[u'] is a direct column or
    // zero, Z[u' + H] the mirror of column H - u' or zero.  For s = 1 the
    // factor exp(+2 pi i r / 64) of u' is applied here and exp(+2 pi i j / N)
    // rides on the second-pass twiddles (see row_fft).
    constexpr int H = N / 2;
    static_assert(EB == 32 && TB == 64 && 32 % (K::CH << K::SWZ_SH) == 0, "split row transform layout");
    const int s = t >> 5, j = t & 31;
    const int rd_end = ncol > j ? (ncol - j + 31) / 32 : 0;  // j + 32 r < ncol
    const int xm = H - j - ncol;                              // H - j - 32 r < ncol  <=>  32 r > xm
    const int rm_beg = xm < 0 ? 0 : xm / 32 + 1;
    // the swizzle term of u = j + 32 r (H - j - 32 r) is that of j (H - j)
    const float4* pd = tile + j * K::CH + K::swz(j, xf);
    const float4* pm = tile + (size_t)(H - j) * K::CH + K::swz(H - j, xf);
    // with a = T[u'][y] = (ab.x, ab.y) and b = T[u'][y+1] = (ab.z, ab.w) of
    // the direct column u', and c, d the same of the mirror column H - u':
    //   Z[u'] +- Z[u' + H] = (P.x - Q.y, P.y + Q.x),
    //   P = a +- conj(c), Q = b +- conj(d)  (one packed FMA each)
    // except at u' = 0, where Z[0] takes the real parts (a.x, b.x)
    const float2 pm1 = make_float2(s == 0 ? 1.f : -1.f, s == 0 ? -1.f : 1.f);
#pragma unroll
    for (int r = 0; r < 32; ++r) {
      float4 ab = make_float4(0.f, 0.f, 0.f, 0.f), cd = make_float4(0.f, 0.f, 0.f, 0.f);
      if (r < rd_end) ab = pd[r * 32 * K::CH];
      if (r >= rm_beg) cd = pm[-r * 32 * K::CH];
      const float2 P = f2_fma(make_float2(cd.x, cd.y), pm1, make_float2(ab.x, ab.y));
      const float2 Q = f2_fma(make_float2(cd.z, cd.w), pm1, make_float2(ab.z, ab.w));
      float2 d = make_float2(P.x - Q.y, P.y + Q.x);
      if (r == 0 && j == 0) {
        const float sg = s == 0 ? 1.f : -1.f;
        d = make_float2(fmaf(sg, cd.x + cd.w, ab.x), fmaf(sg, cd.z - cd.y, ab.z));
      }
      if (s != 0 && r > 0) d = r == 16 ? cmul_i(d) : cmul_c<false>(d, cos_r64(r), sin_r64(r));
      v[r] = d;
    }
  } else if constexpr (TB % (K::CH << K::SWZ_SH) == 0) {
    // the swizzle term of u = t + r T (or N - t - r T) is that of t (N - t)
    const int rd_end = ncol > t ? (ncol - t + TB - 1) / TB : 0;
    const int rm_beg = (N - ncol - t) / TB + 1;
    const float4* pd = tile + t * K::CH + K::swz(t, xf);
    const float4* pm = tile + (size_t)(N - t) * K::CH + K::swz(N - t, xf);
#pragma unroll
    for (int r = 0; r < EB / 2; ++r) {
      float4 ab = make_float4(0.f, 0.f, 0.f, 0.f);
      if (r < rd_end) ab = pd[r * TB * K::CH];
      v[r] = (r == 0 && t == 0) ? make_float2(ab.x, ab.z) : make_float2(ab.x - ab.w, ab.y + ab.z);
    }
#pragma unroll
    for (int r = EB / 2; r < EB; ++r) {
      float4 ab = make_float4(0.f, 0.f, 0.f, 0.f);
      if (r >= rm_beg) ab = pm[-r * TB * K::CH];
      v[r] = make_float2(ab.x + ab.w, ab.z - ab.y);
    }
  } else {
#pragma unroll
    for (int r = 0; r < EB; ++r) {
      const int u = t + r * TB;
      float2 z = make_float2(0.f, 0.f);
      if (u < ncol) {
        const float4 ab = tile[u * K::CH + K::swz(u, xf)];
        z = (u == 0) ? make_float2(ab.x, ab.z) : make_float2(ab.x - ab.w, ab.y + ab.z);
      } else if (N - u < ncol) {
        const int uu = N - u;
        const float4 ab = tile[uu * K::CH + K::swz(uu, xf)];
        z = make_float2(ab.x + ab.w, ab.z - ab.y);
      }
      v[r] = z;
    }
  }
}

// Row pass, after row_zbuild: the inverse FFT of the row pair in `buf`.
template <int N>
__device__ __forceinline__ void row_fft(float2 (&v)[ImgCfg<N>::EB], float2* buf, const float2* __restrict__ tw, int t,
                                        int xf) {
  using K = ImgCfg<N>;
  constexpr int EB = K::EB;
  constexpr int H = N / K::RSPLIT;  // transform length per warp group
  // split transform (see row_zbuild): warp s runs the length-H transform of
  // Y_s in its own buffer; its second pass takes the pair table of
  // exp(+2 pi i k r / H) (s = 0, the table's section at N) or of
  // exp(+2 pi i r (2k + 1) / N) (s = 1, at N + H), so it is given the
  // table base tw + H + s H (the transform reads only its pair table)
  if constexpr (K::RSPLIT == 2) {
    const int s = t >> 5;
    fft_inverse_from_regs<H, false, EB>(v, buf + s * fft_stride<H>(), tw + H + s * H, t & 31, xf);
  } else {
    fft_inverse_from_regs<N, false, EB>(v, buf, tw, t, xf);
  }
}

// Pixel of output register (m, q) of thread t after row_fft: output o of the
// transform, or of sub-transform s as pixel 2 o + s.
template <int N>
__device__ __forceinline__ int row_pix(int t, int m, int q) {
  using K = ImgCfg<N>;
  if constexpr (K::RSPLIT == 2) return 2 * fft_out_index<N / 2, K::EB>(t & 31, m, q) + (t >> 5);
  else return fft_out_index<N, K::EB>(t, m, q);
}

// The two image rows (scaled) of a row pair whose pixels are in v.
template <int N>
__device__ __forceinline__ void row_write(const float2 (&v)[ImgCfg<N>::EB], int t, int xf, int slot, int y0, int tsplit,
                                          int log2l, double W, float* __restrict__ images) {
  using K = ImgCfg<N>;
  constexpr int LP = FftShape<N / K::RSPLIT, K::EB>::LAST_P;
  const float scale = W > 0.0 ? (float)(0.5 / W) : 0.f;
  float* ima = images + ((size_t)slot * N + t_row(y0 + 2 * xf, tsplit, log2l)) * N;
  float* imb = images + ((size_t)slot * N + t_row(y0 + 2 * xf + 1, tsplit, log2l)) * N;
#pragma unroll
  for (int m = 0; m < K::EB / LP; ++m)
#pragma unroll
    for (int q = 0; q < LP; ++q) {
      const float2 z = v[m * LP + dft_perm<LP>(q)];
      const int o = row_pix<N>(t, m, q);
      ima[o] = z.x * scale;
      imb[o] = z.y * scale;
    }
}

// What a row pass keeps of an image (see PassStats).
enum RowMode { kBest, kParts, kClip };

// An image row's (or row pair's) maximum into the image's best, called where
// some lane's maximum lmax is not below the gate (all lanes call; groups of WL
// lanes share an image row): where the group's maximum beats what the image
// has, a lane that holds it finds its lowest index and offers it.  Nearly every
// image of a segment is noise and never gets here.
template <int WL, class Find>
__device__ __forceinline__ void row_best(float lmax, float gate, unsigned long long* __restrict__ best, Find find) {
  const float wmax = warp_max<WL>(lmax);
  if (lmax == wmax && !(lmax < gate)) {
    unsigned long long have;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(have) : "l"(best) : "memory");
    if (best_order(lmax) >= (unsigned)(have >> 32)) atomicMax(best, best_key(lmax, find(lmax)));
  }
}

// Kept-pixel sums of the clipped noise: deviations d from cw.x of the lane's
// values with |d| <= cw.y.
struct KeptSums {
  float s = 0.f, q = 0.f;
  int n = 0;
  __device__ __forceinline__ void add(float v, float2 cw) {
    const float d = v - cw.x;
    if (fabsf(d) <= cw.y) {
      s += d;
      q = fmaf(d, d, q);
      ++n;
    }
  }
};
template <int WL>
__device__ __forceinline__ ClipPartial kept_reduce(const KeptSums& a, const KeptSums& b) {
  float s = a.s + b.s, q = a.q + b.q;
  int n = a.n + b.n;
#pragma unroll
  for (int off = WL / 2; off > 0; off >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, off);
    q += __shfl_xor_sync(0xffffffffu, q, off);
    n += __shfl_xor_sync(0xffffffffu, n, off);
  }
  return ClipPartial{s, q, n, 0};
}

// Statistics of the row pair (T rows i = y0 + 2 xf and i + 1, image rows t_row
// of them) of the image in `slot` whose pixels are in v: the pair's max pixel
// with its lowest index (and under kClip the kept-pixel sums), one StatPartial
// per warp of the transform; under kBest only the image's best.  Finding the
// index and writing a partial cost as much as the maximum itself, and this
// kernel is bound by instruction issue: leaving them out
// (kBest against kParts with the index gated) took the 1024^2 realtime row
// passes from 85.0 to 75.2 ms, 2048^2 batching from 186 to 147, 4096^2 stress
// subset from 8.01 to 7.60.
template <int N, RowMode M>
__device__ __forceinline__ void row_stats(const float2 (&v)[ImgCfg<N>::EB], int t, int xf, int slot, int y0,
                                          int tsplit, int log2l, float gate, const PassStats& ps) {
  using K = ImgCfg<N>;
  constexpr int EB = K::EB, TB = K::TB;
  constexpr int H = N / K::RSPLIT;
  // the noise comes from the grid by Parseval's identity, see k_colfft.  The
  // pair is T rows i, i + 1, image rows ya < yb (adjacent unless the
  // column pass split its transforms: then R apart)
  const int i = y0 + 2 * xf;
  constexpr int LP = FftShape<H, EB>::LAST_P;
  constexpr int EM = EB / LP;
  // max of row y (real parts) and of row y + 1 (imaginary parts), four
  // independent chains each
  float mxa[4] = {-FLT_MAX, -FLT_MAX, -FLT_MAX, -FLT_MAX};
  float mya[4] = {-FLT_MAX, -FLT_MAX, -FLT_MAX, -FLT_MAX};
#pragma unroll
  for (int e = 0; e < EB; e += 2) {
    mxa[(e >> 1) & 3] = fmax3f(mxa[(e >> 1) & 3], v[e].x, v[e + 1].x);
    mya[(e >> 1) & 3] = fmax3f(mya[(e >> 1) & 3], v[e].y, v[e + 1].y);
  }
  const float mx = fmaxf(fmaxf(mxa[0], mxa[1]), fmaxf(mxa[2], mxa[3]));
  const float my = fmaxf(fmaxf(mya[0], mya[1]), fmaxf(mya[2], mya[3]));
  const float lmax = fmaxf(mx, my);
  // the lowest index of the lane's pixels equal to `top`: row ya comes before
  // row yb, and within a row the lane's outputs ascend with (q, m)
  auto find = [&](float top) {
    int best = INT_MAX;
    if (mx == top) {
#pragma unroll
      for (int q = 0; q < LP; ++q)
#pragma unroll
        for (int m = 0; m < EM; ++m)
          if (v[m * LP + dft_perm<LP>(q)].x == top) {
            best = t_row(i, tsplit, log2l) * N + row_pix<N>(t, m, q);
            goto found;
          }
    } else {
#pragma unroll
      for (int q = 0; q < LP; ++q)
#pragma unroll
        for (int m = 0; m < EM; ++m)
          if (v[m * LP + dft_perm<LP>(q)].y == top) {
            best = t_row(i + 1, tsplit, log2l) * N + row_pix<N>(t, m, q);
            goto found;
          }
    }
  found:
    return best;
  };
  constexpr int WL = TB < 32 ? TB : 32;
  if constexpr (M == kBest) {
    if (__any_sync(0xffffffffu, !(lmax < gate))) row_best<WL>(lmax, gate, ps.best + slot, find);
    return;
  }
  // reduce over the transform's T threads (a warp, a part of one, or several
  // warps, one partial each, which the finalisation combines: no barrier)
  const float wmax = warp_max<WL>(lmax);
  int best = INT_MAX;
  if (lmax == wmax) best = find(wmax);
  best = warp_min<WL>(best);
  ClipPartial cp{};
  if constexpr (M == kClip) {
    const float2 cw = ps.clip[slot];
    KeptSums a, b;  // rows y and y + 1 in separate chains
#pragma unroll
    for (int e = 0; e < EB; ++e) {
      a.add(v[e].x, cw);
      b.add(v[e].y, cw);
    }
    cp = kept_reduce<WL>(a, b);
  }
  if ((t & 31) == 0) {
    constexpr int WPT = TB > 32 ? TB / 32 : 1;
    const size_t o = (size_t)slot * K::PARTIALS + ((y0 >> 1) + xf) * WPT + (t >> 5);  // by T row pair
    ps.partials[o] = StatPartial{wmax, best};
    if constexpr (M == kClip) ps.cparts[o] = cp;
  }
}

// Pass B: work item = (image slot, block of RB rows); each pair of rows
// shares one complex inverse FFT.  Blocks loop over items; the column-FFT
// tile T[slot][u][y0 .. y0+RB) of the next item is copied to shared memory
// with cp.async (16-byte chunks, XOR-swizzled per row so the strided reads
// are free of bank conflicts) while the current item is transformed.  Each
// warp of a row pair's transform writes one StatPartial (one per row pair
// when the transform fits a warp, T/32 of them when it spans several): the
// max pixel of its part of the two rows with its lowest index, and under
// kClip the kept-pixel sums (FP32 per thread and across the warp's lanes; the
// finalisation combines an image's partials in FP64).
// With tma_boxes > 0 (N >= 1024 only) thread 0 fetches each item's tile with
// tma_boxes tensor copies of tma_rows u rows from `tmap` ([slot][u][2N
// floats]) and every thread waits on an mbarrier; a wait that gives up sets
// *err, waits once more (bounded) for the copy in flight, and the block
// returns.  Otherwise the threads copy it with cp.async.
// kClip (the one-pass clipped noise): clip[slot] = {mean0, r} in raw pixel
// units, and each row pair also sums d = J - mean0 and d^2 over its pixels J
// with |d| <= r and counts them (FP32 per thread and across the transform's
// threads in a fixed order).
template <int N, RowMode M>
__global__ void __launch_bounds__(ImgCfg<N>::THREADS_B, 2)
    k_rowfft_stats(SegmentGeom g, DevTables tb, const float2* __restrict__ Tbuf, int nimg, int img_base,
                   const double* __restrict__ weight, const PassStats ps, float* __restrict__ images,
                   const __grid_constant__ CUtensorMap tmap, int tma_boxes, int tma_rows, int* __restrict__ err) {
  using K = ImgCfg<N>;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* fbuf = reinterpret_cast<float2*>(smraw);  // [XB][STRIDE_B]
  unsigned char* tb0 = smraw + K::XB * K::STRIDE_B * 8;
  if constexpr (K::TILE_TMA) tb0 += (1024u - (smem_u32(tb0) & 1023u)) & 1023u;  // swizzle atom alignment
  float4* tile = reinterpret_cast<float4*>(tb0);    // [rows][CH]
  __shared__ __align__(8) unsigned long long tbar;
  __shared__ int s_done;  // warps done reading the tile in hand (warp-local transforms)
  const int tid = threadIdx.x;
  const int ncol = g.ncol;
  constexpr int nrb = N / K::RB;
  const int nitems = nimg * nrb;
  const int xf = tid / K::TB;
  const int t = tid - xf * K::TB;
  const int log2l = FftShape<N>::LOG2N - (g.tsplit > 1 ? __ffs(g.tsplit) - 1 : 0);
  const bool use_tma = K::TILE_TMA && tma_boxes > 0;
  // With tensor copies and transforms that synchronise only within a warp,
  // the warps of a block do not wait for one another: each waits for the
  // tile on its own, and the last warp to finish reading it issues the next
  // item's copy.  Otherwise two block barriers per item.
  constexpr bool WARP_LOCAL = K::TILE_TMA && (K::TB <= 32 || K::RSPLIT == 2);
  constexpr int NWB = K::THREADS_B / 32;
  unsigned phase = 0;
  if (use_tma) {
    if (tid == 0) {
      mbar_init(&tbar, 1);
      s_done = 0;
    }
    __syncthreads();
  }
  auto issue_tma = [&](int it) {  // by one thread
    const int sl = it / nrb;
    const int yb = (it - sl * nrb) * K::RB;
    mbar_expect_tx(&tbar, (unsigned)(tma_boxes * tma_rows * K::CH * 16));
    for (int b = 0; b < tma_boxes; ++b)
      tma_load_3d(tile + (size_t)b * tma_rows * K::CH, &tmap, 2 * yb, b * tma_rows, sl, &tbar);
  };
  auto fetch = [&](int it) {
    const int sl = it / nrb;
    const int yb = (it - sl * nrb) * K::RB;
    if (use_tma) {
      if (tid == 0) issue_tma(it);
    } else {
      const float2* src = Tbuf + (size_t)sl * ncol * N + yb;
      for (int i = tid; i < ncol * K::CH; i += K::THREADS_B) {
        const int u = i / K::CH;
        const int c = i - u * K::CH;
        cp_async16(tile + u * K::CH + K::swz(u, c), src + (size_t)u * N + 2 * c);
      }
      cp_async_commit();
    }
  };

  int item = blockIdx.x;
  if (item < nitems) fetch(item);
  for (; item < nitems; item += gridDim.x) {
    if (use_tma && WARP_LOCAL) {
      // a warp whose bounded wait gives up reports it, waits once more (so
      // that a late copy does not land after the block has left) and leaves;
      // no later copy is issued without its arrival below, so the other
      // warps' waits run out in turn
      if (!__all_sync(0xffffffffu, mbar_wait(&tbar, phase))) {
        if ((tid & 31) == 0) atomicExch(err, 1);
        mbar_wait(&tbar, phase);
        return;
      }
      phase ^= 1u;
    } else if (use_tma) {
      const bool ok = mbar_wait(&tbar, phase);
      if (__syncthreads_or(!ok)) {
        // the item's tile copy has not completed: give it one more bounded
        // wait, so that it does not land in shared memory after the block
        // has left, then report the timeout and leave
        if (tid == 0) {
          atomicExch(err, 1);
          mbar_wait(&tbar, phase);
        }
        __syncthreads();
        return;
      }
      phase ^= 1u;
    } else {
      cp_async_wait_all();
      __syncthreads();
    }
    const int slot = item / nrb;
    const int y0 = (item - slot * nrb) * K::RB;
    const float gate = M == kBest ? ps.gate[slot] : 0.f;
    float2 v[K::EB];
    row_zbuild<N>(v, tile, t, xf, ncol);
    if (use_tma && WARP_LOCAL) {
      // tile consumed by this warp; the last of the block's warps resets the
      // count and issues the next item's copy (no warp waits for the tile
      // of item + 2 grid strides before every warp has read item + 1's)
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if ((tid & 31) == 0) {
        __threadfence_block();
        if (atomicAdd(&s_done, 1) == NWB - 1) {
          s_done = 0;
          __threadfence_block();
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          if (item + (int)gridDim.x < nitems) issue_tma(item + gridDim.x);
        }
      }
    } else {
      __syncthreads();  // tile consumed: prefetch the next item
      if (item + (int)gridDim.x < nitems) fetch(item + gridDim.x);
    }
    row_fft<N>(v, fbuf + xf * K::STRIDE_B, tb.twiddle, t, xf);
    if (images != nullptr) row_write<N>(v, t, xf, slot, y0, g.tsplit, log2l, weight[img_base + slot], images);
    row_stats<N, M>(v, t, xf, slot, y0, g.tsplit, log2l, gate, ps);
  }
}

// Pass B over units of up to four transformed images (quads), with the images
// derived from them (sums of two and four): work item = (quad, block of RB rows).  A block takes the quad's images one
// after the other through the transform of k_rowfft_stats.  The pixel rows of
// image k stay with the lane that made them: an even image's are kept, an odd
// one's added to them, which is the row pair of the sum of two images (the
// image of twice the width), and the sums of two make the sum of four in the
// same way.  Every searched one of these images gets its StatPartial here, so
// the widths 2 dt and 4 dt cost no gridding, no column pass and no row
// transform, only additions and the maxima.
// What is kept (64 registers a lane, twice) has no room in registers (the
// transform takes 128, two blocks per SM) or in shared memory (113 KB a block
// are FFT buffers and tile): it goes to tensor memory, which nothing else
// uses here and whose loads and stores do not pass through the L1/shared
// pipe that bounds this kernel.  Two sums deep is what 512 columns hold for 16
// warps (128 columns a warp, four warps on each quarter of the lanes), hence
// quads.
// Measured on whole segments: 177,521 images of 1024^2 (widths 1, 2, 4, 8: six
// in ten transformed) 266.8 to 171.5 ms, 69,139 of 2048^2 (widths 1 .. 16)
// 521.6 to 308.9 ms, 504 of 4096^2 (widths 1 .. 32) 23.2 to 14.1 ms.  Of the
// 1024^2 row passes' 91 ms, keeping and adding take 3 and the sums' maxima 9.
// A block that gives up a bounded wait leaves the item loop and frees its
// tensor memory with the others.
template <int N, RowMode M>
__global__ void __launch_bounds__(ImgCfg<N>::THREADS_B, 2)
    k_rowfft_tree(SegmentGeom g, DevTables tb, const float2* __restrict__ Tbuf, const Unit* __restrict__ units,
                  int nunits, int img_base, int base_base, const PassStats ps,
                  const __grid_constant__ CUtensorMap tmap, int tma_boxes, int tma_rows, int* __restrict__ err) {
  using K = ImgCfg<N>;
  static_assert(K::EB == 32 && K::THREADS_B % 32 == 0, "64 values a lane, whole warps");
  constexpr int NWB = K::THREADS_B / 32;
  constexpr unsigned TCOLS = TreeCfg<N>::COLS;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* fbuf = reinterpret_cast<float2*>(smraw);  // [XB][STRIDE_B]
  unsigned char* tb0 = smraw + K::XB * K::STRIDE_B * 8;
  if constexpr (K::TILE_TMA) tb0 += (1024u - (smem_u32(tb0) & 1023u)) & 1023u;  // swizzle atom alignment
  float4* tile = reinterpret_cast<float4*>(tb0);    // [rows][CH]
  __shared__ __align__(8) unsigned long long tbar;
  __shared__ int s_done;  // warps done reading the tile in hand (warp-local transforms)
  __shared__ unsigned s_tmem;
  const int tid = threadIdx.x;
  const int ncol = g.ncol;
  constexpr int nrb = N / K::RB;
  const int nitems = nunits * nrb;
  const int xf = tid / K::TB;
  const int t = tid - xf * K::TB;
  const int log2l = FftShape<N>::LOG2N - (g.tsplit > 1 ? __ffs(g.tsplit) - 1 : 0);
  const bool use_tma = K::TILE_TMA && tma_boxes > 0;
  constexpr bool WARP_LOCAL = K::TILE_TMA && (K::TB <= 32 || K::RSPLIT == 2);  // see k_rowfft_stats
  unsigned phase = 0;
  if (tid < 32) tmem_alloc(&s_tmem, TCOLS);
  if (tid == 0) {
    mbar_init(&tbar, 1);
    s_done = 0;
  }
  __syncthreads();
  // this warp's lanes and columns: level 0 (single images) and 1 (sums of two)
  const unsigned keep = s_tmem + ((unsigned)((tid >> 5) & 3) << 21) + (unsigned)(tid >> 7) * 128u;
  auto issue_tma = [&](int sl, int yb) {  // by one thread
    mbar_expect_tx(&tbar, (unsigned)(tma_boxes * tma_rows * K::CH * 16));
    for (int b = 0; b < tma_boxes; ++b)
      tma_load_3d(tile + (size_t)b * tma_rows * K::CH, &tmap, 2 * yb, b * tma_rows, sl, &tbar);
  };
  auto fetch = [&](int sl, int yb) {
    if (use_tma) {
      if (tid == 0) issue_tma(sl, yb);
    } else {
      const float2* src = Tbuf + (size_t)sl * ncol * N + yb;
      for (int i = tid; i < ncol * K::CH; i += K::THREADS_B) {
        const int u = i / K::CH;
        const int c = i - u * K::CH;
        cp_async16(tile + u * K::CH + K::swz(u, c), src + (size_t)u * N + 2 * c);
      }
      cp_async_commit();
    }
  };

  int item = blockIdx.x;
  Unit cur = units[item / nrb];  // the grid is at most the number of items
  bool failed = false;
  fetch(cur.base - base_base, (item % nrb) * K::RB);
  while (item < nitems && !failed) {
    const int y0 = (item % nrb) * K::RB;
    const int next = item + (int)gridDim.x;
    Unit nxt = cur;
    if (next < nitems) nxt = units[next / nrb];
    const int top = cur.img[2] >= 0 ? 2 : (cur.img[1] >= 0 ? 1 : 0);
    // lanes 0 .. 3 hold the gates of the quad's images, 4 and 5 those of the
    // sums of two, 6 that of the sum of four
    float gates = 0.f;
    if (M == kBest) {
      const int lane = tid & 31;
      int sl = lane < cur.n ? cur.img[0] + lane : -1;
      if (lane >= 4) sl = lane < 6 && cur.img[1] >= 0 && 2 * (lane - 4) + 1 < cur.n ? cur.img[1] + lane - 4 : -1;
      if (lane == 6) sl = cur.img[2];
      if (sl >= 0) gates = ps.gate[sl - img_base];
    }
    for (int k = 0; k < cur.n; ++k) {
      if (use_tma && WARP_LOCAL) {
        // as in k_rowfft_stats: no copy is issued without this warp's count
        // below, so the other warps' waits run out in turn
        if (!__all_sync(0xffffffffu, mbar_wait(&tbar, phase))) {
          if ((tid & 31) == 0) atomicExch(err, 1);
          mbar_wait(&tbar, phase);
          failed = true;
          break;
        }
        phase ^= 1u;
      } else if (use_tma) {
        const bool ok = mbar_wait(&tbar, phase);
        if (__syncthreads_or(!ok)) {
          if (tid == 0) {
            atomicExch(err, 1);
            mbar_wait(&tbar, phase);
          }
          failed = true;
          break;
        }
        phase ^= 1u;
      } else {
        cp_async_wait_all();
        __syncthreads();
      }
      float2 v[K::EB];
      row_zbuild<N>(v, tile, t, xf, ncol);
      // the tile is read: the next image's (or the next item's first one's)
      const bool more = k + 1 < cur.n || next < nitems;
      const int nsl = (k + 1 < cur.n ? cur.base + k + 1 : nxt.base) - base_base;
      const int nyb = k + 1 < cur.n ? y0 : (next % nrb) * K::RB;
      if (use_tma && WARP_LOCAL) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if ((tid & 31) == 0) {
          __threadfence_block();
          if (atomicAdd(&s_done, 1) == NWB - 1) {
            s_done = 0;
            __threadfence_block();
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            if (more) issue_tma(nsl, nyb);
          }
        }
      } else {
        __syncthreads();
        if (more) fetch(nsl, nyb);
      }
      row_fft<N>(v, fbuf + xf * K::STRIDE_B, tb.twiddle, t, xf);
      int slot = cur.img[0] + k - img_base;
#pragma unroll 1
      for (int lv = 0;;) {
        const float gate = __shfl_sync(0xffffffffu, gates, lv == 0 ? k : (lv == 1 ? 4 + (k >> 1) : 6));
        if (slot >= 0) row_stats<N, M>(v, t, xf, slot, y0, g.tsplit, log2l, gate, ps);
        // level lv's block of images that ends the next level's must be whole
        if (lv >= top || (k | ((2 << lv) - 1)) >= cur.n) break;
        __syncwarp();
        if (((k >> lv) & 1) == 0) {
          tmem_store16(keep + lv * 64, v);
          tmem_store16(keep + lv * 64 + 32, v + 16);
          break;
        }
        tmem_add16(keep + lv * 64, v);
        tmem_add16(keep + lv * 64 + 32, v + 16);
        ++lv;
        const int first = lv == 1 ? cur.img[1] : cur.img[2];
        slot = first < 0 ? -1 : first + (lv == 1 ? k >> 1 : 0) - img_base;
      }
    }
    item = next;
    cur = nxt;
  }
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
  __syncthreads();
  if (tid < 32) tmem_free(s_tmem, TCOLS);
}

// Row pass of image pairs, the first-pass inputs of image row xf of the item:
// Z[u] = T_A[u] + i T_B[u] of two images' tiles, Hermitian-extended as in
// row_zbuild with the images in the place of the rows.
// Tiles are [u][XB] complex values, row r of column u at r ^ duo_swizzle(N, u),
// the same for all columns a lane reads directly and for all it mirrors.
template <int N>
__device__ __forceinline__ void row_zbuild_duo(float2 (&v)[ImgCfg<N>::EB], const float2* __restrict__ tileA,
                                               const float2* __restrict__ tileB, int t, int xf, int ncol) {
  using K = ImgCfg<N>;
  constexpr int EB = K::EB, TB = K::TB, XB = K::XB;
  const float2 zero = make_float2(0.f, 0.f);
  if constexpr (K::RSPLIT == 2) {  // see row_zbuild
    constexpr int H = N / 2;
    static_assert(EB == 32 && TB == 64 && duo_swizzle(N, 32) == 0, "split row transform layout");
    const int s = t >> 5, j = t & 31;
    const int rd_end = ncol > j ? (ncol - j + 31) / 32 : 0;
    const int xm = H - j - ncol;
    const int rm_beg = xm < 0 ? 0 : xm / 32 + 1;
    const int od = j * XB + (xf ^ duo_swizzle(N, j)), om = (H - j) * XB + (xf ^ duo_swizzle(N, H - j));
    const float2 pm1 = make_float2(s == 0 ? 1.f : -1.f, s == 0 ? -1.f : 1.f);
#pragma unroll
    for (int r = 0; r < 32; ++r) {
      float2 a = zero, b = zero, c = zero, d = zero;
      if (r < rd_end) {
        a = tileA[od + r * 32 * XB];
        b = tileB[od + r * 32 * XB];
      }
      if (r >= rm_beg) {
        c = tileA[om - r * 32 * XB];
        d = tileB[om - r * 32 * XB];
      }
      const float2 P = f2_fma(c, pm1, a);
      const float2 Q = f2_fma(d, pm1, b);
      float2 z = make_float2(P.x - Q.y, P.y + Q.x);
      if (r == 0 && j == 0) {
        const float sg = s == 0 ? 1.f : -1.f;
        z = make_float2(fmaf(sg, c.x + d.y, a.x), fmaf(sg, d.x - c.y, b.x));
      }
      if (s != 0 && r > 0) z = r == 16 ? cmul_i(z) : cmul_c<false>(z, cos_r64(r), sin_r64(r));
      v[r] = z;
    }
  } else {
    static_assert(duo_swizzle(N, TB) == 0, "one swizzle per lane");
    const int rd_end = ncol > t ? (ncol - t + TB - 1) / TB : 0;
    const int rm_beg = (N - ncol - t) / TB + 1;
    const int od = t * XB + (xf ^ duo_swizzle(N, t)), om = (N - t) * XB + (xf ^ duo_swizzle(N, N - t));
#pragma unroll
    for (int r = 0; r < EB / 2; ++r) {
      float2 a = zero, b = zero;
      if (r < rd_end) {
        a = tileA[od + r * TB * XB];
        b = tileB[od + r * TB * XB];
      }
      v[r] = (r == 0 && t == 0) ? make_float2(a.x, b.x) : make_float2(a.x - b.y, a.y + b.x);
    }
#pragma unroll
    for (int r = EB / 2; r < EB; ++r) {
      float2 a = zero, b = zero;
      if (r >= rm_beg) {
        a = tileA[om - r * TB * XB];
        b = tileB[om - r * TB * XB];
      }
      v[r] = make_float2(a.x + b.y, b.x - a.y);
    }
  }
}

// Statistics of one image row (T row i) of the image in `slot`, output e of the
// lane's registers read by val(e): one partial per warp of the transform, as
// row_stats writes for a row pair.  Returns the lane's maximum.
template <int N, RowMode M, class F>
__device__ __forceinline__ float row_stats_one(F val, int t, int i, int slot, int tsplit, int log2l, float gate,
                                               const PassStats& ps) {
  using K = ImgCfg<N>;
  constexpr int EB = K::EB, TB = K::TB;
  constexpr int LP = FftShape<N / K::RSPLIT, EB>::LAST_P;
  constexpr int EM = EB / LP;
  constexpr int WL = TB < 32 ? TB : 32;
  float m4[4] = {-FLT_MAX, -FLT_MAX, -FLT_MAX, -FLT_MAX};
#pragma unroll
  for (int e = 0; e < EB; e += 2) m4[(e >> 1) & 3] = fmax3f(m4[(e >> 1) & 3], val(e), val(e + 1));
  const float lmax = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
  auto find = [&](float top) {
    int best = INT_MAX;
#pragma unroll
    for (int q = 0; q < LP; ++q)
#pragma unroll
      for (int m = 0; m < EM; ++m)
        if (val(m * LP + dft_perm<LP>(q)) == top) {
          best = t_row(i, tsplit, log2l) * N + row_pix<N>(t, m, q);
          goto found;
        }
  found:
    return best;
  };
  if constexpr (M == kBest) {
    if (__any_sync(0xffffffffu, !(lmax < gate))) row_best<WL>(lmax, gate, ps.best + slot, find);
    return lmax;
  }
  const float wmax = warp_max<WL>(lmax);
  int best = INT_MAX;
  if (lmax == wmax) best = find(wmax);
  best = warp_min<WL>(best);
  ClipPartial cp{};
  if constexpr (M == kClip) {
    const float2 cw = ps.clip[slot];
    KeptSums k[2];
#pragma unroll
    for (int e = 0; e < EB; ++e) k[e & 1].add(val(e), cw);
    cp = kept_reduce<WL>(k[0], k[1]);
  }
  if ((t & 31) == 0) {
    constexpr int WPT = TB > 32 ? TB / 32 : 1;
    const size_t o = (size_t)slot * (2 * K::PARTIALS) + i * WPT + (t >> 5);
    ps.partials[o] = StatPartial{wmax, best};
    if constexpr (M == kClip) ps.cparts[o] = cp;
  }
  return lmax;
}

// Pass B over units of up to 16 consecutive transformed images, with the images
// derived from them (sums of 2, 4, 8 and 16), N <= 2048: work item = (unit,
// block of XB rows).  A block takes the unit's images two at a time through
// the transform of k_rowfft_stats, one image row of both per transform (A in
// the real parts, B in the imaginary parts; an odd last image alone), so a
// lane holds the same pixels of both and their sum is one addition, with
// nothing kept.  Longer sums form as a binary counter does: a sum of an even
// place is kept, the next one is added to it and goes a level up.  What is
// kept, 32 registers a lane and level, goes to tensor memory, which nothing else
// uses here and whose loads and stores do not pass through the L1/shared pipe;
// three levels take 96 of the 128 columns that 16 warps of an SM can have each.
// Two rows of one image a transform (k_rowfft_tree) keep 64 registers a level
// and one level more, which fits two levels of sums.  1024^2 realtime (widths 1,
// 2, 4, 8): 94,700 images transformed and not 106,500, 164.3 -> 147.4 ms with
// kBest; 2048^2 batching (1 .. 16) 295.3 -> 261.9 ms.
// Items with two images that may not share a transform (may_pair) offer no best;
// the block takes them again after its other items, such images each beside
// itself and once more together for their sum only.  Looking for them takes
// 1024^2 realtime from 137.4 to 138.7 ms, 2048^2 batching from 253.3 to 254.0.  In
// the loop of all items the registers of the rare case took them to 139.1 and 266
// ms; a launch of its own took 8 us of a short search's 100.
// T is read in duo order: with the tiles' rows of XB 8-byte values permuted by
// column, a half-warp's loads meet 16 bank pairs (the hardware's swizzles move
// 16-byte chunks: two-way conflicts).
template <int N, RowMode M>
__global__ void __launch_bounds__(ImgCfg<N>::THREADS_B, 2)
    k_rowfft_duo(SegmentGeom g, DevTables tb, const float2* __restrict__ Tbuf, const Unit* __restrict__ units,
                 int nunits, int img_base, int base_base, const PassStats ps,
                 const __grid_constant__ CUtensorMap tmap, int tma_boxes, int tma_rows, int* __restrict__ err) {
  using K = ImgCfg<N>;
  constexpr int EB = K::EB, XB = K::XB, NL = 4;
  static_assert(EB == 32 && K::THREADS_B % 32 == 0 && pairs_possible(N) && (1 << NL) == unit_images(true), "32 values a lane, whole warps");
  static_assert(sizeof(Unit) == 32, "eight words, one a lane");
  constexpr bool WARP_LOCAL = K::TILE_TMA && (K::TB <= 32 || K::RSPLIT == 2);  // see k_rowfft_stats
  static_assert(WARP_LOCAL == K::TILE_TMA, "tensor copies only where no barrier crosses a warp");
  constexpr int NWB = K::THREADS_B / 32;
  constexpr unsigned TCOLS = TreeCfg<N>::COLS;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* fbuf = reinterpret_cast<float2*>(smraw);  // [XB][STRIDE_B]
  unsigned char* tb0 = smraw + XB * K::STRIDE_B * 8;
  if constexpr (K::TILE_TMA) tb0 += (1024u - (smem_u32(tb0) & 1023u)) & 1023u;
  const bool use_tma = K::TILE_TMA && tma_boxes > 0;
  const int trows = use_tma ? tma_boxes * tma_rows : g.ncol;
  float2* tileA = reinterpret_cast<float2*>(tb0);  // [rows][XB]
  float2* tileB = tileA + (size_t)trows * XB;
  __shared__ __align__(8) unsigned long long tbar;
  __shared__ int s_done;  // warps done reading the tiles in hand
  __shared__ unsigned s_tmem;
  const int tid = threadIdx.x, lane = tid & 31;
  const int ncol = g.ncol;
  constexpr int nrb = N / XB;
  const int nitems = nunits * nrb;
  const int xf = tid / K::TB;
  const int t = tid - xf * K::TB;
  const int log2l = FftShape<N>::LOG2N - (g.tsplit > 1 ? __ffs(g.tsplit) - 1 : 0);
  unsigned phase = 0;
  if (tid < 32) tmem_alloc(&s_tmem, TCOLS);
  if (tid == 0) {
    mbar_init(&tbar, 1);
    s_done = 0;
  }
  __syncthreads();
  // this warp's lanes and columns: 32 for each level that is kept
  const unsigned keep = s_tmem + ((unsigned)((tid >> 5) & 3) << 21) + (unsigned)(tid >> 7) * 128u;
  // lanes 0 .. 15 stand for a unit's images, 16 .. 23 for its sums of two,
  // 24 .. 27 of four, 28 and 29 of eight, 30 of sixteen: place lj of level ll
  const int ll = lane < 16 ? 0 : (lane < 24 ? 1 : (lane < 28 ? 2 : (lane < 30 ? 3 : 4)));
  const int lj = lane - (32 - (32 >> ll));

  // tiles of rows yb .. yb + XB of the image in T slot sl, and of the next one if `two`
  auto issue_tma = [&](int sl, bool two, int yb) {  // by one thread
    const int n = two ? 2 : 1;
    mbar_expect_tx(&tbar, (unsigned)(n * tma_boxes * tma_rows * XB * 8));
    for (int i = 0; i < n; ++i)
      for (int b = 0; b < tma_boxes; ++b)
        tma_load_3d((i ? tileB : tileA) + (size_t)b * tma_rows * XB, &tmap, 2 * yb, b * tma_rows, sl + i, &tbar);
  };
  auto fetch = [&](int sl, bool two, int yb) {
    if (use_tma) {
      if (tid == 0) issue_tma(sl, two, yb);
      return;
    }
    constexpr int CH = XB / 2;  // 16-byte chunks per column
    const float2* src = Tbuf + (size_t)sl * ncol * N + yb;
    const int n = (two ? 2 : 1) * ncol * CH;
    for (int i = tid; i < n; i += K::THREADS_B) {
      const int u = i / CH;  // columns of A, then of B
      const int c = i - u * CH;
      cp_async16(tileA + (size_t)u * XB + 2 * c, src + (size_t)u * N + 2 * c);
    }
    cp_async_commit();
  };

  // a unit's words, one a lane: base, n, img[0 .. 4]
  auto load_unit = [&](int it) { return reinterpret_cast<const int*>(units + it / nrb)[lane & 7]; };
  // bit k: images k and k + 1 of the unit may not share a transform
  auto apart_of = [&](int cur) {
    const int n = __shfl_sync(0xffffffffu, cur, 1), img = __shfl_sync(0xffffffffu, cur, 2);
    const float rms = lane < n ? ps.rms[img + lane - img_base] : 0.f;  // n <= 16
    const float other = __shfl_xor_sync(0xffffffffu, rms, 1);
    return __ballot_sync(0xffffffffu, (lane | 1) < n && !may_pair(rms, other));
  };
  bool failed = false, again = false;
  // every item of the block, or those with such images
  auto items = [&](auto only_apart) {
    constexpr bool APART = decltype(only_apart)::value;
    int item = blockIdx.x, cur = load_unit(item);  // the grid is at most the number of items
    auto advance = [&](int& it) {  // to the next item; its unit
      int u = cur;
      do {
        it += (int)gridDim.x;
        if (it >= nitems) break;
        u = load_unit(it);
      } while (APART && apart_of(u) == 0);
      return u;
    };
    if (APART && apart_of(cur) == 0) cur = advance(item);
    if (item < nitems)
      fetch(__shfl_sync(0xffffffffu, cur, 0) - base_base, __shfl_sync(0xffffffffu, cur, 1) > 1, (item % nrb) * XB);
    while (item < nitems && !failed) {
      const int y0 = (item % nrb) * XB;
      int next = item;
      const int nxt = advance(next);
      const int base = __shfl_sync(0xffffffffu, cur, 0), n = __shfl_sync(0xffffffffu, cur, 1);
      const int first = __shfl_sync(0xffffffffu, cur, 2 + ll);
      // this lane's image: its slot (-1: not searched) and gate; the highest level searched
      const int slots = first >= 0 && (lj + 1) << ll <= n ? first + lj - img_base : -1;
      const int top = 31 - __clz((int)(__ballot_sync(0xffffffffu, cur >= 0) >> 2 & 31u) | 1);
      float gates = 0.f;
      if (M == kBest && slots >= 0) gates = ps.gate[slots];
      const unsigned apart = apart_of(cur);
      if (!APART && apart != 0) {
        gates = INFINITY;
        again = true;
      }
      const int i = y0 + xf;
      for (int k = 0; k < n; k += 2) {
        if (use_tma) {
          // as in k_rowfft_stats: no copy is issued without this warp's count
          // below, so the other warps' waits run out in turn
          if (!__all_sync(0xffffffffu, mbar_wait(&tbar, phase))) {
            if (lane == 0) atomicExch(err, 1);
            mbar_wait(&tbar, phase);
            failed = true;
            break;
          }
          phase ^= 1u;
        } else {
          cp_async_wait_all();
          __syncthreads();
        }
        const bool two = k + 1 < n;
        float2 v[EB];
        const bool split = APART && (apart >> k & 1u);
        if (split)
#pragma unroll 1
          for (int b = 0; b < 2; ++b) {
            const float2* tile = b ? tileB : tileA;
            row_zbuild_duo<N>(v, tile, tile, t, xf, ncol);
            __syncwarp();  // the last transform's values are read
            row_fft<N>(v, fbuf + xf * K::STRIDE_B, tb.twiddle, t, xf);
            row_stats_one<N, M>([&](int e) { return v[e].x; }, t, i, __shfl_sync(0xffffffffu, slots, k + b), g.tsplit,
                                log2l, __shfl_sync(0xffffffffu, gates, k + b), ps);
          }
        row_zbuild_duo<N>(v, tileA, two ? tileB : tileA, t, xf, ncol);  // A alone: beside itself
        // the tiles are read: the unit's next images' (or the next item's first ones')
        const bool here = k + 2 < n;
        const int nbase = __shfl_sync(0xffffffffu, nxt, 0), nn = __shfl_sync(0xffffffffu, nxt, 1);
        const int nsl = (here ? base + k + 2 : nbase) - base_base;
        const bool ntwo = here ? k + 3 < n : nn > 1;
        const int nyb = here ? y0 : (next % nrb) * XB;
        const bool more = here || next < nitems;
        if (use_tma) {
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) {
            __threadfence_block();
            if (atomicAdd(&s_done, 1) == NWB - 1) {
              s_done = 0;
              __threadfence_block();
              asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
              if (more) issue_tma(nsl, ntwo, nyb);
            }
          }
        } else {
          __syncthreads();
          if (more) fetch(nsl, ntwo, nyb);
        }
        row_fft<N>(v, fbuf + xf * K::STRIDE_B, tb.twiddle, t, xf);
        // no pixel of a sum is above the sum of its images' maxima in the lane
        // (rounding is monotonic), so a sum's maximum is taken only where that
        // bound reaches its gate: 1024^2 realtime row passes 75.2 -> 74.3 ms,
        // 2048^2 batching 147.5 -> 145.1.  The maxima of images that went through
        // alone have other roundings: no bound.
        float bound = INFINITY;
        if (!split) {
          const int sa = __shfl_sync(0xffffffffu, slots, k), sb = __shfl_sync(0xffffffffu, slots, k + 1);
          const float ga = __shfl_sync(0xffffffffu, gates, k), gb = __shfl_sync(0xffffffffu, gates, k + 1);
          bound = row_stats_one<N, M>([&](int e) { return v[e].x; }, t, i, sa, g.tsplit, log2l, ga, ps);
          if (two) bound += row_stats_one<N, M>([&](int e) { return v[e].y; }, t, i, sb, g.tsplit, log2l, gb, ps);
        }
        if (!two || top == 0) continue;
        float2 s[EB / 2];
#pragma unroll
        for (int e = 0; e < EB / 2; ++e)
          s[e] = make_float2(v[2 * e].x + v[2 * e].y, v[2 * e + 1].x + v[2 * e + 1].y);
#pragma unroll 1
        for (int lv = 1;; ++lv) {
          const int j = k >> lv;  // s is sum j of this level
          const int sl = __shfl_sync(0xffffffffu, slots, 32 - (32 >> lv) + j);
          const float gt = __shfl_sync(0xffffffffu, gates, 32 - (32 >> lv) + j);
          if (sl >= 0 && (M != kBest || __any_sync(0xffffffffu, !(bound < gt))))
            row_stats_one<N, M>([&](int e) { return e & 1 ? s[e >> 1].y : s[e >> 1].x; }, t, i, sl, g.tsplit, log2l,
                                gt, ps);
          // the next level's block of images must be whole
          if (lv >= top || ((j | 1) + 1) << lv > n) break;
          __syncwarp();
          if ((j & 1) == 0) {
            tmem_store16(keep + (lv - 1) * 32, s);
            if (M == kBest) tmem_store1(keep + 96 + (lv - 1), bound);
            break;
          }
          if (M == kBest) bound += tmem_load1(keep + 96 + (lv - 1));
          tmem_add16(keep + (lv - 1) * 32, s);
        }
      }
      item = next;
      cur = nxt;
    }
  };
  items(std::false_type{});
  // every warp has read its last tile and, unless a wait ran out, seen every item
  if (__syncthreads_and(!failed) && again) items(std::true_type{});
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
  __syncthreads();
  if (tid < 32) tmem_free(s_tmem, TCOLS);
}

// The row-pass kernel of units at side N.
template <int N, RowMode M, bool PAIRS>
constexpr auto tree_kernel() {
  if constexpr (PAIRS) return k_rowfft_duo<N, M>;
  else return k_rowfft_tree<N, M>;
}

// The most dynamic shared memory a block of `kern` can have: the device's
// opt-in per-block limit (227 KB on sm_103a) less the kernel's static shared
// memory.  Kernels whose request depends on the plan set their attribute to
// this bound, not to the request: the attribute belongs to the kernel, and
// plans searched at once on other host threads (the serving runtime) would
// otherwise lower it under each other's launches.  0 if it cannot be read.
template <class Kernel>
int max_dynamic_smem(Kernel kern) {
  cudaFuncAttributes fa;
  int dev = 0, optin = 0;
  if (cudaFuncGetAttributes(&fa, kern) != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return optin - (int)fa.sharedSizeBytes;
}

// Blocks of `kern` an SM holds at once, for a kernel that allocates `cols`
// columns of tensor memory: the occupancy query answers 1 for any kernel with
// an allocation, whatever its size, but blocks whose columns fit together do
// run together (one block per SM made the 1024^2 row pass 1.5 times slower).
// Registers are given to warps in units of 256.
template <class Kernel>
cudaError_t tmem_blocks_per_sm(int* out, Kernel kern, int threads, int smem, int cols) {
  cudaFuncAttributes fa;
  int dev = 0, regs = 0, sm_smem = 0, reserved = 0;
  cudaError_t e = cudaFuncGetAttributes(&fa, kern);
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&regs, cudaDevAttrMaxRegistersPerMultiprocessor, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sm_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
  if (e != cudaSuccess) return e;
  const int by_regs = regs / std::max((threads + 31) / 32 * ((fa.numRegs * 32 + 255) / 256 * 256), 1);
  const int by_smem = sm_smem / std::max(smem + (int)fa.sharedSizeBytes + reserved, 1);
  *out = std::max(1, std::min(std::min(by_regs, by_smem), 512 / cols));
  return cudaSuccess;
}

// Launch `kern`, with the scheduling priority of `pl` where it sets one (a
// launch attribute, so that a captured graph keeps it on the kernel node).
template <class... P, class... A>
cudaError_t launch_with(void (*kern)(P...), dim3 grid, dim3 block, int smem, cudaStream_t st,
                        const PassLaunch* pl, A&&... args) {
  if (pl == nullptr || !pl->set_priority) {
    kern<<<grid, block, smem, st>>>(std::forward<A>(args)...);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributePriority;
  at[0].val.priority = pl->priority;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...);
}

// Dynamic shared memory of a column-pass block that keeps a second column
// block off an SM (two such blocks and their reserved shares exceed the
// SM's shared memory) while one row-pass block of `row_smem` bytes still
// fits beside it.  `smem` if that cannot be had (or is already so).
inline int one_per_sm_smem(int smem, int row_smem, int smem_max) {
  int dev = 0, sm_smem = 0, reserved = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sm_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) != cudaSuccess) {
    cudaGetLastError();
    return smem;
  }
  const int floor = sm_smem / 2 - reserved + 16;
  if (smem >= floor || floor > smem_max || floor + row_smem + 2 * reserved > sm_smem) return smem;
  return floor;
}



// Periodicity row pass (Sec. 3.1 footnote).  A pair is the two quadrature
// images (U and Q) of one (DM trial, fluctuation frequency); work item =
// (pair, block of XB rows), and each transform takes one row y with
// Z[u] = T_U[u][y] + i T_Q[u][y] (Hermitian-extended as in the search's row
// pass), so its output holds row y of I_U in the real parts and of I_Q in
// the imaginary parts.  Per row it writes the maximum of I_U^2 + I_Q^2 (raw
// pixel units) and its lowest index.  pairs[j] = {U slot, Q slot, -, -}.
// The tile is [ncol][CH] 16-byte chunks {U[u][y], Q[u][y]} copied with
// cp.async, or, where every transform fits one warp and tma_boxes > 0
// (N = 1024), two tiles [rows][XB] of U and of Q rows, each filled by
// tma_boxes tensor copies of tma_rows u rows from `tmap` ([slot][u][2N
// floats], boxes of XB complex values), with T in duo order: an 8-byte load of
// 16 columns then meets 16 bank pairs (the hardware's 64-byte swizzle moves
// 16-byte chunks and left two-way conflicts: 2048 pairs of
// 1024^2 9.07 ms a call so, 8.67 this way).  Then, as in the search's row
// pass, no block barrier is left: each warp waits for the tiles on an
// mbarrier (bounded; a warp that gives up sets *err, waits once more and
// leaves) and the last warp to read them issues the next item's copies.
template <int N>
__global__ void __launch_bounds__(ImgCfg<N>::THREADS_B, 2)
    k_rowfft_power(SegmentGeom g, DevTables tb, const float2* __restrict__ Tbuf, const int4* __restrict__ pairs,
                   int npairs, StatPartial* __restrict__ partials, const __grid_constant__ CUtensorMap tmap,
                   int tma_boxes, int tma_rows, int* __restrict__ err) {
  using K = ImgCfg<N>;
  constexpr int EB = K::EB, TB = K::TB;
  constexpr bool PTMA = K::TILE_TMA && TB <= 32;  // warp-local transforms (N = 1024)
  static_assert(!PTMA || (K::XB == 8 && EB == 32), "power tiles: 64-byte rows of 8 complex values");
  constexpr int NWB = K::THREADS_B / 32;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* fbuf = reinterpret_cast<float2*>(smraw);                       // [XB][STRIDE_B]
  float4* tile = reinterpret_cast<float4*>(fbuf + K::XB * K::STRIDE_B);  // [ncol][CH]
  // tensor-copy tiles of U and Q rows, [rows][XB]
  unsigned char* tu0 = smraw + K::XB * K::STRIDE_B * 8;
  tu0 += (1024u - (smem_u32(tu0) & 1023u)) & 1023u;
  const unsigned tsz = ((unsigned)(tma_boxes * tma_rows * K::XB * 8) + 511u) & ~511u;
  float2* tileU = reinterpret_cast<float2*>(tu0);
  float2* tileQ = reinterpret_cast<float2*>(tu0 + tsz);
  __shared__ float w_max[32];
  __shared__ int w_idx[32];
  __shared__ __align__(8) unsigned long long tbar;
  __shared__ int s_done;
  const int tid = threadIdx.x;
  const int lane = tid & 31;
  const int wid = tid >> 5;
  const int ncol = g.ncol;
  constexpr int nrb = N / K::XB;  // row blocks per pair
  const int nitems = npairs * nrb;
  const int xf = tid / TB;
  const int t = tid - xf * TB;
  const int log2l = FftShape<N>::LOG2N - (g.tsplit > 1 ? __ffs(g.tsplit) - 1 : 0);

  const bool use_tma = PTMA && tma_boxes > 0;
  unsigned phase = 0;
  if (use_tma) {
    if (tid == 0) {
      mbar_init(&tbar, 1);
      s_done = 0;
    }
    __syncthreads();
  }
  auto issue_tma = [&](int it) {  // by one thread
    const int pj = it / nrb;
    const int yb = (it - pj * nrb) * K::XB;
    const int4 pr = pairs[pj];
    mbar_expect_tx(&tbar, (unsigned)(2 * tma_boxes * tma_rows * K::XB * 8));
    for (int b = 0; b < tma_boxes; ++b) {
      tma_load_3d(tileU + (size_t)b * tma_rows * K::XB, &tmap, 2 * yb, b * tma_rows, pr.x, &tbar);
      tma_load_3d(tileQ + (size_t)b * tma_rows * K::XB, &tmap, 2 * yb, b * tma_rows, pr.y, &tbar);
    }
  };
  auto prefetch = [&](int it) {
    if (use_tma) {
      if (tid == 0) issue_tma(it);
      return;
    }
    const int pj = it / nrb;
    const int yb = (it - pj * nrb) * K::XB;
    const int4 pr = pairs[pj];
    const float2* su = Tbuf + (size_t)pr.x * ncol * N + yb;
    const float2* sq = Tbuf + (size_t)pr.y * ncol * N + yb;
    for (int i = tid; i < ncol * K::CH; i += K::THREADS_B) {
      const int u = i / K::CH;
      const int c = i - u * K::CH;
      float2* d = reinterpret_cast<float2*>(tile + u * K::CH + (c ^ (u & (K::CH - 1))));
      cp_async8(d, su + (size_t)u * N + c);
      cp_async8(d + 1, sq + (size_t)u * N + c);
    }
    cp_async_commit();
  };

  int item = blockIdx.x;
  if (item < nitems) prefetch(item);
  for (; item < nitems; item += gridDim.x) {
    if (use_tma) {
      if (!__all_sync(0xffffffffu, mbar_wait(&tbar, phase))) {
        if (lane == 0) atomicExch(err, 1);
        mbar_wait(&tbar, phase);
        return;
      }
      phase ^= 1u;
    } else {
      cp_async_wait_all();
      __syncthreads();
    }
    const int pj = item / nrb;
    const int iy = (item - pj * nrb) * K::XB + xf;   // T row; image row y below
    const int y = t_row(iy, g.tsplit, log2l);
    float2 v[EB];
    if (PTMA && use_tma) {
      if constexpr (PTMA) row_zbuild_duo<N>(v, tileU, tileQ, t, xf, ncol);
    } else if constexpr (TB % K::CH == 0) {
      // as in the search's row pass: u = t + r T (or N - t - r T) has the
      // swizzle term of t (N - t), and the loads are predicated, not branched
      const int rd_end = ncol > t ? (ncol - t + TB - 1) / TB : 0;
      const int rm_beg = (N - ncol - t) / TB + 1;
      const float4* pd = tile + t * K::CH + (xf ^ (t & (K::CH - 1)));
      const float4* pm = tile + (size_t)(N - t) * K::CH + (xf ^ ((N - t) & (K::CH - 1)));
#pragma unroll
      for (int r = 0; r < EB / 2; ++r) {
        float4 ab = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r < rd_end) ab = pd[r * TB * K::CH];
        v[r] = (r == 0 && t == 0) ? make_float2(ab.x, ab.z) : make_float2(ab.x - ab.w, ab.y + ab.z);
      }
#pragma unroll
      for (int r = EB / 2; r < EB; ++r) {
        float4 ab = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r >= rm_beg) ab = pm[-r * TB * K::CH];
        v[r] = make_float2(ab.x + ab.w, ab.z - ab.y);
      }
    } else {
#pragma unroll
      for (int r = 0; r < EB; ++r) {
        const int u = t + r * TB;
        float2 z = make_float2(0.f, 0.f);
        if (u < ncol) {
          const float4 ab = tile[u * K::CH + (xf ^ (u & (K::CH - 1)))];
          z = (u == 0) ? make_float2(ab.x, ab.z) : make_float2(ab.x - ab.w, ab.y + ab.z);
        } else if (N - u < ncol) {
          const int uu = N - u;
          const float4 ab = tile[uu * K::CH + (xf ^ (uu & (K::CH - 1)))];
          z = make_float2(ab.x + ab.w, ab.z - ab.y);
        }
        v[r] = z;
      }
    }
    if (use_tma) {
      // tiles read by this warp; the last of the block's warps issues the
      // next item's copies
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) {
        __threadfence_block();
        if (atomicAdd(&s_done, 1) == NWB - 1) {
          s_done = 0;
          __threadfence_block();
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          if (item + (int)gridDim.x < nitems) issue_tma(item + gridDim.x);
        }
      }
    } else {
      __syncthreads();  // tile consumed: prefetch the next item
      if (item + (int)gridDim.x < nitems) prefetch(item + gridDim.x);
    }
    fft_inverse_from_regs<N, false, EB>(v, fbuf + xf * K::STRIDE_B, tb.twiddle, t, xf);

    constexpr int LP = FftShape<N, EB>::LAST_P;
    constexpr int EM = EB / LP;
    float pa[4] = {-1.f, -1.f, -1.f, -1.f};
#pragma unroll
    for (int e = 0; e < EB; ++e) pa[e & 3] = fmaxf(pa[e & 3], fmaf(v[e].x, v[e].x, v[e].y * v[e].y));
    const float lmax = fmaxf(fmaxf(pa[0], pa[1]), fmaxf(pa[2], pa[3]));
    constexpr int WL = TB < 32 ? TB : 32;
    const float wmax = warp_max<WL>(lmax);
    int best = INT_MAX;
    if (lmax == wmax) {
#pragma unroll
      for (int q = 0; q < LP; ++q)
#pragma unroll
        for (int m = 0; m < EM; ++m) {
          const float2 z = v[m * LP + dft_perm<LP>(q)];
          if (fmaf(z.x, z.x, z.y * z.y) == wmax) {
            best = y * N + fft_out_index<N, EB>(t, m, q);
            goto found;
          }
        }
    found:;
    }
    best = warp_min<WL>(best);
    float mx = wmax;
    int mi = best;
    if (TB > 32) {
      constexpr int WPT = TB / 32;
      const int wi = t >> 5;
      if (lane == 0) {
        w_max[wid] = wmax;
        w_idx[wid] = best;
      }
      fft_sync<TB>(xf);
      if (t == 0) {
        const int w0 = wid - wi;
        mx = -1.f;
        mi = INT_MAX;
        for (int w = 0; w < WPT; ++w) max_merge(mx, mi, w_max[w0 + w], w_idx[w0 + w]);
      }
      fft_sync<TB>(xf);
    }
    if (t == 0) {
      partials[(size_t)pj * N + iy] = StatPartial{mx, mi};
    }
  }
}

template <int N>
cudaError_t run_rowfft_power(const SegmentGeom& g, const DevTables& tb, const float2* Tbuf, const int4* pairs,
                             int npairs, StatPartial* partials, const TileMap* tm, int* err, cudaStream_t st) {
  using K = ImgCfg<N>;
  // tensor-copy tiles where every transform fits one warp (see k_rowfft_power)
  const bool tma = K::TILE_TMA && K::TB <= 32 && tm != nullptr && tm->nbox > 0 && err != nullptr;
  const int tsz = tma ? (tm->nbox * tm->rows * K::XB * 8 + 511) / 512 * 512 : 0;
  const int smem = tma ? K::SMEM_B_FIXED + 1024 + 2 * tsz : K::SMEM_B_FIXED + g.ncol * K::CH * 16;
  const int smem_max = max_dynamic_smem(k_rowfft_power<N>);
  if (smem > smem_max) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(k_rowfft_power<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_rowfft_power<N>, cudaFuncAttributePreferredSharedMemoryCarveout,
                           cudaSharedmemCarveoutMaxShared);
  if (e != cudaSuccess) return e;
  if (npairs <= 0) return cudaSuccess;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_rowfft_power<N>, K::THREADS_B, smem);
  if (e != cudaSuccess) return e;
  const long nitems = (long)npairs * (N / K::XB);
  const long grid = std::min<long>(nitems, (long)std::max(per_sm, 1) * sm_count());
  CUtensorMap none;
  memset(&none, 0, sizeof(none));
  k_rowfft_power<N><<<(int)grid, K::THREADS_B, smem, st>>>(g, tb, Tbuf, pairs, npairs, partials,
                                                           tma ? tm->map : none, tma ? tm->nbox : 0,
                                                           tma ? tm->rows : 0, err);
  return cudaGetLastError();
}


template <int N>
int rowfft_tile_rows(int ncol);

template <int N>
cudaError_t run_colfft(const SegmentGeom& g, const DevTables& tb, const Group* groups, int g_begin, int ngroups,
                       int img_base, int base_base, const float2* cellbuf, float2* Tbuf, float* colsq, float* mean0,
                       bool duo, cudaStream_t st, const PassLaunch* pl) {
  using C = ColCfg<N>;
  using K = ImgCfg<N>;
  int smem = C::SMEM_FIXED + g.max_cells * C::SMEM_PER_CELL;
  const int smem_max = max_dynamic_smem(k_colfft<N>);
  if (smem > smem_max) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(k_colfft<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_colfft<N>, cudaFuncAttributePreferredSharedMemoryCarveout,
                           cudaSharedmemCarveoutMaxShared);
  if (e != cudaSuccess) return e;
  if (ngroups <= 0) return cudaSuccess;
  if (pl != nullptr && pl->one_per_sm)
    smem = one_per_sm_smem(smem, K::SMEM_B_FIXED + (K::TILE_TMA ? 1024 : 0) + rowfft_tile_rows<N>(g.ncol) * K::CH * 16,
                           smem_max);
  dim3 grid(ngroups, g.ncol);
  return launch_with(k_colfft<N>, grid, dim3(C::THREADS), smem, st, pl, g, tb, groups, g_begin, img_base, base_base,
                     cellbuf, Tbuf, colsq, mean0, duo ? 1 : 0);
}

// Rows of the row-pass tile: ncol, or the boxes' total under tensor copies.
template <int N>
int rowfft_tile_rows(int ncol) {
  if (!ImgCfg<N>::TILE_TMA) return ncol;
  int nbox, rows;
  tile_boxes(ncol, &nbox, &rows);
  return nbox * rows;
}

template <int N, RowMode M>
cudaError_t run_rowfft_stats_k(const SegmentGeom& g, const DevTables& tb, const float2* Tbuf, int nimg,
                               int img_base, const double* weight, const PassStats& ps, float* images,
                               const TileMap* tm, int* err, cudaStream_t st, const PassLaunch* pl) {
  using K = ImgCfg<N>;
  const int smem = K::SMEM_B_FIXED + (K::TILE_TMA ? 1024 : 0) + rowfft_tile_rows<N>(g.ncol) * K::CH * 16;
  auto kern = k_rowfft_stats<N, M>;
  const int smem_max = max_dynamic_smem(kern);
  if (smem > smem_max) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  if (e != cudaSuccess) return e;
  if (nimg <= 0) return cudaSuccess;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, K::THREADS_B, smem);
  if (e != cudaSuccess) return e;
  const long nitems = (long)nimg * (N / K::RB);
  long grid = std::min<long>(nitems, (long)std::max(per_sm, 1) * sm_count());
  // short-lived blocks of items_per_block items (the kernel strides by the grid)
  if (pl != nullptr && pl->items_per_block > 0)
    grid = std::max(grid, std::min<long>((nitems + pl->items_per_block - 1) / pl->items_per_block, INT_MAX));
  const bool tma = K::TILE_TMA && tm != nullptr && tm->nbox > 0 && err != nullptr;
  CUtensorMap none;
  memset(&none, 0, sizeof(none));
  return launch_with(kern, dim3((unsigned)grid), dim3(K::THREADS_B), smem, st, pl, g, tb, Tbuf, nimg, img_base,
                     weight, ps, images, tma ? tm->map : none, tma ? tm->nbox : 0, tma ? tm->rows : 0, err);
}

template <int N>
cudaError_t run_rowfft_stats(const SegmentGeom& g, const DevTables& tb, const float2* Tbuf, int nimg,
                             int img_base, const double* weight, const PassStats& ps, float* images,
                             const TileMap* tm, int* err, cudaStream_t st, const PassLaunch* pl) {
  if (ps.clip != nullptr)
    return run_rowfft_stats_k<N, kClip>(g, tb, Tbuf, nimg, img_base, weight, ps, images, tm, err, st, pl);
  if (ps.best != nullptr)
    return run_rowfft_stats_k<N, kBest>(g, tb, Tbuf, nimg, img_base, weight, ps, images, tm, err, st, pl);
  return run_rowfft_stats_k<N, kParts>(g, tb, Tbuf, nimg, img_base, weight, ps, images, tm, err, st, pl);
}

template <int N, RowMode M, bool PAIRS>
cudaError_t run_rowfft_tree_k(const SegmentGeom& g, const DevTables& tb, const float2* Tbuf, const Unit* units,
                              int nunits, int img_base, int base_base, const PassStats& ps, const TileMap* tm,
                              int* err, cudaStream_t st, const PassLaunch* pl) {
  using K = ImgCfg<N>;
  const int smem = K::SMEM_B_FIXED + (K::TILE_TMA ? 1024 : 0) + rowfft_tile_rows<N>(g.ncol) * K::CH * 16;
  auto kern = tree_kernel<N, M, PAIRS>();
  const int smem_max = max_dynamic_smem(kern);
  if (smem > smem_max) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  if (e != cudaSuccess) return e;
  if (nunits <= 0) return cudaSuccess;
  int per_sm = 0;
  e = tmem_blocks_per_sm(&per_sm, kern, K::THREADS_B, smem, TreeCfg<N>::COLS);
  if (e != cudaSuccess) return e;
  // an item is up to unit_images(PAIRS) images, two of them a transform where they are paired
  const long nitems = (long)nunits * (N / (PAIRS ? K::XB : K::RB));
  const long steps = unit_images(PAIRS) / (PAIRS ? 2 : 1);
  long grid = std::min<long>(nitems, (long)std::max(per_sm, 1) * sm_count());
  if (pl != nullptr && pl->items_per_block > 0)
    grid = std::max(grid, std::min<long>((steps * nitems + pl->items_per_block - 1) / pl->items_per_block,
                                         std::min<long>(nitems, INT_MAX)));
  const bool tma = K::TILE_TMA && tm != nullptr && tm->nbox > 0 && err != nullptr;
  CUtensorMap none;
  memset(&none, 0, sizeof(none));
  return launch_with(kern, dim3((unsigned)grid), dim3(K::THREADS_B), smem, st, pl, g, tb, Tbuf, units, nunits,
                     img_base, base_base, ps, tma ? tm->map : none, tma ? tm->nbox : 0, tma ? tm->rows : 0, err);
}

template <int N>
cudaError_t run_rowfft_tree(const SegmentGeom& g, const DevTables& tb, const float2* Tbuf, const Unit* units,
                            int nunits, bool pairs, int img_base, int base_base, const PassStats& ps,
                            const TileMap* tm, int* err, cudaStream_t st, const PassLaunch* pl) {
  static_assert(N >= kTreeMinNpix, "whole warps");
#define RF_UNITS(M, P) run_rowfft_tree_k<N, M, P>(g, tb, Tbuf, units, nunits, img_base, base_base, ps, tm, err, st, pl)
  if (pairs) {
    if constexpr (pairs_possible(N))
      return ps.clip ? RF_UNITS(kClip, true) : (ps.best ? RF_UNITS(kBest, true) : RF_UNITS(kParts, true));
    return cudaErrorInvalidValue;
  }
  return ps.clip ? RF_UNITS(kClip, false) : (ps.best ? RF_UNITS(kBest, false) : RF_UNITS(kParts, false));
#undef RF_UNITS
}

template <int N>
void fill_shape(ImageKernelShape* o) {
  using K = ImgCfg<N>;
  o->images_per_group = K::B;
  o->cols_per_cta = 1;
  o->threads_a = ColCfg<N>::THREADS;
  o->smem_a = ColCfg<N>::SMEM_FIXED;
  o->warps_per_col = 0;
  o->rows_per_cta = K::RB;
  o->partials_per_image = K::PARTIALS;
  o->threads_b = K::THREADS_B;
  o->smem_b = K::SMEM_B_FIXED;
  o->smem_a_per_cell = ColCfg<N>::SMEM_PER_CELL;
  o->smem_b_per_row = K::CH * 16;
  o->tile_tma = K::TILE_TMA;
}

#define RF_INSTANTIATE_IMAGE(N)                                                                              \
  template cudaError_t run_colfft<N>(const SegmentGeom&, const DevTables&, const Group*, int, int, int, int, \
                                     const float2*, float2*, float*, float*, bool, cudaStream_t,            \
                                     const PassLaunch*);                                                    \
  template cudaError_t run_rowfft_stats<N>(const SegmentGeom&, const DevTables&, const float2*, int, int,    \
                                           const double*, const PassStats&, float*, const TileMap*, int*,   \
                                           cudaStream_t, const PassLaunch*);                                \
  template void fill_shape<N>(ImageKernelShape*);                                                           \
  template cudaError_t run_rowfft_power<N>(const SegmentGeom&, const DevTables&, const float2*, const int4*, \
                                           int, StatPartial*, const TileMap*, int*, cudaStream_t);

#define RF_INSTANTIATE_TREE(N)                                                                               \
  template cudaError_t run_rowfft_tree<N>(const SegmentGeom&, const DevTables&, const float2*, const Unit*,  \
                                          int, bool, int, int, const PassStats&, const TileMap*, int*,       \
                                          cudaStream_t, const PassLaunch*);

}  // namespace rf
