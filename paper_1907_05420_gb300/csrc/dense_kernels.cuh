// Building blocks of the blocked right-looking dense LDL^T (panel width
// kDenseNB = 64), shared by the factor of the Schur complement S (one matrix)
// and by the dense tail of the block factors (one matrix per block, batched
// over blockIdx with a stride).  Matrices are column-major with leading
// dimension n; only the lower triangle is read or written.  A panel k0 has
// kb pivot columns (kb < 64 for a last ragged panel; the rows below the
// pivots may extend past the last pivot column: the tail's augmented rows).
// Per panel:
//   k_dense_diag_t:   LDL^T of the kb x kb diagonal block;
//   k_dense_panel_t:  L21 = A21 L11^{-T} D1^{-1} and Y = L21 D1 (rows below);
//   k_dense_update:   A22 -= Y L21^T on the lower 16 x 16 tiles (FP64).
// A division by a pivot is a multiplication by its reciprocal.
// Included by the translation units that launch them (internal linkage).
#pragma once
#include "handle.h"
#include "pivot.cuh"

namespace kkt {

namespace {

constexpr int kPanelW = kDenseNB;

// Static-pivot rule of the block factors: a pivot with |d| < pivot_eps *
// max|A_b| is replaced by +-pivot_eps * max|A_b|, with the sign the inertia of
// a quasidefinite block gives its column (+ primal, - multiplier).  A null
// anorm turns the rule off (the factor of S).
struct PivotRule {
  const double* anorm = nullptr;   // per matrix of the batch
  double pivot_eps = 0.0;
  const int32_t* primal = nullptr; // per column of the matrix: 1 if primal
};

// LDL^T of the diagonal block at (k0, k0) of matrix blockIdx.x, in shared
// memory, in sub-panels of kSub = 8 columns:
//   (1) the sub-panel with all its rows, right-looking, by four warps (one per
//       SM sub-partition) that hold it in registers: a lane per row, the
//       columns dealt out over the warps (two warps per column set while more
//       than 32 rows are left, four sets of columns afterwards).  One barrier
//       per pivot: the warps that own the pivot's column publish it in shared
//       memory, every thread forms the same 1 / d and its own l = u / d, and the
//       next pivot's column is updated and published first;
//   (2) the trailing triangle of the block takes A[i][j] -= sum_c L[i][c] U[j][c]
//       over the sub-panel, spread over all threads (rows p and R-1-p of the
//       triangle of order R together hold R + 1 entries).
// What bounds it: FP64 on one SM.  An FP64 operation keeps its sub-partition's
// pipe busy for 64 cycles per warp, so the chain of a pivot (the reciprocal,
// l, the next column's entry, a barrier: about 540 cycles) and the 64^3 / 6
// multiply-adds of the block both count.  Sub-panels of 8 keep few of those in
// the chain's steps; 16 took 10% longer.  64 FP64 pivots of one matrix take
// 31 us (69 with a barrier pair per pivot, the reciprocal on one thread and a
// thread per row below a sub-panel's diagonal block), 32 pivots 9.6 us (26.8);
// FP32, where only barriers and shared memory count, 10.8 us per 64 (24.5).
constexpr int kSub = 8;

__device__ __forceinline__ void bar_sync_warps03() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

// Phase (1) for the thread that holds row `row` and the columns q G + g of the
// sub-panel at column c0 (cb <= 16 pivots).  Entries above the diagonal and
// rows past the block are carried along and never stored.
// RULE: the pivot rule applies; repl holds the replacement of each of the
// block's pivots, +-thr, and thr's bit pattern is compared with the pivot's
// (non-negative doubles order like their bits, and a comparison of integers
// leaves the FP64 pipe alone).  There are no branches around the multiply-adds:
// a column that is done takes the last one or two updates of its set along,
// unused.
template <class T, int G, bool RULE>
__device__ __forceinline__ int diag_subpanel(T (&A)[kPanelW][kPanelW + 1], T (&U)[kPanelW][kSub + 1],
                                             T (&col)[2][kPanelW], const T* repl, int c0, int cb, int row, int g) {
  constexpr int NQ = kSub / G;
  int pert = 0;
  T a[NQ];
#pragma unroll
  for (int q = 0; q < NQ; q++) a[q] = A[row][c0 + q * G + g];
  if (g == 0) col[0][row] = a[0];
  bar_sync_warps03();
#pragma unroll
  for (int k = 0; k < kSub; k++) {
    if (k < cb) {
      const T* ck = col[k & 1];
      const T u = ck[row];
      T d = ck[c0 + k];
      T uj[NQ];  // all loads first
#pragma unroll
      for (int q = (k + 1) / G; q < NQ; q++) uj[q] = ck[c0 + q * G + g];
      if constexpr (RULE) {
        const T t = repl[c0 + k];
        const long long mag = 0x7fffffffffffffffLL;
        const bool small = (__double_as_longlong((double)d) & mag) < (__double_as_longlong((double)t) & mag);
        d = small ? t : d;
        pert += small;
      }
      const T l = u * pivot_recip(d);
#pragma unroll
      for (int q = (k + 1) / G; q < NQ; q++) {
        a[q] -= l * uj[q];
        // the next pivot's column is published as soon as it is updated
        if (q == (k + 1) / G && g == (k + 1) % G) col[(k + 1) & 1][row] = a[q];
      }
      if (g == k % G) {  // (above the diagonal: unused entries)
        U[row][k] = u;
        A[row][c0 + k] = row == c0 + k ? d : l;
      }
      bar_sync_warps03();
    }
  }
  return pert;
}

template <class T, bool RULE>
__global__ void __launch_bounds__(256, 1) k_dense_diag_t(T* __restrict__ S0, int n, int k0, int kb,
                                                      int64_t bstride, PivotRule rule,
                                                      unsigned long long* __restrict__ counters) {
  __shared__ T A[kPanelW][kPanelW + 1];
  __shared__ T U[kPanelW][kSub + 1];
  __shared__ T col[2][kPanelW];
  __shared__ T repl[RULE ? kPanelW : 1];
  T* S = S0 + (int64_t)blockIdx.x * bstride;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  {
    // 16 loads per thread issued together, then stored
    T v[16];
#pragma unroll
    for (int u = 0; u < 16; u++) {
      const int q = tid + u * 256, c = q >> 6, r = q & 63;
      v[u] = (r >= c && r < kb && c < kb) ? S[(int64_t)(k0 + r) + (int64_t)(k0 + c) * n] : T(0);
    }
    if (RULE && tid < kb) {
      // a threshold that is not positive (or NaN) leaves every pivot alone
      const double thr = rule.pivot_eps * rule.anorm[blockIdx.x];
      repl[tid] = thr > 0.0 ? (T)(rule.primal[k0 + tid] ? thr : -thr) : T(0);
    }
#pragma unroll
    for (int u = 0; u < 16; u++) {
      const int q = tid + u * 256, c = q >> 6, r = q & 63;
      A[r][c] = v[u];
    }
  }
  int pert = 0;
  __syncthreads();
  for (int c0 = 0; c0 < kb; c0 += kSub) {
    const int cb = min(kSub, kb - c0);
    if (warp < 4) {  // (1)
      if (kb > 32 && c0 < 32)
        pert += diag_subpanel<T, 2, RULE>(A, U, col, repl, c0, cb, (warp & 1) * 32 + lane, warp >> 1);
      else
        pert += diag_subpanel<T, 4, RULE>(A, U, col, repl, c0, cb, (c0 & 32) + lane, warp);
    }
    __syncthreads();
    const int r0 = c0 + cb, R = kb - r0;
    if (R > 0) {  // (2) (only the last sub-panel is ragged: cb == kSub here)
      for (int q = tid; q < R * (R + 1) / 2; q += 256) {
        const int p = q / (R + 1), off = q - p * (R + 1);
        const int i = off < R - p ? R - 1 - p : p, j = off < R - p ? off : off - (R - p);
        T acc = T(0);
#pragma unroll
        for (int c = 0; c < kSub; c++) acc += A[r0 + i][c0 + c] * U[r0 + j][c];
        A[r0 + i][r0 + j] -= acc;
      }
      __syncthreads();
    }
  }
  {
#pragma unroll
    for (int u = 0; u < 16; u++) {
      const int q = tid + u * 256, c = q >> 6, r = q & 63;
      if (r >= c && r < kb && c < kb) S[(int64_t)(k0 + r) + (int64_t)(k0 + c) * n] = A[r][c];
    }
  }
  const T dd = tid < kb ? A[tid][tid] : T(0);
  const int pos = __syncthreads_count(dd > T(0));
  const int neg = __syncthreads_count(dd < T(0));
  if (tid == 0) {
    atomicAdd(&counters[kPos], (unsigned long long)pos);
    atomicAdd(&counters[kNeg], (unsigned long long)neg);
    if (kb - pos - neg) atomicAdd(&counters[kZero], (unsigned long long)(kb - pos - neg));
    if (pert) atomicAdd(&counters[kPerturbed], (unsigned long long)pert);
  }
}

// TF32 operand images of the trailing update, written by the panel kernels
// themselves (FP32 only): the shared-memory layout of the tensor-core update's
// 128-row A blocks (Y) and 64-row B blocks (L21), K-major 8-row x 16-byte core
// matrices, 16 cores along K.  Rows are counted from the first trailing row;
// columns at or past kb are zero.  A null A skips the images.
struct Tf32Images {
  uint8_t* A = nullptr;
  uint8_t* B = nullptr;
};

__device__ __forceinline__ int64_t tf32_img_off(int rho, int c, int rows_blk) {
  const int blk = rho / rows_blk, rr = rho - blk * rows_blk;
  return (int64_t)blk * (rows_blk / 8) * 16 * 128 + ((rr >> 3) * 16 + (c >> 2)) * 128 + (rr & 7) * 16 + (c & 3) * 4;
}

// Rows k0+kb .. rend-1 of matrix blockIdx.y, one thread per row (ROWS rows
// per CTA): solve y L11^T = a with y in registers and L11 in shared memory
// (every thread of a warp reads the same L11 entry), then Y = y and
// L21 = y D1^{-1}.  Y has the matrix's leading dimension n and its rows.
template <class T, int ROWS>
__global__ void __launch_bounds__(ROWS) k_dense_panel_t(T* __restrict__ S0, T* __restrict__ Y0, int n,
                                                        int k0, int kb, int rend, int64_t bstride,
                                                        int64_t ystride, Tf32Images img) {
  __shared__ T L11[kPanelW][kPanelW];  // [j][c], zero outside the strict lower triangle
  __shared__ T dinv[kPanelW];
  T* S = S0 + (int64_t)blockIdx.y * bstride;
  T* Y = Y0 + (int64_t)blockIdx.y * ystride;
  for (int q = threadIdx.x; q < kPanelW * kPanelW; q += blockDim.x) {
    const int c = q / kPanelW, j = q - c * kPanelW;
    L11[j][c] = (j > c && j < kb) ? S[(int64_t)(k0 + j) + (int64_t)(k0 + c) * n] : T(0);
  }
  for (int c = threadIdx.x; c < kPanelW; c += blockDim.x)
    dinv[c] = c < kb ? T(1) / S[(int64_t)(k0 + c) + (int64_t)(k0 + c) * n] : T(0);
  __syncthreads();
  const int row = k0 + kb + blockIdx.x * ROWS + threadIdx.x;
  if (row >= rend) return;
  T y[kPanelW];
#pragma unroll
  for (int c = 0; c < kPanelW; c++) y[c] = c < kb ? S[row + (int64_t)(k0 + c) * n] : T(0);
  // y_j = a_j - sum_{c<j} y_c L_jc, subtracted in increasing c
#pragma unroll
  for (int j = 1; j < kPanelW; j++) {
    T acc = y[j];
#pragma unroll
    for (int c = 0; c < j; c++) acc -= y[c] * L11[j][c];
    y[j] = acc;
  }
#pragma unroll
  for (int c = 0; c < kPanelW; c++)
    if (c < kb) {
      Y[row + (int64_t)c * n] = y[c];
      S[row + (int64_t)(k0 + c) * n] = y[c] * dinv[c];
    }
  if constexpr (sizeof(T) == 4) {
    if (img.A) {
      const int rho = row - (k0 + kb);
#pragma unroll
      for (int kq = 0; kq < kPanelW / 4; kq++) {
        float4 a, l;
        a.x = y[4 * kq];
        a.y = y[4 * kq + 1];
        a.z = y[4 * kq + 2];
        a.w = y[4 * kq + 3];
        l.x = y[4 * kq] * dinv[4 * kq];
        l.y = y[4 * kq + 1] * dinv[4 * kq + 1];
        l.z = y[4 * kq + 2] * dinv[4 * kq + 2];
        l.w = y[4 * kq + 3] * dinv[4 * kq + 3];
        *reinterpret_cast<float4*>(img.A + tf32_img_off(rho, 4 * kq, 128)) = a;
        *reinterpret_cast<float4*>(img.B + tf32_img_off(rho, 4 * kq, 64)) = l;
      }
    }
  }
}

// The same solve with one warp per row: lane l holds y_l and y_{l+32}, and
// column c's value reaches the other lanes by shuffle.  The dependency chain
// of a row is 64 steps long instead of 2016 multiply-adds, which is what counts
// for few rows (and in FP64, whose dependent multiply-add latency is long).
// From column 32 on only y_{l+32} is left to update.  WARPS rows per CTA.
template <class T, int WARPS>
__global__ void __launch_bounds__(32 * WARPS) k_dense_panel_w(T* __restrict__ S0, T* __restrict__ Y0, int n, int k0,
                                                       int kb, int rend, int64_t bstride, int64_t ystride,
                                                       Tf32Images img) {
  __shared__ T L11[kPanelW][kPanelW + 1];
  __shared__ T dinv[kPanelW];
  T* S = S0 + (int64_t)blockIdx.y * bstride;
  T* Y = Y0 + (int64_t)blockIdx.y * ystride;
  const int lane = threadIdx.x & 31;
  const int row = k0 + kb + blockIdx.x * WARPS + (threadIdx.x >> 5);
  const bool live = row < rend;
  T y0 = live && lane < kb ? S[row + (int64_t)(k0 + lane) * n] : T(0);
  T y1 = live && lane + 32 < kb ? S[row + (int64_t)(k0 + lane + 32) * n] : T(0);
  for (int q = threadIdx.x; q < kPanelW * kPanelW; q += blockDim.x) {
    const int j = q / kPanelW, i = q - j * kPanelW;
    if (i < kb && j < i) L11[i][j] = S[(int64_t)(k0 + i) + (int64_t)(k0 + j) * n];
  }
  for (int c = threadIdx.x; c < kb; c += blockDim.x) dinv[c] = pivot_recip(S[(int64_t)(k0 + c) + (int64_t)(k0 + c) * n]);
  __syncthreads();
  if (!live) return;
  const int k32 = min(kb, 32);
  for (int c = 0; c < k32; c++) {
    const T yc = __shfl_sync(0xffffffffu, y0, c);
    if (lane > c && lane < kb) y0 -= yc * L11[lane][c];
    if (lane + 32 < kb) y1 -= yc * L11[lane + 32][c];
  }
  for (int c = 32; c < kb; c++) {
    const T yc = __shfl_sync(0xffffffffu, y1, c - 32);
    if (lane + 32 > c && lane + 32 < kb) y1 -= yc * L11[lane + 32][c];
  }
  if (lane < kb) {
    Y[row + (int64_t)lane * n] = y0;
    S[row + (int64_t)(k0 + lane) * n] = y0 * dinv[lane];
  }
  if (lane + 32 < kb) {
    Y[row + (int64_t)(lane + 32) * n] = y1;
    S[row + (int64_t)(k0 + lane + 32) * n] = y1 * dinv[lane + 32];
  }
  if constexpr (sizeof(T) == 4) {
    if (img.A) {
      const int rho = row - (k0 + kb);
      const float l0 = lane < kb ? y0 * dinv[lane] : 0.f, l1 = lane + 32 < kb ? y1 * dinv[lane + 32] : 0.f;
      *reinterpret_cast<float*>(img.A + tf32_img_off(rho, lane, 128)) = y0;
      *reinterpret_cast<float*>(img.A + tf32_img_off(rho, lane + 32, 128)) = y1;
      *reinterpret_cast<float*>(img.B + tf32_img_off(rho, lane, 64)) = l0;
      *reinterpret_cast<float*>(img.B + tf32_img_off(rho, lane + 32, 64)) = l1;
    }
  }
}

// A launch with a scheduling priority (a launch attribute, so that it also
// holds for the kernel node when the launch is captured in a graph).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_prio(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                               int prio, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributePriority;
  attr[0].val.priority = prio;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// The diagonal block of nb matrices (with the pivot rule if it is on).
template <class T>
inline void launch_dense_diag(T* S, int n, int k0, int kb, int nb, int64_t bstride, const PivotRule& rule,
                              unsigned long long* counters, cudaStream_t st, int prio = 0) {
  launch_prio(rule.anorm ? k_dense_diag_t<T, true> : k_dense_diag_t<T, false>, dim3(nb), dim3(256), 0, st, prio, S, n,
              k0, kb, bstride, rule, counters);
}

// Rows below the diagonal block of nb matrices.  A thread per row issues the
// fewest instructions (no idle lanes) but its dependency chain is long (88 us
// in FP64, 14 in FP32); a warp per row has a 64-step chain.  FP64: 200 rows
// take 10.4 us with four warps per CTA, 12.4 with eight, 88 with a thread per
// row; 14,400 rows 92, 88 and 88; 57,600 rows 337, 328 and 229.  FP32: 4,096
// rows 12.3 us with a warp per row, 13.8 with a thread; 9,000 rows 16.5 and
// 14.4.
constexpr int kPanelRowsFour = 152 * 32;     // FP64: up to these rows, four warps per CTA
constexpr int kPanelRowsThread = 152 * 96;   // FP64: from these rows on, a thread per row
constexpr int kPanelRowsThreadF32 = 6144;    // FP32
template <class T>
inline void launch_dense_panel(T* S, T* Y, int n, int k0, int kb, int rend, int nb, int64_t bstride,
                               int64_t ystride, cudaStream_t st, int prio = 0, Tf32Images img = Tf32Images{}) {
  const int m = rend - k0 - kb;
  if (m <= 0) return;
  if constexpr (sizeof(T) == 4) {
    if ((int64_t)m * nb >= kPanelRowsThreadF32) {
      launch_prio(k_dense_panel_t<T, 128>, dim3((m + 127) / 128, nb), dim3(128), 0, st, prio, S, Y, n, k0, kb,
                  rend, bstride, ystride, img);
      return;
    }
  } else {
    if ((int64_t)m * nb >= kPanelRowsThread) {
      launch_prio(k_dense_panel_t<T, 32>, dim3((m + 31) / 32, nb), dim3(32), 0, st, prio, S, Y, n, k0, kb, rend,
                  bstride, ystride, img);
      return;
    }
  }
  if (sizeof(T) == 8 && (int64_t)m * nb <= kPanelRowsFour)
    launch_prio(k_dense_panel_w<T, 4>, dim3((m + 3) / 4, nb), dim3(128), 0, st, prio, S, Y, n, k0, kb, rend, bstride,
                ystride, img);
  else
    launch_prio(k_dense_panel_w<T, 8>, dim3((m + 7) / 8, nb), dim3(256), 0, st, prio, S, Y, n, k0, kb, rend, bstride,
                ystride, img);
}

// Trailing update of matrix blockIdx.y on the lower 16 x 16 tiles below the
// panel, one entry per thread: A[i][j] -= sum_c Y[i][c] L[j][c] for
// k0+kb <= j <= i < rend.  What bounds it: the FP64 pipe, at two multiply-adds
// per SM and cycle so narrow that two shared-memory loads per multiply-add hide
// behind it; register tiles buy nothing, and 64 x 64 tiles cost a narrow
// trailing matrix the chip (one such tile keeps its SM 63 us).  One matrix with
// 200 rows: 8 us (64 x 64 tiles: 78); 96 matrices with 800 rows, 3.9 GFLOP:
// 3.30 ms, 0.95 of the FP64 rate (3.78).
constexpr int kUpdTile = 16;

template <class T>
__global__ void __launch_bounds__(kUpdTile * kUpdTile)
    k_dense_update(T* __restrict__ S0, const T* __restrict__ Y0, int n, int k0, int kb, int rend,
                         int64_t bstride, int64_t ystride) {
  __shared__ T Ys[kPanelW][kUpdTile + 1];
  __shared__ T Ls[kPanelW][kUpdTile + 1];
  T* S = S0 + (int64_t)blockIdx.y * bstride;
  const T* Y = Y0 + (int64_t)blockIdx.y * ystride;
  const int base = k0 + kb;
  // tile (ti, tj), tj <= ti, of the packed lower triangle
  const int t = blockIdx.x;
  int ti = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  while (ti * (ti + 1) / 2 > t) ti--;
  while ((ti + 1) * (ti + 2) / 2 <= t) ti++;
  const int i0 = base + ti * kUpdTile, j0 = base + (t - ti * (ti + 1) / 2) * kUpdTile;
  const int r = threadIdx.x % kUpdTile, g = threadIdx.x / kUpdTile;
  T ys[kPanelW / kUpdTile], ls[kPanelW / kUpdTile];  // all loads first
#pragma unroll
  for (int u = 0; u < kPanelW / kUpdTile; u++) {
    const int c = g + u * kUpdTile;
    ys[u] = c < kb && i0 + r < rend ? Y[(i0 + r) + (int64_t)c * n] : T(0);
    ls[u] = c < kb && j0 + r < rend ? S[(j0 + r) + (int64_t)(k0 + c) * n] : T(0);
  }
  const int i = i0 + r, j = j0 + g;  // consecutive threads, consecutive rows
  const bool live = i < rend && j <= i;
  const T cur = live ? S[i + (int64_t)j * n] : T(0);
#pragma unroll
  for (int u = 0; u < kPanelW / kUpdTile; u++) {
    Ys[g + u * kUpdTile][r] = ys[u];
    Ls[g + u * kUpdTile][r] = ls[u];
  }
  __syncthreads();
  T acc = T(0);
  if (kb == kPanelW) {
#pragma unroll 16
    for (int c = 0; c < kPanelW; c++) acc += Ys[c][r] * Ls[c][g];
  } else {
    for (int c = 0; c < kb; c++) acc += Ys[c][r] * Ls[c][g];
  }
  if (live) S[i + (int64_t)j * n] = cur - acc;
}

template <class T>
inline void launch_dense_update(T* S, const T* Y, int n, int k0, int kb, int rend, int nb, int64_t bstride,
                                int64_t ystride, cudaStream_t st) {
  const int tiles = (rend - k0 - kb + kUpdTile - 1) / kUpdTile;
  k_dense_update<T><<<dim3(tiles * (tiles + 1) / 2, nb), kUpdTile * kUpdTile, 0, st>>>(S, Y, n, k0, kb, rend, bstride,
                                                                                       ystride);
}

}  // namespace

}  // namespace kkt
