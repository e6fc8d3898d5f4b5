// (c) Dense LDL^T of the Schur complement, S = L_s D_s L_s^T, and the solve
// S x_g = t (Algorithm 1; eqs. SCform and SCsolve).
//
// S is n x n, column-major, lower triangle.  Blocked right-looking, block
// width kDenseNB = 64, per block column k0:
//   diagonal block: LDL^T of the 64 x 64 block with rows in registers, and
//   panel: L21 = A21 L11^{-T} D1^{-1}, Y = L21 D1 kept for the update
//     (k_dense_diag_t / k_dense_panel_t in dense_kernels.cuh, shared with the
//     tensor-core modes and the dense tail of the block factors);
//   k_dense_update: A22 -= Y L21^T on the lower-triangle 16 x 16 tiles (FP64).
// No pivoting: S is positive definite when the blocks are quasidefinite and C
// is positive definite; a zero pivot is counted and reported.
#include <cooperative_groups.h>

#include "dense_kernels.cuh"

namespace kkt {

namespace cg = cooperative_groups;

namespace {

constexpr int NB = kDenseNB;

// forward substitution with unit lower L: diagonal block of one block column
__global__ void k_dense_fwd_diag(const double* __restrict__ S, double* __restrict__ x, int n, int k0) {
  const int kb = min(NB, n - k0);
  if (threadIdx.x != 0) return;
  for (int c = 0; c < kb; c++) {
    double v = x[k0 + c];
    for (int c2 = 0; c2 < c; c2++) v -= S[(k0 + c) + (int64_t)(k0 + c2) * n] * x[k0 + c2];
    x[k0 + c] = v;
  }
}

// x[i] -= sum_{c in block} L[i][c] x[c] for rows below the block
__global__ void k_dense_fwd_update(const double* __restrict__ S, double* __restrict__ x, int n, int k0) {
  const int kb = min(NB, n - k0);
  const int i = k0 + kb + blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double acc = 0.0;
  for (int c = 0; c < kb; c++) acc += S[i + (int64_t)(k0 + c) * n] * x[k0 + c];
  x[i] -= acc;
}

__global__ void k_dense_diag_scale(const double* __restrict__ S, double* __restrict__ x, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    x[i] /= S[i + (int64_t)i * n];
}

// dot[c] = sum_{i >= k0+kb} L[i][k0+c] x[i]
__global__ void k_dense_bwd_dot(const double* __restrict__ S, const double* __restrict__ x,
                                double* __restrict__ dot, int n, int k0) {
  const int kb = min(NB, n - k0);
  const int c = blockIdx.x;
  if (c >= kb) return;
  __shared__ double red[256];
  double acc = 0.0;
  const double* col = S + (int64_t)(k0 + c) * n;
  for (int i = k0 + kb + threadIdx.x; i < n; i += blockDim.x) acc += col[i] * x[i];
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) dot[c] = red[0];
}

__global__ void k_dense_bwd_diag(const double* __restrict__ S, double* __restrict__ x,
                                 const double* __restrict__ dot, int n, int k0) {
  const int kb = min(NB, n - k0);
  if (threadIdx.x != 0) return;
  for (int c = kb - 1; c >= 0; c--) {
    double v = x[k0 + c] - dot[c];
    for (int c2 = c + 1; c2 < kb; c2++) v -= S[(k0 + c2) + (int64_t)(k0 + c) * n] * x[k0 + c2];
    x[k0 + c] = v;
  }
}

// Inverses X_t = L_tt^{-1} of the unit lower 64 x 64 diagonal blocks of a
// factor (row-major per block, zero above the diagonal and outside the
// matrix) and the reciprocal pivots 1 / D.  With them each step of the block
// triangular solves applies its diagonal block as a product instead of a
// 64-step substitution.  Row i of X is e_i - sum_{k<i} L_ik X_k (right-looking
// over k, one barrier per k).
// Batched over blockIdx.y (matrix b at L0 + b * bstride with leading dimension
// ld, its inverses at X0 + b * xstride); dinv may be null.
template <class T>
__global__ void __launch_bounds__(256) k_diag_inverse(const T* __restrict__ L0, int n, int ld, int64_t bstride,
                                                      double* __restrict__ X0, int64_t xstride,
                                                      double* __restrict__ dinv) {
  extern __shared__ double dsm[];
  double(*Ls)[65] = reinterpret_cast<double(*)[65]>(dsm);
  double(*Xs)[65] = reinterpret_cast<double(*)[65]>(dsm + 64 * 65);
  const T* L = L0 + (int64_t)blockIdx.y * bstride;
  double* X = X0 + (int64_t)blockIdx.y * xstride;
  const int t = blockIdx.x, r0 = t * 64, rows = min(64, n - r0), tid = threadIdx.x;
  for (int q = tid; q < 64 * 64; q += blockDim.x) {
    const int c = q / 64, i = q - c * 64;
    Ls[i][c] = (i > c && i < rows) ? (double)L[(int64_t)(r0 + i) + (int64_t)(r0 + c) * ld] : 0.0;
    Xs[i][c] = (i == c && i < rows) ? 1.0 : 0.0;
  }
  if (dinv && tid < rows) dinv[r0 + tid] = 1.0 / (double)L[(int64_t)(r0 + tid) * (ld + 1)];
  __syncthreads();
  for (int k = 0; k + 1 < rows; k++) {
    const int cnt = (rows - 1 - k) * (k + 1);
    for (int q = tid; q < cnt; q += blockDim.x) {
      const int i = k + 1 + q / (k + 1), j = q % (k + 1);
      Xs[i][j] -= Ls[i][k] * Xs[k][j];
    }
    __syncthreads();
  }
  for (int q = tid; q < 64 * 64; q += blockDim.x) X[(int64_t)t * 4096 + q] = Xs[q / 64][q % 64];
}

// ---- pipelined triangular solves with a dense factor ----
//
// One launch per direction for the factor of S or for the dense tails of all
// blocks.  A cluster of four CTAs owns a 64-row block t, 16 rows each; clusters
// take the blocks in the order of an atomic ticket (all matrices' first block,
// then all second ones, ...), so that a cluster only ever waits for blocks of
// clusters that started before it.  A solution entry is its own flag: the
// vector the blocks publish in holds kUnset until an entry is stored, and every
// thread polls just the four entries it multiplies, so a block's hand-over
// costs one store and one load through L2, with no fence and no barrier.  Polls
// are bounded: a wait that runs out records a timeout instead of spinning on.
//
// What bounds them: the chain of blocks.  Per block the products with all
// earlier blocks but the last are done while waiting; the right-hand side that
// they leave is exchanged through distributed shared memory and multiplied with
// X_t = L_tt^{-1}.  FUSED (the factor of S, whose chain is long): the last one's
// product uses Z_t = X_t L_{t,t-1} (backward: X_t^T L_{t+1,t}^T), formed once per
// factor, so that nothing but one 64-wide product and its reduction lies between
// two hand-overs.  The tails have short chains and many matrices, for which Z
// would cost more than it saves.
// Measured (one right-hand side): S of order 9,600 by its envelope, FP64, 226 and
// 250 us per direction (900 and 1,266 with a flag and a fence per block, one CTA
// per block and both products in the chain); the dense FP32 factor 295 and 316
// us (851 and 1,156; 339 and 329 with sleeps of 2 us at most); 96 tails of order
// 724 117 and 109 us (211 and 157 with a cluster per tail that meets at a barrier
// per block), 24 tails of order 6,938 1.36 and 1.27 ms (4.9 and 3.4).
constexpr long long kSpinBudgetCycles = 4000000000LL;  // about 2 s at 2 GHz
constexpr unsigned long long kUnset = ~0ULL;           // a NaN no arithmetic gives
constexpr int kTrsvCluster = 4;                        // CTAs per 64-row block
constexpr int kTrsvRows = 64 / kTrsvCluster;           // rows per CTA

__device__ __forceinline__ unsigned long long ld_relaxed(const double* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void publish(double* p, double v) {
  unsigned long long b = (unsigned long long)__double_as_longlong(v);
  if (b == kUnset) b = 0x7ff8000000000000ULL;  // a NaN passed on from the input
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(b) : "memory");
}

// The four entries p[0], p[st], p[2 st], p[3 st] once all are published (those
// with index e + k st >= lim read as zero).  dist: blocks between this one and
// the awaited one; a distant wait sleeps between its polls, so that the blocks
// at the front of the chain have L2 to themselves.
__device__ __forceinline__ void poll4(const double* p, int st, int e, int lim, int dist, int* err, bool& dead,
                                      double (&y)[4]) {
  unsigned long long v[4];
  long long t0 = 0;
  for (int spin = 0;; spin++) {
    bool all = true;
#pragma unroll
    for (int k = 0; k < 4; k++) v[k] = e + k * st < lim ? ld_relaxed(p + k * st) : 0ULL;
#pragma unroll
    for (int k = 0; k < 4; k++) all = all && v[k] != kUnset;
    if (all || dead) break;
    if (spin == 0) t0 = clock64();
    if (dist > 2) __nanosleep(min(250 * (dist - 2), 10000));
    if ((spin & 63) == 63 && (clock64() - t0 > kSpinBudgetCycles || *((volatile int*)err) != 0)) {
      atomicExch(err, 1);
      dead = true;
    }
  }
#pragma unroll
  for (int k = 0; k < 4; k++) y[k] = __longlong_as_double((long long)v[k]);
}

// FORWARD: L y = in; else L^T x = D^{-1} in (dinv; null: no scaling).  Matrix b
// of the batch at L0 + b bstride (order n, leading dimension ld), its inverses
// X_t at X0 + b xstride, its vectors at in0 + b vstride and out0 + b vstride
// (out0 may be null), published in pub0 + b 64 nb.  jr: the envelope of S (first
// column block of row block t, or one past the last row block of column block
// t).  For an FP32 factor the products with L are formed in FP32 (x_j rounded to
// FP32) and added to the FP64 row sums once per block: the FP32 factor's own
// error is some 1e-4 relative, far above the 1e-7 of these products.
template <bool FORWARD, class T, bool FUSED>
__global__ void __cluster_dims__(kTrsvCluster, 1, 1) __launch_bounds__(256, 3)
    k_trsv(const T* __restrict__ L0, int n, int ld, int64_t bstride, int nbatch, const double* __restrict__ X0,
           int64_t xstride, const double* __restrict__ Z, const double* in0, double* out0, int64_t vstride,
           double* pub0, const double* __restrict__ dinv, const int* __restrict__ jr, unsigned* ticket, int* err) {
  __shared__ double rhs[64];  // the block's right-hand side, written by the whole cluster
  __shared__ double part[8][kTrsvRows], part2[8][kTrsvRows];
  __shared__ int s_tk;
  cg::cluster_group cluster = cg::this_cluster();
  const int q = (int)cluster.block_rank(), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nb = (n + 63) / 64;
  if (q == 0 && tid == 0) s_tk = ticket ? (int)(atomicAdd(ticket, 1u) + 1u) : (int)(blockIdx.x / kTrsvCluster);
  cluster.sync();  // every CTA of the cluster runs from here on
  const int tk = *cluster.map_shared_rank(&s_tk, 0);
  const int step = tk / nbatch, b = tk - step * nbatch, t = FORWARD ? step : nb - 1 - step;
  const int r0 = t * 64 + q * kTrsvRows;  // this CTA's first row
  const int rows = min(kTrsvRows, n - r0);  // may be <= 0 in a ragged last block
  const T* L = L0 + (int64_t)b * bstride;
  double* pub = pub0 + (int64_t)b * nb * 64;
  bool dead = false;
  // products with X and Z: row r of this CTA, columns 4 pid .. 4 pid + 3
  const int r = tid & 15, pid = tid >> 4;
  double xr[4], zr[4];
  const double* Xt = X0 + (int64_t)b * xstride + (int64_t)t * 4096;
  const int jn = FORWARD ? t - 1 : t + 1;
  const int jfar = FORWARD ? (jr ? jr[t] : 0) : (jr ? jr[t] : nb) - 1;  // farthest block with a product
  const bool any = FORWARD ? jfar <= jn : jfar >= jn;
#pragma unroll
  for (int k = 0; k < 4; k++) {
    const int c = 4 * pid + k, row = q * kTrsvRows + r;
    xr[k] = FORWARD ? Xt[row * 64 + c] : Xt[c * 64 + row];
    zr[k] = FUSED && any ? Z[((int64_t)(FORWARD ? 0 : nb) + t) * 4096 + row * 64 + c] : 0.0;
  }
  // products with L: own row (column, backward) of this CTA and four entries
  // e0 + k es of a block, so that neighbouring lanes read neighbouring entries
  const int own = FORWARD ? tid & 15 : tid >> 4, e0 = FORWARD ? 4 * (tid >> 4) : tid & 15, es = FORWARD ? 1 : 16;
  const bool live = own < rows;
  auto load = [&](int j, T(&v)[4]) {
#pragma unroll
    for (int k = 0; k < 4; k++) {
      const int e = j * 64 + e0 + k * es;
      v[k] = live && e < n ? (FORWARD ? L[(int64_t)(r0 + own) + (int64_t)e * ld] : L[(int64_t)e + (int64_t)(r0 + own) * ld])
                           : T(0);
    }
  };
  const int dj = FORWARD ? 1 : -1;
  const int nfar = any ? (FORWARD ? jn - jfar : jfar - jn) + (FUSED ? 0 : 1) : 0;
  double acc = 0.0;
  T lv[4];
  if (nfar > 0) load(jfar, lv);
  for (int u = 0; u < nfar; u++) {
    const int j = jfar + u * dj;
    T cur[4];
#pragma unroll
    for (int k = 0; k < 4; k++) cur[k] = lv[k];
    if (u + 1 < nfar) load(j + dj, lv);
    double y[4];
    const int e = j * 64 + e0;
    poll4(pub + e, es, e, n, FORWARD ? t - j : j - t, err, dead, y);
    if constexpr (sizeof(T) == 8) {
#pragma unroll
      for (int k = 0; k < 4; k++) acc += cur[k] * y[k];
    } else {
      T a = T(0);
#pragma unroll
      for (int k = 0; k < 4; k++) a += cur[k] * (T)y[k];
      acc += (double)a;
    }
  }
  const int64_t vo = (int64_t)b * vstride + r0;
  if (FORWARD) {
    acc += __shfl_xor_sync(0xffffffffu, acc, 16);
    if (lane < 16) part[warp][lane] = acc;
  } else {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((lane & 15) == 0) part[0][own] = acc;
  }
  __syncthreads();
  if (tid < kTrsvRows) {
    double v = 0.0;
    if (tid < rows) {
      v = in0[vo + tid];
      if (!FORWARD && dinv) v *= dinv[r0 + tid];
      if (FORWARD) {
#pragma unroll
        for (int w = 0; w < 8; w++) v -= part[w][tid];
      } else {
        v -= part[0][tid];
      }
    }
#pragma unroll
    for (int k = 0; k < kTrsvCluster; k++) cluster.map_shared_rank(rhs, k)[q * kTrsvRows + tid] = v;
  }
  cluster.sync();
  double a2 = 0.0;
#pragma unroll
  for (int k = 0; k < 4; k++) a2 += xr[k] * rhs[4 * pid + k];
  if (FUSED && any) {
    double y[4];
    const int e = jn * 64 + 4 * pid;
    poll4(pub + e, 1, e, n, 1, err, dead, y);
#pragma unroll
    for (int k = 0; k < 4; k++) a2 -= zr[k] * y[k];
  }
  a2 += __shfl_xor_sync(0xffffffffu, a2, 16);
  if (lane < 16) part2[warp][lane] = a2;
  __syncthreads();
  if (warp == 0) {
    const int h = (lane >> 4) * 4;
    double v = (part2[h][r] + part2[h + 1][r]) + (part2[h + 2][r] + part2[h + 3][r]);
    v += __shfl_xor_sync(0xffffffffu, v, 16);
    if (lane < rows && lane < kTrsvRows) {
      publish(pub + r0 + lane, v);
      if (out0) out0[vo + lane] = v;
    }
  }
}

// Z of the fused solves: block t, direction blockIdx.y, rows 16 blockIdx.z ..:
// forward Z_t = X_t L_{t,t-1}, backward Z_t = X_t^T L_{t+1,t}^T (X_t is lower
// triangular).
template <class T>
__global__ void __launch_bounds__(256) k_trsv_couple(const T* __restrict__ L, int n, const double* __restrict__ X,
                                                     double* __restrict__ Z) {
  __shared__ double Ls[64][65];  // [k][c]
  __shared__ double Xs[64][17];  // [k][row of this CTA]
  const int t = blockIdx.x, nb = gridDim.x, q = blockIdx.z, tid = threadIdx.x;
  const bool fwd = blockIdx.y == 0;
  const int hi = fwd ? t : t + 1;  // the block row of the off-diagonal block
  if (hi == 0 || hi >= nb) return;  // (a block outside the envelope of S is zero, and so is its product)
  const T* B = L + (int64_t)hi * 64 + (int64_t)(hi - 1) * 64 * n;
  const int rows = min(64, n - hi * 64);
  for (int p = tid; p < 4096; p += 256) {
    const int i = p & 63, j = p >> 6;  // entry (i, j) of the block
    const double v = i < rows ? (double)B[i + (int64_t)j * n] : 0.0;
    if (fwd) Ls[i][j] = v;
    else Ls[j][i] = v;
  }
  for (int p = tid; p < 1024; p += 256) {
    const int k = fwd ? p & 63 : p >> 4, i = fwd ? p >> 6 : p & 15;
    Xs[k][i] = fwd ? X[(int64_t)t * 4096 + (q * 16 + i) * 64 + k] : X[(int64_t)t * 4096 + k * 64 + q * 16 + i];
  }
  __syncthreads();
  const int c = tid & 63, g = (tid >> 6) * 4;
  const int k0 = fwd ? 0 : q * 16 + g, k1 = fwd ? q * 16 + g + 4 : 64;
  double acc[4] = {};
  for (int k = k0; k < k1; k++) {
    const double l = Ls[k][c];
#pragma unroll
    for (int i = 0; i < 4; i++) acc[i] += Xs[k][g + i] * l;
  }
#pragma unroll
  for (int i = 0; i < 4; i++) Z[((int64_t)blockIdx.y * nb + t) * 4096 + (q * 16 + g + i) * 64 + c] = acc[i];
}

}  // namespace

cudaError_t launch_dense_ldlt(Handle& h, unsigned long long* counters, cudaStream_t st) {
  const int n = h.nC;
  for (int k0 = 0; k0 < n; k0 += NB) {
    const int kb = std::min(NB, n - k0);
    const int rend = h.panel_rend.empty() ? n : h.panel_rend[k0 / NB];
    // diagonal block (rows in registers) and panel (warp per row), FP64
    cudaError_t e = launch_dense_diag_panel_f64(h, k0, kb, rend, counters, st);
    if (e != cudaSuccess) return e;
    const int rest = rend - k0 - kb;
    if (rest > 0) {
      const int kt = kt_begin(h, kFamDenseF64, update_flops(rest, 0, rest, kb), st);
      launch_dense_update<double>(h.S, h.Ypanel, n, k0, kb, rend, 1, 0, 0, st);
      kt_end(h, kt, st);
      h.launches++;
    }
  }
  cudaError_t e = cudaGetLastError();
  return e != cudaSuccess ? e : launch_diag_inverse(h, false, st);
}

namespace {

// x = S^{-1} t with the factor in type T; x may be t.
template <class T>
cudaError_t dense_solve_in(Handle& h, const T* L, const double* t, double* x, cudaStream_t st) {
  const int n = h.nC;
  if (n == 0) return cudaSuccess;
  const int nb = (n + NB - 1) / NB;
  double *y1 = h.trsv_s, *y2 = h.trsv_s + (int64_t)nb * 64;  // the vectors both directions publish in
  unsigned* ticket = nullptr;
  if (nb > 1) {  // one block waits for nothing: no flags, no tickets
    ticket = reinterpret_cast<unsigned*>(h.trsv_s + 2 * (int64_t)nb * 64);
    cudaError_t e = cudaMemsetAsync(h.trsv_s, 0xff, sizeof(double) * trsv_doubles(nb, 2), st);
    if (e != cudaSuccess) return e;
  }
  k_trsv<true, T, true><<<nb * kTrsvCluster, 256, 0, st>>>(L, n, n, 0, 1, h.Xinv, 0, h.Zs, t, nullptr, 0, y1, nullptr,
                                                           h.d.trsv_jlo, ticket, h.dev_err);
  k_trsv<false, T, true><<<nb * kTrsvCluster, 256, 0, st>>>(L, n, n, 0, 1, h.Xinv, 0, h.Zs, y1, x, 0, y2, h.Sdinv,
                                                            h.d.trsv_jhi, ticket ? ticket + 1 : nullptr, h.dev_err);
  h.launches += 2;
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_dense_solve(Handle& h, const double* t, double* x, cudaStream_t st) {
  return dense_solve_in<double>(h, h.S, t, x, st);
}

// x = S32^{-1} t with the FP32 factor of the TF32/BF16 modes (FP64 accumulation)
cudaError_t launch_dense_solve_f32(Handle& h, const double* t, double* x, cudaStream_t st) {
  return dense_solve_in<float>(h, h.S32, t, x, st);
}

// The triangular solves of the N dense tails, in place on zt (the tail's first
// entry of block 0; blocks nA apart).
cudaError_t launch_tail_trsv(Handle& h, bool forward, double* zt, cudaStream_t st) {
  const int nb = (h.nT + NB - 1) / NB;
  unsigned* ticket = nullptr;
  if (nb > 1) {
    ticket = reinterpret_cast<unsigned*>(h.trsv_t + (int64_t)h.N * nb * 64);
    cudaError_t e = cudaMemsetAsync(h.trsv_t, 0xff, sizeof(double) * trsv_doubles(h.N * nb, 1), st);
    if (e != cudaSuccess) return e;
  }
  const int64_t t2 = (int64_t)h.nTa * h.nTa, xs = (int64_t)nb * 4096;
  const int grid = h.N * nb * kTrsvCluster;
  if (forward)
    k_trsv<true, double, false><<<grid, 256, 0, st>>>(h.Tt, h.nT, h.nTa, t2, h.N, h.Xtail, xs, nullptr, zt, zt, h.nA,
                                                      h.trsv_t, nullptr, nullptr, ticket, h.dev_err);
  else
    k_trsv<false, double, false><<<grid, 256, 0, st>>>(h.Tt, h.nT, h.nTa, t2, h.N, h.Xtail, xs, nullptr, zt, zt, h.nA,
                                                       h.trsv_t, nullptr, nullptr, ticket, h.dev_err);
  h.launches++;
  return cudaGetLastError();
}

// Doubles of a publishing buffer: `vectors` vectors of 64 nb entries and the tickets.
int64_t trsv_doubles(int64_t nb, int vectors) { return (int64_t)vectors * nb * 64 + 2; }

cudaError_t launch_dense_solve_ws(Handle& h, const double* t, double* x, double* dot,
                                  cudaStream_t st) {
  const int n = h.nC;
  if (n == 0) return cudaSuccess;
  cudaError_t e = cudaMemcpyAsync(x, t, sizeof(double) * n, cudaMemcpyDeviceToDevice, st);
  if (e != cudaSuccess) return e;
  for (int k0 = 0; k0 < n; k0 += NB) {
    const int kb = std::min(NB, n - k0);
    k_dense_fwd_diag<<<1, 32, 0, st>>>(h.S, x, n, k0);
    h.launches++;
    const int rest = n - k0 - kb;
    if (rest > 0) {
      k_dense_fwd_update<<<(rest + 255) / 256, 256, 0, st>>>(h.S, x, n, k0);
      h.launches++;
    }
  }
  k_dense_diag_scale<<<(n + 255) / 256, 256, 0, st>>>(h.S, x, n);
  h.launches++;
  const int last = ((n - 1) / NB) * NB;
  for (int k0 = last; k0 >= 0; k0 -= NB) {
    k_dense_bwd_dot<<<NB, 256, 0, st>>>(h.S, x, dot, n, k0);
    k_dense_bwd_diag<<<1, 32, 0, st>>>(h.S, x, dot, n, k0);
    h.launches += 2;
  }
  return cudaGetLastError();
}

// The diagonal-block inverses and reciprocal pivots of the current factor of S
// (FP64 in S, or FP32 in S32), for the block triangular solves.
constexpr int kInvSmem = 2 * 64 * 65 * (int)sizeof(double);

// Kernel attributes set once (before any launch, outside stream capture).
cudaError_t dense_prepare() {
  cudaError_t e = cudaFuncSetAttribute(k_diag_inverse<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, kInvSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_diag_inverse<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, kInvSmem);
  return e;
}

cudaError_t launch_diag_inverse(Handle& h, bool f32, cudaStream_t st) {
  const int n = h.nC;
  if (n == 0) return cudaSuccess;
  const int nb = (n + NB - 1) / NB;
  const int smem = kInvSmem;
  if (f32) k_diag_inverse<float><<<nb, 256, smem, st>>>(h.S32, n, n, 0, h.Xinv, 0, h.Sdinv);
  else k_diag_inverse<double><<<nb, 256, smem, st>>>(h.S, n, n, 0, h.Xinv, 0, h.Sdinv);
  h.launches++;
  if (nb > 1) {
    if (f32) k_trsv_couple<float><<<dim3(nb, 2, 4), 256, 0, st>>>(h.S32, n, h.Xinv, h.Zs);
    else k_trsv_couple<double><<<dim3(nb, 2, 4), 256, 0, st>>>(h.S, n, h.Xinv, h.Zs);
    h.launches++;
  }
  return cudaGetLastError();
}

// The diagonal-block inverses of the N dense tails (order nT, leading
// dimension nTa), for the tail's block triangular solves.
cudaError_t launch_tail_inverse(Handle& h, cudaStream_t st) {
  const int nbT = (h.nT + NB - 1) / NB;
  const int smem = kInvSmem;
  k_diag_inverse<double><<<dim3(nbT, h.N), 256, smem, st>>>(h.Tt, h.nT, h.nTa, (int64_t)h.nTa * h.nTa, h.Xtail,
                                                           (int64_t)nbT * 4096, nullptr);
  h.launches++;
  return cudaGetLastError();
}

}  // namespace kkt
