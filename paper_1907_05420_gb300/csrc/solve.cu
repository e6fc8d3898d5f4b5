// (d) Local solves and the right-hand-side reduction (eqs. SCsolve and
// SCsolve1; Algorithm 1), plus the FP64 residual of the
// iterative refinement on the full K.
//
// One application of the factored K^{-1} to r = [r_0..r_{N-1}; r_g]:
//   z_i = L_i^{-1} P^T r_i                       (k_fsolve_lvl, level by level)
//   u_i = W_i^T D_i^{-1} z_i                     (k_reduce_u: E^T A_i^{-1} r_i)
//   t   = r_g - sum_i M_i^T u_i                  (k_reduce_t, block order)
//   x_g = S^{-1} t                               (dense solve)
//   z_i -= W_i (M_i x_g)                         (k_apply_xg: L^{-1} P^T B_i x_g)
//   x_i = P L_i^{-T} D_i^{-1} z_i                (k_diag_scale, k_bsolve_lvl)
// which is x_i = A_i^{-1} (r_i - B_i x_g).  Every output is summed by one thread
// or one warp in a fixed order.
#include "handle.h"

namespace kkt {

namespace {

__global__ void k_permute_in(const double* __restrict__ r, const int32_t* __restrict__ perm,
                             double* __restrict__ z, int nA, int N) {
  const int64_t total = (int64_t)nA * N;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = q / nA, kk = q - b * nA;
    z[q] = r[b * nA + perm[kk]];
  }
}

__global__ void k_permute_out(const double* __restrict__ z, const int32_t* __restrict__ perm,
                              double* __restrict__ x, int nA, int N) {
  const int64_t total = (int64_t)nA * N;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = q / nA, kk = q - b * nA;
    x[b * nA + perm[kk]] = z[q];
  }
}

// kkt_solve_noalloc's level solves, over every supernode (a dense tail's factor is
// in the panels too).  One warp per (supernode, block): z[cols(s)] -= sum_d
// L_d[rows in s] z[cols(d)]; then the unit-lower solve with the diagonal block.
__global__ void __launch_bounds__(128) k_fsolve_level(const int32_t* __restrict__ sn_list, int nsn,
                                                      DevSym d, const double* __restrict__ Lx,
                                                      int64_t pt, double* __restrict__ z, int nA,
                                                      int N) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (warp >= nsn * N) return;
  const int si = warp % nsn, b = warp / nsn;
  const int s = sn_list[si];
  const int m = (int)(d.sn_rowptr[s + 1] - d.sn_rowptr[s]);
  const int f = d.sn_first[s], w = d.sn_first[s + 1] - f;
  const double* P = Lx + b * pt + d.sn_valoff[s];
  double* zb = z + (int64_t)b * nA;
  for (int64_t u = d.upd_ptr[s]; u < d.upd_ptr[s + 1]; u++) {
    const int dd = d.upd_src[u];
    const int r0 = d.upd_r0[u], r1 = d.upd_r1[u];
    const int md = (int)(d.sn_rowptr[dd + 1] - d.sn_rowptr[dd]);
    const int fd = d.sn_first[dd], wd = d.sn_first[dd + 1] - fd;
    const double* Pd = Lx + b * pt + d.sn_valoff[dd];
    const int32_t* Rd = d.sn_rows + d.sn_rowptr[dd];
    const int j = r0 + lane;  // r1 - r0 <= w <= 32
    if (j < r1) {
      double acc = 0.0;
      for (int kk = 0; kk < wd; kk++) acc += Pd[(int64_t)kk * md + j] * zb[fd + kk];
      zb[Rd[j]] -= acc;
    }
    __syncwarp();
  }
  double zc = lane < w ? zb[f + lane] : 0.0;
  for (int c = 0; c + 1 < w; c++) {
    const double zcc = __shfl_sync(0xffffffffu, zc, c);
    if (lane > c && lane < w) zc -= P[(int64_t)c * m + lane] * zcc;
  }
  if (lane < w) zb[f + lane] = zc;
}

// Row j's products with the solution's entries in the descendants' columns:
// records p, p + step, ... below p1.
__device__ __forceinline__ double row_products(const RowRec* __restrict__ rec, int64_t p, int64_t p1, int step,
                                               const double* __restrict__ Lb, const double* zb) {
  double acc = 0.0;
  for (; p < p1; p += step) {
    const RowRec R = rec[p];
    const double* a = Lb + (R.off_wd >> 6);
    const double* v = zb + R.fd;
    const int wd = (int)(R.off_wd & 63);
#pragma unroll 4
    for (int k = 0; k < wd; k++) acc += a[(int64_t)k * R.md] * v[k];
  }
  return acc;
}

// One level of the forward solve.  The first small_ctas CTAs take the level's
// small supernodes (the first nsmall of the list), eight lanes per (supernode,
// block), lane = row: each walks its row's records, then they solve with the
// diagonal block by shuffles; the pairs of a warp are mostly blocks of one
// supernode.  The other CTAs take one (supernode, block) each: lane = row, the
// warps deal out the row's records, the partial sums are added in warp order and
// one warp solves with the diagonal block.
// What bounds it: latency, a few dependent loads per record.  A warp per small
// supernode leaves most lanes idle; one thread per small supernode walks all its
// rows one after the other (as slow).  All levels of the 2,383-bus grid, 96
// blocks: forward 0.25 ms (0.37 with a warp or CTA per supernode, 0.39 with a
// thread per small one), backward 0.23 (0.58 and 0.38).
constexpr int kSolveWarps = 8;

__global__ void __launch_bounds__(kSolveWarps * 32)
    k_fsolve_lvl(const SnDesc* __restrict__ sn, int nsmall, int nsn, int small_ctas, const int64_t* __restrict__ fr_ptr,
                 const RowRec* __restrict__ fr_rec, const double* __restrict__ Lx, int64_t pt, double* z, int nA, int N) {
  __shared__ double part[kSolveWarps][32];
  if ((int)blockIdx.x < small_ctas) {
    const int64_t q = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 3;
    const int c = threadIdx.x & 7;
    const bool live = q < (int64_t)nsmall * N;
    const int si = live ? (int)(q / N) : 0, b = live ? (int)(q - (int64_t)si * N) : 0;
    const SnDesc D = sn[si];
    const double* Lb = Lx + b * pt;
    const double* P = Lb + D.val;
    double* zb = z + (int64_t)b * nA;
    const bool row = live && c < D.w;
    double l[kSmallSnCols - 1], acc = 0.0;
#pragma unroll
    for (int k = 0; k + 1 < kSmallSnCols; k++) l[k] = row && k < c ? P[(int64_t)k * D.m + c] : 0.0;
    if (row) acc = zb[D.f + c] - row_products(fr_rec, fr_ptr[D.f + c], fr_ptr[D.f + c + 1], 1, Lb, zb);
#pragma unroll
    for (int k = 0; k + 1 < kSmallSnCols; k++) {
      const double y = __shfl_sync(0xffffffffu, acc, k, 8);
      if (row && k < c) acc -= l[k] * y;
    }
    if (row) zb[D.f + c] = acc;
    return;
  }
  const int pair = blockIdx.x - small_ctas, nbig = nsn - nsmall;
  const SnDesc D = sn[nsmall + pair % nbig];
  const int b = pair / nbig, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const double* Lb = Lx + b * pt;
  const double* P = Lb + D.val;
  double* zb = z + (int64_t)b * nA;
  part[warp][lane] = lane < D.w ? row_products(fr_rec, fr_ptr[D.f + lane] + warp, fr_ptr[D.f + lane + 1], kSolveWarps,
                                               Lb, zb)
                                : 0.0;
  __syncthreads();
  if (warp == 0) {
    double zc = 0.0;
    if (lane < D.w) {
      double sum = 0.0;
      for (int q = 0; q < kSolveWarps; q++) sum += part[q][lane];
      zc = zb[D.f + lane] - sum;
    }
    for (int c = 0; c + 1 < D.w; c++) {
      const double zcc = __shfl_sync(0xffffffffu, zc, c);
      if (lane > c && lane < D.w) zc -= P[(int64_t)c * D.m + lane] * zcc;
    }
    if (lane < D.w) zb[D.f + lane] = zc;
  }
}

// The tail's share of the forward solve: z_j -= sum over row j's records, four
// lanes per (tail row, block) that deal out the records.  96 tails of order 724:
// 65 us (209 with a CTA per (tail supernode, block) that routed the products to
// their rows by shuffles, 102 with one lane).
__global__ void __launch_bounds__(128)
    k_tail_fgather(const int64_t* __restrict__ fr_ptr, const RowRec* __restrict__ fr_rec, const double* __restrict__ Lx,
                   int64_t pt, double* z, int nA, int tail_col, int nT, int N) {
  const int64_t q = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 2;
  const bool live = q < (int64_t)nT * N;
  const int j = tail_col + (live ? (int)(q / N) : 0), b = live ? (int)(q % N) : 0, l = threadIdx.x & 3;
  double* zb = z + (int64_t)b * nA;
  double acc = live ? row_products(fr_rec, fr_ptr[j] + l, fr_ptr[j + 1], 4, Lx + b * pt, zb) : 0.0;
  acc += __shfl_xor_sync(0xffffffffu, acc, 1);
  acc += __shfl_xor_sync(0xffffffffu, acc, 2);
  if (live && l == 0) zb[j] -= acc;
}

// One level of the backward solve, split as the forward one: eight lanes per
// small (supernode, block), lane = column; else a CTA per pair, warp w on the
// columns c = w mod 8, up to four of them together so that each x is gathered
// once.
__global__ void __launch_bounds__(kSolveWarps * 32)
    k_bsolve_lvl(const SnDesc* __restrict__ sn, int nsmall, int nsn, int small_ctas, const int32_t* __restrict__ sn_rows,
                 const double* __restrict__ Lx, int64_t pt, double* z, int nA, int N) {
  __shared__ double dots[32];
  if ((int)blockIdx.x < small_ctas) {
    const int64_t q = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 3;
    const int c = threadIdx.x & 7;
    const bool live = q < (int64_t)nsmall * N;
    const int si = live ? (int)(q / N) : 0, b = live ? (int)(q - (int64_t)si * N) : 0;
    const SnDesc D = sn[si];
    const int32_t* R = sn_rows + D.rows;
    double* zb = z + (int64_t)b * nA;
    const bool col = live && c < D.w;
    const double* P = Lx + b * pt + D.val + (int64_t)(col ? c : 0) * D.m;  // this lane's column
    double l[kSmallSnCols], x = col ? zb[D.f + c] : 0.0;
#pragma unroll
    for (int k = 1; k < kSmallSnCols; k++) l[k] = col && c < k && k < D.w ? P[k] : 0.0;
    if (col) {
#pragma unroll 8
      for (int r = D.w; r < D.m; r++) x -= P[r] * zb[R[r]];
    }
#pragma unroll
    for (int k = kSmallSnCols - 1; k > 0; k--) {
      const double xk = __shfl_sync(0xffffffffu, x, k, 8);
      if (c < k && k < D.w) x -= l[k] * xk;
    }
    if (col) zb[D.f + c] = x;
    return;
  }
  const int pair = blockIdx.x - small_ctas, nbig = nsn - nsmall;
  const SnDesc D = sn[nsmall + pair % nbig];
  const int b = pair / nbig, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const double* P = Lx + b * pt + D.val;
  const int32_t* R = sn_rows + D.rows;
  double* zb = z + (int64_t)b * nA;
  double acc[4] = {};
  if (warp < D.w) {
#pragma unroll 4
    for (int r = D.w + lane; r < D.m; r += 32) {
      const double xr = zb[R[r]];
#pragma unroll
      for (int u = 0; u < 4; u++)
        if (warp + u * kSolveWarps < D.w) acc[u] += P[(int64_t)(warp + u * kSolveWarps) * D.m + r] * xr;
    }
#pragma unroll
    for (int u = 0; u < 4; u++) {
      if (warp + u * kSolveWarps < D.w) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], o);
        if (lane == 0) dots[warp + u * kSolveWarps] = acc[u];
      }
    }
  }
  __syncthreads();
  if (warp == 0) {
    double mine = lane < D.w ? zb[D.f + lane] - dots[lane] : 0.0;
    for (int c = D.w - 1; c >= 0; c--) {
      const double xc = __shfl_sync(0xffffffffu, mine, c);
      if (lane < c) mine -= P[(int64_t)lane * D.m + c] * xc;
    }
    if (lane < D.w) zb[D.f + lane] = mine;
  }
}

// z /= D (D from the panel diagonals)
__global__ void k_diag_scale(const int64_t* __restrict__ col_dpos, const double* __restrict__ Lx,
                             int64_t pt, double* __restrict__ z, int nA, int N) {
  const int64_t total = (int64_t)nA * N;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = q / nA, j = q - b * nA;
    z[q] /= Lx[b * pt + col_dpos[j]];
  }
}

// one warp per (supernode, block), top-down:
// x[cols(s)] = L_ss^{-T} (y[cols(s)] - L_off^T x[offrows(s)])
__global__ void __launch_bounds__(128) k_bsolve_level(const int32_t* __restrict__ sn_list, int nsn,
                                                      DevSym d, const double* __restrict__ Lx,
                                                      int64_t pt, double* __restrict__ z, int nA,
                                                      int N) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (warp >= nsn * N) return;
  const int si = warp % nsn, b = warp / nsn;
  const int s = sn_list[si];
  const int m = (int)(d.sn_rowptr[s + 1] - d.sn_rowptr[s]);
  const int f = d.sn_first[s], w = d.sn_first[s + 1] - f;
  const double* P = Lx + b * pt + d.sn_valoff[s];
  const int32_t* R = d.sn_rows + d.sn_rowptr[s];
  double* zb = z + (int64_t)b * nA;
  double mine = lane < w ? zb[f + lane] : 0.0;
  for (int c = 0; c < w; c++) {
    const double* col = P + (int64_t)c * m;
    double acc = 0.0;
    for (int r = w + lane; r < m; r += 32) acc += col[r] * zb[R[r]];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == c) mine -= acc;
  }
  for (int c = w - 1; c >= 0; c--) {
    const double xc = __shfl_sync(0xffffffffu, mine, c);
    if (lane < c) mine -= P[(int64_t)lane * m + c] * xc;
  }
  if (lane < w) zb[f + lane] = mine;
}

// u_b[t] = sum_rho W_b[rho][t] z_b[w_col[rho]] / D[rho]; one CTA per (block,
// 32 columns).  The rows of the augmented tail (from row nd on) are dense: their
// z / D is staged in shared memory kReduceRows rows at a time, and warp w sums the
// rows w mod 16.  The rows before them carry a few columns each: every lane walks
// its column's list, the warps dealing out the entries.  The 16 partials are
// added in warp order.  96 blocks, 2,579 rows of 100 columns: 35 us (150 over
// the dense rows and columns of all W; 52 with z / D formed by every lane).
constexpr int kReduceWarps = 16, kReduceRows = 1024;

__global__ void __launch_bounds__(32 * kReduceWarps) k_reduce_u(const double* __restrict__ W, const double* __restrict__ z,
                                                  const double* __restrict__ wdinv,
                                                  const int32_t* __restrict__ w_col, const int32_t* __restrict__ wr_ptr,
                                                  const int32_t* __restrict__ wr_row, int nd, int nw, int k, int nA,
                                                  double* __restrict__ u) {
  __shared__ double part[kReduceWarps][32];
  __shared__ double zd[kReduceRows];
  const int b = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = blockIdx.x * 32 + lane;
  const double* Wb = W + (int64_t)b * nw * k;
  const double* zb = z + (int64_t)b * nA;
  const double* db = wdinv + (int64_t)b * nw;
  double acc = 0.0;
  if (t < k) {
    const int p1 = wr_ptr[t + 1];
    for (int p = wr_ptr[t] + warp; p < p1; p += kReduceWarps) {
      const int rho = wr_row[p];
      acc += Wb[(int64_t)rho * k + t] * (zb[w_col[rho]] * db[rho]);
    }
  }
  for (int r0 = nd; r0 < nw; r0 += kReduceRows) {
    const int rows = min(kReduceRows, nw - r0);
    __syncthreads();
    for (int r = threadIdx.x; r < rows; r += blockDim.x) zd[r] = zb[w_col[r0 + r]] * db[r0 + r];
    __syncthreads();
    if (t < k) {
      const double* Wr = Wb + (int64_t)r0 * k + t;
#pragma unroll 8
      for (int r = warp; r < rows; r += kReduceWarps) acc += Wr[(int64_t)r * k] * zd[r];
    }
  }
  part[warp][lane] = acc;
  __syncthreads();
  if (warp == 0 && t < k) {
    double sum = 0.0;
    for (int q = 0; q < kReduceWarps; q++) sum += part[q][lane];
    u[(int64_t)b * k + t] = sum;
  }
}

// The kernels over the coupling columns take LANES lanes per column: 32 where a
// column has many entries (SCOPF: hundreds, and a dense C; coupling_lanes), one
// where it has two.  The lanes add up in a fixed order.
template <int LANES>
__device__ __forceinline__ double lanes_sum(double v) {
#pragma unroll
  for (int o = LANES / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// t[c] = r_g[c] - sum_{e in column c} b[e] u[block(e)][t(e)]
template <int LANES>
__global__ void k_reduce_t(const double* __restrict__ rg, const int32_t* __restrict__ t_ptr,
                           const int32_t* __restrict__ t_e, const int32_t* __restrict__ e_t,
                           const int32_t* __restrict__ e_block, const double* __restrict__ b_vals,
                           const double* __restrict__ u, int k, int nC, double* __restrict__ tg) {
  const int c = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / LANES), l = threadIdx.x % LANES;
  double acc = 0.0;
  if (c < nC)
    for (int q = t_ptr[c] + l; q < t_ptr[c + 1]; q += LANES) {
      const int e = t_e[q];
      acc += b_vals[e] * u[(int64_t)e_block[e] * k + e_t[e]];
    }
  acc = lanes_sum<LANES>(acc);
  if (c < nC && l == 0) tg[c] = rg[c] - acc;
}

// v_b[t] = sum_{e in block b, index t} b[e] x_g[col(e)]
__global__ void k_mx(const int32_t* __restrict__ bt_ptr, const int32_t* __restrict__ b_col,
                     const double* __restrict__ b_vals, const double* __restrict__ xg, int k, int N,
                     double* __restrict__ v) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= k * N) return;
  const int b = q / k, t = q - b * k;
  const int32_t* bp = bt_ptr + (int64_t)b * (k + 1);
  double acc = 0.0;
  for (int e = bp[t]; e < bp[t + 1]; e++) acc += b_vals[e] * xg[b_col[e]];
  v[q] = acc;
}

// z_b[w_col[rho]] -= sum_t W_b[rho][t] v_b[t], eight lanes per row: over all
// columns for the rows of the augmented tail (from row nd on), over the columns
// of the row's supernode for the others.  96 blocks, 2,579 rows of 100 columns:
// 37 us (68 with a thread per row over all columns), 17 of 2,258 rows of 1,632
// columns 49 (243).
__global__ void __launch_bounds__(256)
    k_apply_xg(const double* __restrict__ W, const double* __restrict__ v, const int32_t* __restrict__ w_col,
               const int32_t* __restrict__ w_sn, const int32_t* __restrict__ wt_ptr, const int32_t* __restrict__ wt_idx,
               int nd, int nw, int k, int nA, int N, double* __restrict__ z) {
  const int64_t q = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 3;
  const int l = threadIdx.x & 7;
  const bool live = q < (int64_t)nw * N;
  const int b = live ? (int)(q / nw) : 0, rho = live ? (int)(q - (int64_t)b * nw) : 0;
  const double* Wr = W + ((int64_t)b * nw + rho) * k;
  const double* vb = v + (int64_t)b * k;
  double acc = 0.0;
  if (live && rho >= nd) {
#pragma unroll 8
    for (int t = l; t < k; t += 8) acc += Wr[t] * vb[t];
  } else if (live) {
    const int s = w_sn[rho], e1 = wt_ptr[s + 1];
    for (int e = wt_ptr[s] + l; e < e1; e += 8) acc += Wr[wt_idx[e]] * vb[wt_idx[e]];
  }
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (live && l == 0) z[(int64_t)b * nA + w_col[rho]] -= acc;
}

// ---- residual rho = r - K x ----

__global__ void k_resid_blocks(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                               const int32_t* __restrict__ src, const double* __restrict__ a_vals,
                               int64_t nnzA, const double* __restrict__ r, const double* __restrict__ x,
                               double* __restrict__ rho, int nA, int N) {
  const int64_t total = (int64_t)nA * N;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = q / nA;
    const int row = (int)(q - b * nA);
    const double* a = a_vals + b * nnzA;
    const double* xb = x + b * nA;
    double acc = 0.0;
    for (int p = rowptr[row]; p < rowptr[row + 1]; p++) acc += a[src[p]] * xb[col[p]];
    rho[q] = r[q] - acc;
  }
}

// rows of E: subtract B_i x_g
__global__ void k_resid_b(const int32_t* __restrict__ bt_ptr, const int32_t* __restrict__ b_row,
                          const int32_t* __restrict__ b_col, const double* __restrict__ b_vals,
                          const double* __restrict__ xg, int k, int nA, int N,
                          double* __restrict__ rho) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= k * N) return;
  const int b = q / k, t = q - b * k;
  const int32_t* bp = bt_ptr + (int64_t)b * (k + 1);
  if (bp[t] == bp[t + 1]) return;
  double acc = 0.0;
  for (int e = bp[t]; e < bp[t + 1]; e++) acc += b_vals[e] * xg[b_col[e]];
  rho[(int64_t)b * nA + b_row[bp[t]]] -= acc;
}

// coupling rows: rho_g = r_g - sum_i B_i^T x_i - C x_g
template <int LANES>
__global__ void k_resid_g(const int32_t* __restrict__ t_ptr, const int32_t* __restrict__ t_e,
                          const int32_t* __restrict__ e_block, const int32_t* __restrict__ b_row,
                          const double* __restrict__ b_vals, const double* __restrict__ c_vals,
                          int c_kind, const double* __restrict__ r, const double* __restrict__ x,
                          int nA, int N, int nC, double* __restrict__ rho) {
  const int c = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / LANES), l = threadIdx.x % LANES;
  const int64_t g = (int64_t)N * nA;
  double acc = 0.0;
  if (c < nC) {
    for (int q = t_ptr[c] + l; q < t_ptr[c + 1]; q += LANES) {
      const int e = t_e[q];
      acc += b_vals[e] * x[(int64_t)e_block[e] * nA + b_row[e]];
    }
    if (c_kind == 0) {
      if (l == 0) acc += c_vals[c] * x[g + c];
    } else {
      for (int c2 = l; c2 < nC; c2 += LANES) {
        const double cv = c2 <= c ? c_vals[(int64_t)c * nC + c2] : c_vals[(int64_t)c2 * nC + c];
        acc += cv * x[g + c2];
      }
    }
  }
  acc = lanes_sum<LANES>(acc);
  if (c < nC && l == 0) rho[g + c] = r[g + c] - acc;
}

__device__ __forceinline__ void atomic_max_nonneg(double* addr, double v) {
  // non-negative doubles order like their bit patterns; a NaN with a clear
  // sign bit orders above +Inf, so it survives the maximum
  atomicMax(reinterpret_cast<unsigned long long*>(addr), (unsigned long long)__double_as_longlong(v));
}

// max(a, b) that keeps a NaN of either argument (fmax drops it), so that a
// non-finite entry reaches the norm and the convergence test sees it
__device__ __forceinline__ double max_keep_nan(double a, double b) { return (a > b || a != a) ? a : b; }

// red[0] = ||a||_inf, red[1] = ||b||_inf, red[2] = ||c||_inf; NaN if an entry is NaN
__global__ void k_norms3(const double* __restrict__ a, const double* __restrict__ b,
                         const double* __restrict__ c, int64_t n, double* __restrict__ red) {
  __shared__ double sh[3][256];
  double m0 = 0, m1 = 0, m2 = 0;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n;
       q += (int64_t)gridDim.x * blockDim.x) {
    m0 = max_keep_nan(m0, fabs(a[q]));
    m1 = max_keep_nan(m1, fabs(b[q]));
    m2 = max_keep_nan(m2, fabs(c[q]));
  }
  sh[0][threadIdx.x] = m0;
  sh[1][threadIdx.x] = m1;
  sh[2][threadIdx.x] = m2;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s)
      for (int k = 0; k < 3; k++) sh[k][threadIdx.x] = max_keep_nan(sh[k][threadIdx.x], sh[k][threadIdx.x + s]);
    __syncthreads();
  }
  if (threadIdx.x == 0)
    for (int k = 0; k < 3; k++) atomic_max_nonneg(&red[k], sh[k][0]);
}

// The CTA's maximum of m (NaN kept) into *out with one atomic: one per thread
// on the same address took 416 us for a million rows, one per CTA 76.
__device__ __forceinline__ void block_max_to(double* out, double m) {
  __shared__ double sh[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max_keep_nan(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x < 32) {
    m = threadIdx.x < blockDim.x / 32 ? sh[threadIdx.x] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max_keep_nan(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (threadIdx.x == 0) atomic_max_nonneg(out, m);
  }
}

// What kkt_solve's convergence test reads, straight into pinned host memory (one
// launch instead of a copy for each).
__global__ void k_publish(const double* __restrict__ red, const double* __restrict__ knorm,
                          const int* __restrict__ dev_err, const int* __restrict__ cum_err, double* host) {
  const int l = threadIdx.x;
  if (l < 3) host[l] = red[l];
  if (l == 3) host[3] = knorm[0];
  if (l == 4) *reinterpret_cast<int*>(host + 4) = *dev_err;
  if (l == 5) *reinterpret_cast<int*>(host + 5) = cum_err ? *cum_err : 0;
}

// ||K||_inf: row sums of |K| (NaN if an entry of A or B is NaN)
__global__ void k_knorm_blocks(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ src,
                               const double* __restrict__ a_vals, int64_t nnzA,
                               const int32_t* __restrict__ bt_ptr, const int32_t* __restrict__ b_row,
                               const double* __restrict__ b_vals, const int32_t* __restrict__ E,
                               int k, int nA, int N, double* __restrict__ out) {
  const int64_t total = (int64_t)nA * N;
  double m = 0.0;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = q / nA;
    const int row = (int)(q - b * nA);
    const double* a = a_vals + b * nnzA;
    double acc = 0.0;
    for (int p = rowptr[row]; p < rowptr[row + 1]; p++) acc += fabs(a[src[p]]);
    m = max_keep_nan(m, acc);
  }
  // rows of E also carry B's entries
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < (int64_t)k * N;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int b = (int)(q / k), t = (int)(q - (int64_t)b * k);
    const int32_t* bp = bt_ptr + (int64_t)b * (k + 1);
    if (bp[t] == bp[t + 1]) continue;
    const double* a = a_vals + (int64_t)b * nnzA;
    const int row = E[t];
    double acc = 0.0;
    for (int p = rowptr[row]; p < rowptr[row + 1]; p++) acc += fabs(a[src[p]]);
    for (int e = bp[t]; e < bp[t + 1]; e++) acc += fabs(b_vals[e]);
    m = max_keep_nan(m, acc);
  }
  block_max_to(out, m);
}

template <int LANES>
__global__ void k_knorm_g(const int32_t* __restrict__ t_ptr, const int32_t* __restrict__ t_e,
                          const double* __restrict__ b_vals, const double* __restrict__ c_vals,
                          int c_kind, int nC, double* __restrict__ out) {
  const int c = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / LANES), l = threadIdx.x % LANES;
  double acc = 0.0;
  if (c < nC) {
    for (int q = t_ptr[c] + l; q < t_ptr[c + 1]; q += LANES) acc += fabs(b_vals[t_e[q]]);
    if (c_kind == 0) {
      if (l == 0) acc += fabs(c_vals[c]);
    } else {
      for (int c2 = l; c2 < nC; c2 += LANES)
        acc += fabs(c2 <= c ? c_vals[(int64_t)c * nC + c2] : c_vals[(int64_t)c2 * nC + c]);
    }
  }
  block_max_to(out, lanes_sum<LANES>(acc));
}

__global__ void k_axpy(double* __restrict__ y, const double* __restrict__ x, int64_t n) {
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n;
       q += (int64_t)gridDim.x * blockDim.x)
    y[q] += x[q];
}

// Deterministic dot products (a fixed reduction order for a given n): each
// of kDotBlocks CTAs sums a strided part of the vectors in a fixed order and
// reduces it by a tree; one CTA adds the partial sums by a tree.
constexpr int kDotBlocks = 512;

__global__ void __launch_bounds__(256) k_dot_partial(const double* __restrict__ a, const double* __restrict__ b,
                                                     int64_t n, double* __restrict__ partial) {
  __shared__ double sh[256];
  double acc = 0.0;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x)
    acc += a[q] * b[q];
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[blockIdx.x] = sh[0];
}

__global__ void __launch_bounds__(kDotBlocks) k_dot_final(const double* __restrict__ partial, double* __restrict__ out) {
  __shared__ double sh[kDotBlocks];
  sh[threadIdx.x] = partial[threadIdx.x];
  __syncthreads();
  for (int s = kDotBlocks / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[0] = sh[0];
}

// y += a x
__global__ void k_axpby(double* __restrict__ y, double a, const double* __restrict__ x, int64_t n) {
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x)
    y[q] += a * x[q];
}

// y = a x
__global__ void k_scale_into(double* __restrict__ y, double a, const double* __restrict__ x, int64_t n) {
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x)
    y[q] = a * x[q];
}

// Lanes per coupling column: a warp from 16 entries per column on, and for a
// dense C (a row of nC entries).  1,021 buses with 16 outages (304 columns of some
// 121 entries): t 13 us (214 with a thread per column), the residual's coupling
// rows 14 (204), their norm 9 (101).  A solve of the cumulative coupling on 200
// buses, a thread and a warp per column: 211 and 207 us with 9 entries, 231 and 218
// with 17, 331 and 289 with 49; with the two of the adjacent coupling the same to
// 0.5%, where a thread keeps the launches small.
inline int coupling_lanes(const Handle& h) { return h.c_kind == 1 || h.nnzB >= 16 * (int64_t)h.nC ? 32 : 1; }
inline int coupling_grid(const Handle& h) { return (int)(((int64_t)h.nC * coupling_lanes(h) + 255) / 256); }

// CTAs of one level of the block solves: the small supernodes, then one per
// (other supernode, block).
struct LevelGrid {
  int first, nsn, nsmall, small_ctas, ctas;
};

inline LevelGrid level_grid(const Handle& h, int l) {
  LevelGrid g;
  g.first = h.flvl_ptr[l];
  g.nsn = h.flvl_ptr[l + 1] - g.first;
  g.nsmall = h.flvl_small[l];
  g.small_ctas = (int)(((int64_t)g.nsmall * h.N * 8 + kSolveWarps * 32 - 1) / (kSolveWarps * 32));
  g.ctas = g.small_ctas + (g.nsn - g.nsmall) * h.N;
  return g;
}

inline int grid_for(int64_t n, int bs = 256) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((n + bs - 1) / bs, 152 * 16));
}

}  // namespace

// The application is split where it first needs the factor of S: the front
// (forward block solves and right-hand-side reduction) needs only the block
// factors and W; the back does the rest.
cudaError_t launch_apply_front(Handle& h, const double* r, cudaStream_t st) {
  const int nA = h.nA, N = h.N, k = h.cpl.k, nw = h.cpl.nw;
  const int64_t pt = h.sym.panel_total;
  const int64_t nb = (int64_t)nA * N;
  {
    k_permute_in<<<grid_for(nb), 256, 0, st>>>(r, h.d.perm, h.z, nA, N);
    h.launches++;
  }
  // with a dense tail, the levels cover the supernodes outside it and the
  // tail's triangular solves are dense (the tail factor's triangles)
  const bool tail = h.nT > 0;
  for (int l = 0; l < h.sym.nlevels; l++) {
    const LevelGrid g = level_grid(h, l);
    if (g.ctas == 0) continue;
    k_fsolve_lvl<<<g.ctas, kSolveWarps * 32, 0, st>>>(h.d.flvl_desc + g.first, g.nsmall, g.nsn, g.small_ctas,
                                                      h.d.fr_ptr, h.d.fr_rec, h.Lx, pt, h.z, nA, N);
    h.launches++;
  }
  if (tail) {
    cudaError_t e = launch_tail_fsolve(h, h.z, st);
    if (e != cudaSuccess) return e;
  }
  if (h.nC > 0) {
    if (k > 0 && nw > 0) {
      dim3 g((k + 31) / 32, N);
      {
    k_reduce_u<<<g, 32 * kReduceWarps, 0, st>>>(h.W, h.z, h.wdinv, h.d.w_col, h.d.wr_ptr, h.d.wr_row, h.nw_nt, nw, k,
                                                nA, h.u);
    h.launches++;
  }
    } else if (k > 0) {
      cudaMemsetAsync(h.u, 0, sizeof(double) * (size_t)k * N, st);
    }
    {
    (coupling_lanes(h) == 32 ? k_reduce_t<32> : k_reduce_t<1>)<<<coupling_grid(h), 256, 0, st>>>(
        r + nb, h.d.t_ptr, h.d.t_e, h.d.e_t, h.d.e_block, h.b_vals, h.u, k, h.nC, h.tg);
    h.launches++;
  }
  }
  return cudaGetLastError();
}

cudaError_t launch_apply_back(Handle& h, double* out, cudaStream_t st, bool solve_s) {
  const int nA = h.nA, N = h.N, k = h.cpl.k, nw = h.cpl.nw;
  const int64_t pt = h.sym.panel_total;
  const int64_t nb = (int64_t)nA * N;
  const bool tail = h.nT > 0;
  if (h.nC > 0) {
    // without solve_s, h.xg already holds x_g (a sharded solve's broadcast)
    cudaError_t e = !solve_s ? cudaSuccess
                    : h.cum     ? launch_cum_solve(h, h.tg, h.xg, st)
                    : (h.s_factor == 1 ? launch_dense_solve_f32(h, h.tg, h.xg, st)
                                       : launch_dense_solve(h, h.tg, h.xg, st));
    if (e != cudaSuccess) return e;
    if (k > 0 && nw > 0) {
      {
    k_mx<<<(k * N + 255) / 256, 256, 0, st>>>(h.d.bt_ptr, h.d.b_col, h.b_vals, h.xg, k, N, h.v);
    h.launches++;
  }
      {
    k_apply_xg<<<(int)(((int64_t)nw * N * 8 + 255) / 256), 256, 0, st>>>(
        h.W, h.v, h.d.w_col, h.d.w_sn, h.d.wt_ptr, h.d.wt_idx, h.nw_nt, nw, k, nA, N, h.z);
    h.launches++;
  }
    }
  }
  {
    k_diag_scale<<<grid_for(nb), 256, 0, st>>>(h.d.col_dpos, h.Lx, pt, h.z, nA, N);
    h.launches++;
  }
  if (tail) {
    cudaError_t e = launch_tail_bsolve(h, h.z, st);
    if (e != cudaSuccess) return e;
  }
  for (int l = h.sym.nlevels - 1; l >= 0; l--) {
    const LevelGrid g = level_grid(h, l);
    if (g.ctas == 0) continue;
    k_bsolve_lvl<<<g.ctas, kSolveWarps * 32, 0, st>>>(h.d.flvl_desc + g.first, g.nsmall, g.nsn, g.small_ctas,
                                                      h.d.sn_rows, h.Lx, pt, h.z, nA, N);
    h.launches++;
  }
  {
    k_permute_out<<<grid_for(nb), 256, 0, st>>>(h.z, h.d.perm, out, nA, N);
    h.launches++;
  }
  if (h.nC > 0)
    cudaMemcpyAsync(out + nb, h.xg, sizeof(double) * h.nC, cudaMemcpyDeviceToDevice, st);
  return cudaGetLastError();
}

// The tail's share of the forward solve and its dense triangular solves.
cudaError_t launch_tail_fsolve(Handle& h, double* z, cudaStream_t st) {
  k_tail_fgather<<<(int)(((int64_t)h.nT * h.N * 4 + 127) / 128), 128, 0, st>>>(
      h.d.fr_ptr, h.d.fr_rec, h.Lx, h.sym.panel_total, z, h.nA, h.sym.tail_col, h.nT, h.N);
  h.launches++;
  cudaError_t e = cudaGetLastError();
  return e != cudaSuccess ? e : launch_tail_trsv(h, true, z + h.sym.tail_col, st);
}

cudaError_t launch_tail_bsolve(Handle& h, double* z, cudaStream_t st) {
  return launch_tail_trsv(h, false, z + h.sym.tail_col, st);
}

cudaError_t launch_apply_inverse(Handle& h, const double* r, double* out, cudaStream_t st) {
  cudaError_t e = launch_apply_front(h, r, st);
  return e != cudaSuccess ? e : launch_apply_back(h, out, st);
}

cudaError_t launch_residual(Handle& h, const double* r, const double* x, double* rho, cudaStream_t st) {
  const int nA = h.nA, N = h.N, k = h.cpl.k;
  const int64_t nb = (int64_t)nA * N;
  {
    k_resid_blocks<<<grid_for(nb), 256, 0, st>>>(h.d.full_rowptr, h.d.full_col, h.d.full_src, h.a_vals,
                                               h.nnzA, r, x, rho, nA, N);
    h.launches++;
  }
  if (h.nC > 0) {
    if (k > 0)
      {
    k_resid_b<<<(k * N + 255) / 256, 256, 0, st>>>(h.d.bt_ptr, h.d.b_row, h.d.b_col, h.b_vals,
                                                     x + nb, k, nA, N, rho);
    h.launches++;
  }
    {
    (coupling_lanes(h) == 32 ? k_resid_g<32> : k_resid_g<1>)<<<coupling_grid(h), 256, 0, st>>>(
        h.d.t_ptr, h.d.t_e, h.d.e_block, h.d.b_row, h.b_vals, h.c_vals, h.c_kind, r, x, nA, N, h.nC, rho);
    h.launches++;
  }
  }
  return cudaGetLastError();
}

cudaError_t launch_knorm(Handle& h, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(h.knorm, 0, sizeof(double), st);
  if (e != cudaSuccess) return e;
  const int64_t nb = (int64_t)h.nA * h.N;
  {
    k_knorm_blocks<<<grid_for(nb), 256, 0, st>>>(h.d.full_rowptr, h.d.full_src, h.a_vals, h.nnzA,
                                               h.d.bt_ptr, h.d.b_row, h.b_vals, h.d.E, h.cpl.k,
                                               h.nA, h.N, h.knorm);
    h.launches++;
  }
  if (h.nC > 0)
    {
    (coupling_lanes(h) == 32 ? k_knorm_g<32> : k_knorm_g<1>)<<<coupling_grid(h), 256, 0, st>>>(
        h.d.t_ptr, h.d.t_e, h.b_vals, h.c_vals, h.c_kind, h.nC, h.knorm);
    h.launches++;
  }
  return cudaGetLastError();
}

cudaError_t launch_axpy(Handle& h, double* y, const double* x, int64_t n, cudaStream_t st) {
  {
    k_axpy<<<grid_for(n), 256, 0, st>>>(y, x, n);
    h.launches++;
  }
  return cudaGetLastError();
}

cudaError_t launch_norms(Handle& h, const double* rho, const double* x, const double* rhs,
                         cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(h.red, 0, sizeof(double) * 3, st);
  if (e != cudaSuccess) return e;
  const int64_t nK = (int64_t)h.nA * h.N + h.nC;
  {
    k_norms3<<<grid_for(nK), 256, 0, st>>>(rho, x, rhs, nK, h.red);
    h.launches++;
  }
  return cudaGetLastError();
}

cudaError_t launch_publish(Handle& h, cudaStream_t st) {
  k_publish<<<1, 32, 0, st>>>(h.red, h.knorm, h.dev_err, h.cum ? h.cum_err : nullptr, h.host_red);
  h.launches++;
  return cudaGetLastError();
}

cudaError_t launch_dot(Handle& h, const double* a, const double* b, int64_t n, double* out, cudaStream_t st) {
  k_dot_partial<<<kDotBlocks, 256, 0, st>>>(a, b, n, h.red + 16);
  k_dot_final<<<1, kDotBlocks, 0, st>>>(h.red + 16, out);
  h.launches += 2;
  return cudaGetLastError();
}

cudaError_t launch_axpby(Handle& h, double* y, double a, const double* x, int64_t n, cudaStream_t st) {
  k_axpby<<<grid_for(n), 256, 0, st>>>(y, a, x, n);
  h.launches++;
  return cudaGetLastError();
}

cudaError_t launch_scale_into(Handle& h, double* y, double a, const double* x, int64_t n, cudaStream_t st) {
  k_scale_into<<<grid_for(n), 256, 0, st>>>(y, a, x, n);
  h.launches++;
  return cudaGetLastError();
}

cudaError_t launch_apply_inverse_ws(Handle& h, const double* r, double* out,
                                    const SolveWorkspace& ws, cudaStream_t st) {
  const int nA = h.nA, N = h.N, k = h.cpl.k, nw = h.cpl.nw;
  const int64_t pt = h.sym.panel_total;
  const int64_t nb = (int64_t)nA * N;
  k_permute_in<<<grid_for(nb), 256, 0, st>>>(r, h.d.perm, ws.z, nA, N);
  h.launches++;
  for (int l = 0; l < h.sym.nlevels; l++) {
    const int s0 = h.lvl_ptr[l], nsn = h.lvl_ptr[l + 1] - s0;
    const int warps = nsn * N;
    k_fsolve_level<<<(warps + 3) / 4, 128, 0, st>>>(h.d.lvl_sn + s0, nsn, h.d, h.Lx, pt, ws.z, nA, N);
    h.launches++;
  }
  if (h.nC > 0) {
    if (k > 0 && nw > 0) {
      dim3 g((k + 31) / 32, N);
      k_reduce_u<<<g, 32 * kReduceWarps, 0, st>>>(h.W, ws.z, h.wdinv, h.d.w_col, h.d.wr_ptr, h.d.wr_row, h.nw_nt, nw,
                                                  k, nA, ws.u);
      h.launches++;
    } else if (k > 0) {
      cudaError_t e = cudaMemsetAsync(ws.u, 0, sizeof(double) * (size_t)k * N, st);
      if (e != cudaSuccess) return e;
    }
    (coupling_lanes(h) == 32 ? k_reduce_t<32> : k_reduce_t<1>)<<<coupling_grid(h), 256, 0, st>>>(
        r + nb, h.d.t_ptr, h.d.t_e, h.d.e_t, h.d.e_block, h.b_vals, ws.u, k, h.nC, ws.tg);
    h.launches++;
    cudaError_t e = h.cum ? launch_cum_solve(h, ws.tg, ws.xg, st) : launch_dense_solve_ws(h, ws.tg, ws.xg, ws.dot, st);
    if (e != cudaSuccess) return e;
    if (k > 0 && nw > 0) {
      k_mx<<<(k * N + 255) / 256, 256, 0, st>>>(h.d.bt_ptr, h.d.b_col, h.b_vals, ws.xg, k, N, ws.v);
      k_apply_xg<<<(int)(((int64_t)nw * N * 8 + 255) / 256), 256, 0, st>>>(
          h.W, ws.v, h.d.w_col, h.d.w_sn, h.d.wt_ptr, h.d.wt_idx, h.nw_nt, nw, k, nA, N, ws.z);
      h.launches += 2;
    }
  }
  k_diag_scale<<<grid_for(nb), 256, 0, st>>>(h.d.col_dpos, h.Lx, pt, ws.z, nA, N);
  h.launches++;
  for (int l = h.sym.nlevels - 1; l >= 0; l--) {
    const int s0 = h.lvl_ptr[l], nsn = h.lvl_ptr[l + 1] - s0;
    const int warps = nsn * N;
    k_bsolve_level<<<(warps + 3) / 4, 128, 0, st>>>(h.d.lvl_sn + s0, nsn, h.d, h.Lx, pt, ws.z, nA, N);
    h.launches++;
  }
  k_permute_out<<<grid_for(nb), 256, 0, st>>>(ws.z, h.d.perm, out, nA, N);
  h.launches++;
  if (h.nC > 0) {
    cudaError_t e = cudaMemcpyAsync(out + nb, ws.xg, sizeof(double) * h.nC, cudaMemcpyDeviceToDevice, st);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

}  // namespace kkt
