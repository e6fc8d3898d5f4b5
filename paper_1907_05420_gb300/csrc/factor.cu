// (a) Batched numeric LDL^T of the N blocks A_i = P L_i D_i L_i^T P^T
// (the block factorization of Algorithm 1), all blocks sharing one supernodal
// structure.
//
// Storage: block b's factor is one contiguous array of supernode panels;
// panel s is column-major m_s x w_s (its rows are sn_rows[s], the first w_s of
// them its own columns).  The diagonal of the w_s x w_s top block holds D,
// the rest of the panel holds L (unit diagonal implied).
//
// Schedule: supernodes are processed level by level of the supernodal
// elimination tree.  Per level two launches:
//   k_factor_update: left-looking updates of every supernode s of the level
//     from its descendants d,  P_s[rel(i), j - f_s] -= sum_k L_d[i,k] D_d[k] L_d[j,k],
//     one CTA per (32-row tile of s, block) so that the wide supernodes at the
//     top of the tree spread over many SMs;
//   k_panel_factor: dense LDL^T of the panels (1x1 pivots; a pivot below
//     pivot_eps*max|A_i| is replaced by the expected-sign value and counted).
// The top of the tree (the dense tail, a suffix of the supernodes) is left out
// of the level loop: once the rest is factored, its updates from outside the
// tail are applied and the tail is factored as one dense triangle per block
// (tail.cu).
// Every entry is written by one thread in a fixed order: the result does not
// depend on scheduling.
#include "handle.h"
#include "pivot.cuh"

namespace kkt {

namespace {

__global__ void k_scatter_a(const double* __restrict__ a_vals, int64_t nnzA,
                            const int64_t* __restrict__ a_map, double* __restrict__ Lx,
                            int64_t pt, int N) {
  const int64_t total = nnzA * (int64_t)N;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total;
       q += (int64_t)gridDim.x * blockDim.x) {
    int64_t b = q / nnzA, p = q - b * nnzA;
    Lx[b * pt + a_map[p]] = a_vals[q];
  }
}

// Inertia-correction shift of the copied values: +dw on the diagonal of the
// primal rows of every block, -dc on the dual rows, dcs on C's diagonal (+dw
// for primal coupling variables, -dc for multipliers).  One thread per
// (block, row) or C entry.
__global__ void k_shift_diag(double* __restrict__ a_vals, int64_t nnzA, const int32_t* __restrict__ diag_pos,
                             int nA, int nP, int N, double* __restrict__ c_vals, int nC, int c_kind, double dw,
                             double dc, double dcs) {
  const int64_t na = (int64_t)N * nA;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < na + nC;
       q += (int64_t)gridDim.x * blockDim.x) {
    if (q < na) {
      const int64_t b = q / nA;
      const int r = (int)(q - b * nA);
      a_vals[b * nnzA + diag_pos[r]] += r < nP ? dw : -dc;
    } else {
      const int64_t i = q - na;
      c_vals[c_kind == 0 ? i : i * nC + i] += dcs;
    }
  }
}

// max |a| of each block (threshold base of the pivot perturbation)
__global__ void k_block_absmax(const double* __restrict__ a_vals, int64_t nnzA,
                               double* __restrict__ anorm) {
  __shared__ double red[256];
  const double* a = a_vals + blockIdx.x * nnzA;
  double m = 0.0;
  for (int64_t p = threadIdx.x; p < nnzA; p += blockDim.x) m = fmax(m, fabs(a[p]));
  red[threadIdx.x] = m;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + s]);
    __syncthreads();
  }
  if (threadIdx.x == 0) anorm[blockIdx.x] = red[0];
}

// One CTA per (32-row tile of supernode s, block; 128 threads).  The tile's update is
// accumulated in shared memory over the descendants d that meet the tile (in
// update order) and subtracted from the panel once.  For each update the rows
// of d that land in the tile ([ia, ib), listed per tile at analysis with only
// the updates that meet it) and the rows that land in s's columns ([r0, r1))
// are staged in shared memory, the latter pre-multiplied by D_d.
constexpr int kTileRows = kFactorTileRows;
constexpr int kFactorThreads = 128;

__global__ void __launch_bounds__(kFactorThreads) k_factor_update(const int32_t* __restrict__ work,
                                                       const UpdPair* __restrict__ pairs, DevSym d,
                                                       double* __restrict__ Lx, int64_t pt,
                                                       const double* __restrict__ LDx, int64_t ldt) {
  __shared__ double acc[kTileRows][kMaxSnWidth + 1];
  __shared__ double Li[kTileRows][kMaxSnWidth + 1];
  __shared__ double Lj[kMaxSnWidth][kMaxSnWidth + 1];
  __shared__ int rs[kTileRows], tc[kMaxSnWidth];
  const int item = blockIdx.x, b = blockIdx.y, tid = threadIdx.x;
  const int s = work[4 * item], lo = work[4 * item + 1], hi = work[4 * item + 2];
  const int p0 = work[4 * item + 3], p1 = work[4 * item + 7];  // this item's updates, to the next item's
  const int ms = (int)(d.sn_rowptr[s + 1] - d.sn_rowptr[s]);
  const int f = d.sn_first[s], ws = d.sn_first[s + 1] - f;
  const int nrow = hi - lo;
  const double* Lb = Lx + b * pt;
  const double* LDb = LDx + b * ldt;
  double* P = Lx + b * pt + d.sn_valoff[s];
  for (int q = tid; q < kTileRows * (kMaxSnWidth + 1); q += blockDim.x) (&acc[0][0])[q] = 0.0;
  // The next update's operands, read while this one's products run (its record
  // was read one update earlier): of each operand this thread's first kAhead
  // entries, all of them for the narrow descendants that most updates have.  Read
  // between the two barriers instead, they are a trip to L2 in the chain of every
  // update: all levels of 2,383 buses x 96 periods 1.17 -> 0.98 ms, of 301 x 48
  // 0.134 -> 0.110, of 9,241 x 24 4.4 -> 3.7 ms.
  constexpr int kAhead = 2;
  double li[kAhead], lj[kAhead];
  int pi[kAhead], pj[kAhead], rsn = 0, tcn = 0;
  const auto fetch = [&](const UpdPair& R) {
    const int ni = R.ib - R.ia, nj = R.r1 - R.r0, wd = R.wd, md = R.md;
    const double* Pd = Lb + R.val + R.ia;
    const double* PDd = LDb + R.val + R.r0;  // the same panel's L D (descendants lie outside the tail)
#pragma unroll
    for (int u = 0; u < kAhead; u++) {
      const int q = tid + u * kFactorThreads;
      pi[u] = pj[u] = -1;
      if (q < ni * wd) {
        const int kk = q / ni, i = q - kk * ni;
        li[u] = Pd[(int64_t)kk * md + i];
        pi[u] = i * (kMaxSnWidth + 1) + kk;
      }
      if (q < nj * wd) {
        const int kk = q / nj, j = q - kk * nj;
        lj[u] = PDd[(int64_t)kk * md + j];
        pj[u] = j * (kMaxSnWidth + 1) + kk;
      }
    }
    if (tid < ni) rsn = d.upd_rel[R.rel + R.ia + tid - R.r0] - lo;
    if (tid < nj) tcn = d.sn_rows[R.rows + R.r0 + tid] - f;
  };
  UpdPair Rn{}, Rnn{};
  if (p0 < p1) {
    Rn = pairs[p0];
    if (p0 + 1 < p1) Rnn = pairs[p0 + 1];
    fetch(Rn);
  }
  for (int p = p0; p < p1; p++) {
    const UpdPair R = Rn;
    const int ni = R.ib - R.ia, nj = R.r1 - R.r0, wd = R.wd, md = R.md;
    __syncthreads();  // the previous update's reads of Li/Lj are done
#pragma unroll
    for (int u = 0; u < kAhead; u++) {
      if (pi[u] >= 0) (&Li[0][0])[pi[u]] = li[u];
      if (pj[u] >= 0) (&Lj[0][0])[pj[u]] = lj[u];
    }
    for (int q = tid + kAhead * kFactorThreads; q < ni * wd; q += kFactorThreads) {
      const int kk = q / ni, i = q - kk * ni;
      Li[i][kk] = Lb[R.val + (int64_t)kk * md + R.ia + i];
    }
    for (int q = tid + kAhead * kFactorThreads; q < nj * wd; q += kFactorThreads) {
      const int kk = q / nj, j = q - kk * nj;
      Lj[j][kk] = LDb[R.val + (int64_t)kk * md + R.r0 + j];
    }
    if (tid < ni) rs[tid] = rsn;
    if (tid < nj) tc[tid] = tcn;
    __syncthreads();
    if (p + 1 < p1) {
      Rn = Rnn;
      if (p + 2 < p1) Rnn = pairs[p + 2];
      fetch(Rn);
    }
    for (int q = tid; q < ni * nj; q += blockDim.x) {
      const int i = q % ni, j = q / ni;
      if (R.ia + i < R.r0 + j) continue;  // above the diagonal of the target
      double sum = 0.0;
      for (int kk = 0; kk < wd; kk++) sum += Li[i][kk] * Lj[j][kk];
      acc[rs[i]][tc[j]] += sum;
    }
  }
  __syncthreads();
  for (int q = tid; q < nrow * ws; q += blockDim.x) {
    const int r = q % nrow, c = q / nrow;
    P[(int64_t)c * ms + lo + r] -= acc[r][c];
  }
}

// Dense LDL^T of the panels of one level (1x1 pivots; right-looking order of the
// operations on every entry), and L D of each panel for the updates of its
// ancestors: column c's entries times d_c, the product the updates would
// otherwise form per target tile.  The leaves are thousands of panels of a few
// columns and rows, the top of the tree a few of up to 32 columns and thousands
// of rows, so a launch has two kinds of CTAs:
//   small panels (at most kPanelSmall entries): eight lanes each, staged in shared
//     memory, the blocks of one supernode side by side;
//   items of a larger panel: its w x w triangle in shared memory, then one row per
//     thread in registers against it.  A panel of more than kPanelRows rows below
//     its triangle has an item for the triangle and, in a second launch, one per
//     tile of kPanelTile rows.
// Bound by the FP64 pipe and, at the top, by the chain of pivots.  With one CTA of
// 256 threads per panel, working on it in global memory, all levels of 2,383 buses
// x 96 periods took 1.55 ms, of 301 x 48 0.18 ms and of 9,241 x 24 10 ms (there
// panels of 32 columns and thousands of rows); now 0.63, 0.093 and 1.39 ms.
constexpr int kPanelThreads = 128;
constexpr int kPanelGroups = kPanelThreads / 8;

struct PanelSmallShared {
  double t[kPanelGroups][kPanelSmall + 1];
};
struct PanelTileShared {
  double T[kMaxSnWidth][kMaxSnWidth + 1];
  double U[kMaxSnWidth][kMaxSnWidth];  // U[c][r] = l_rc d_c (0 from column w on)
  double D[kMaxSnWidth], Di[kMaxSnWidth];  // d_c and 1 / d_c (0 from column w on)
};

// 0, which perturbs nothing, unless the product is positive (0 * Inf is not)
__device__ __forceinline__ double panel_threshold(double pivot_eps, double anorm) {
  const double thr = pivot_eps * anorm;
  return thr > 0.0 ? thr : 0.0;
}

// The pivot as it is used: a magnitude below thr becomes +-thr (thr >= 0).  Bit
// patterns of non-negative numbers order as the numbers do; a NaN stays.
// cnt: positive, negative, zero or NaN, perturbed.
__device__ __forceinline__ double panel_pivot(double dv, double thr, bool primal, int* cnt, bool count) {
  const long long inf = 0x7ff0000000000000LL;
  const long long mag = __double_as_longlong(dv) & 0x7fffffffffffffffLL;
  const bool pert = mag < __double_as_longlong(thr);
  if (pert) dv = primal ? thr : -thr;
  if (count) {
    const long long v = __double_as_longlong(dv), m = v & 0x7fffffffffffffffLL;
    atomicAdd(&cnt[m == 0 || m > inf ? 2 : (v > 0 ? 0 : 1)], 1);
    if (pert) atomicAdd(&cnt[3], 1);
  }
  return dv;
}

__device__ __forceinline__ void panel_small(PanelSmallShared& sh, const SnDesc* __restrict__ small, int nsmall, int cta,
                                            const int32_t* __restrict__ col_primal, double* __restrict__ Lx,
                                            int64_t pt, double* __restrict__ LDx, int64_t ldt,
                                            const double* __restrict__ anorm, double pivot_eps, int N, int* cnt) {
  const int g = threadIdx.x >> 3, l = threadIdx.x & 7;
  const int64_t q = (int64_t)cta * kPanelGroups + g;
  const bool on = q < (int64_t)nsmall * N;
  const int b = on ? (int)(q % N) : 0;
  SnDesc S{};
  if (on) S = small[q / N];
  const int w = on ? S.w : 0, m = S.m;
  double* T = sh.t[g];
  double* P = Lx + b * pt + S.val;
  double* PD = LDx + b * ldt + S.val;
  const double thr = on ? panel_threshold(pivot_eps, anorm[b]) : 0.0;
  for (int e = l; e < w * m; e += 8) T[e] = P[e];
  const int wmax = __reduce_max_sync(0xffffffffu, w);
  __syncwarp();
  for (int c = 0; c < wmax; c++) {
    const bool act = c < w;
    double* colc = T + c * m;
    double dv = 0.0;
    if (act) {
      dv = panel_pivot(colc[c], thr, col_primal[S.f + c] != 0, cnt, l == 0);
      const double di = pivot_recip(dv);
      for (int r = c + 1 + l; r < m; r += 8) colc[r] *= di;
    }
    __syncwarp();
    if (act) {
      if (l == 0) colc[c] = dv;
      for (int c2 = c + 1; c2 < w; c2++) {
        const double l2 = colc[c2] * dv;
        for (int r = c2 + l; r < m; r += 8) T[c2 * m + r] -= colc[r] * l2;
      }
    }
    __syncwarp();
  }
  for (int c = 0; c < w; c++) {
    const double dv = T[c * m + c];
    for (int r = l; r < m; r += 8) {
      const double v = T[c * m + r];
      P[c * m + r] = v;
      PD[c * m + r] = v * dv;
    }
  }
}

// one row per thread, eight columns of it in registers at a time (the sums read
// earlier columns again from L1; their FP64 operations take far longer)
__device__ __forceinline__ void panel_rows(const PanelTileShared& sh, double* P, double* PD, int m, int w, int r0,
                                           int r1) {
  constexpr int W = 8;
  for (int r = r0 + threadIdx.x; r < r1; r += kPanelThreads) {
    for (int c0 = 0; c0 < w; c0 += W) {
      double a[W];
#pragma unroll
      for (int c = 0; c < W; c++) a[c] = c0 + c < w ? P[(int64_t)(c0 + c) * m + r] : 0.0;
#pragma unroll 4
      for (int k = 0; k < c0; k++) {
        const double lk = P[(int64_t)k * m + r];
#pragma unroll
        for (int c = 0; c < W; c++) a[c] -= lk * sh.U[k][c0 + c];
      }
#pragma unroll
      for (int c = 0; c < W; c++) {
        a[c] *= sh.Di[c0 + c];
#pragma unroll
        for (int c2 = c + 1; c2 < W; c2++) a[c2] -= a[c] * sh.U[c0 + c][c0 + c2];
      }
#pragma unroll
      for (int c = 0; c < W; c++)
        if (c0 + c < w) {
          P[(int64_t)(c0 + c) * m + r] = a[c];
          PD[(int64_t)(c0 + c) * m + r] = a[c] * sh.D[c0 + c];
        }
    }
  }
}

__device__ __forceinline__ void panel_tile(PanelTileShared& sh, const PanelItem it, int b,
                                           const int32_t* __restrict__ col_primal, double* __restrict__ Lx, int64_t pt,
                                           double* __restrict__ LDx, int64_t ldt, const double* __restrict__ anorm,
                                           double pivot_eps, int* cnt) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, m = it.m, w = it.w;
  double* P = Lx + b * pt + it.val;
  double* PD = LDx + b * ldt + it.val;
  for (int e = tid; e < kMaxSnWidth * kMaxSnWidth; e += kPanelThreads) {
    const int c = e / kMaxSnWidth, r = e % kMaxSnWidth;
    if (r < w && c <= r) sh.T[r][c] = P[(int64_t)c * m + r];
    sh.U[c][r] = 0.0;
  }
  if (tid < kMaxSnWidth) sh.Di[tid] = 0.0;
  __syncthreads();
  if (it.factor) {
    const double thr = panel_threshold(pivot_eps, anorm[b]);
    for (int c = 0; c < w; c++) {
      const double dv = panel_pivot(sh.T[c][c], thr, col_primal[it.first + c] != 0, cnt, tid == 0);
      const double di = pivot_recip(dv);
      if (tid < w - c - 1) {
        const int r = c + 1 + tid;
        const double lr = sh.T[r][c] * di;
        sh.T[r][c] = lr;
        sh.U[c][r] = lr * dv;
      }
      if (tid == 0) {
        sh.D[c] = dv;
        sh.Di[c] = di;
      }
      __syncthreads();
      const int r = c + 1 + lane;
      for (int c2 = c + 1 + warp; c2 < w; c2 += kPanelThreads / 32)
        if (r >= c2 && r < w) sh.T[r][c2] -= sh.T[r][c] * sh.U[c][c2];
      __syncthreads();
    }
    for (int e = tid; e < w * w; e += kPanelThreads) {
      const int c = e / w, r = e - c * w;
      const int64_t pos = (int64_t)c * m + r;
      const double v = r == c ? sh.D[c] : (r > c ? sh.T[r][c] : P[pos]);
      if (r >= c) P[pos] = v;
      PD[pos] = v * sh.D[c];
    }
  } else {
    if (tid < w) {
      sh.D[tid] = sh.T[tid][tid];
      sh.Di[tid] = pivot_recip(sh.T[tid][tid]);
    }
    for (int e = tid; e < w * w; e += kPanelThreads) {
      const int c = e / w, r = e - c * w;
      if (r > c) sh.U[c][r] = sh.T[r][c] * sh.T[c][c];
    }
    __syncthreads();
  }
  panel_rows(sh, P, PD, m, w, it.r0, it.r1);
}

__global__ void __launch_bounds__(kPanelThreads, 5)
k_panel_factor(const SnDesc* __restrict__ small, int nsmall, int small_ctas, const PanelItem* __restrict__ items,
               const int32_t* __restrict__ col_primal, double* __restrict__ Lx, int64_t pt, double* __restrict__ LDx,
               int64_t ldt, const double* __restrict__ anorm, double pivot_eps, int N,
               unsigned long long* __restrict__ counters) {
  __shared__ union Shared {
    __device__ Shared() {}
    PanelSmallShared s;
    PanelTileShared t;
  } sh;
  __shared__ int cnt[4];
  if (threadIdx.x < 4) cnt[threadIdx.x] = 0;
  __syncthreads();
  if ((int)blockIdx.x < small_ctas) {
    panel_small(sh.s, small, nsmall, blockIdx.x, col_primal, Lx, pt, LDx, ldt, anorm, pivot_eps, N, cnt);
  } else {
    const int q = blockIdx.x - small_ctas;
    panel_tile(sh.t, items[q / N], q % N, col_primal, Lx, pt, LDx, ldt, anorm, pivot_eps, cnt);
  }
  __syncthreads();
  if (threadIdx.x < 4 && cnt[threadIdx.x]) atomicAdd(&counters[threadIdx.x], (unsigned long long)cnt[threadIdx.x]);
}

}  // namespace

cudaError_t launch_shift_diag(Handle& h, double dw, double dc, double dcs, cudaStream_t st) {
  const int64_t total = (int64_t)h.N * h.nA + h.nC;
  if (total == 0) return cudaSuccess;
  const int grid = (int)std::min<int64_t>((total + 255) / 256, 152 * 8);
  k_shift_diag<<<grid, 256, 0, st>>>(h.a_vals, h.nnzA, h.d.diag_pos, h.nA, h.nP, h.N, h.c_vals, h.nC, h.c_kind,
                                     dw, dc, dcs);
  h.launches++;
  return cudaGetLastError();
}

cudaError_t launch_scatter_a(Handle& h, cudaStream_t st) {
  const int64_t pt = h.sym.panel_total;
  cudaError_t e = cudaMemsetAsync(h.Lx, 0, sizeof(double) * pt * h.N, st);
  if (e != cudaSuccess) return e;
  int64_t total = h.nnzA * h.N;
  int grid = (int)std::min<int64_t>((total + 255) / 256, 152 * 16);
  {
    k_scatter_a<<<grid, 256, 0, st>>>(h.a_vals, h.nnzA, h.d.a_map, h.Lx, pt, h.N);
    h.launches++;
  }
  {
    k_block_absmax<<<h.N, 256, 0, st>>>(h.a_vals, h.nnzA, h.anorm);
    h.launches++;
  }
  return cudaGetLastError();
}

cudaError_t launch_factor_levels(Handle& h, cudaStream_t st) {
  const int64_t pt = h.sym.panel_total;
  // supernodes outside the dense tail, level by level
  for (int l = 0; l < h.sym.nlevels; l++) {
    const int w0 = h.fwork_lvl_ptr[l], w1 = h.fwork_lvl_ptr[l + 1];
    if (l > 0 && w1 > w0) {
      dim3 grid(w1 - w0, h.N);
      const int kt = kt_begin(h, kFamFactorUpd, h.N * h.fupd_flops[l], st);
      k_factor_update<<<grid, kFactorThreads, 0, st>>>(h.d.fwork + 4 * w0, h.d.fpairs, h.d, h.Lx, pt, h.LDx,
                                                        h.ld_total);
      kt_end(h, kt, st);
      h.launches++;
    }
    // small panels and the triangles of the others, then the rows of the longest
    const PanelLevel L = h.panel_lvl[l];
    for (int second = 0; second < 2; second++) {
      const int nsmall = second ? 0 : L.nsmall, nitem = second ? L.nrows : L.nitems;
      const int64_t small_ctas = ((int64_t)nsmall * h.N + kPanelGroups - 1) / kPanelGroups;
      const int64_t ctas = small_ctas + (int64_t)nitem * h.N;
      if (ctas == 0) continue;
      k_panel_factor<<<(unsigned)ctas, kPanelThreads, 0, st>>>(
          h.d.panel_small + L.small0, nsmall, (int)small_ctas, h.d.panel_items + L.item0 + (second ? L.nitems : 0),
          h.d.col_primal, h.Lx, pt, h.LDx, h.ld_total, h.anorm, h.opt.pivot_eps, h.N, h.counters);
      h.launches++;
    }
  }
  if (h.nT > 0) {
    // the dense tail, its updates from the rest of the tree (all factored by now)
    // first; an augmented tail needs the W rows outside the tail and its own rows Z
    if (h.tail_aug) {
      cudaError_t e = launch_w_solve_before_tail(h, st);
      if (e != cudaSuccess) return e;
    }
    cudaError_t e = launch_dense_tail(h, st);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

}  // namespace kkt
