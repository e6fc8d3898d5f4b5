// (a) Dense tail of the block factors.
//
// The last supernodes of the postorder (the top of the elimination tree) have
// row sets inside the tail columns [c_T, n) and are nearly dense there, so the
// tail of every block is factored as one dense nT x nT lower triangle
// (nT = n - c_T) instead of supernode by supernode: the work is the same
// LDL^T (Algorithm 1's block factorization) with the explicit zeros of the
// tail included, done by the blocked dense kernels that factor S
// (dense_kernels.cuh), batched over the N blocks.
//
// Per factor: the tail panels (A's values) are gathered into the zeroed dense
// triangles, which then take the updates from outside the tail; each 64-wide
// panel step factors the diagonal blocks of all N triangles (with the
// static-pivot rule and the inertia counts of the sparse panels), forms L21 and
// Y = L21 D, and updates the trailing triangles, in FP64 on the CUDA cores (tail
// mode 1) or in emulated FP64 on the tensor cores (tail mode 2, the update of
// dense_tc.cu: 7 base-256 digit slices per operand); the factor is scattered back
// into the supernodal panels, which the solves use.
// Entries of the triangles outside the supernodal structure stay exact zeros
// (every product that reaches them has a zero factor).
//
// Augmented tail: each triangle gets k more rows, Z^T, where Z holds the
// tail's rows of P^T E - L_{T,rest} W_rest (the right-hand sides of W after
// the updates from outside the tail; zero rows for tail columns outside the
// reach of E).  Factoring only the nT tail pivots of [T Z; Z^T 0] is the
// incomplete factorization of Sec. 4.2 (eq. augmented) restricted to the tail:
// the augmented rows become W_T^T D_T^{-1} with W_T = L_T^{-1} Z, and the
// trailing k x k block becomes -W_T^T D_T^{-1} W_T, the tail's share of G.  So
// the tail's W solve and contraction run inside the tail factor.
#include "dense_kernels.cuh"

namespace kkt {

namespace {

// panels of the tail supernodes <-> dense triangles (order nTa, the first nT
// columns), lower part only
template <bool TO_DENSE>
__global__ void __launch_bounds__(256) k_tail_move(DevSym d, double* __restrict__ Lx, int64_t pt,
                                                   double* __restrict__ T, int nTa, int tail_col,
                                                   int tail_sn) {
  const int s = tail_sn + blockIdx.x, b = blockIdx.y;
  const int m = (int)(d.sn_rowptr[s + 1] - d.sn_rowptr[s]);
  const int f = d.sn_first[s], w = d.sn_first[s + 1] - f;
  double* P = Lx + b * pt + d.sn_valoff[s];
  const int32_t* R = d.sn_rows + d.sn_rowptr[s];
  double* Tb = T + (int64_t)b * nTa * nTa;
  for (int q = threadIdx.x; q < m * w; q += blockDim.x) {
    const int c = q / m, i = q - c * m;
    const int row = R[i], col = f + c;
    if (row < col) continue;  // strictly upper part of the diagonal block: unused
    double* t = Tb + (int64_t)(row - tail_col) + (int64_t)(col - tail_col) * nTa;
    if (TO_DENSE) *t = P[q];
    else P[q] = *t;
  }
}

// Augmented rows: T_b[nT + t][j] = Z_b[j][t] (tail column j's W row before
// the tail solve; zero for a column outside the reach of E), and after the
// factor the tail's W rows from them: row nT + t of the factor holds
// (W_T^T D_T^{-1})[t][j], so W_b[row(j)][t] = T_b[nT + t][j] * D_j.
template <bool TO_DENSE>
__global__ void k_tail_aug_rows(double* __restrict__ W, int nw, int k, double* __restrict__ T, int nT,
                                int nTa, const int32_t* __restrict__ wrow) {
  const int b = blockIdx.y;
  double* Tb = T + (int64_t)b * nTa * nTa;
  double* Wb = W + (int64_t)b * nw * k;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < nT * k; q += gridDim.x * blockDim.x) {
    const int j = q / k, t = q - j * k;
    const int r = wrow[j];
    if (r < 0) continue;
    double* a = Tb + (int64_t)(nT + t) + (int64_t)j * nTa;
    if (TO_DENSE) *a = Wb[(int64_t)r * k + t];
    else Wb[(int64_t)r * k + t] = *a * Tb[(int64_t)j + (int64_t)j * nTa];
  }
}

// The updates of the dense tails from the descendants outside them (all but the
// heavy ones), T[i][j] -= sum_d sum_k L_d[i][k] D_d[k] L_d[j][k], one warp per
// (4-row tile with updates, block): the warp walks the descendants that meet
// the tile, sums their products into its own tile in shared memory (lanes over
// the entries a descendant adds, operands straight from global memory, each
// warp on its own: no barrier between descendants) and subtracts it from the
// dense triangle at the end.
// What bounds it: latency, about two round trips to L2 per descendant and tile,
// hidden by 40 warps per SM with small tiles; then the FP64 pipe, 72% busy on 24
// tails of order 732 and 68% on 8 of order 7,009, where L1 is at 78%.  The CTA-wide staging of
// k_factor_update, with two barriers per descendant, took 138 us for 48 tails of
// order 130 (60 here), 2.8 ms for 96 of order 724 (1.5) and, without their heavy
// descendants, 56 ms for 24 of order 6,938 (13.4); loading the next descendant
// ahead into registers cost more warps than it hid latency (39 ms).
constexpr int kTailUpdWarps = 4;
inline int tail_upd_smem(int cols) { return kTailUpdWarps * cols * (kTailTileRows + 1) * (int)sizeof(double); }

template <int COLS>
__global__ void __launch_bounds__(32 * kTailUpdWarps, 10)
    k_tail_update(const int32_t* __restrict__ work, int nitems, const TailPair* __restrict__ pairs,
                  const int32_t* __restrict__ sn_rows, const double* __restrict__ Lx, int64_t pt,
                  const double* __restrict__ LDx, int64_t ldt, double* __restrict__ T, int nT, int nTa, int tail_col) {
  extern __shared__ __align__(16) double accs[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, b = blockIdx.y;
  const int item = blockIdx.x * kTailUpdWarps + warp;
  if (item >= nitems) return;
  double* acc = accs + warp * COLS * (kTailTileRows + 1);  // [column][row]
  const int i0 = work[3 * item] * kTailTileRows, j0 = work[3 * item + 1] * COLS;
  const int p0 = work[3 * item + 2], p1 = work[3 * item + 5];
  for (int q = lane; q < COLS * (kTailTileRows + 1); q += 32) acc[q] = 0.0;
  const double* Lb = Lx + b * pt;
  const double* LDb = LDx + b * ldt;
  const int ri0 = tail_col + i0, rj0 = tail_col + j0;
  TailPair Rn = pairs[p0];
  __syncwarp();
  for (int p = p0; p < p1; p++) {
    const TailPair R = Rn;
    if (p + 1 < p1) Rn = pairs[p + 1];
    const int ne = R.ni * R.nj, md = R.md, wd = R.wd;
    for (int q = lane; q < ne; q += 32) {
      const int j = (int)(((uint32_t)q * R.inv) >> 16), i = q - j * R.ni;
      const int row = sn_rows[R.ri + i] - ri0, col = sn_rows[R.rj + j] - rj0;
      const double* a = Lb + R.li + i;
      const double* c = LDb + R.lj + j;
      double sum = 0.0;
      int k = 0;
      for (; k + 4 <= wd; k += 4, a += 4 * md, c += 4 * md) {
        const double a0 = a[0], a1 = a[md], a2 = a[2 * md], a3 = a[3 * md];
        const double c0 = c[0], c1 = c[md], c2 = c[2 * md], c3 = c[3 * md];
        sum += a0 * c0;
        sum += a1 * c1;
        sum += a2 * c2;
        sum += a3 * c3;
      }
      if (k < wd) {  // one to three columns left, loaded together
        const bool b1 = k + 1 < wd, b2 = k + 2 < wd;
        const double a0 = a[0], a1 = b1 ? a[md] : 0.0, a2 = b2 ? a[2 * md] : 0.0;
        const double c0 = c[0], c1 = b1 ? c[md] : 0.0, c2 = b2 ? c[2 * md] : 0.0;
        sum += a0 * c0;
        if (b1) sum += a1 * c1;
        if (b2) sum += a2 * c2;
      }
      if (i0 + row >= j0 + col) acc[col * (kTailTileRows + 1) + row] += sum;
    }
    __syncwarp();
  }
  double* Tb = T + (int64_t)b * nTa * nTa;
  const int row = lane & (kTailTileRows - 1), i = i0 + row;
  constexpr int kStep = 32 / kTailTileRows;
#pragma unroll 8
  for (int c = lane / kTailTileRows; c < COLS; c += kStep) {
    const int j = j0 + c;
    if (i < nT && j <= i) Tb[(int64_t)i + (int64_t)j * nTa] -= acc[c * (kTailTileRows + 1) + row];
  }
}

}  // namespace

cudaError_t launch_dense_tail(Handle& h, cudaStream_t st) {
  const int nT = h.nT, nTa = h.nTa, N = h.N;
  const int tail_sn = h.sym.tail_sn, tail_col = h.sym.tail_col;
  const int nsn = h.sym.nsuper - tail_sn;
  const int64_t pt = h.sym.panel_total, t2 = (int64_t)nTa * nTa, ys = (int64_t)nTa * kPanelW;
  const int k = h.cpl.k, nw = h.cpl.nw;
  const dim3 agrid((int)std::min<int64_t>(((int64_t)nT * k + 255) / 256, 64), N);
  cudaError_t e = cudaMemsetAsync(h.Tt, 0, sizeof(double) * t2 * N, st);
  if (e != cudaSuccess) return e;
  k_tail_move<true><<<dim3(nsn, N), 256, 0, st>>>(h.d, h.Lx, pt, h.Tt, nTa, tail_col, tail_sn);
  h.launches++;
  if (h.tail_aug) {
    k_tail_aug_rows<true><<<agrid, 256, 0, st>>>(h.W, nw, k, h.Tt, nT, nTa, h.d.tail_wrow);
    h.launches++;
  }
  if (h.tail_items > 0) {
    const int kt = kt_begin(h, kFamFactorUpd, N * h.tupd_flops, st);
    const int cols = tail_tile_cols(nT);
    (cols == 128 ? k_tail_update<128> : k_tail_update<64>)<<<
        dim3((h.tail_items + kTailUpdWarps - 1) / kTailUpdWarps, N), 32 * kTailUpdWarps, tail_upd_smem(cols), st>>>(
        h.d.twork, h.tail_items, h.d.tpairs, h.d.sn_rows, h.Lx, pt, h.LDx, h.ld_total, h.Tt, nT, nTa, tail_col);
    kt_end(h, kt, st);
    h.launches++;
  }
  if (h.tail_mode == 2) {
    e = launch_tail_heavy_update(h, st);
    if (e == cudaSuccess) e = launch_tail_factor_emulated(h, st);
    if (e != cudaSuccess) return e;
  }
  const PivotRule rule{h.anorm, h.opt.pivot_eps, h.d.col_primal + tail_col};
  for (int k0 = 0; h.tail_mode == 1 && k0 < nT; k0 += kPanelW) {
    const int kb = std::min(kPanelW, nT - k0);
    const int kd = kt_begin(h, kFamDiag, N * (2.0 / 3.0) * kb * kb * kb, st);
    launch_dense_diag<double>(h.Tt, nTa, k0, kb, N, t2, rule, h.counters, st);
    kt_end(h, kd, st);
    h.launches++;
    const int rest = nTa - k0 - kb;
    if (rest > 0) {
      launch_dense_panel<double>(h.Tt, h.TY, nTa, k0, kb, nTa, N, t2, ys, st);
      const int kt = kt_begin(h, kFamDenseF64, N * update_flops(rest, 0, rest, kb), st);
      launch_dense_update<double>(h.Tt, h.TY, nTa, k0, kb, nTa, N, t2, ys, st);
      kt_end(h, kt, st);
      h.launches += 2;
    }
  }
  k_tail_move<false><<<dim3(nsn, N), 256, 0, st>>>(h.d, h.Lx, pt, h.Tt, nTa, tail_col, tail_sn);
  h.launches++;
  if (h.tail_aug) {
    k_tail_aug_rows<false><<<agrid, 256, 0, st>>>(h.W, nw, k, h.Tt, nT, nTa, h.d.tail_wrow);
    h.launches++;
  }
  e = cudaGetLastError();
  return e != cudaSuccess ? e : launch_tail_inverse(h, st);
}

}  // namespace kkt
