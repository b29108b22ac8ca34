// Refined truncation solve (TN_SOLVE_REFINED): FP64 result from an FP32 start.
//
// The truncated SVD of the bond matrix K = R_v R_w^T (Methods, "The simple
// update procedure") is taken as the eigen-decomposition
// H = K K^H = R_v conj(G_w) R_v^H = U diag(sigma^2) U^H, where G_v = R_v^H R_v
// and G_w are the Gram matrices of the gate-split environment-weighted site
// matrices, built from the open-p environments N_p of both sides.  The gate is
// split on the projectors of v's physical index as in solve32.cu, which makes
// G_v block diagonal.  Phases:
//
//   1. chol64_kernel: FP64 pivoted Cholesky of the two chi x chi blocks of G_v,
//      P^T G_b P = L_b L_b^H, so that R_b = L_b^H P^T.
//   2. solve32_kernel in basis mode: the same R_v rounded to FP32, the FP32
//      Cholesky of G_w, K^T = R_w R_v^T and the one-sided Jacobi of K in FP32
//      shared memory.  It yields only a starting basis: the columns of K J
//      normalised (U_0, n x n, by decreasing sigma, the columns below
//      1e-3 sigma_1 re-orthonormalised in FP32) and sigma^2.
//   3. refine_kernel: one Newton step in FP64 for the kept chi columns, the
//      refinement of Ogita and Aishima ("Iterative refinement for symmetric
//      eigenvalue decomposition", Japan J. Indust. Appl. Math. 35, 2018), in
//      the basis U_A of the active columns of U_0 (sigma above 1e-6 sigma_1):
//        P = H U_k,  S = U_A^H P,  R = I - U_A^H U_k               (FP64)
//        lambda_j = S_jj / (1 - R_jj)
//        E_ij = (S_ij + lambda_j R_ij) / (lambda_j - lambda_i)  for i != j,
//               R_ij / 2 when the pair is not separated; E_jj = R_jj / 2
//        u_j' = u_j + U_A E_Aj + (I - P_A) P_j / lambda_j
//      The last term is the Newton correction toward the complement of
//      span(U_A), on which H is about zero; to first order it is
//      P_j / lambda_j - U_A (S_Aj / lambda_j + R_Aj).  The step converges
//      quadratically: a start orthogonal to about 1e-6 leaves an error of
//      order (1e-6 / relative gap)^2.  It is taken for the head columns
//      (sigma >= 1e-3 sigma_1).  Below that the FP32 start is limited by the
//      FP32 Gram inputs themselves, and the Rayleigh quotients of the squared
//      problem are dominated by the head's rounding, so tail columns keep
//      their start's eigenvalues and take only the corrections that keep
//      them orthogonal to the head (E_ij = R_ij - conj(E_ji)) and to each
//      other (R_ij / 2).
//   4. legs_kernel: FP64 leg matrices from the refined basis,
//      C_v = R_v^+ U_k sqrt(S) by triangular solves and
//      C_w = R_v^T conj(U_k) / sqrt(sigma ||sigma||); the outputs D_v[p] and
//      D_w[q] (FP32 planar), the spectrum S = sigma / ||sigma|| in decreasing
//      order, and both gate-edge messages diag(S).
//
// Only phase 2 computes in FP32.  The quantities the outputs are computed from
// (R_v, H U, the Rayleigh quotients, the corrected eigenvectors and the leg
// matrices) are FP64.
#include <math.h>

#include <algorithm>

#include "chol_rows.cuh"
#include "common.cuh"
#include "tnbp.h"

namespace tnbp {
namespace {

struct cd {
  double x, y;
};
__device__ __forceinline__ cd cz() { return {0.0, 0.0}; }
__device__ __forceinline__ cd cconj(cd a) { return {a.x, -a.y}; }
__device__ __forceinline__ cd cadd(cd a, cd b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ cd csub(cd a, cd b) { return {a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ cd cscale(cd a, double s) { return {a.x * s, a.y * s}; }
__device__ __forceinline__ cd cmul(cd a, cd b) {
  return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
// acc += a * b
__device__ __forceinline__ void cfma(cd& acc, cd a, cd b) {
  acc.x = fma(a.x, b.x, acc.x);
  acc.x = fma(-a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y);
  acc.y = fma(a.y, b.x, acc.y);
}
__device__ __forceinline__ double cabs2(cd a) { return a.x * a.x + a.y * a.y; }
__device__ __forceinline__ cd shfl_xor(cd v, int o) {
  return {__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o)};
}

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kJU = 4;              // output columns per thread in the basis update
constexpr int kSmemChi = 64;   // up to here the FP32 basis and the FP64 Cholesky run in
                               // shared memory; above, in the edge's global workspace
constexpr int kMaxChi = 256;
constexpr int kSmemBudget = 200 * 1024;
// Head columns, sigma >= 1e-3 sigma_1: the FP32 start is accurate enough there
// for one Newton step to reach FP64 accuracy.  Below, the start is limited by
// the FP32 Gram inputs themselves (their rounding puts an absolute floor of
// about sqrt(eps_32) sigma_1 under the singular values), and the Rayleigh
// quotient of the squared problem H would be dominated by the head's
// rounding, so tail columns keep their start's values and are only kept
// orthogonal.
constexpr double kHead = 1e-6;
// Separation test of a pair: the start's eigenvalue lambda_0[i] carries the
// FP32 rounding of its column, about kNoise sqrt(lambda_0[0] lambda_0[i])
// (a few FP32 ulps of sigma_1 times sigma_i, with a margin).  A pair whose gap
// is not clearly above that, or whose Newton correction would exceed 1/4, is
// treated as degenerate: only kept orthogonal (R_ij / 2).  Rotations inside
// the kept set are a gauge freedom of the two-site matrix, so leaving such a
// pair unrotated changes no contraction of the state.
constexpr double kNoise = 2e-6;

// ------------------------------------------------------------ FP64 Cholesky
// Block b = blockIdx.y of edge blockIdx.z: G_b = conj(N_b^v) -> L_b, perm_b,
// rank_b; ctas CTAs per block (one up to kSmemChi, a cluster above), CV columns
// per lane and RW rows per row warp.  The factor is collected by original row, in
// shared memory or in the edge's S block of the workspace, and copied to pivot
// order at the end.
constexpr int kCholThreads = 512 + 32;  // 16 row warps and the pivot warp

template <int CV, int RW>
__global__ void __launch_bounds__(kCholThreads, 1) chol64_kernel(SolveArgs a, int ctas) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double2 column[2 * 32 * CV];
  __shared__ int perm_s[32 * CV];
  const int rank = blockIdx.x, b = blockIdx.y, edge = blockIdx.z, chi = a.chi;
  const int64_t c2 = (int64_t)chi * chi;
  const float* g = a.gram + (int64_t)edge * 8 * c2 + (int64_t)b * 2 * c2;
  const RefineLayout lay = refine_layout(chi);
  double* base = a.work + (int64_t)edge * lay.stride;
  int* ints = reinterpret_cast<int*>(base + lay.ints);
  // the basis kernel that follows may start (its first phase does not read
  // these factors; it waits for this grid before it does)
  cudaTriggerProgrammaticLaunchCompletion();
  double2* rows = ctas == 1 ? reinterpret_cast<double2*>(smem_raw)
                            : reinterpret_cast<double2*>(base + lay.S) + (int64_t)b * c2;
  const int first = rank * kCholThreads + threadIdx.x, step = ctas * kCholThreads;
  for (int64_t idx = first; idx < c2; idx += step) rows[idx] = make_double2(0.0, 0.0);
  if (ctas == 1) __syncthreads();
  else chol::cluster_sync();
  const int r = chol::pivoted_cholesky<CV, RW>(
      chi, ctas, rank, column, a.gram_cut,
      [&](int i, int j) {
        const int64_t o = (int64_t)i * chi + j;
        return make_double2((double)g[o], -(double)g[c2 + o]);
      },
      [&](int i, int k, double2 l) { rows[(int64_t)i * chi + k] = l; }, perm_s);
  if (ctas == 1) __syncthreads();
  else chol::cluster_sync();
  double2* L = reinterpret_cast<double2*>(base + lay.L) + (int64_t)b * c2;
  for (int64_t idx = first; idx < c2; idx += step) {
    const int t = (int)(idx / chi);
    L[idx] = rows[(int64_t)perm_s[t] * chi + (idx - (int64_t)t * chi)];
  }
  if (rank == 0) {
    for (int t = threadIdx.x; t < chi; t += kCholThreads) ints[b * chi + t] = perm_s[t];
    if (threadIdx.x == 0) ints[2 * chi + b] = r;
  }
}

// One CTA per block holds chi <= 64 (16 row warps x 4 rows); a cluster of 4
// holds chi <= 128 and one of 8 chi <= 256 at two rows per warp.  Measured (ncu):
// chi = 64, 51 edges 0.23 ms (0.27 with the block in shared memory and four
// barriers a step); chi = 128, two edges 0.61 ms (1.82 with one CTA per block in
// global memory).  Bound by the FP64 pipe at chi = 64 (two DFMAs a clock).
cudaError_t launch_chol64(const SolveArgs& a, cudaStream_t st) {
  const int ctas = a.chi <= kSmemChi ? 1 : a.chi <= 128 ? 4 : 8;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ctas, 2, a.n_edges);
  cfg.blockDim = dim3(kCholThreads);
  cfg.dynamicSmemBytes = ctas == 1 ? sizeof(double2) * (size_t)a.chi * a.chi : 0;
  cfg.stream = st;
  cudaLaunchAttribute cl[1];
  cl[0].id = cudaLaunchAttributeClusterDimension;
  cl[0].val.clusterDim.x = ctas;
  cl[0].val.clusterDim.y = 1;
  cl[0].val.clusterDim.z = 1;
  cfg.attrs = cl;
  cfg.numAttrs = ctas > 1 ? 1 : 0;
  if (ctas == 1) return cudaLaunchKernelEx(&cfg, chol64_kernel<2, 4>, a, ctas);
  if (ctas == 4) return cudaLaunchKernelEx(&cfg, chol64_kernel<4, 2>, a, ctas);
  return cudaLaunchKernelEx(&cfg, chol64_kernel<8, 2>, a, ctas);
}

// ------------------------------------------------------------ refinement
struct EdgeView {
  int chi, n, act;
  const cd* L;         // [2][chi][chi] lower triangular
  const int* perm;     // [2][chi]
  const int* rank;     // [2]
  const cd* U;         // [n][n]: column m at U + n m
  cd* U1;              // [chi][n]: refined kept columns
  const double* lam0;  // [n]
  double* lam1;        // [chi]
  const double* misc;  // [0] sum of sigma^2 of the start
  const float* gw;     // [q][re|im][chi][chi] the open-q environments N_q^w (FP32 inputs)
};

__device__ EdgeView edge_view(const SolveArgs& a, int edge) {
  const RefineLayout lay = refine_layout(a.chi);
  double* base = a.work + (int64_t)edge * lay.stride;
  EdgeView v;
  v.chi = a.chi;
  v.n = 2 * a.chi;
  const int* ints = reinterpret_cast<const int*>(base + lay.ints);
  v.perm = ints;
  v.rank = ints + 2 * a.chi;
  v.act = ints[2 * a.chi + 2];
  v.L = reinterpret_cast<const cd*>(base + lay.L);
  v.U = reinterpret_cast<const cd*>(base + lay.U);
  v.U1 = reinterpret_cast<cd*>(base + lay.U1);
  v.lam0 = base + lay.lam0;
  v.lam1 = base + lay.lam1;
  v.misc = base + lay.misc;
  v.gw = a.gram + (int64_t)edge * 8 * (int64_t)a.chi * a.chi + 4 * (int64_t)a.chi * a.chi;
  return v;
}

// out(i, j) = sum_{r in [lo(i), hi(i))} arow(i, r) * B[j * ldb + bidx(i, r)]
// for the rows i < nrows and the columns j0 .. j0 + J - 1 of B; store(i, j,
// value).  Bound by the FP64 pipe (two lanes a clock: a warp's instruction takes
// it for 16 clocks whatever its active lanes), so the split keeps the FP64
// instructions few: a row is taken by L lanes, the fewest that still give every
// warp rows, whose partial sums need log2(L) additions per column at the end;
// four of a lane's operands are loaded ahead.
template <int L, int J, int kAhead, class RF, class AF, class BF, class SF>
__device__ __forceinline__ void rows_block(int nrows, int j0, const cd* B, int ldb, RF range,
                                           AF arow, BF bidx, SF store) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int sub = lane & (L - 1);
  for (int i0 = warp * (32 / L); i0 < nrows; i0 += kWarps * (32 / L)) {
    const int i = i0 + lane / L;
    int lo = 0, hi = 0;
    if (i < nrows) range(i, lo, hi);
    cd acc[J];
#pragma unroll
    for (int jj = 0; jj < J; ++jj) acc[jj] = cz();
    const cd* bj = B + (int64_t)j0 * ldb;
    int r = lo + sub;
    for (; r + (kAhead - 1) * L < hi; r += kAhead * L) {
      cd av[kAhead];
#pragma unroll
      for (int u = 0; u < kAhead; ++u) av[u] = arow(i, r + u * L);
#pragma unroll
      for (int u = 0; u < kAhead; ++u) {
        const cd* bp = bj + bidx(i, r + u * L);
#pragma unroll
        for (int jj = 0; jj < J; ++jj) cfma(acc[jj], av[u], bp[jj * ldb]);
      }
    }
    for (; r < hi; r += L) {
      const cd av = arow(i, r);
      const cd* bp = bj + bidx(i, r);
#pragma unroll
      for (int jj = 0; jj < J; ++jj) cfma(acc[jj], av, bp[jj * ldb]);
    }
    __syncwarp();
#pragma unroll
    for (int jj = 0; jj < J; ++jj) {
#pragma unroll
      for (int o = L / 2; o > 0; o >>= 1) acc[jj] = cadd(acc[jj], shfl_xor(acc[jj], o));
      if (i < nrows && sub == (jj & (L - 1))) store(i, j0 + jj, acc[jj]);
    }
  }
}

// All cw columns.  SMALL (n <= 64): every CTA runs each product about once, and
// what it costs is fetching its instructions, so the loops stay short: eight
// lanes a row, two columns at a time.  Otherwise two lanes a row (eight up to 64
// rows), eight columns at a time and the rest in smaller groups.
template <int L, class RF, class AF, class BF, class SF>
__device__ __forceinline__ void rows_cols(int nrows, int cw, const cd* B, int ldb, RF range,
                                          AF arow, BF bidx, SF store) {
  int j = 0;
  for (; j + 8 <= cw; j += 8) rows_block<L, 8, 4>(nrows, j, B, ldb, range, arow, bidx, store);
  if (j + 4 <= cw) {
    rows_block<L, 4, 4>(nrows, j, B, ldb, range, arow, bidx, store);
    j += 4;
  }
  if (j + 2 <= cw) {
    rows_block<L, 2, 4>(nrows, j, B, ldb, range, arow, bidx, store);
    j += 2;
  }
  if (j < cw) rows_block<L, 1, 4>(nrows, j, B, ldb, range, arow, bidx, store);
}

template <bool SMALL, class RF, class AF, class BF, class SF>
__device__ __forceinline__ void row_products(int nrows, int cw, const cd* B, int ldb, RF range,
                                             AF arow, BF bidx, SF store) {
  if (SMALL) {
    int j = 0;
    for (; j + 2 <= cw; j += 2) rows_block<8, 2, 1>(nrows, j, B, ldb, range, arow, bidx, store);
    if (j < cw) rows_block<8, 1, 1>(nrows, j, B, ldb, range, arow, bidx, store);
  } else if (nrows > 64) {
    rows_cols<2>(nrows, cw, B, ldb, range, arow, bidx, store);
  } else {
    rows_cols<8>(nrows, cw, B, ldb, range, arow, bidx, store);
  }
}

// One Newton step for the kept columns [j0, j1) of one edge.  Shared-memory
// buffers (column-major, column j at j * n): Uc (the start's columns), B1
// (Y = R_v^H U_c, then P = H U_c), B2 (T = N_q^w Y'_q, then S, then the
// update coefficients), B3 (Y'_q, then Z = conj(G_w) Y, then R); lamc the
// columns' Rayleigh quotients (negated start eigenvalue for tail columns),
// lamf the final eigenvalues.
template <bool SMALL>
__device__ void refine_chunk(const SolveArgs& a, const EdgeView& v, int j0, int j1, cd* Uc, cd* B1,
                             cd* B2, cd* B3, double* lamc, double* lamf) {
  const int chi = v.chi, n = v.n, A = v.act;
  const int64_t c2 = (int64_t)chi * chi;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int jl = min(j1, min(chi, A));
  for (int j = max(j0, jl) + tid; j < j1; j += blockDim.x) v.lam1[j] = 0.0;
  if (j0 >= jl) return;
  const int cw = jl - j0;
  for (int idx = tid; idx < cw * n; idx += blockDim.x) Uc[idx] = v.U[(int64_t)j0 * n + idx];
  __syncthreads();
  // Y = R_v^H U_c: Y[(k, perm_k[s])] = sum_{t <= s, t < rank_k} L_k[s][t] U[(k, t)]
  row_products<SMALL>(
      n, cw, Uc, n,
      [&](int i, int& lo, int& hi) {
        const int k = i / chi, s = i - k * chi;
        lo = 0;
        hi = min(s + 1, v.rank[k]);
      },
      [&](int i, int t) {
        const int k = i / chi, s = i - k * chi;
        return v.L[k * c2 + (int64_t)s * chi + t];
      },
      [&](int i, int t) { return (i / chi) * chi + t; },
      [&](int i, int j, cd val) {
        const int k = i / chi, s = i - k * chi;
        B1[j * n + k * chi + v.perm[k * chi + s]] = val;
      });
  __syncthreads();
  // Z = conj(G_w) Y through the rank-one phase structure of G_w: with the
  // global phase of b(q) chosen so that b_q(q) = 1 and b_k(q) = -i s (k != q),
  // conj(G_w) = sum_q c(q) c(q)^H (x) N_q^w, c(0) = (1, -i s), c(1) = (-i s, 1),
  // so Z = sum_q c(q) (x) N_q^w Y'_q with Y'_q = c(q)^H Y:
  //   Y'_0 = Y_0 + i s Y_1,  Y'_1 = i s Y_0 + Y_1      (into B3)
  //   T_q = N_q^w Y'_q                                  (into B2; two chi x chi products)
  //   Z_0 = T_0 - i s T_1,   Z_1 = -i s T_0 + T_1       (into B3)
  // The factors +-i s are exact, so this is conj(G_w) Y with half the products.
  const double sg = (double)a.sign;
  for (int idx = tid; idx < cw * n; idx += blockDim.x) {
    const int j = idx / n, i = idx - j * n;
    const int q = i / chi, e = i - q * chi;
    const cd y0 = B1[j * n + e], y1 = B1[j * n + chi + e];
    const cd other = q == 0 ? y1 : y0;             // the term multiplied by i s
    const cd mine = q == 0 ? y0 : y1;
    B3[j * n + i] = {mine.x - sg * other.y, mine.y + sg * other.x};
  }
  __syncthreads();
  row_products<SMALL>(
      n, cw, B3, n, [&](int, int& lo, int& hi) { lo = 0; hi = chi; },
      [&](int i, int r) {
        const int q = i / chi, e = i - q * chi;
        const int64_t o = (int64_t)q * 2 * c2 + (int64_t)e * chi + r;
        return cd{(double)v.gw[o], (double)v.gw[c2 + o]};
      },
      [&](int i, int r) { return (i / chi) * chi + r; },
      [&](int i, int j, cd val) { B2[j * n + i] = val; });
  __syncthreads();
  for (int idx = tid; idx < cw * n; idx += blockDim.x) {
    const int j = idx / n, i = idx - j * n;
    const int k = i / chi, e = i - k * chi;
    const cd t0 = B2[j * n + e], t1 = B2[j * n + chi + e];
    const cd other = k == 0 ? t1 : t0;             // the term multiplied by -i s
    const cd mine = k == 0 ? t0 : t1;
    B3[j * n + i] = {mine.x + sg * other.y, mine.y - sg * other.x};
  }
  __syncthreads();
  // P = R_v Z: P[(b, t)] = sum_{s >= t} conj(L_b[s][t]) Z[(b, perm_b[s])], zero for t >= rank_b
  row_products<SMALL>(
      n, cw, B3, n,
      [&](int i, int& lo, int& hi) {
        const int b = i / chi, t = i - b * chi;
        lo = t;
        hi = t < v.rank[b] ? chi : t;
      },
      [&](int i, int s) {
        const int b = i / chi, t = i - b * chi;
        return cconj(v.L[b * c2 + (int64_t)s * chi + t]);
      },
      [&](int i, int s) {
        const int b = i / chi;
        return b * chi + v.perm[b * chi + s];
      },
      [&](int i, int j, cd val) { B1[j * n + i] = val; });
  __syncthreads();
  // S = U_A^H P and R = I - U_A^H U_c
  row_products<SMALL>(
      A, cw, B1, n, [&](int, int& lo, int& hi) { lo = 0; hi = n; },
      [&](int i, int r) { return cconj(v.U[(int64_t)i * n + r]); }, [&](int, int r) { return r; },
      [&](int i, int j, cd val) { B2[j * n + i] = val; });
  row_products<SMALL>(
      A, cw, Uc, n, [&](int, int& lo, int& hi) { lo = 0; hi = n; },
      [&](int i, int r) { return cconj(v.U[(int64_t)i * n + r]); }, [&](int, int r) { return r; },
      [&](int i, int j, cd val) {
        B3[j * n + i] = {(i == j0 + j ? 1.0 : 0.0) - val.x, -val.y};
      });
  __syncthreads();
  // head columns (lambda_0 >= kHead lambda_0[0]) take the Newton step with
  // the Rayleigh quotient lambda_j = S_jj / (1 - R_jj); tail columns keep
  // their start's eigenvalue (lamc = -lambda_0 marks them)
  const double lhead = kHead * v.lam0[0];
  for (int j = tid; j < cw; j += blockDim.x) {
    const int jg = j0 + j;
    if (v.lam0[jg] >= lhead) {
      const double s = B2[j * n + jg].x, r = B3[j * n + jg].x;
      const double lam = s / (1.0 - r);
      lamc[j] = (lam > 0.0 && isfinite(lam)) ? lam : 0.0;
    } else {
      lamc[j] = -v.lam0[jg];
    }
  }
  __syncthreads();
  // Update coefficients c_ij (into B2), one warp per column j.  Head column:
  // c_ij = E_ij - S_ij / lambda_j - R_ij with the Newton E_ij (R_ij / 2 for
  // pairs that are not separated), and the final eigenvalue
  // lambda_j - sum_i |E_ij|^2 (lambda_i - lambda_j): the Rayleigh quotient of
  // the start carries that second-order contamination from the components
  // the step removes.  Tail column: c_ij = R_ij - conj(E_ji) against a head
  // column i (the mirror of the head column's correction, which keeps the
  // pair orthogonal to first order) and R_ij / 2 against a tail column.
  const double s00 = sqrt(fmax(v.lam0[0], 0.0));
  for (int j = warp; j < cw; j += kWarps) {
    const int jg = j0 + j;
    const double lj = lamc[j];
    const double ilj = lj > 0.0 ? 1.0 / lj : 0.0;
    double corr = 0.0;
    for (int i = lane; i < A; i += 32) {
      const cd s = B2[j * n + i], r = B3[j * n + i];
      const double li = v.lam0[i];
      cd c = cz();
      if (lj > 0.0) {
        cd e;
        if (i == jg) {
          e = cscale(r, 0.5);
        } else {
          const cd num = cadd(s, cscale(r, lj));
          const double den = lj - li;
          const double noise = kNoise * s00 * sqrt(fmax(li, 0.0));
          if (16.0 * cabs2(num) < den * den && fabs(den) > noise) {
            e = cscale(num, 1.0 / den);
            corr += cabs2(e) * (li - lj);
          } else {
            e = cscale(r, 0.5);
          }
        }
        c = csub(csub(e, cscale(s, ilj)), r);
      } else if (lj < 0.0) {
        if (i != jg && li >= lhead) {
          const cd num = cadd(cconj(s), cscale(cconj(r), li));
          const double den = li + lj;  // lambda_i - lambda_j
          const double noise = kNoise * s00 * (sqrt(li) + sqrt(-lj));
          const cd eji = (16.0 * cabs2(num) < den * den && fabs(den) > noise)
                             ? cscale(num, 1.0 / den)
                             : cscale(cconj(r), 0.5);
          c = csub(r, cconj(eji));
        } else {
          c = cscale(r, 0.5);
        }
      }
      B2[j * n + i] = c;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) corr += __shfl_xor_sync(0xffffffffu, corr, o);
    if (lane == 0) lamf[j] = lj > 0.0 ? lj - corr : v.lam0[jg];
  }
  __syncthreads();
  // u_j' = u_j + P_j / lambda_j + sum_{i < A} u_i c_ij for head columns,
  // u_j + sum_i u_i c_ij for tail columns; a head column without a positive
  // Rayleigh quotient keeps its start
  constexpr int JU = SMALL ? 1 : kJU, AHEAD = SMALL ? 2 : 8;
  const int ng = (cw + JU - 1) / JU;
  for (int idx = tid; idx < n * ng; idx += blockDim.x) {
    const int r = idx % n, jb = (idx / n) * JU;
    cd acc[JU];
#pragma unroll
    for (int jj = 0; jj < JU; ++jj) acc[jj] = cz();
    const int nj = min(JU, cw - jb);
    for (int i0 = 0; i0 < A; i0 += AHEAD) {
      cd u[AHEAD];
#pragma unroll
      for (int t = 0; t < AHEAD; ++t) u[t] = i0 + t < A ? v.U[(int64_t)(i0 + t) * n + r] : cz();
#pragma unroll
      for (int t = 0; t < AHEAD; ++t) {
        if (i0 + t >= A) break;
#pragma unroll
        for (int jj = 0; jj < JU; ++jj)
          if (jj < nj) cfma(acc[jj], u[t], B2[(jb + jj) * n + i0 + t]);
      }
    }
#pragma unroll
    for (int jj = 0; jj < JU; ++jj) {
      const int j = jb + jj;
      if (jj >= nj) continue;
      const double lj = lamc[j];
      cd out = Uc[j * n + r];
      if (lj > 0.0) out = cadd(cadd(out, cscale(B1[j * n + r], 1.0 / lj)), acc[jj]);
      else if (lj < 0.0) out = cadd(out, acc[jj]);
      v.U1[(int64_t)(j0 + j) * n + r] = out;
    }
  }
  for (int j = tid; j < cw; j += blockDim.x) v.lam1[j0 + j] = lamf[j];
  __syncthreads();
}

// Bound by the FP64 pipe.  Measured (ncu): chi = 64, 51 edges 1.78 ms (2.21 with
// eight lanes on every row and every group of eight columns reduced whole);
// chi = 37, 24 edges 0.24 ms (0.42); with the short loops of SMALL chi = 21, 7
// edges 38 us (63 with the unrolled ones, 101 at first), chi = 16, 48 edges 66 us
// (100, 127).
// The kept-column slots of all edges, ne * chi, split evenly over the grid: each
// block takes a contiguous range (split further at edge boundaries and into
// pieces of at most cwmax columns).
template <bool SMALL>
__global__ void __launch_bounds__(kThreads, 1) refine_kernel(SolveArgs a, int cwmax) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int chi = a.chi, n = 2 * chi;
  cd* Uc = reinterpret_cast<cd*>(smem_raw);
  cd* B1 = Uc + (int64_t)cwmax * n;
  cd* B2 = B1 + (int64_t)cwmax * n;
  cd* B3 = B2 + (int64_t)cwmax * n;
  double* lamc = reinterpret_cast<double*>(B3 + (int64_t)cwmax * n);
  double* lamf = lamc + cwmax;
  const int64_t T = (int64_t)a.n_edges * chi;
  const int64_t g0 = (int64_t)blockIdx.x * T / gridDim.x;
  const int64_t g1 = (int64_t)(blockIdx.x + 1) * T / gridDim.x;
  for (int64_t g = g0; g < g1;) {
    const int e = (int)(g / chi), j0 = (int)(g % chi);
    const int jend = (int)min((int64_t)chi, j0 + (g1 - g));
    const EdgeView v = edge_view(a, e);
    for (int s = j0; s < jend; s += cwmax) refine_chunk<SMALL>(a, v, s, min(jend, s + cwmax), Uc, B1, B2, B3, lamc, lamf);
    g += jend - j0;
  }
}

// ------------------------------------------------------------ leg matrices
// Same split of the kept-column slots.  Per edge: the kept set (the chi
// candidates with sigma above svd_cut * the largest), ||sigma||, and each
// column's slot in decreasing order.  Per chunk of refined columns u (both
// blocks b), in FP64:
//   Y = L_b u_b          (R_v^H u, so that C_w = R_v^T conj(u) = conj(Y)), and
//   W with L_b^H W = u_b (back substitution: C_v = R_v^+ u),
// then D_v[b][perm_b[s]][pos] = W[(b, s)] sqrt(sigma / ||sigma||) and
// D_w[q][e][pos] = sum_b b_b(q) conj(Y[(b, pinv_b(e))]) / sqrt(sigma ||sigma||)
// with b_b(q) = exp(s i pi/4 s_b s_q), as the gate split gives.
// Measured (ncu): chi = 64, 51 edges 0.53 ms (0.56 with the substitution over the
// whole block, two barriers a step), chi = 37, 24 edges 0.15 ms (0.21), chi = 21,
// 7 edges 45 us (59).
template <bool SMALL>
__global__ void __launch_bounds__(kThreads, 2) legs_kernel(SolveArgs a, int cwmax) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int chi = a.chi, n = 2 * chi;
  cd* Ub = reinterpret_cast<cd*>(smem_raw);        // [cwmax][n] refined columns
  cd* Yb = Ub + (int64_t)cwmax * n;                // [cwmax][n]
  double* lam_s = reinterpret_cast<double*>(Yb + (int64_t)cwmax * n);  // [chi]
  int* pos_s = reinterpret_cast<int*>(lam_s + chi);                     // [chi]
  int* pinv = pos_s + chi;                                             // [2][chi]
  unsigned char* keep_s = reinterpret_cast<unsigned char*>(pinv + 2 * chi);  // [chi]
  __shared__ double scal[4];  // nrm, smax, kept count, discarded weight
  const int64_t c2 = (int64_t)chi * chi;
  const int tid = threadIdx.x;
  const int64_t T = (int64_t)a.n_edges * chi;
  const int64_t g0 = (int64_t)blockIdx.x * T / gridDim.x;
  const int64_t g1 = (int64_t)(blockIdx.x + 1) * T / gridDim.x;
  const double sg = (double)a.sign;
  const double c45 = 0.70710678118654752440;
  for (int64_t g = g0; g < g1;) {
    const int e = (int)(g / chi), j0 = (int)(g % chi);
    const int j1 = (int)min((int64_t)chi, j0 + (g1 - g));
    g += j1 - j0;
    const EdgeView v = edge_view(a, e);
    const int cand = min(chi, v.act);
    for (int m = tid; m < chi; m += blockDim.x) lam_s[m] = m < cand ? v.lam1[m] : 0.0;
    for (int i = tid; i < 2 * chi; i += blockDim.x) pinv[(i / chi) * chi + v.perm[i]] = i % chi;
    __syncthreads();
    if (tid == 0) {
      double smax = 0.0;
      for (int m = 0; m < cand; ++m) smax = fmax(smax, lam_s[m] > 0.0 ? sqrt(lam_s[m]) : 0.0);
      double kept = 0.0, tot = 0.0;
      int nk = 0;
      for (int m = 0; m < chi; ++m) {
        const double s = lam_s[m] > 0.0 ? sqrt(lam_s[m]) : 0.0;
        const bool k = m < cand && s > 0.0 && s > a.svd_cut * smax;
        keep_s[m] = k;
        if (k) { kept += lam_s[m]; ++nk; }
        tot += m < cand ? fmax(lam_s[m], 0.0) : fmax(v.lam0[m], 0.0);
      }
      for (int m = chi; m < n; ++m) tot += fmax(v.lam0[m], 0.0);
      scal[0] = sqrt(kept);
      scal[1] = smax;
      scal[2] = nk;
      scal[3] = tot > 0.0 ? fmax(tot - kept, 0.0) / tot : 0.0;
    }
    __syncthreads();
    const int nk = (int)scal[2];
    for (int m = tid; m < chi; m += blockDim.x) {
      int p = 0;
      if (keep_s[m]) {
        for (int q = 0; q < chi; ++q)
          p += keep_s[q] && (lam_s[q] > lam_s[m] || (lam_s[q] == lam_s[m] && q < m));
      } else {
        p = nk;
        for (int q = 0; q < m; ++q) p += !keep_s[q];
      }
      pos_s[m] = p;
    }
    const double nrm = scal[0];
    const bool ok = nrm > 0.0 && isfinite(nrm);
    if (j0 == 0 && tid == 0) {
      double* st = a.stats + 4 * e;
      st[0] = scal[3];
      st[1] = nk;
      st[2] = scal[1];
      if (!ok) atomicOr(a.flags, 1);
    }
    float* dv = a.dmat + (int64_t)e * 8 * c2;
    float* dw = dv + 4 * c2;
    for (int js = j0; js < j1; js += cwmax) {
      const int cw = min(cwmax, j1 - js);
      for (int idx = tid; idx < cw * n; idx += blockDim.x) {
        const int jj = idx / n;
        Ub[idx] = keep_s[js + jj] ? v.U1[(int64_t)js * n + idx] : cz();
      }
      __syncthreads();
      // Y = L_b u_b (from the unmodified columns) first
      row_products<SMALL>(
          n, cw, Ub, n,
          [&](int i, int& lo, int& hi) {
            const int b = i / chi, t = i - b * chi;
            lo = 0;
            hi = min(t + 1, v.rank[b]);
          },
          [&](int i, int k) {
            const int b = i / chi, t = i - b * chi;
            return v.L[b * c2 + (int64_t)t * chi + k];
          },
          [&](int i, int k) { return (i / chi) * chi + k; },
          [&](int i, int j, cd val) { Yb[j * n + i] = val; });
      __syncthreads();
      // W: solve L_b^H w = u_b for every column of the chunk by back
      // substitution over s = rank_b - 1 .. 0, in place in Ub: w[s] = u[s] /
      // L[s][s], then u[t] -= conj(L[s][t]) w[s] for t < s.  One warp per
      // (column, block) holds the column in registers (lane t % 32) and passes
      // w[s] on by shuffle, so that a step waits for no other warp; the next
      // row of L is loaded ahead.
      for (int task = tid >> 5; task < 2 * cw; task += kWarps) {
        const int b = task & 1, jj = task >> 1, lane = tid & 31;
        cd* uc = Ub + jj * n + b * chi;
        const cd* Lb = v.L + b * c2;
        for (int base = (v.rank[b] - 1) / 32 * 32; base >= 0 && v.rank[b] > 0; base -= 32) {
          // the triangle of columns base .. base + 31, then the rows above it
          const int t = base + lane;
          cd u = t < v.rank[b] ? uc[t] : cz();
          const int last = min(v.rank[b], base + 32) - 1;
          const double inv = t <= last ? 1.0 / Lb[(int64_t)t * chi + t].x : 0.0;
          cd row = cz();
          if (t <= last) row = Lb[(int64_t)last * chi + t];
          for (int sidx = last; sidx >= base; --sidx) {
            cd next = cz();
            if (sidx > base && t < sidx) next = Lb[(int64_t)(sidx - 1) * chi + t];
            const double is = __shfl_sync(0xffffffffu, inv, sidx & 31);
            cd w = {__shfl_sync(0xffffffffu, u.x, sidx & 31),
                    __shfl_sync(0xffffffffu, u.y, sidx & 31)};
            w = cscale(w, is);
            if (t == sidx) {
              u = w;
            } else if (t < sidx) {
              const cd l = cconj(row);
              u.x = fma(-l.x, w.x, u.x);
              u.x = fma(l.y, w.y, u.x);
              u.y = fma(-l.x, w.y, u.y);
              u.y = fma(-l.y, w.x, u.y);
            }
            row = next;
          }
          if (t <= last) uc[t] = u;
          __syncwarp();
          for (int t2 = lane; t2 < base; t2 += 32) {
            cd x = uc[t2];
            for (int sidx = last; sidx >= base; --sidx) {
              const cd l = cconj(Lb[(int64_t)sidx * chi + t2]);
              const cd w = uc[sidx];
              x.x = fma(-l.x, w.x, x.x);
              x.x = fma(l.y, w.y, x.x);
              x.y = fma(-l.x, w.y, x.y);
              x.y = fma(-l.y, w.x, x.y);
            }
            uc[t2] = x;
          }
          __syncwarp();
        }
      }
      __syncthreads();
      cd* Wb_ = Ub;  // W now occupies Ub (entries past each block's rank unused)
      // D_v and D_w columns, one thread per (column, e)
      for (int idx = tid; idx < cw * chi; idx += blockDim.x) {
        const int jj = idx / chi, ei = idx - jj * chi, m = js + jj;
        const int p = pos_s[m];
        const bool keep = ok && keep_s[m];
        const double sgm = keep ? sqrt(lam_s[m]) : 0.0;
        const double fv = keep ? sqrt(sgm / nrm) : 0.0;
        const double fw = keep ? 1.0 / sqrt(sgm * nrm) : 0.0;
        const int64_t o = (int64_t)ei * chi + p;
        cd w0 = cz(), w1 = cz();
        for (int b = 0; b < 2; ++b) {
          const int s = pinv[b * chi + ei];
          const cd z = (keep && s < v.rank[b]) ? cscale(Wb_[jj * n + b * chi + s], fv) : cz();
          dv[(int64_t)b * 2 * c2 + o] = (float)z.x;
          dv[(int64_t)b * 2 * c2 + c2 + o] = (float)z.y;
          const cd y = Yb[jj * n + b * chi + s];
          const cd cwv = {y.x * fw, -y.y * fw};
          const double sb = (b == 0) ? 1.0 : -1.0;
          w0 = cadd(w0, cmul({c45, sg * sb * c45}, cwv));
          w1 = cadd(w1, cmul({c45, -sg * sb * c45}, cwv));
        }
        dw[o] = (float)w0.x;
        dw[c2 + o] = (float)w0.y;
        dw[2 * c2 + o] = (float)w1.x;
        dw[3 * c2 + o] = (float)w1.y;
      }
      for (int jj = tid; jj < cw; jj += blockDim.x) {
        const int m = js + jj, p = pos_s[m];
        const bool keep = ok && keep_s[m];
        if (a.s_out) a.s_out[(int64_t)e * chi + p] = keep ? sqrt(lam_s[m]) / nrm : 0.0;
      }
      if (ok && a.msg) {
        float* m0 = a.msg + (int64_t)a.msg_vw[2 * e] * 2 * c2;
        float* m1 = a.msg + (int64_t)a.msg_vw[2 * e + 1] * 2 * c2;
        for (int idx = tid; idx < cw * chi; idx += blockDim.x) {
          const int jj = idx / chi, k = idx - jj * chi, m = js + jj;
          const int p = pos_s[m];
          const float val = (k == p && keep_s[m]) ? (float)(sqrt(lam_s[m]) / nrm) : 0.f;
          m0[(int64_t)p * chi + k] = val; m0[c2 + (int64_t)p * chi + k] = 0.f;
          m1[(int64_t)p * chi + k] = val; m1[c2 + (int64_t)p * chi + k] = 0.f;
        }
      }
      __syncthreads();
    }
  }
}

// Shared-memory limits of the refined solve's kernels, raised once per device to
// the largest request any chi <= kMaxChi makes, so that concurrent launches (the
// job server's slots) never lower a limit another thread relies on.
constexpr size_t kCholSmemMax = sizeof(double2) * kSmemChi * kSmemChi;
constexpr size_t kRefineSmemMax = kSmemBudget + 4096;
constexpr size_t kLegsSmemMax = kSmemBudget / 2 + 8192;

int sm_count() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 148;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 148;
  return sms > 0 ? sms : 148;
}

}  // namespace

cudaError_t refine_prepare() {
  static DeviceOnce once;
  return once([] {
    cudaError_t result = cudaFuncSetAttribute(
        chol64_kernel<2, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCholSmemMax);
    for (auto k : {refine_kernel<false>, refine_kernel<true>})
      if (result == cudaSuccess)
        result = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)kRefineSmemMax);
    for (auto k : {legs_kernel<false>, legs_kernel<true>})
      if (result == cudaSuccess)
        result = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)kLegsSmemMax);
    return result;
  });
}

bool solve_refined_supported(int chi) {
  if (chi >= 1 && chi <= kSmemChi) return solve32_supported(chi);
  return chi <= kMaxChi && (2 * chi) % 32 == 0;  // the global-memory basis kernel
}

cudaError_t launch_solve_refined_basis(const SolveArgs& a, cudaStream_t st) {
  if (a.n_edges <= 0) return cudaSuccess;
  if (!solve_refined_supported(a.chi)) return cudaErrorInvalidValue;
  // 1. FP64 Cholesky of the v-side Gram blocks
  cudaError_t e = refine_prepare();
  if (e != cudaSuccess) return e;
  if ((e = launch_chol64(a, st)) != cudaSuccess) return e;
  // 2. FP32 starting basis
  SolveArgs b = a;
  b.basis = 1;
  return a.chi <= kSmemChi ? launch_solve32(b, st) : launch_basis_gmem(b, st);
}

cudaError_t launch_solve_refined_newton(const SolveArgs& a, cudaStream_t st) {
  if (a.n_edges <= 0) return cudaSuccess;
  if (!solve_refined_supported(a.chi)) return cudaErrorInvalidValue;
  const int chi = a.chi, n = 2 * chi;
  const bool small = n <= 64;
  // 3. FP64 Newton step, the kept-column slots balanced over the SMs
  const int64_t T = (int64_t)a.n_edges * chi;
  const int cw_fit = (int)(kSmemBudget / (sizeof(cd) * 4 * (size_t)n + 2 * sizeof(double)));
  int grid = (int)std::min<int64_t>(T, sm_count());
  grid = (int)std::max<int64_t>(grid, (T + cw_fit - 1) / cw_fit);
  const int cwmax = (int)((T + grid - 1) / grid);
  const size_t sm_ref = sizeof(cd) * 4 * (size_t)cwmax * n + 2 * sizeof(double) * cwmax;
  cudaError_t e = refine_prepare();
  if (e != cudaSuccess) return e;
  if (sm_ref > kRefineSmemMax) return cudaErrorInvalidValue;
  if (small) refine_kernel<true><<<grid, kThreads, sm_ref, st>>>(a, cwmax);
  else refine_kernel<false><<<grid, kThreads, sm_ref, st>>>(a, cwmax);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  // 4. FP64 leg matrices, spectrum and messages.  The back substitution is a
  // chain of chi dependent passes: two CTAs per SM (half the columns each)
  // overlap their latencies.
  int grid_l = (int)std::min<int64_t>(T, 2 * (int64_t)sm_count());
  const int cw_fit_l = (int)((kLegsSmemMax - 8192) / (sizeof(cd) * 2 * (size_t)n));
  grid_l = (int)std::max<int64_t>(grid_l, (T + cw_fit_l - 1) / cw_fit_l);
  const int cw_l = (int)((T + grid_l - 1) / grid_l);
  const size_t sm_legs = sizeof(cd) * 2 * (size_t)cw_l * n + sizeof(double) * chi +
                         sizeof(int) * 3 * chi + chi + 16;
  if (sm_legs > kLegsSmemMax) return cudaErrorInvalidValue;
  if (small) legs_kernel<true><<<grid_l, kThreads, sm_legs, st>>>(a, cw_l);
  else legs_kernel<false><<<grid_l, kThreads, sm_legs, st>>>(a, cw_l);
  return cudaGetLastError();
}

cudaError_t launch_solve_refined(const SolveArgs& a, cudaStream_t st) {
  cudaError_t e = launch_solve_refined_basis(a, st);
  if (e != cudaSuccess) return e;
  return launch_solve_refined_newton(a, st);
}

}  // namespace tnbp
