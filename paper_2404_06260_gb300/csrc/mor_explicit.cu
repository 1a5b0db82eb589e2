// Paper-literal weights on the GPU (Sec. 4, Lemma 4.1, Eq. (14)) for subdomains small
// enough for dense factors: batched dense Cholesky factorisations, triangular solves
// and the pieces of the explicit weighted SVD.
//
//   - k_ell_to_dense: scatter a sliced-ELL block into a dense per-subdomain matrix
//     (row-major, leading dimension = its order) with caller-given local indices;
//   - k_potrf_diag / _panel / _update: right-looking blocked Cholesky A = L L^T in place,
//     64-column panels, batched over subdomains of different orders (Golub & Van Loan
//     Alg. 4.2.2 by blocks);
//   - k_transpose_block: copy of a square block, transposed (the triangular solves
//     walk columns of a factor as contiguous rows of its transpose);
//   - k_trsv_cols: two vectors per warp: forward (L x = b) or backward (U x = b)
//     substitution, column-oriented;
//   - k_trsv_rows: one row per warp: x R = y with R upper (row-major), for
//     X = Y R_BB^{-1};
//   - k_trmv_upper: y = U z per vector;
//   - k_node_normals: the Gaussian test matrix S of the paper's sketch on B.
// Everything is binary64.
#include "mor_dev.cuh"
#include "mor_kernels.h"

#include <algorithm>

namespace mor {
namespace {

constexpr int kNB = 64;  // Cholesky panel width and update tile

// D[doff[sd] + (rloc[r] - r_sub[sd]) * ld[sd] + (cloc[c] - c_sub[sd])] = A[r, c] for
// the stored entries of rows r in [0, n_rows) whose local row rloc[r] - r_sub[sd] lies
// in [0, r_n[sd]) and whose local column cloc[c] - c_sub[sd] lies in [0, ncols[sd]).
// sd = row_sd[r].
__global__ void k_ell_to_dense(int64_t n_rows, const int32_t* __restrict__ row_sd,
                               const int32_t* __restrict__ rloc,
                               const int32_t* __restrict__ cloc, EllView<double> A,
                               const int32_t* __restrict__ r_sub,
                               const int32_t* __restrict__ r_n,
                               const int32_t* __restrict__ c_sub,
                               const int32_t* __restrict__ ncols,
                               const int32_t* __restrict__ ld, const int64_t* __restrict__ doff,
                               double* __restrict__ D) {
  const int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (r >= n_rows) return;
  const int sd = row_sd[r];
  const int lr = rloc[r] - r_sub[sd];
  if (lr < 0 || lr >= r_n[sd]) return;
  const int w = A.width[r >> 5];
  const int64_t base = doff[sd] + (int64_t)lr * ld[sd];
  for (int j = 0; j < w; ++j) {
    const int64_t at = ell_at(r, j, A.W);
    const int c = A.col[at];
    if (c < 0) continue;
    const int lc = cloc[c] - c_sub[sd];
    if (lc < 0 || lc >= ncols[sd]) continue;
    D[base + lc] = A.val[at];
  }
}

// b / d within one unit in the last place from r = 1 / d rounded: the product b r and one
// step of Markstein's correction, whose remainder is exact (P. Markstein, IBM J. Res. Dev.
// 34, 1990).  The reciprocal of a pivot is formed once for all the entries it divides.  That
// holds while r is a normal number, the remainder does not underflow (b = 0 or above 2^-959)
// and the quotient does not overflow; elsewhere, and for infinities and NaN, it divides: in a
// function of its own, as the compiler would otherwise run the division beside the product.
// (Division everywhere: diagonal block 49 -> 76 us, panel 42 -> 82, column solve 261 -> 355.)
__device__ __noinline__ double div_slow(double b, double d) { return b / d; }
__device__ __forceinline__ double div_by(double b, double d, double r) {
  const double q = b * r;
  const int eb = (__double2hiint(b) >> 20) & 0x7FF, ed = (__double2hiint(d) >> 20) & 0x7FF;
  const bool safe = (unsigned)(ed - 2) <= 2042u && eb - ed < 1000 && (eb >= 64 || !nonzero(b)) &&
                    eb < 2047;
  if (!safe) return div_slow(b, d);
  return fma(fma(-d, q, b), r, q);
}

// Diagonal block j0 of every subdomain's matrix (order n[sd]), nb columns: factored as
// L D L^T in registers (lower triangle, one multiply-add per entry and column), the square
// roots of the pivots at the end, in parallel.  A non-positive pivot sets *bad.  A chain of
// nb steps: a square root in front of every division and the update's index arithmetic
// made a step 4,500 clocks.  8 blocks of 64: 49 us, with the panel below 91 instead of 300.
constexpr int kPotrfOwn = (kNB * (kNB + 1) / 2 + 255) / 256;  // entries per thread
__global__ void __launch_bounds__(256)
    k_potrf_diag(double* D, const int64_t* __restrict__ doff, const int32_t* __restrict__ nn,
                 int j0, int* bad) {
  __shared__ double col[2][kNB], colp[kNB];  // column c, and column c / a_cc
  __shared__ double rs[kNB];                 // 1 / sqrt of the pivots
  const int sd = blockIdx.x, n = nn[sd];
  if (j0 >= n) return;
  const int nb = min(kNB, n - j0);
  double* A = D + doff[sd] + (int64_t)j0 * n + j0;
  const int tid = threadIdx.x;
  double a[kPotrfOwn];
  int ri[kPotrfOwn], ci[kPotrfOwn];  // entry (ri, ci), ci <= ri; ci = -1: none
#pragma unroll
  for (int m = 0; m < kPotrfOwn; ++m) {
    const int idx = tid + m * 256;
    a[m] = 0.0;
    ri[m] = ci[m] = -1;
    if (idx < nb * (nb + 1) / 2) {
      // columns from the last to the first: the entries of the columns still to come are
      // the first ones, and whole warps run out of work as the factorisation proceeds
      int c = (int)((sqrtf(8.0f * (float)idx + 1.0f) - 1.0f) * 0.5f);
      while ((c + 1) * (c + 2) / 2 <= idx) ++c;
      while (c * (c + 1) / 2 > idx) --c;
      ci[m] = nb - 1 - c;
      ri[m] = ci[m] + idx - c * (c + 1) / 2;
      a[m] = A[(int64_t)ri[m] * n + ci[m]];
      if (ci[m] == 0) col[0][ri[m]] = a[m];
    }
  }
  for (int c = 0; c < nb; ++c) {
    __syncthreads();
    const double* cc = col[c & 1];
    double* cn = col[(c + 1) & 1];
    if (tid >= c && tid < nb) {
      double d = cc[c];
      if (!(d > 0.0)) {
        if (tid == c) atomicExch(bad, 1);
        d = 1.0;
      }
      const double r = 1.0 / d;
      colp[tid] = div_by(cc[tid], d, r);
      if (tid == c) rs[c] = d;
    }
    __syncthreads();
#pragma unroll
    for (int m = 0; m < kPotrfOwn; ++m)
      if (ci[m] > c) {
        a[m] -= cc[ri[m]] * colp[ci[m]];
        if (ci[m] == c + 1) cn[ri[m]] = a[m];
      }
  }
  __syncthreads();
  // rs holds the pivots d; L_rc = a_rc / sqrt(d_c)
  if (tid < nb) {
    const double l = sqrt(rs[tid]);
    colp[tid] = l;
    rs[tid] = 1.0 / l;
  }
  __syncthreads();
#pragma unroll
  for (int m = 0; m < kPotrfOwn; ++m)
    if (ci[m] >= 0) {
      const int r = ri[m], c = ci[m];
      A[(int64_t)r * n + c] = r == c ? colp[c] : div_by(a[m], colp[c], rs[c]);
      if (r != c) A[(int64_t)c * n + r] = 0.0;
    }
}

// The panel below diagonal block j0: rows i >= j0 + nb satisfy L[i, j0:j0+nb] L_dd^T =
// A[i, j0:j0+nb].  32 rows per block, four lanes per row, each with every fourth column in
// registers: x_c comes by shuffle and its multiply-adds on the columns behind it are
// independent.  grid (n_sd, row chunks).  One thread per row and one block per subdomain
// cost most of 300 us a panel; 42 now (8 subdomains of order up to 340).
constexpr int kPanelRows = 32;
__global__ void __launch_bounds__(4 * kPanelRows)
    k_potrf_panel(double* D, const int64_t* __restrict__ doff, const int32_t* __restrict__ nn,
                  int j0) {
  __shared__ double Lt[kNB][kNB + 4];  // Lt[c][s] = L_dd[s][c]
  __shared__ double rc[kNB];
  const int sd = blockIdx.x, n = nn[sd];
  const int i0 = j0 + kNB + blockIdx.y * kPanelRows;
  if (i0 >= n) return;  // rows below: the block has kNB columns
  double* A = D + doff[sd];
  const int tid = threadIdx.x, h = tid & 3;
  for (int idx = tid; idx < kNB * kNB; idx += 4 * kPanelRows) {
    const int s = idx / kNB, c = idx % kNB;
    Lt[c][s] = A[(int64_t)(j0 + s) * n + j0 + c];
  }
  __syncthreads();
  if (tid < kNB) rc[tid] = 1.0 / Lt[tid][tid];
  const int i = i0 + (tid >> 2);
  double* row = A + (int64_t)min(i, n - 1) * n + j0;
  double x[kNB / 4];
#pragma unroll
  for (int q = 0; q < kNB / 4; ++q) x[q] = i < n ? row[4 * q + h] : 0.0;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < kNB / 4; ++q)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int c = 4 * q + e;
      double v = div_by(x[q], Lt[c][c], rc[c]);
      v = __shfl_sync(0xFFFFFFFFu, v, e, 4);
      if (h == e) x[q] = v;
      if (h > e) x[q] = fma(-v, Lt[c][4 * q + h], x[q]);
#pragma unroll
      for (int p = q + 1; p < kNB / 4; ++p) x[p] = fma(-v, Lt[c][4 * p + h], x[p]);
    }
  if (i < n)
#pragma unroll
    for (int q = 0; q < kNB / 4; ++q) row[4 * q + h] = x[q];
}

// trailing update of panel j0: A[I, J] -= P_I P_J^T for the 64 x 64 tiles I >= J of the
// rows and columns after the panel (P = the panel's columns); grid (n_sd, tiles)
__global__ void __launch_bounds__(256)
    k_potrf_update(double* D, const int64_t* __restrict__ doff, const int32_t* __restrict__ nn,
                   int j0) {
  extern __shared__ double sm[];
  double* PI = sm;                        // kNB x (kNB + 1)
  double* PJ = sm + kNB * (kNB + 1);
  const int sd = blockIdx.x, n = nn[sd];
  const int t0 = j0 + kNB;
  if (t0 >= n) return;
  const int T = (n - t0 + kNB - 1) / kNB;
  // tile index -> (I, J), I >= J, row-major over the lower triangle of tiles
  const int t = blockIdx.y;
  int I = (int)((sqrt(8.0 * t + 1.0) - 1.0) * 0.5);
  while ((I + 1) * (I + 2) / 2 <= t) ++I;
  while (I * (I + 1) / 2 > t) --I;
  const int J = t - I * (I + 1) / 2;
  if (I >= T) return;
  double* A = D + doff[sd];
  const int i0 = t0 + I * kNB, c0 = t0 + J * kNB;
  const int tid = threadIdx.y * 16 + threadIdx.x;
  for (int idx = tid; idx < kNB * kNB; idx += 256) {
    const int r = idx / kNB, q = idx % kNB;
    PI[r * (kNB + 1) + q] = (i0 + r < n) ? A[(int64_t)(i0 + r) * n + j0 + q] : 0.0;
    PJ[r * (kNB + 1) + q] = (c0 + r < n) ? A[(int64_t)(c0 + r) * n + j0 + q] : 0.0;
  }
  __syncthreads();
  double acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = 0.0;
  const int ty = threadIdx.y, tx = threadIdx.x;
  for (int q = 0; q < kNB; ++q) {
    double xa[4], yb[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) xa[a] = PI[(ty * 4 + a) * (kNB + 1) + q];
#pragma unroll
    for (int b = 0; b < 4; ++b) yb[b] = PJ[(tx * 4 + b) * (kNB + 1) + q];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) acc[a][b] += xa[a] * yb[b];
  }
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const int r = i0 + ty * 4 + a;
    if (r >= n) continue;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int c = c0 + tx * 4 + b;
      if (c < n && c <= r) A[(int64_t)r * n + c] -= acc[a][b];
    }
  }
}

// Out_sd[r, c] = In_sd[c + s0, r + s0] for r, c < m[sd] (the block starting at (s0, s0)
// with s0 = soff[sd] of an order-n[sd] matrix), lower triangle only of In (upper part
// of the output zero for a lower In block)
__global__ void k_transpose_block(const double* __restrict__ In, const int64_t* __restrict__ ioff,
                                  const int32_t* __restrict__ nn, const int32_t* __restrict__ soff,
                                  const int32_t* __restrict__ mm, double* __restrict__ Out,
                                  const int64_t* __restrict__ ooff, int transpose) {
  const int sd = blockIdx.y, n = nn[sd], s0 = soff[sd], m = mm[sd];
  const double* A = In + ioff[sd];
  double* B = Out + ooff[sd];
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < (int64_t)m * m;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int r = (int)(idx / m), c = (int)(idx % m);
    // the lower-triangular source entry (i, j), i >= j
    const int i = transpose ? c : r, j = transpose ? r : c;
    B[idx] = (i >= j) ? A[(int64_t)(i + s0) * n + j + s0] : 0.0;
  }
}

// Two vectors per warp: x = F^{-1} b with F triangular of order n[sd], given through T whose
// row j is column j of F (contiguous).  forward (F lower): x_j = b_j / F_jj, then b_l -=
// F_lj x_j for l > j; backward (F upper): the same for l < j from the last row.  The vectors
// are columns `col` of rows [roff[sd], roff[sd] + n) of X (leading dimension ldx), solved in
// place, staged in shared memory beside the reciprocals of the diagonal.  Bound by binary64
// issue: with one vector per block its eight warps each repeated the division of every step,
// 8 of its 9 operations: 1.14 -> 0.26 ms a solve (8 subdomains of order about 250, 100
// to 160 vectors each).  grid (n_sd, columns / (2 warps)).
__global__ void __launch_bounds__(128)
    k_trsv_cols(const double* __restrict__ Tm, const int64_t* __restrict__ toff,
                const int32_t* __restrict__ nn, const int32_t* __restrict__ tld,
                const int32_t* __restrict__ tsh, double* X, const int64_t* __restrict__ roff,
                int ldx, const int32_t* __restrict__ ncol, int forward, int n_max) {
  extern __shared__ double sh[];
  const int sd = blockIdx.x, nw = blockDim.x / 32, lane = threadIdx.x & 31;
  const int col0 = blockIdx.y * 2 * nw;
  if (col0 >= ncol[sd]) return;
  const int n = nn[sd], ld = tld[sd], shift = tsh[sd];
  const double* T = Tm + toff[sd] + (int64_t)shift * ld + shift;
  double* rd = sh;
  for (int i = threadIdx.x; i < n; i += blockDim.x) rd[i] = 1.0 / T[(int64_t)i * ld + i];
  const int nv = min(2 * nw, ncol[sd] - col0);
  double* x = X + roff[sd] * ldx + col0;
  for (int idx = threadIdx.x; idx < n * nv; idx += blockDim.x) {
    const int i = idx / nv, v = idx - i * nv;
    sh[(int64_t)(1 + v) * n_max + i] = x[(int64_t)i * ldx + v];
  }
  __syncthreads();
  const int v0 = 2 * (threadIdx.x / 32);
  if (v0 < nv) {
    double* b0 = sh + (int64_t)(1 + v0) * n_max;
    double* b1 = v0 + 1 < nv ? b0 + n_max : b0;  // an odd last vector runs alone
    const bool two = v0 + 1 < nv;
    for (int s = 0; s < n; ++s) {
      const int j = forward ? s : n - 1 - s;
      const double* tj = T + (int64_t)j * ld;
      // odd lanes divide for the second vector
      const double xv = div_by((lane & 1) ? b1[j] : b0[j], tj[j], rd[j]);
      const double x0 = __shfl_sync(0xFFFFFFFFu, xv, 0);
      const double x1 = __shfl_sync(0xFFFFFFFFu, xv, 1);
      const int l0 = forward ? j + 1 : 0, l1 = forward ? n : j;
      for (int l = l0 + lane; l < l1; l += 32) {
        const double t = tj[l];
        b0[l] = fma(-t, x0, b0[l]);
        if (two) b1[l] = fma(-t, x1, b1[l]);
      }
      if (lane == 0) b0[j] = x0;
      if (two && lane == 1) b1[j] = x1;
      __syncwarp();
    }
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < n * nv; idx += blockDim.x) {
    const int i = idx / nv, v = idx - i * nv;
    x[(int64_t)i * ldx + v] = sh[(int64_t)(1 + v) * n_max + i];
  }
}

// one row per warp: the row y (length m[sd]) of X (rows [roff[sd], roff[sd] + rows[sd]),
// leading dimension ldx) becomes x with x R = y, R upper of order m given row-major
// (x_j = (y_j - sum_{l<j} x_l R_lj) / R_jj, column-oriented over the rows of R:
// x_j = y_j / R_jj, then y_l -= R_jl x_j for l > j)
__global__ void __launch_bounds__(256)
    k_trsv_rows(const double* __restrict__ R, const int64_t* __restrict__ roff_r,
                const int32_t* __restrict__ mm, double* X, const int64_t* __restrict__ roff,
                int ldx, const int* __restrict__ sd_of_warp, const int* __restrict__ row_of_warp,
                int n_warps) {
  extern __shared__ double ysh[];
  const int w = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  const int lane = threadIdx.x & 31;
  if (w >= n_warps) return;
  const int sd = sd_of_warp[w], row = row_of_warp[w];
  const int m = mm[sd];
  double* y = ysh + (threadIdx.x / 32) * ldx;
  double* xr = X + (roff[sd] + row) * (int64_t)ldx;
  const double* Rm = R + roff_r[sd];
  for (int l = lane; l < m; l += 32) y[l] = xr[l];
  __syncwarp();
  for (int j = 0; j < m; ++j) {
    const double* rj = Rm + (int64_t)j * m;
    const double xj = y[j] / rj[j];
    for (int l = j + 1 + lane; l < m; l += 32) y[l] -= rj[l] * xj;
    __syncwarp();
    if (lane == 0) y[j] = xj;
    __syncwarp();
  }
  for (int l = lane; l < m; l += 32) xr[l] = y[l];
}

// y = U z per vector, U upper of order n[sd] (row-major): y_a = sum_{b >= a} U_ab z_b;
// z = column `col` of rows [roff[sd], +n) of Z, y into the same place of Y
__global__ void __launch_bounds__(256)
    k_trmv_upper(const double* __restrict__ U, const int64_t* __restrict__ uoff,
                 const int32_t* __restrict__ nn, const double* __restrict__ Z, double* Y,
                 const int64_t* __restrict__ roff, int ld, const int32_t* __restrict__ ncol) {
  extern __shared__ double z[];
  const int sd = blockIdx.x, col = blockIdx.y;
  if (col >= ncol[sd]) return;
  const int n = nn[sd];
  const double* Us = U + uoff[sd];
  for (int i = threadIdx.x; i < n; i += blockDim.x) z[i] = Z[(roff[sd] + i) * ld + col];
  __syncthreads();
  for (int a = threadIdx.x; a < n; a += blockDim.x) {
    const double* ua = Us + (int64_t)a * n;
    double s = 0.0;
    for (int b2 = a; b2 < n; ++b2) s += ua[b2] * z[b2];
    Y[(roff[sd] + a) * ld + col] = s;
  }
}

// S[b, j] of the paper's sketch for the B rows in ascending node order: the first
// normal of Philox(counter (node, j, sd, 1), key = seed); rows [boff[sd], +m[sd]) of
// out (leading dimension ld), columns j < kk[sd]
__global__ void k_node_normals(int n_sd, const int32_t* __restrict__ bnode,
                               const int64_t* __restrict__ boff, const int32_t* __restrict__ mm,
                               const int32_t* __restrict__ kk, int k, uint64_t seed,
                               uint32_t sd_base, double* __restrict__ out, int ld) {
  const int sd = blockIdx.y;
  const int m = mm[sd];
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < (int64_t)m * k;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int r = (int)(idx / k), j = (int)(idx % k);
    double v = 0.0;
    if (j < kk[sd]) {
      uint32_t c[4] = {(uint32_t)bnode[boff[sd] + r], (uint32_t)j, (uint32_t)sd + sd_base, 1u};
      philox4x32_10(c, (uint32_t)(seed & 0xFFFFFFFFull), (uint32_t)(seed >> 32));
      float z0, z1;
      box_muller(c[0], c[1], z0, z1);
      v = (double)z0;
    }
    out[(boff[sd] + r) * ld + j] = v;
  }
}

}  // namespace

void launch_ell_to_dense(int64_t n_rows, const int32_t* row_sd, const int32_t* rloc,
                         const int32_t* cloc, const EllView<double>& A, const int32_t* r_sub,
                         const int32_t* r_n, const int32_t* c_sub, const int32_t* ncols,
                         const int32_t* ld, const int64_t* doff, double* D, cudaStream_t st) {
  if (n_rows <= 0) return;
  count_launch();
  k_ell_to_dense<<<(unsigned)((n_rows + 255) / 256), 256, 0, st>>>(
      n_rows, row_sd, rloc, cloc, A, r_sub, r_n, c_sub, ncols, ld, doff, D);
}

void launch_potrf(int n_sd, int n_max, double* D, const int64_t* doff, const int32_t* nn,
                  int* bad, cudaStream_t st) {
  if (n_sd <= 0) return;
  static bool attr = false;
  const size_t sm = sizeof(double) * 2 * kNB * (kNB + 1);
  if (!attr) {
    cudaFuncSetAttribute(k_potrf_update, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    attr = true;
  }
  for (int j0 = 0; j0 < n_max; j0 += kNB) {
    count_launch();
    k_potrf_diag<<<n_sd, 256, 0, st>>>(D, doff, nn, j0, bad);
    const int T = (n_max - j0 - kNB + kNB - 1) / kNB;
    if (T > 0) {
      count_launch(2);
      k_potrf_panel<<<dim3(n_sd, (n_max - j0 - kNB + kPanelRows - 1) / kPanelRows),
                      4 * kPanelRows, 0, st>>>(D, doff, nn, j0);
      k_potrf_update<<<dim3(n_sd, T * (T + 1) / 2), dim3(16, 16), sm, st>>>(D, doff, nn, j0);
    }
  }
}

void launch_transpose_block(int n_sd, int m_max, const double* In, const int64_t* ioff,
                            const int32_t* nn, const int32_t* soff, const int32_t* mm,
                            double* Out, const int64_t* ooff, int transpose, cudaStream_t st) {
  if (n_sd <= 0 || m_max <= 0) return;
  count_launch();
  const int64_t n = (int64_t)m_max * m_max;
  const unsigned bx = (unsigned)std::min<int64_t>((n + 255) / 256, 1024);
  k_transpose_block<<<dim3(bx, n_sd), 256, 0, st>>>(In, ioff, nn, soff, mm, Out, ooff,
                                                    transpose);
}

void launch_trsv_cols(int n_sd, int n_max, int ncol_max, const double* T, const int64_t* toff,
                      const int32_t* nn, const int32_t* tld, const int32_t* tsh, double* X,
                      const int64_t* roff, int ldx, const int32_t* ncol, int forward,
                      cudaStream_t st) {
  if (n_sd <= 0 || ncol_max <= 0) return;
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_trsv_cols, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
    attr = true;
  }
  // two vectors per warp and the reciprocals in 220 KB: four warps up to order 3,128, one at
  // the largest (6,144)
  int nw = 4;
  while (nw > 1 && sizeof(double) * (1 + 2 * nw) * (size_t)n_max > 220 * 1024) --nw;
  count_launch();
  k_trsv_cols<<<dim3(n_sd, (ncol_max + 2 * nw - 1) / (2 * nw)), 32 * nw,
                sizeof(double) * (1 + 2 * nw) * (size_t)n_max, st>>>(
      T, toff, nn, tld, tsh, X, roff, ldx, ncol, forward, n_max);
}

void launch_trsv_rows(const double* R, const int64_t* roff_r, const int32_t* mm, double* X,
                      const int64_t* roff, int ldx, const int* sd_of_warp,
                      const int* row_of_warp, int n_warps, cudaStream_t st) {
  if (n_warps <= 0) return;
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_trsv_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    attr = true;
  }
  count_launch();
  const int wpb = 8;
  k_trsv_rows<<<(n_warps + wpb - 1) / wpb, 32 * wpb, sizeof(double) * wpb * ldx, st>>>(
      R, roff_r, mm, X, roff, ldx, sd_of_warp, row_of_warp, n_warps);
}

void launch_trmv_upper(int n_sd, int n_max, int ncol_max, const double* U, const int64_t* uoff,
                       const int32_t* nn, const double* Z, double* Y, const int64_t* roff,
                       int ld, const int32_t* ncol, cudaStream_t st) {
  if (n_sd <= 0 || ncol_max <= 0) return;
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_trmv_upper, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    attr = true;
  }
  count_launch();
  k_trmv_upper<<<dim3(n_sd, ncol_max), 256, sizeof(double) * n_max, st>>>(U, uoff, nn, Z, Y,
                                                                          roff, ld, ncol);
}

void launch_node_normals(int n_sd, int m_max, const int32_t* bnode, const int64_t* boff,
                         const int32_t* mm, const int32_t* kk, int k, uint64_t seed,
                         uint32_t sd_base, double* out, int ld, cudaStream_t st) {
  if (n_sd <= 0 || m_max <= 0 || k <= 0) return;
  count_launch();
  const int64_t n = (int64_t)m_max * k;
  const unsigned bx = (unsigned)std::min<int64_t>((n + 255) / 256, 1024);
  k_node_normals<<<dim3(bx, n_sd), 256, 0, st>>>(n_sd, bnode, boff, mm, kk, k, seed, sd_base,
                                                 out, ld);
}

}  // namespace mor
