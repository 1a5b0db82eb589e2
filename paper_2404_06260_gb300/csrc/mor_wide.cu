// Dense per-subdomain linear algebra of step 2 for wide sketches (k up to 511 columns,
// the k_i = floor(M_i / 8) sketch size of Sec. 7.1 and App. C) and for the |B| x |B|
// Gram of the explicit SVD (|B| up to 1024), where the small shared-memory kernels of
// mor_dense.cu do not fit:
//   - tall-skinny Grams X^T Y over the rows of each subdomain, 64 x 64 output tiles,
//     split over row chunks and reduced in chunk order (deterministic);
//   - row-block products X M_sd in 128-row x 64-column output tiles.
// Everything is binary64.
#include "mor_kernels.h"

namespace mor {
namespace {

constexpr int kWT = 64;      // output tile of the Gram and of the row product
constexpr int kWRows = 16;   // rows staged per step of the Gram

// part[(sd * S + s)][i * n + j] = sum over the rows of chunk s of subdomain sd of
// X[r, i] Y[r, j] for the 64 x 64 tiles on and below the diagonal: every product here is
// symmetric, up to rounding (X^T X, X^T H X, V^T A V) or to the tolerance of the adjoint
// solves, where the whole square averaged was measured no more accurate.  Block
// (16, 16), thread (tx, ty) rows ty + 16 a and columns tx + 16 b of the tile; the 16-wide
// strips past n are left out.  Bound by binary64 issue, so by what is multiplied: the whole
// square in tiles padded to 64 took 1.95 ms for 14 subdomains of up to 261 columns, 0.91 now.
__global__ void __launch_bounds__(256)
    k_gram_wide(DTiles tl, int S, const double* __restrict__ X, int ldx, int n,
                const double* __restrict__ Y, int ldy, double* __restrict__ part) {
  __shared__ double Xs[kWRows][kWT + 1];
  __shared__ double Ys[kWRows][kWT + 1];
  const int sd = blockIdx.x / S, s = blockIdx.x % S;
  // tile (ti, tj), tj <= ti, of the lower triangle by rows
  int ti = 0;
  while ((ti + 1) * (ti + 2) / 2 <= (int)blockIdx.y) ++ti;
  const int i0 = ti * kWT, j0 = ((int)blockIdx.y - ti * (ti + 1) / 2) * kWT;
  const int na = (min(kWT, n - i0) + 15) / 16, nb = (min(kWT, n - j0) + 15) / 16;
  const int lo = tl.lo[sd], hi = tl.hi[sd];
  const int nt = hi - lo;
  const int t0 = lo + (int)((int64_t)nt * s / S), t1 = lo + (int)((int64_t)nt * (s + 1) / S);
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * 16 + tx;
  double acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = 0.0;
  for (int t = t0; t < t1; ++t) {
    const int r0 = tl.r0[t], r1 = tl.r1[t];
    for (int base = r0; base < r1; base += kWRows) {
      const int nr = min(kWRows, r1 - base);
      for (int idx = tid; idx < kWRows * kWT; idx += 256) {
        const int rr = idx / kWT, c = idx % kWT;
        const bool in = rr < nr;
        Xs[rr][c] = (in && i0 + c < n) ? X[(int64_t)(base + rr) * ldx + i0 + c] : 0.0;
        Ys[rr][c] = (in && j0 + c < n) ? Y[(int64_t)(base + rr) * ldy + j0 + c] : 0.0;
      }
      __syncthreads();
#pragma unroll 4
      for (int rr = 0; rr < kWRows; ++rr) {
        double xa[4], yb[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) xa[a] = Xs[rr][ty + 16 * a];
#pragma unroll
        for (int b = 0; b < 4; ++b) yb[b] = Ys[rr][tx + 16 * b];
#pragma unroll
        for (int a = 0; a < 4; ++a)
          if (a < na) {
#pragma unroll
            for (int b = 0; b < 4; ++b)
              if (b < nb) acc[a][b] += xa[a] * yb[b];
          }
      }
      __syncthreads();
    }
  }
  double* P = part + (int64_t)(sd * S + s) * n * n;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int i = i0 + ty + 16 * a, j = j0 + tx + 16 * b;
      if (i < n && j < n) P[(int64_t)i * n + j] = acc[a][b];
    }
}

// G[sd][i * ldg + j] and its mirror image = sum over s of part[(sd * S + s)][i * n + j],
// j <= i, s in order
__global__ void k_gram_wide_reduce(int S, int n, const double* __restrict__ part,
                                   double* __restrict__ G, int ldg, int64_t sd_stride) {
  const int sd = blockIdx.y;
  const int64_t nn = (int64_t)n * n;
  double* Gs = G + (int64_t)sd * sd_stride;
  for (int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; o < nn;
       o += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(o / n), j = (int)(o % n);
    if (j > i) continue;
    double acc = 0.0;
    for (int s = 0; s < S; ++s) acc += part[(int64_t)(sd * S + s) * nn + o];
    Gs[(int64_t)i * ldg + j] = acc;
    Gs[(int64_t)j * ldg + i] = acc;
  }
}

// Y[row, j] = sum_l X[row, l] M_sd[l, j] for j < nout, 0 for nout <= j < ldy; block
// (16, 16) over a 128-row x 64-column output tile (each thread 8 rows x 4 columns)
constexpr int kRMRows = 128, kRMK = 16;
__global__ void __launch_bounds__(256)
    k_rowmul_wide(DTiles tl, const double* __restrict__ X, int ldx, int nin,
                  const double* __restrict__ M, int ldm, double* __restrict__ Y, int ldy,
                  int nout) {
  __shared__ double Xs[kRMRows][kRMK + 1];
  __shared__ double Ms[kRMK][kWT + 1];
  const int tile = blockIdx.x, sd = tl.sd[tile];
  const int r0 = tl.r0[tile], r1 = tl.r1[tile];
  const int nr = r1 - r0;
  const int j0 = blockIdx.y * kWT;
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * 16 + tx;
  const double* Msd = M + (int64_t)sd * ldm * ldm;
  double acc[8][4];
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = 0.0;
  if (j0 < nout) {
    for (int l0 = 0; l0 < nin; l0 += kRMK) {
      for (int idx = tid; idx < kRMRows * kRMK; idx += 256) {
        const int rr = idx / kRMK, l = idx % kRMK;
        Xs[rr][l] = (rr < nr && l0 + l < nin) ? X[(int64_t)(r0 + rr) * ldx + l0 + l] : 0.0;
      }
      for (int idx = tid; idx < kRMK * kWT; idx += 256) {
        const int l = idx / kWT, c = idx % kWT;
        Ms[l][c] = (l0 + l < nin && j0 + c < nout) ? Msd[(int64_t)(l0 + l) * ldm + j0 + c]
                                                   : 0.0;
      }
      __syncthreads();
#pragma unroll 4
      for (int l = 0; l < kRMK; ++l) {
        double mb[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) mb[b] = Ms[l][tx * 4 + b];
#pragma unroll
        for (int a = 0; a < 8; ++a) {
          const double xv = Xs[ty * 8 + a][l];
#pragma unroll
          for (int b = 0; b < 4; ++b) acc[a][b] += xv * mb[b];
        }
      }
      __syncthreads();
    }
  }
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    const int rr = ty * 8 + a;
    if (rr >= nr) continue;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int j = j0 + tx * 4 + b;
      if (j < ldy) Y[(int64_t)(r0 + rr) * ldy + j] = (j < nout) ? acc[a][b] : 0.0;
    }
  }
}

}  // namespace

int gram_wide_chunks(int n_sd, int n) {
  const int nt = (n + kWT - 1) / kWT, tiles = nt * (nt + 1) / 2;
  int S = (4 * 152 + n_sd * tiles - 1) / (n_sd * tiles);
  return S < 1 ? 1 : (S > 16 ? 16 : S);
}

void launch_gram_wide(const DTiles& tiles, int n_sd, const double* X, int ldx, int n,
                      const double* Y, int ldy, double* part, double* G, int ldg,
                      int64_t sd_stride, cudaStream_t st) {
  if (tiles.n <= 0 || n_sd <= 0) return;
  const int S = gram_wide_chunks(n_sd, n);
  const int nt = (n + kWT - 1) / kWT;
  count_launch(2);
  k_gram_wide<<<dim3(n_sd * S, nt * (nt + 1) / 2), dim3(16, 16), 0, st>>>(tiles, S, X, ldx, n,
                                                                        Y, ldy, part);
  const int64_t nn = (int64_t)n * n;
  const int bx = (int)((nn + 255) / 256 < 64 ? (nn + 255) / 256 : 64);
  k_gram_wide_reduce<<<dim3(bx, n_sd), 256, 0, st>>>(S, n, part, G, ldg, sd_stride);
}

void launch_rowmul_wide(const DTiles& tiles, const double* X, int ldx, int nin,
                        const double* M, int ldm, double* Y, int ldy, int nout,
                        cudaStream_t st) {
  if (tiles.n <= 0) return;
  count_launch();
  k_rowmul_wide<<<dim3(tiles.n, (ldy + kWT - 1) / kWT), dim3(16, 16), 0, st>>>(
      tiles, X, ldx, nin, M, ldm, Y, ldy, nout);
}

}  // namespace mor
