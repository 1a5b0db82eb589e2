// The symmetric eigensolver of step 2 (the H_i-orthonormalisation, the singular values of
// Eq. (24) or Eq. (14) and the diagonal-block update, Sec. 6): batched positive
// semidefinite matrices, one per subdomain, of order up to 1024.
//
// Method: a diagonally pivoted Cholesky factor G = L L^T, then one-sided Jacobi on the
// columns of L (Veselic & Hari, Numer. Math. 56, 1989; Demmel & Veselic, SIAM J. Matrix
// Anal. 13, 1992): rotations make the columns W = L V orthogonal, and W_j = sigma_j u_j
// gives eigenvalue sigma_j^2 and eigenvector u_j, accurate relative to themselves as those
// of the two-sided threshold iteration.  The eigenvectors need no accumulation, a rotation
// touches two columns instead of two rows, two columns and two more of V, and the pivoted
// factor starts nearly orthogonal: 6 to 9 sweeps with the last, which finds nothing to rotate,
// at the orders and conditions of the workloads (4 at order 13).
//  - Scaling: G by a power of two to a largest diagonal entry in [1, 2).
//  - A column whose pivot falls below n 2^-53 of its own diagonal entry (or below kEigTiny)
//    is rounding noise and takes no part.  The r columns of the factor give the r largest
//    eigenvalues, however small; the others are 0, and their eigenvectors complete the basis:
//    the unit vectors e_j of the columns left out, made orthogonal to all before them by
//    Gram-Schmidt, repeated while a pass takes half of the vector (Giraud, Langou, Rozloznik
//    & van den Eshof, Numer. Math. 101, 2005).
//  - A pair rotates while |w_p.w_q| > sqrt(n) 2^-53 |w_p| |w_q| (the rounding level of the
//    product); the iteration stops after a sweep without rotations (at most 40).
//  - The tangent is formed in binary32 and only the orthogonality of the rotation in
//    binary64: c = (1 + t^2)^(-1/2) by one third-order Householder step from a binary32
//    root, s = t c.  An angle off by 2^-24 leaves 2^-24 of the product to the next sweep.
//
// What bounds it: binary64 issue (a warp instruction keeps a quarter of the SM busy for 64
// clocks) and, for small orders, the chain product -> tangent -> rotation of each round.
// Orders up to 48, and up to kEigSmem where the subdomains alone fill the chip: one CTA per
// subdomain, the factor in shared memory, 8 lanes per pair (k_sym_eig).  Others: a cluster per
// subdomain works on pairs of column blocks staged from L2 (k_sym_eig_blocks).
// Per batch, against the two-sided iteration with the matrix in shared memory (up to 80) or
// in L2 and one CTA per subdomain: 64 matrices of order 42 2.13 -> 1.06 ms, 40 of 74 8.5 ->
// 2.0 ms, 14 of 203 145 -> 8 ms, 8 of 127 and rank about 60 169 -> 4.0 ms (the noise directions of
// an explicit Gram never met the two-sided threshold and ran all 40 sweeps; here they take no
// part in the sweeps).
#include <cooperative_groups.h>

#include <algorithm>

#include "mor_kernels.h"

namespace mor {
namespace {

constexpr int kEigSmem = 128;  // largest order of k_sym_eig (128^2 binary64 in shared memory)
constexpr int kEigMax = 1024;
constexpr int kEigSweeps = 40;
constexpr int kEigLanes = 8;  // lanes per column pair in k_sym_eig
// smallest pivot: products of two columns at the rounding level stay normal numbers
constexpr double kEigTiny = 0x1p-600;

// d^(-1/2) for d in [2^-100, 2^100]: Householder's third-order iteration from binary32
__device__ __forceinline__ double inv_sqrt(double d) {
  const double y = (double)rsqrtf((float)d);
  const double e = fma(-d * y, y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}

// 2^-e with |x| in [2^e, 2^(e+1))
__device__ __forceinline__ double pow2_below(double x) {
  const int e = (int)((__double_as_longlong(x) >> 52) & 0x7FF);
  return __longlong_as_double((long long)(2046 - e) << 52);
}

// about 2^-22 accurate; 0 for negative and zero x
__device__ __forceinline__ float fast_sqrt(float x) { return x > 0.0f ? x * rsqrtf(x) : 0.0f; }

// A column is d * w with 1 / d kept beside d, so that a rotation takes one multiply-add
// per entry: c (p - t q) = (c d_p) (w_p - t d_q / d_p w_q).  d returns to 1 when the column
// is next loaded or its norm taken.
struct JCol {
  double sq;     // squared norm of d * w, updated by the rotations
  double d, di;  // scale and its inverse
};

// The rotation that orthogonalises columns p and q, in two parts around the tangent, the one
// thing that waits for the product pq = w_p.w_q: w_p -= t rq w_q, w_q += t rp w_p (old).
struct JPair {
  double dd;       // d_p d_q
  double diff;     // |q|^2 - |p|^2
  double rp, rq;   // d_p / d_q, d_q / d_p
  float level;     // |d_p d_q pq| 2^k above which the pair rotates
  int k;           // |p| |q| 2^k lies in [1, 4)
  bool far;        // norms more than 2^50 apart
};
// x 2^k by the exponent bits (no binary64 operation); 0 below the normal range, huge above
__device__ __forceinline__ double times_pow2(double x, int k) {
  const int hi = __double2hiint(x), e = ((hi >> 20) & 0x7FF) + k;
  if (((hi >> 20) & 0x7FF) == 0 || e <= 0) return 0.0;
  return __hiloint2double(e < 2047 ? hi + k * (1 << 20) : (hi & 0x800FFFFF) | 0x7FE00000,
                          __double2loint(x));
}
// norm^2 = m 4^e with m in [1, 4); a square lost to cancellation counts as the smallest number
__device__ __forceinline__ float norm_split(double sq, int& e) {
  const int hi = max(__double2hiint(sq), 0x00100000);
  e = ((hi >> 20) - 1023) >> 1;
  return (float)__hiloint2double(hi - e * (1 << 21), __double2loint(sq));
}
__device__ __forceinline__ JPair jacobi_prepare(const JCol& p, const JCol& q, float tol) {
  JPair s;
  s.dd = p.d * q.d;
  s.diff = q.sq - p.sq;
  s.rp = p.d * q.di;
  s.rq = q.d * p.di;
  int ep, eq;
  const float mp = norm_split(p.sq, ep), mq = norm_split(q.sq, eq);
  s.level = tol * (fast_sqrt(mp) * fast_sqrt(mq));
  s.k = -(ep + eq);
  s.far = abs(ep - eq) > 50;
  return s;
}
// the tangent, 0 when the product is at the rounding level (only the angle: binary32 roots
// and quotients by the fast instructions are exact enough); apq = d_p d_q pq.  Product and
// norms go to binary32 relative to |p| |q|: columns of a graded or rank-deficient matrix
// have norms whose products binary32 does not hold.
__device__ __forceinline__ double jacobi_tangent(const JPair& s, double pq, double& apq) {
  apq = s.dd * pq;
  const float o = (float)times_pow2(apq, s.k);
  if (!(fabsf(o) > s.level)) return 0.0;
  if (s.far) return apq / s.diff;  // the tangent to 2^-90
  const float tau = 0.5f * __fdividef((float)times_pow2(s.diff, s.k), o);
  const float a = fabsf(tau);
  const float tt = a > 1e8f ? __fdividef(0.5f, a)
                            : __fdividef(1.0f, a + fast_sqrt(fmaf(a, a, 1.0f)));
  return (double)(tau >= 0.0f ? tt : -tt);
}
// the columns' state after the rotation
__device__ __forceinline__ void jacobi_finish(JCol& p, JCol& q, double t, double apq) {
  const double h = fma(t, t, 1.0), c = inv_sqrt(h), ci = h * c;
  p.sq = fma(-t, apq, p.sq);
  q.sq = fma(t, apq, q.sq);
  p.d *= c;
  q.d *= c;
  p.di *= ci;
  q.di *= ci;
}

// pair k of round `round` of the circle method over m (even) players
__device__ __forceinline__ void circle_pair(int m, int round, int k, int& p, int& q) {
  const int x1 = m - 1 - k;
  int a = k - 1 + round, b = x1 - 1 + round;
  if (a >= m - 1) a -= m - 1;
  if (b >= m - 1) b -= m - 1;
  p = k == 0 ? 0 : a + 1;
  q = b + 1;
}

// rank by descending value (ties by index) of ev[i] >= 0 among the n values (negative: last)
__device__ __forceinline__ int rank_of(const double* ev, int n, int i) {
  const long long li = __double_as_longlong(ev[i]);  // they order like their bits
  int r = 0;
  for (int j = 0; j < n; ++j) {
    const long long lj = __double_as_longlong(ev[j]);
    r += lj > li || (lj == li && j < i);
  }
  return r;
}

// a matrix with an infinity or a NaN: every result is NaN
__device__ __forceinline__ void fill_nan(int ld, int n, double* ev, double* V) {
  const double nan = __longlong_as_double(0x7ff8000000000000LL);
  for (int64_t idx = threadIdx.x; idx < (int64_t)ld * ld; idx += blockDim.x)
    V[idx] = idx / ld < n && idx % ld < n ? nan : 0.0;
  for (int i = threadIdx.x; i < ld; i += blockDim.x) ev[i] = i < n ? nan : 0.0;
}

// One CTA per subdomain; columns of lds = kEigLanes * E doubles (rows beyond n zero).
template <int E>
__global__ void __launch_bounds__(E <= 12 ? 384 : 512)
    k_sym_eig(const double* __restrict__ A, int ld, int n, double* evals, double* evecs) {
  constexpr int lds = kEigLanes * E;
  extern __shared__ __align__(16) double eig_sh[];
  double* w = eig_sh;                 // n columns
  double* g0 = w + (size_t)n * lds;   // diagonal of G
  JCol* jc = reinterpret_cast<JCol*>(g0 + n);
  double* nrm = g0 + n;  // factor: open columns < 0; at last the eigenvalues (over jc)
  int* act = reinterpret_cast<int*>(jc + n);
  __shared__ int s_m, s_p, s_rot;
  __shared__ double s_scale;
  const int sd = blockIdx.x, tid = threadIdx.x, nth = blockDim.x, lane = tid & 31;
  const double* As = A + (int64_t)sd * ld * ld;
  if (tid < 32) {
    double mx = 0.0;
    for (int i = lane; i < n; i += 32) mx = fmax(mx, As[(int64_t)i * ld + i]);
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) s_scale = mx > 0x1p-1000 && mx < 0x1p1000 ? pow2_below(mx) : 1.0;
  }
  __syncthreads();
  const double scale = s_scale;
  double* ev = evals + (int64_t)sd * ld;
  double* V = evecs + (int64_t)sd * ld * ld;
  bool bad = false;
  for (int idx = tid; idx < n * lds; idx += nth) {
    const int j = idx / lds, i = idx - j * lds;
    double v = 0.0;
    if (i < n) v = 0.5 * (As[(int64_t)i * ld + j] + As[(int64_t)j * ld + i]) * scale;
    bad = bad || !isfinite(v);
    w[idx] = v;
    if (i == j) g0[j] = v;
  }
  if (__syncthreads_or(bad)) return fill_nan(ld, n, ev, V);
  // ---- pivoted Cholesky: column p of w becomes the factor's column, with zeros in the rows
  // factored before; nrm[j] < 0 marks a column still to be factored ----
  const double noise = (double)n * 0x1p-53;
  for (int j = tid; j < n; j += nth) nrm[j] = -1.0;
  if (tid == 0) s_m = 0;
  __syncthreads();
  for (int step = 0; step < n; ++step) {
    if (tid < 32) {
      // the largest remaining diagonal entry above its noise level: positive doubles order
      // like their bits, whose low byte gives way to the index
      long long best = 0;
      for (int j = lane; j < n; j += 32) {
        const double d = w[j * lds + j];
        if (nrm[j] < 0.0 && d > noise * g0[j] && d > kEigTiny) {
          const long long key = (__double_as_longlong(d) & ~255LL) | j;
          best = best > key ? best : key;
        }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const long long x = __shfl_xor_sync(0xffffffffu, best, o);
        best = best > x ? best : x;
      }
      if (lane == 0) s_p = best > 0 ? (int)(best & 255) : -1;
    }
    __syncthreads();
    const int p = s_p;
    if (p < 0) break;
    double* wp = w + p * lds;
    const double d = wp[p];
    const double y = d > 0x1p-90 ? inv_sqrt(d) : 1.0 / sqrt(d);
    __syncthreads();
    for (int i = tid; i < n; i += nth) wp[i] = nrm[i] < 0.0 ? wp[i] * y : 0.0;
    __syncthreads();
    if (tid == 0) {
      nrm[p] = 1.0;
      act[step] = p;  // the pairs run in pivot order: one or two sweeps fewer
      s_m = step + 1;
    }
    for (int idx = tid; idx < n * lds; idx += nth) {
      const int j = idx / lds, i = idx - j * lds;
      if (j != p && nrm[j] < 0.0) w[idx] = fma(-wp[j], wp[i], w[idx]);
    }
    __syncthreads();
  }
  // the columns left out become unit vectors, behind the pivots in the list
  const int m = s_m, me = m + (m & 1);
  for (int j = 0; j < n; ++j)
    if (nrm[j] < 0.0)
      for (int i = tid; i < lds; i += nth) w[j * lds + i] = i == j ? 1.0 : 0.0;
  if (tid < 32) {
    int c = m;
    for (int j0 = 0; j0 < n; j0 += 32) {
      const bool in = j0 + lane < n && nrm[j0 + lane] < 0.0;
      const unsigned b = __ballot_sync(0xffffffffu, in);
      if (in) act[c + __popc(b & ((1u << lane) - 1))] = j0 + lane;
      c += __popc(b);
    }
  }
  __syncthreads();
  // ---- one-sided Jacobi ----
  const int grp = tid / kEigLanes, gl = tid % kEigLanes, ngrp = nth / kEigLanes;
  const float tol = sqrtf((float)n) * 0x1p-53f;
  auto squares = [&](int j) {  // squared norm of column j by the 8 lanes of a group
    double s = 0.0;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const double v = w[j * lds + gl + kEigLanes * e];
      s = fma(v, v, s);
    }
    for (int o = 1; o < kEigLanes; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
  };
  for (int sweep = 0; sweep < kEigSweeps; ++sweep) {
    for (int k0 = 0; k0 < n; k0 += ngrp) {  // whole warps stay together for the shuffles
      const int j = min(k0 + grp, n - 1);
      const bool in = k0 + grp < n;
      if (sweep > 0 && in) {
        const double d = jc[j].d;
#pragma unroll
        for (int e = 0; e < E; ++e) w[j * lds + gl + kEigLanes * e] *= d;
      }
      __syncwarp();
      const double s = squares(j);
      if (gl == 0 && in) jc[j] = JCol{s, 1.0, 1.0};
    }
    if (tid == 0) s_rot = 0;
    __syncthreads();
    if (m < 2) break;
    for (int round = 0; round < me - 1; ++round) {
      for (int k0 = 0; k0 < me / 2; k0 += ngrp) {
        const int k = k0 + grp;
        int p = -1, q = -1;
        if (k < me / 2) circle_pair(me, round, k, p, q);
        const bool on = p >= 0 && p < m && q < m;
        p = on ? act[p] : 0;
        q = on ? act[q] : 0;
        JCol cp = jc[p], cq = jc[q];
        const JPair pr = jacobi_prepare(cp, cq, tol);
        double a[E], b[E], s0 = 0.0, s1 = 0.0;
#pragma unroll
        for (int e = 0; e < E; ++e) {
          a[e] = w[p * lds + gl + kEigLanes * e];
          b[e] = w[q * lds + gl + kEigLanes * e];
          if (e & 1)
            s1 = fma(a[e], b[e], s1);
          else
            s0 = fma(a[e], b[e], s0);
        }
        double pq = s0 + s1;
        for (int o = 1; o < kEigLanes; o <<= 1) pq += __shfl_xor_sync(0xffffffffu, pq, o);
        double apq;
        const double t = jacobi_tangent(pr, pq, apq);
        if (!on || !nonzero(t)) continue;
        const double al = t * pr.rq, be = t * pr.rp;
#pragma unroll
        for (int e = 0; e < E; ++e) {
          w[p * lds + gl + kEigLanes * e] = fma(-al, b[e], a[e]);
          w[q * lds + gl + kEigLanes * e] = fma(be, a[e], b[e]);
        }
        jacobi_finish(cp, cq, t, apq);
        if (gl == 0) {
          jc[p] = cp;
          jc[q] = cq;
          s_rot = 1;
        }
      }
      __syncthreads();
    }
    const int rotated = s_rot;
    __syncthreads();
    if (!rotated) break;
  }
  // ---- normalised columns, and the completion of the basis ----
  for (int k0 = 0; k0 < n; k0 += ngrp) {
    const int j = act[min(k0 + grp, n - 1)];
    const double d = jc[j].d;  // 1 unless the last sweep still rotated
    const double s = d * d * squares(j);
    const bool in = k0 + grp < m;
    const double f = in ? d / sqrt(s) : 1.0;
    __syncwarp();
    if (in)
#pragma unroll
      for (int e = 0; e < E; ++e) w[j * lds + gl + kEigLanes * e] *= f;
    if (gl == 0 && k0 + grp < n) g0[j] = in ? s : -1.0;  // from here the eigenvalues
  }
  __syncthreads();
  double* cf = reinterpret_cast<double*>(jc);  // coefficients on the columns before
  int* rk = reinterpret_cast<int*>(cf + n);
  for (int t = m; t < n; ++t) {
    const int j = act[t];
    double* wj = w + j * lds;
    bool any = false;
    for (int k = tid; k < t; k += nth) {
      cf[k] = w[act[k] * lds + j];
      any = any || nonzero(cf[k]);
    }
    if (!__syncthreads_or(any)) continue;  // a null column: e_j as it is
    double s0 = 1.0, s1 = 1.0;
    for (int pass = 0; pass < 4; ++pass) {
      if (pass > 0) {
        for (int k0 = 0; k0 < t; k0 += ngrp) {
          const double* wk = w + act[min(k0 + grp, t - 1)] * lds;
          double s = 0.0;
#pragma unroll
          for (int e = 0; e < E; ++e) s = fma(wk[gl + kEigLanes * e], wj[gl + kEigLanes * e], s);
          for (int o = 1; o < kEigLanes; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
          if (gl == 0 && k0 + grp < t) cf[k0 + grp] = s;
        }
        __syncthreads();
      }
      for (int x = tid; x < n; x += nth) {
        double v = wj[x];
        for (int k = 0; k < t; ++k) v = fma(-cf[k], w[act[k] * lds + x], v);
        wj[x] = v;
      }
      __syncthreads();
      s0 = s1;
      s1 = squares(j);
      if (pass > 0 && s1 >= 0.25 * s0) break;
    }
    __syncthreads();
    for (int x = tid; x < n; x += nth) wj[x] *= 1.0 / sqrt(s1);
    __syncthreads();
  }
  // ---- eigenvalues in descending order ----
  for (int k = tid; k < n; k += nth) rk[act[k]] = k < m ? rank_of(g0, n, act[k]) : k;
  __syncthreads();
  for (int i = tid; i < ld; i += nth) {
    if (i < n)
      ev[rk[i]] = g0[i] > 0.0 ? g0[i] / scale : 0.0;
    else
      ev[i] = 0.0;
  }
  for (int64_t idx = tid; idx < (int64_t)ld * ld; idx += nth) {
    const int r = (int)(idx / ld), j = (int)(idx - (int64_t)r * ld);
    if (r >= n || j >= n)
      V[idx] = 0.0;
    else
      V[(int64_t)r * ld + rk[j]] = w[j * lds + r];
  }
}

// A cluster of C CTAs per subdomain.  Cholesky: CTA c keeps the columns j = c mod C
// (shared memory, or its part of `work` where they do not fit) and the pivot's owner
// writes the finished column to W, in pivot order; two cluster barriers per column.
// Jacobi: the columns of W in blocks of b; a round of the circle method over the blocks
// gives every CTA pairs of blocks, which it stages in shared memory, rotates (all pairs of
// both blocks in the first round of a sweep, the pairs across them in the others) and writes
// back; one cluster barrier per round.  In a round of column pairs the first warps keep one
// thread per pair for the rotations, the others form the products (eight lanes per pair and
// row segment) and apply the rotations (a warp per pair), so that the columns' state is read
// and updated beside that work; with everything done by 16 lanes per pair the rotation's 30
// binary64 instructions were a third of the issue.  A pair is tested at the same place of
// every sweep: one whose columns have not turned since its last test is skipped, and a block
// pair without any such column is not staged.  Against 16 lanes per pair for everything: 40
// matrices of order 74 2.64 -> 2.00 ms, 14 of 203 9.7 -> 8.1, 8 of 127 6.2 -> 5.4.
constexpr size_t kEigBlkSmem = 200 * 1024;
constexpr int kEigParts = 4;  // row segments of a product at most (and two for the rotations)
__global__ void __launch_bounds__(768)
    k_sym_eig_blocks(const double* __restrict__ A, int ld, int n, int b, int R, int in_smem,
                     double* evals, double* evecs, double* work) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  cl.barrier_arrive();  // waited for before the first store to another CTA's shared memory
  extern __shared__ __align__(16) double eig_sh[];
  __shared__ long long s_key[2][8];
  __shared__ int s_rot[2][8];
  __shared__ int s_flag;
  __shared__ double s_red[32];
  const int C = (int)cl.num_blocks(), c = (int)cl.block_rank();
  const int sd = blockIdx.x / C;
  const int tid = threadIdx.x, nth = blockDim.x, lane = tid & 31, warp = tid >> 5;
  const int nw = nth >> 5;
  const double* As = A + (int64_t)sd * ld * ld;
  double* ev = evals + (int64_t)sd * ld;
  double* V = evecs + (int64_t)sd * ld * ld;
  // global: W (columns), eigenvalues | open flags, diagonal of G, and the columns to factor
  double* base = work + (int64_t)sd * (2 * (int64_t)n * n + 16 * n);
  double* W = base;
  double* gn = base + (int64_t)n * n;
  double* gd = gn + n;
  int* gturn = reinterpret_cast<int*>(gd + 2 * n);  // tick of a column's last rotation
  double* stage = in_smem ? eig_sh + (size_t)((n + C - 1) / C) * n : eig_sh;  // pivot column
  double* F = in_smem ? eig_sh
                      : base + (int64_t)n * n + 4 * n + (int64_t)c * ((n + C - 1) / C) * n;
  // power-of-two scale by the largest diagonal entry
  double mx = 0.0;
  for (int i = tid; i < n; i += nth) mx = fmax(mx, As[(int64_t)i * ld + i]);
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) s_red[warp] = mx;
  __syncthreads();
  mx = 0.0;
  for (int k = 0; k < nw; ++k) mx = fmax(mx, s_red[k]);
  const double scale = mx > 0x1p-1000 && mx < 0x1p1000 ? pow2_below(mx) : 1.0;
  const int own = (n - c + C - 1) / C;  // columns c, c + C, ...
  bool bad = false;
  for (int64_t idx = tid; idx < (int64_t)own * n; idx += nth) {
    const int k = (int)(idx / n), i = (int)(idx - (int64_t)k * n), j = c + C * k;
    const double v = 0.5 * (As[(int64_t)i * ld + j] + As[(int64_t)j * ld + i]) * scale;
    F[idx] = v;
    bad = bad || !isfinite(v);
    if (i == j) {
      __stcg(gd + j, v);
      __stcg(gn + j, -1.0);  // still to be factored
      __stcg(gturn + j, 0);
    }
  }
  bad = __syncthreads_or(bad) != 0;
  cl.barrier_wait();  // every CTA of the cluster has started
  if (tid < C) *cl.map_shared_rank(&s_rot[0][c], tid) = bad;
  cl.sync();
  for (int g = 0; g < C; ++g) bad = bad || s_rot[0][g];
  if (bad) {
    if (c == 0) fill_nan(ld, n, ev, V);
    cl.sync();
    return;
  }
  const double noise = (double)n * 0x1p-53;
  int r = 0;  // pivots taken
  for (; r < n; ++r) {
    const int par = r & 1;
    if (warp == 0) {
      long long best = 0;
      for (int k = lane; k < own; k += 32) {
        const int j = c + C * k;
        const double d = F[(int64_t)k * n + j];
        if (__ldcg(gn + j) < 0.0 && d > noise * __ldcg(gd + j) && d > kEigTiny) {
          const long long key = (__double_as_longlong(d) & ~2047LL) | j;
          best = best > key ? best : key;
        }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const long long x = __shfl_xor_sync(0xffffffffu, best, o);
        best = best > x ? best : x;
      }
      if (lane < C) *cl.map_shared_rank(&s_key[par][c], lane) = best;
    }
    cl.sync();
    long long best = 0;
    for (int g = 0; g < C; ++g) best = best > s_key[par][g] ? best : s_key[par][g];
    if (best <= 0) break;
    const int p = (int)(best & 2047);
    if (p % C == c) {
      const double* fp = F + (int64_t)(p / C) * n;
      const double d = fp[p];
      const double y = d > 0x1p-90 ? inv_sqrt(d) : 1.0 / sqrt(d);
      for (int i = tid; i < n; i += nth)  // the rows factored before are zero
        __stcg(W + (int64_t)r * n + i, __ldcg(gn + i) < 0.0 ? fp[i] * y : 0.0);
    }
    cl.sync();
    if (p % C == c && tid == 0) __stcg(gn + p, 1.0);
    for (int i = tid; i < n; i += nth) stage[i] = __ldcg(W + (int64_t)r * n + i);
    __syncthreads();
    // one warp per own column that is still open
    for (int k = warp; k < own; k += nw) {
      const int j = c + C * k;
      if (j == p || !(__ldcg(gn + j) < 0.0)) continue;
      const double lj = stage[j];
      for (int i = lane; i < n; i += 32)
        F[(int64_t)k * n + i] = fma(-lj, stage[i], F[(int64_t)k * n + i]);
    }
    __syncthreads();
  }
  // the columns left out, behind the pivots in index order: e_j for now
  const int m = r;
  int* left = gturn + n;
  for (int j = 0, at = r; j < n; ++j) {
    if (!(__ldcg(gn + j) < 0.0)) continue;
    if (at % C == c) {
      for (int i = tid; i < n; i += nth) __stcg(W + (int64_t)at * n + i, i == j ? 1.0 : 0.0);
      if (tid == 0) __stcg(left + at, j);
    }
    ++at;
  }
  cl.sync();
  // ---- one-sided Jacobi on block pairs ----
  b = max(1, min(b, (m + 2 * C - 1) / (2 * C)));
  const int nb = 2 * ((m + 2 * b - 1) / (2 * b));  // blocks (even), the last ones may be short
  const float tol = sqrtf((float)n) * 0x1p-53f;
  double* blk = eig_sh;                                       // 2 b columns of n
  JCol* jc = reinterpret_cast<JCol*>(blk + (size_t)2 * b * n);
  double* s_pq = reinterpret_cast<double*>(jc + 2 * b);  // products: R parts of b | b, b: t rq, t rp
  int* s_turn = reinterpret_cast<int*>(s_pq + kEigParts * b);
  const int PG = (b + 3) / 4, rs = ((n + R - 1) / R + 7) & ~7;  // groups of 4 pairs, segment
  const int T = nb * 2 * b;                                     // ticks per sweep
  const int ws = (b + 31) / 32, w1 = warp - ws, nw1 = nw - ws;  // ws warps for the rotations
  auto warp_sum = [&](double v) {
    for (int o = 1; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
  for (int sweep = 0; sweep < kEigSweeps; ++sweep) {
    if (tid == 0) s_flag = 0;
    __syncthreads();
    for (int round = 0; round < nb - 1; ++round) {
      for (int k = c; k < nb / 2; k += C) {
        int I, J;
        circle_pair(nb, round, k, I, J);
        const int i0 = min(m, I * b), ni = min(m, i0 + b) - i0;
        const int j0 = min(m, J * b), nj = min(m, j0 + b) - j0;
        const int tick0 = (sweep * nb + round) * 2 * b;
        __syncthreads();  // the last pair's columns and ticks are written back
        // nothing of either block has turned since the pair was here
        bool turned = sweep == 0;
        for (int x = tid; x < ni + nj; x += nth) {
          const int tk = __ldcg(gturn + (x < ni ? i0 + x : j0 + x - ni));
          s_turn[x < ni ? x : b + x - ni] = tk;
          turned = turned || tk >= tick0 - T;
        }
        if (!__syncthreads_or(turned)) continue;
#pragma unroll 4
        for (int idx = tid; idx < ni * n; idx += nth)
          blk[idx] = __ldcg(W + (int64_t)i0 * n + idx);
#pragma unroll 4
        for (int idx = tid; idx < nj * n; idx += nth)
          blk[b * n + idx] = __ldcg(W + (int64_t)j0 * n + idx);
        __syncthreads();
        // staged column x: x < b of block I, x - b of block J
        auto present = [&](int x) { return x < b ? x < ni : x - b < nj; };
        for (int x = warp; x < 2 * b; x += nw) {
          if (!present(x)) continue;
          double s = 0.0;
          for (int i = lane; i < n; i += 32) s = fma(blk[x * n + i], blk[x * n + i], s);
          s = warp_sum(s);
          if (lane == 0) jc[x] = JCol{s, 1.0, 1.0};
        }
        __syncthreads();
        const bool all = round == 0;
        const int rounds = all ? 2 * b - 1 : b;
        bool rot = false;
        for (int q = 0; q < rounds; ++q) {
          auto pair = [&](int x, int& u, int& v) {
            if (all) {
              circle_pair(2 * b, q, x, u, v);
            } else {
              u = x;
              v = x + q;
              v = b + (v >= b ? v - b : v);
            }
            return present(u) && present(v);
          };
          const int last = tick0 + q - T;  // the pairs' last test
          auto due = [&](int u, int v) {
            return sweep == 0 || s_turn[u] >= last || s_turn[v] >= last;
          };
          // thread x < b: pair x
          int u = 0, v = 0;
          const bool mine = tid < b && pair(tid, u, v) && due(u, v);
          JCol cp, cq;
          JPair pr;
          if (mine) {
            cp = jc[u];
            cq = jc[v];
            pr = jacobi_prepare(cp, cq, tol);
          }
          for (int wk = w1 < 0 ? PG * R : w1; wk < PG * R; wk += nw1) {
            const int x = (wk % PG) * 4 + (lane >> 3), seg = wk / PG;
            int xu = 0, xv = 0;
            const bool on = x < b && pair(x, xu, xv) && due(xu, xv);
            if (!__any_sync(0xffffffffu, on)) continue;
            const double *wp = blk + xu * n, *wq = blk + xv * n;
            const int iend = on ? min(n, (seg + 1) * rs) : 0;
            double s0 = 0.0, s1 = 0.0;
            int i = seg * rs + (lane & 7);
            for (; i + 8 < iend; i += 16) {
              s0 = fma(wp[i], wq[i], s0);
              s1 = fma(wp[i + 8], wq[i + 8], s1);
            }
            if (i < iend) s0 = fma(wp[i], wq[i], s0);
            double pq = s0 + s1;
            for (int o = 1; o < 8; o <<= 1) pq += __shfl_xor_sync(0xffffffffu, pq, o);
            if ((lane & 7) == 0 && on) s_pq[seg * b + x] = pq;
          }
          __syncthreads();
          double t = 0.0, apq = 0.0;
          if (mine) {
            double pq = s_pq[tid];
            for (int g = 1; g < R; ++g) pq += s_pq[g * b + tid];
            t = jacobi_tangent(pr, pq, apq);
          }
          if (tid < b) {
            s_pq[tid] = mine ? t * pr.rq : 0.0;
            s_pq[b + tid] = mine ? t * pr.rp : 0.0;
          }
          __syncthreads();
          if (nonzero(t)) {
            jacobi_finish(cp, cq, t, apq);
            jc[u] = cp;
            jc[v] = cq;
            s_turn[u] = s_turn[v] = tick0 + q;
            rot = true;
          }
          for (int x = w1 < 0 ? b : w1; x < b; x += nw1) {
            const double al = s_pq[x], be = s_pq[b + x];
            if (!nonzero(al)) continue;
            int xu, xv;
            pair(x, xu, xv);
            double *wp = blk + xu * n, *wq = blk + xv * n;
#pragma unroll 4
            for (int i = lane; i < n; i += 32) {
              const double x1 = wp[i], x2 = wq[i];
              wp[i] = fma(-al, x2, x1);
              wq[i] = fma(be, x1, x2);
            }
          }
          __syncthreads();
        }
        if (rot) s_flag = 1;
        for (int x = tid; x < ni + nj; x += nth)
          __stcg(gturn + (x < ni ? i0 + x : j0 + x - ni), s_turn[x < ni ? x : b + x - ni]);
        for (int idx = tid; idx < ni * n; idx += nth)
          __stcg(W + (int64_t)i0 * n + idx, blk[idx] * jc[idx / n].d);
        for (int idx = tid; idx < nj * n; idx += nth)
          __stcg(W + (int64_t)j0 * n + idx, blk[b * n + idx] * jc[b + idx / n].d);
      }
      cl.sync();
    }
    if (tid < C) *cl.map_shared_rank(&s_rot[sweep & 1][c], tid) = s_flag;
    cl.sync();
    int any = 0;
    for (int g = 0; g < C; ++g) any |= s_rot[sweep & 1][g];
    if (!any) break;
  }
  // ---- normalised columns (CTA c: columns c, c + C, ...) ----
  for (int k = warp; k < own; k += nw) {
    const int j = c + C * k;
    double* wj = W + (int64_t)j * n;
    double s = 0.0;
    for (int i = lane; i < n; i += 32) {
      const double v = __ldcg(wj + i);
      s = fma(v, v, s);
    }
    s = warp_sum(s);
    if (lane == 0) __stcg(gn + j, j < m ? s : -1.0);  // from here the eigenvalues
    if (j < m) {
      const double f = 1.0 / sqrt(s);
      for (int i = lane; i < n; i += 32) __stcg(wj + i, __ldcg(wj + i) * f);
    }
  }
  cl.sync();
  // ---- completion of the basis: CTA c forms rows x0 to x1 of the vector, a warp every nw-th
  // column's share; the coefficients of a repeated pass and the norms are summed over the
  // cluster in `parts` ----
  double* cf = eig_sh;                    // coefficients on the columns before
  double* acc = cf + n;                   // 32 rows per warp
  double* vown = acc + 32 * nw;           // own rows of the vector
  double* parts = base + (int64_t)n * n + 4 * n;
  const int x0 = n * c / C, nx = n * (c + 1) / C - x0;
  for (int t = m; t < n; ++t) {
    const int j = __ldcg(left + t);
    bool any = false;
    for (int k = tid; k < t; k += nth) {
      cf[k] = __ldcg(W + (int64_t)k * n + j);
      any = any || nonzero(cf[k]);
    }
    for (int x = tid; x < nx; x += nth) vown[x] = x0 + x == j ? 1.0 : 0.0;
    if (!__syncthreads_or(any)) continue;  // a null column: e_j as it is (for every CTA)
    double s0 = 1.0, s1 = 1.0;
    for (int pass = 0; pass < 4; ++pass) {
      if (pass > 0) {
        for (int k = warp; k < t; k += nw) {
          double s = 0.0;
          for (int x = lane; x < nx; x += 32)
            s = fma(__ldcg(W + (int64_t)k * n + x0 + x), vown[x], s);
          s = warp_sum(s);
          if (lane == 0) __stcg(parts + (int64_t)c * n + k, s);
        }
        cl.sync();
        for (int k = tid; k < t; k += nth) {
          double s = 0.0;
          for (int g = 0; g < C; ++g) s += __ldcg(parts + (int64_t)g * n + k);
          cf[k] = s;
        }
        __syncthreads();
      }
      for (int xb = 0; xb < nx; xb += 32) {
        double s = 0.0;
        if (xb + lane < nx)
          for (int k = warp; k < t; k += nw)
            s = fma(cf[k], __ldcg(W + (int64_t)k * n + x0 + xb + lane), s);
        acc[warp * 32 + lane] = s;
        __syncthreads();
        if (warp == 0 && xb + lane < nx) {
          for (int u = 1; u < nw; ++u) s += acc[u * 32 + lane];
          vown[xb + lane] -= s;
        }
        __syncthreads();
      }
      if (warp == 0) {
        double s = 0.0;
        for (int x = lane; x < nx; x += 32) s = fma(vown[x], vown[x], s);
        s = warp_sum(s);
        if (lane == 0) __stcg(parts + (int64_t)C * n + c, s);
      }
      cl.sync();
      s0 = s1;
      s1 = 0.0;
      for (int g = 0; g < C; ++g) s1 += __ldcg(parts + (int64_t)C * n + g);
      if (pass > 0 && s1 >= 0.25 * s0) break;
    }
    const double f = 1.0 / sqrt(s1);
    for (int x = tid; x < nx; x += nth) __stcg(W + (int64_t)t * n + x0 + x, vown[x] * f);
    cl.sync();
  }
  // ---- eigenvalues in descending order ----
  double* evs = eig_sh;
  for (int i = tid; i < n; i += nth) evs[i] = __ldcg(gn + i);
  __syncthreads();
  for (int k = warp; k < own; k += nw) {
    const int j = c + C * k;
    int rank = j;
    if (lane == 0 && j < m) rank = rank_of(evs, n, j);
    rank = __shfl_sync(0xffffffffu, rank, 0);
    if (lane == 0) ev[rank] = j < m ? evs[j] / scale : 0.0;
    for (int i = lane; i < n; i += 32)
      V[(int64_t)i * ld + rank] = __ldcg(W + (int64_t)j * n + i);
  }
  if (c == 0) {
    for (int i = n + tid; i < ld; i += nth) ev[i] = 0.0;
    for (int64_t idx = tid; idx < (int64_t)ld * ld; idx += nth) {
      const int i = (int)(idx / ld), j = (int)(idx - (int64_t)i * ld);
      if (i >= n || j >= n) V[idx] = 0.0;
    }
  }
  cl.sync();  // no CTA leaves while another may still write to it
}

template <int E>
void launch_small(int n_sd, const double* A, int ld, int n, double* evals, double* evecs,
                  cudaStream_t st) {
  const int nth = std::max(64, (std::max(1, (n + 1) / 2) * kEigLanes + 31) / 32 * 32);
  auto smem = [](int m) {
    return sizeof(double) * ((size_t)m * kEigLanes * E + m) + sizeof(JCol) * m + sizeof(int) * m;
  };
  // (one limit for every order: threads may launch different ones at the same time)
  cudaFuncSetAttribute(k_sym_eig<E>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)smem(kEigLanes * E));
  k_sym_eig<E><<<n_sd, nth, smem(n), st>>>(A, ld, n, evals, evecs);
}

}  // namespace

// CTAs per subdomain: as many as fill the chip once, with at least 16 columns each; one up
// to order 48, where the chain of a round counts and not its arithmetic (64 matrices of
// order 42: 1.06 ms with one CTA each, 1.18 with two; 40 of 74: 3.6 with one, 2.6 with three)
static int eig_ctas(int n_sd, int n) {
  if (n <= 48) return 1;
  return std::max(1, std::min({8, 152 / std::max(1, n_sd), n / 16}));
}

size_t sym_eig_work(int n) { return 2 * (size_t)n * n + 16 * (size_t)n; }

void launch_sym_eig(int n_sd, const double* A, int ld, int n, double* evals, double* evecs,
                    double* work, cudaStream_t st) {
  if (n_sd <= 0 || n <= 0 || n > kEigMax) return;
  count_launch();
  int C = eig_ctas(n_sd, n);
  if (n <= kEigSmem && C == 1) {
    if (n <= 16) return launch_small<2>(n_sd, A, ld, n, evals, evecs, st);
    if (n <= 32) return launch_small<4>(n_sd, A, ld, n, evals, evecs, st);
    if (n <= 48) return launch_small<6>(n_sd, A, ld, n, evals, evecs, st);
    if (n <= 64) return launch_small<8>(n_sd, A, ld, n, evals, evecs, st);
    if (n <= 80) return launch_small<10>(n_sd, A, ld, n, evals, evecs, st);
    if (n <= 96) return launch_small<12>(n_sd, A, ld, n, evals, evecs, st);
    return launch_small<16>(n_sd, A, ld, n, evals, evecs, st);
  }
  // a staged column, its state, its share of the products and its last turn
  const size_t col = sizeof(double) * (size_t)n + sizeof(JCol) + sizeof(double) * kEigParts / 2 +
                     sizeof(int);
  const int b = std::max(1, std::min((n + 2 * C - 1) / (2 * C), (int)(kEigBlkSmem / (2 * col))));
  const size_t factor = sizeof(double) * (size_t)((n + C - 1) / C) * n;
  int in_smem = factor <= kEigBlkSmem ? 1 : 0;
  // the staged blocks; the factor and a column; the completion's coefficients, 32 rows for
  // each of at most 24 warps, and a vector's share
  const size_t sm = std::max({2 * b * col, (in_smem ? factor : 0) + sizeof(double) * (size_t)n,
                              sizeof(double) * (2 * (size_t)n + 32 * 24)});
  // row segments of a product by the binary64 issue of the busiest quarter of the SM: each
  // warp takes n / 8R multiply-adds and four additions
  const int PG = (b + 3) / 4;
  auto cost = [&](int r) { return (PG * r + 3) / 4 * ((n + 8 * r - 1) / (8 * r) + 4); };
  int R = 1;
  for (int r = 2; r <= kEigParts; r *= 2)
    if (cost(r) < cost(R)) R = r;
  const int nth = std::min(768, std::max(256, 32 * ((b + 31) / 32 + std::max(PG * R, b))));
  auto fn = k_sym_eig_blocks;
  // one limit for every order, as above: the factor or the blocks, and a column
  cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)(kEigBlkSmem + sizeof(double) * kEigMax));
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)C;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(n_sd * C));
  cfg.blockDim = dim3((unsigned)nth);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, fn, A, ld, n, b, R, in_smem, evals, evecs, work);
}

}  // namespace mor
