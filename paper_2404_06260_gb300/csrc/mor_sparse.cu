// Sliced-ELL multi-right-hand-side products and the batched Jacobi-preconditioned CG
// used for every local solve of step 2 (A_II and H^+ systems of Sec. 4 and Sec. 6).
//
// Vectors are row-major blocks [rows x kp] (kp = right-hand sides padded to a multiple
// of 4).  A CUDA block owns one row tile of one subdomain; thread (tx, ty) handles the
// 16-byte column chunk tx of rows r0 + ty, r0 + ty + RB, ...  Every (subdomain, column)
// pair runs its own CG recurrence; per-tile column sums go to a partial array and the
// last tile of a subdomain to finish (atomic ticket) reduces them in tile order, so the
// reductions are deterministic and need no extra launch.
#include "mor_kernels.h"
#include "mor_tc.cuh"

#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <mutex>
#include <vector>
#include "mor_plan.h"

namespace mor {
namespace {

template <typename T>
struct alignas(16) Pack {
  static constexpr int N = 16 / sizeof(T);
  T v[N];
};

template <typename T>
__device__ __forceinline__ Pack<T> ld(const T* p) {
  return *reinterpret_cast<const Pack<T>*>(p);
}
template <typename T>
__device__ __forceinline__ void st(T* p, const Pack<T>& x) {
  *reinterpret_cast<Pack<T>*>(p) = x;
}

struct Geo {
  int tx, ty, nch, rb, tid, nth;
};
__device__ __forceinline__ Geo geo() {
  Geo g;
  g.tx = threadIdx.x;
  g.ty = threadIdx.y;
  g.nch = blockDim.x;
  g.rb = blockDim.y;
  g.tid = g.ty * g.nch + g.tx;
  g.nth = g.nch * g.rb;
  return g;
}

// two consecutive slots of one row of a staged sliced-ELL tile: values first, so that a
// binary32 record is one 16-byte shared-memory load
template <typename T>
struct alignas(16) Slot2 {
  T v[2];
  int32_t c[2];
};

// shared memory layout: red[nth * N] of T, scratch[nth] doubles, sums[3*kp] doubles,
// then the staged sliced-ELL tile: slots[((W + 1) / 2) * kTileRows] pair records,
// pair-major (record h of row rr at h * kTileRows + rr)
template <typename T>
struct Smem {
  T* red;
  double* scratch;
  double* sums;
  Slot2<T>* slots;
};
__host__ __device__ constexpr __forceinline__ size_t align16(size_t x) {
  return (x + 15) & ~(size_t)15;
}
template <typename T>
__device__ __forceinline__ Smem<T> smem_layout(const Geo& g, int kp, int W) {
  extern __shared__ __align__(16) unsigned char raw[];
  Smem<T> s;
  size_t o = 0;
  s.red = reinterpret_cast<T*>(raw + o);
  o += align16(16 * (size_t)g.nth);
  s.scratch = reinterpret_cast<double*>(raw + o);
  s.sums = s.scratch + g.nth;
  o += align16(sizeof(double) * ((size_t)g.nth + 3 * kp));
  s.slots = reinterpret_cast<Slot2<T>*>(raw + o);
  return s;
}
template <typename T>
__host__ __device__ constexpr __forceinline__ size_t smem_bytes(int nch, int rb, int kp, int W) {
  size_t nth = (size_t)nch * rb;
  return align16(16 * nth) + align16(sizeof(double) * (nth + 3 * kp)) +
         sizeof(Slot2<T>) * (size_t)kTileRows * ((W + 1) / 2);
}

// column sums over ty of per-thread N-wide accumulators -> out[tx*N + e] (double)
template <typename T, int N>
__device__ void block_colsum(const Geo& g, const T (&acc)[N], T* red, double* out,
                             bool write = true) {
#pragma unroll
  for (int e = 0; e < N; ++e) red[g.tid * N + e] = acc[e];
  __syncthreads();
  int p2 = 1;
  while (p2 < g.rb) p2 <<= 1;
  for (int s = p2 >> 1; s > 0; s >>= 1) {
    if (g.ty < s && g.ty + s < g.rb)
#pragma unroll
      for (int e = 0; e < N; ++e) red[g.tid * N + e] += red[(g.tid + s * g.nch) * N + e];
    __syncthreads();
  }
  if (g.ty == 0 && write)
#pragma unroll
    for (int e = 0; e < N; ++e) out[g.tx * N + e] = (double)red[g.tx * N + e];
}

// true in the last of n blocks to come here (for every thread); the counter returns to
// zero.  One thread's acquire-release ticket behind the block barrier orders the blocks'
// earlier writes before the last block's later reads (which pass by L1: __ldcg).
__device__ __forceinline__ bool take_ticket(const Geo& g, int* counter, int n) {
  __shared__ int is_last;
  __syncthreads();
  if (g.tid == 0) {
    int prev;
    asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;"
                 : "=r"(prev)
                 : "l"(counter)
                 : "memory");
    is_last = prev == n - 1;
    if (is_last) *counter = 0;
  }
  __syncthreads();
  return is_last != 0;
}

// sums[q*kp + c] = sum over rows lo..hi-1 of part[q][t*kp + c], q < NS, in a fixed order: S
// threads share a column (at most 4: their sums are then added one after the other, and a
// binary64 addition takes 66 clocks), eight loads in flight each
template <int NS>
__device__ void rows_colsum(const Geo& g, const double* const (&part)[NS], int kp, int lo, int hi,
                            double* scratch, double* sums) {
  const int cols = NS * kp;
  for (int c0 = 0; c0 < cols; c0 += g.nth) {
    const int cw = min(cols - c0, g.nth);
    const int S = min(4, g.nth / cw);
    const int sidx = g.tid / cw, x = c0 + g.tid - sidx * cw;
    double acc = 0.0;
    if (sidx < S) {
      const int q = x / kp, c = x - q * kp;
      const double* P = part[0];
#pragma unroll
      for (int u = 1; u < NS; ++u) P = q == u ? part[u] : P;
      for (int t = lo + sidx; t < hi; t += 8 * S) {
        double v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
          v[u] = t + u * S < hi ? __ldcg(P + (int64_t)(t + u * S) * kp + c) : 0.0;
#pragma unroll
        for (int u = 0; u < 8; ++u) acc += v[u];
      }
    }
    scratch[g.tid] = acc;
    __syncthreads();
    for (int cc = g.tid; cc < cw; cc += g.nth) {
      double s = scratch[cc];
      for (int q = 1; q < S; ++q) s += scratch[q * cw + cc];
      sums[c0 + cc] = s;
    }
    __syncthreads();
  }
}

// The column sums of a subdomain's tiles lo..hi-1 (part[q][t*kp + c], this block wrote tile
// `tile`) into sums[q*kp + c], q < NS; true in the one block that ends up with them.  Two
// levels, in a fixed order: the last block of every kRedGroup tiles adds those to a group
// sum, the last group adds the groups.  One block adding a subdomain's 170 to 250 tiles
// alone was a tail of 10 us per sum behind every kernel (binary64 additions at 2 per clock
// behind a dozen dependent loads); the two short ones take 4.  Few tiles: one level.
constexpr int kRedGroup = 16;
template <int NS>
__device__ bool tile_sums(const Geo& g, const double* const (&part)[NS], double* gpart,
                          int* gcount, int* count, int kp, int tile, int lo, int hi,
                          double* scratch, double* sums) {
  const int nt = hi - lo;
  if (nt <= 2 * kRedGroup) {
    if (!take_ticket(g, count, nt)) return false;
    rows_colsum<NS>(g, part, kp, lo, hi, scratch, sums);
    return true;
  }
  const int ng = (nt + kRedGroup - 1) / kRedGroup, gi = (tile - lo) / kRedGroup;
  const int g0 = lo + gi * kRedGroup, g1 = min(hi, g0 + kRedGroup);
  if (!take_ticket(g, gcount + lo + gi, g1 - g0)) return false;
  // group sums of a subdomain: NS blocks of ng rows from row lo NS of gpart
  double* gp = gpart + (int64_t)lo * NS * kp;
  rows_colsum<NS>(g, part, kp, g0, g1, scratch, sums);
  for (int x = g.tid; x < NS * kp; x += g.nth) {
    const int q = x / kp, c = x - q * kp;
    __stcg(gp + ((int64_t)q * ng + gi) * kp + c, sums[x]);
  }
  if (!take_ticket(g, count, ng)) return false;
  const double* gparts[NS];
#pragma unroll
  for (int q = 0; q < NS; ++q) gparts[q] = gp + (int64_t)q * ng * kp;
  rows_colsum<NS>(g, gparts, kp, 0, ng, scratch, sums);
  return true;
}

// CG coefficients: binary64 state with a binary32 copy
__device__ __forceinline__ void set_coef(double* c64, float* c32, int i, double v) {
  c64[i] = v;
  c32[i] = (float)v;
}
// the N coefficients of pack tx of subdomain sd in the working precision
template <typename T>
__device__ __forceinline__ Pack<T> coef_pack(const double* c64, const float* c32, int sd,
                                             int kp, int tx) {
  constexpr int N = Pack<T>::N;
  if constexpr (sizeof(T) == 4) {
    return ld(reinterpret_cast<const T*>(c32) + sd * kp + tx * N);
  } else {
    return ld(reinterpret_cast<const T*>(c64) + sd * kp + tx * N);
  }
}

// the N columns of pack tx of subdomain sd have all converged (their work can be skipped:
// converged columns have alpha = 0 and are reset at the next residual replacement)
template <typename T>
__device__ __forceinline__ bool pack_done(const CgState& s, int sd, int kp, int tx) {
  constexpr int N = Pack<T>::N;
  const int* d = s.done + sd * kp + tx * N;
  bool all = true;
#pragma unroll
  for (int e = 0; e < N; ++e) all = all && d[e] != 0;
  return all;
}

__device__ __forceinline__ void count_active(const Geo& g, const int* done, int sd, int kp,
                                             int* active) {
  __shared__ int cnt;
  if (g.tid == 0) cnt = 0;
  __syncthreads();
  for (int c = g.tid; c < kp; c += g.nth)
    if (!done[sd * kp + c]) atomicAdd(&cnt, 1);
  __syncthreads();
  if (g.tid == 0) active[sd] = cnt;
}

// ---------------------------------------------------------------------------------
// Sliced-ELL products on a row tile.  The tile's slots (column index and value) are
// first staged in shared memory with coalesced loads (consecutive threads take
// consecutive rows of one slot pair), which takes the index load off the critical path
// of the gathers; a row's slots 2h and 2h + 1 form one record, so one shared load feeds
// two gathers.  Thread (tx, ty) then computes the 16-byte column chunk tx of rows
// ty, ty + RB, ...: the slots of a batch are gathered (predicated, independent loads)
// before their multiply-adds, which run in slot order.  k_spmm: Y = A X.
// k_cg_spmm_pq: q = A p with the column sums of p.q.  k_residual64: r = b - A x with
// the column sums of r.r.
template <typename T>
__device__ __forceinline__ void stage_tile(const Geo& g, int r0, int nrows,
                                           const EllView<T>& A, Slot2<T>* slots) {
  const int W = A.W, W2 = (W + 1) / 2;
  const bool full = nrows == kTileRows;  // full tiles: pair and row by shifts
  for (int idx = g.tid; idx < nrows * W2; idx += g.nth) {
    int h, rr;
    if (full) {
      h = idx / kTileRows;  // kTileRows is a power of two: compiles to a shift
      rr = idx & (kTileRows - 1);
    } else {
      h = idx / nrows;
      rr = idx - h * nrows;
    }
    int64_t r = (int64_t)r0 + rr;
    const int w = A.width[r >> 5];
    Slot2<T> rec;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      int j = 2 * h + u;
      rec.c[u] = -1;
      rec.v[u] = T(0);
      if (j < w) {
        int64_t at = ell_at(r, j, W);
        rec.c[u] = A.col[at];
        rec.v[u] = A.val[at];
      }
    }
    slots[h * kTileRows + rr] = rec;
  }
}

// row rr of the staged tile (slice width w) times X: column chunk tx.  R records (2 R
// slots) are gathered per batch before their multiply-adds, which run in slot order
// (the sum is the same for every R).
template <typename T, int R = 1>
__device__ __forceinline__ Pack<T> spmm_row(int rr, int w, int tx, const Slot2<T>* slots,
                                            const T* __restrict__ X, int kp) {
  constexpr int N = Pack<T>::N;
  Pack<T> acc;
#pragma unroll
  for (int e = 0; e < N; ++e) acc.v[e] = T(0);
  const int w2 = (w + 1) >> 1;
  for (int h0 = 0; h0 < w2; h0 += R) {
    Slot2<T> rec[R];
    Pack<T> xv[2 * R];
#pragma unroll
    for (int g = 0; g < R; ++g) {
      if (h0 + g < w2) {
        rec[g] = slots[(h0 + g) * kTileRows + rr];
      } else {
        rec[g].c[0] = rec[g].c[1] = -1;
        rec[g].v[0] = rec[g].v[1] = T(0);
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        if (rec[g].c[u] >= 0) {
          xv[2 * g + u] = ld(X + (int64_t)rec[g].c[u] * kp + tx * N);
        } else {
#pragma unroll
          for (int e = 0; e < N; ++e) xv[2 * g + u].v[e] = T(0);
        }
      }
    }
#pragma unroll
    for (int g = 0; g < R; ++g)
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int e = 0; e < N; ++e) acc.v[e] += rec[g].v[u] * xv[2 * g + u].v[e];
  }
  return acc;
}

template <typename T>
__global__ void k_spmm(DTiles tl, EllView<T> A, const T* __restrict__ X, T* __restrict__ Y,
                       int kp) {
  constexpr int N = Pack<T>::N;
  Geo g = geo();
  Smem<T> sm = smem_layout<T>(g, kp, A.W);
  const int tile = blockIdx.x;
  const int r0 = tl.r0[tile], r1 = tl.r1[tile];
  stage_tile(g, r0, r1 - r0, A, sm.slots);
  __syncthreads();
  for (int rr = g.ty; rr < r1 - r0; rr += g.rb) {
    int64_t row = r0 + rr;
    st(Y + row * kp + g.tx * N,
       spmm_row(rr, A.width[row >> 5], g.tx, sm.slots, X, kp));
  }
}

// binary64 residual row: A x and sum_j |a_ij x_j| in one pass over the staged slots
// (batches of four records, eight slots)
__device__ __forceinline__ void spmm_row_res(int rr, int w, int tx, const Slot2<double>* slots,
                                             const double* __restrict__ X, int kp,
                                             Pack<double>& acc, Pack<double>& aabs) {
  constexpr int N = Pack<double>::N;
  constexpr int H = 4;
#pragma unroll
  for (int e = 0; e < N; ++e) acc.v[e] = aabs.v[e] = 0.0;
  const int w2 = (w + 1) >> 1;
  for (int h0 = 0; h0 < w2; h0 += H) {
    Pack<double> xv[2 * H];
    double av[2 * H];
#pragma unroll
    for (int hh = 0; hh < H; ++hh) {
      Slot2<double> rec;
      if (h0 + hh < w2) {
        rec = slots[(h0 + hh) * kTileRows + rr];
      } else {
        rec.c[0] = rec.c[1] = -1;
        rec.v[0] = rec.v[1] = 0.0;
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        av[2 * hh + u] = rec.v[u];
        if (rec.c[u] >= 0) {
          xv[2 * hh + u] = ld(X + (int64_t)rec.c[u] * kp + tx * N);
        } else {
#pragma unroll
          for (int e = 0; e < N; ++e) xv[2 * hh + u].v[e] = 0.0;
        }
      }
    }
#pragma unroll
    for (int u = 0; u < 2 * H; ++u)
#pragma unroll
      for (int e = 0; e < N; ++e) {
        double t = av[u] * xv[u].v[e];
        acc.v[e] += t;
        aabs.v[e] += fabs(t);
      }
  }
}

// at most TH threads per block; 40 registers leave room for 1536 threads per SM (six
// blocks of 256, twelve of 128).  R: records gathered per batch (spmm_row)
template <typename T, int R = 1, int TH = 256>
__global__ void __launch_bounds__(TH, TH <= 256 ? 1536 / TH : 1)
    k_cg_spmm_pq(DTiles tl, EllView<T> A, const T* __restrict__ p, T* __restrict__ q, int kp,
                 CgState s) {
  constexpr int N = Pack<T>::N;
  Geo g = geo();
  Smem<T> sm = smem_layout<T>(g, kp, A.W);
  const int tile = blockIdx.x, sd = tl.sd[tile];
  if (s.active[sd] == 0) return;  // every column of this subdomain has converged
  const int r0 = tl.r0[tile], r1 = tl.r1[tile];
  stage_tile(g, r0, r1 - r0, A, sm.slots);
  __syncthreads();
  T acc[N];
#pragma unroll
  for (int e = 0; e < N; ++e) acc[e] = T(0);
  const int rend = pack_done<T>(s, sd, kp, g.tx) ? 0 : r1 - r0;
  for (int rr = g.ty; rr < rend; rr += g.rb) {
    int64_t row = r0 + rr;
    Pack<T> qv = spmm_row<T, R>(rr, A.width[row >> 5], g.tx, sm.slots, p, kp);
    int64_t o = row * kp + g.tx * N;
    st(q + o, qv);
    Pack<T> pv = ld(p + o);
#pragma unroll
    for (int e = 0; e < N; ++e) acc[e] += pv.v[e] * qv.v[e];
  }
  block_colsum<T, N>(g, acc, sm.red, s.part1 + (int64_t)tile * kp);
  const double* const parts[1] = {s.part1};
  if (!tile_sums<1>(g, parts, s.gpart, s.gcount, s.counter + sd, kp, tile, tl.lo[sd], tl.hi[sd],
                    sm.scratch, sm.sums))
    return;
  for (int c = g.tid; c < kp; c += g.nth) {
    int i = sd * kp + c;
    double a = 0.0;
    if (!s.done[i]) {
      // exact line search along p: alpha = p.r / p.Ap (equals r.z / p.Ap in exact CG,
      // and stays a descent step after a residual replacement kept p)
      double pq = sm.sums[c];
      if (pq > 0.0)
        a = s.pr[i] / pq;
      else
        s.done[i] = 1;  // breakdown (p = 0 or indefinite): stop this column
    }
    set_coef(s.alpha, s.alpha32, i, a);
  }
}

// the N columns of pack tx met the binary64 test in the last sweep of this solve (seen: there
// was one): their x64 has not changed since, nor have their residual and its sums
template <int N>
__device__ __forceinline__ bool pack_settled(const RefineState& s, int sd, int kp, int tx,
                                             int seen) {
  bool all = seen != 0;
#pragma unroll
  for (int e = 0; e < N; ++e) all = s.scale[sd * kp + tx * N + e] == 0.0 && all;
  return all;
}

template <bool kFloor>
__global__ void k_residual64(DTiles tl, EllView<double> A, const double* __restrict__ b,
                             const double* __restrict__ x, double* __restrict__ r, int kp,
                             int nc, double rtol2, int seen, RefineState s,
                             const double* __restrict__ anorm) {
  constexpr int N = 2;
  Geo g = geo();
  Smem<double> sm = smem_layout<double>(g, kp, A.W);
  const int tile = blockIdx.x, sd = tl.sd[tile];
  if (seen && s.active[sd] == 0) return;  // settled in the last sweep
  const int r0 = tl.r0[tile], r1 = tl.r1[tile];
  stage_tile(g, r0, r1 - r0, A, sm.slots);
  __syncthreads();
  const bool settled = pack_settled<N>(s, sd, kp, g.tx, seen);
  double acc[N] = {0.0, 0.0}, aca[N] = {0.0, 0.0}, axx[N] = {0.0, 0.0};
  for (int rr = g.ty; rr < (settled ? 0 : r1 - r0); rr += g.rb) {
    int64_t row = r0 + rr;
    Pack<double> ax, aabs;
    {
      Pack<double> xo = ld(x + row * kp + g.tx * N);
#pragma unroll
      for (int e = 0; e < N; ++e) axx[e] += xo.v[e] * xo.v[e];
    }
    if constexpr (kFloor)
      spmm_row_res(rr, A.width[row >> 5], g.tx, sm.slots, x, kp, ax, aabs);
    else
      ax = spmm_row(rr, A.width[row >> 5], g.tx, sm.slots, x, kp);
    int64_t o = row * kp + g.tx * N;
    Pack<double> bv = ld(b + o), rv;
#pragma unroll
    for (int e = 0; e < N; ++e) {
      rv.v[e] = bv.v[e] - ax.v[e];
      acc[e] += rv.v[e] * rv.v[e];
      if constexpr (kFloor) {
        double f = aabs.v[e] + fabs(bv.v[e]);
        aca[e] += f * f;
      }
    }
    st(r + o, rv);
  }
  // a settled pack keeps the last sweep's sums
  block_colsum<double, N>(g, acc, sm.red, s.part + (int64_t)tile * kp, !settled);
  __syncthreads();
  block_colsum<double, N>(g, axx, sm.red, s.part3 + (int64_t)tile * kp, !settled);
  if constexpr (kFloor) {
    __syncthreads();
    block_colsum<double, N>(g, aca, sm.red, s.part2 + (int64_t)tile * kp);
  }
  if constexpr (kFloor) {
    const double* const parts[3] = {s.part, s.part3, s.part2};
    if (!tile_sums<3>(g, parts, s.gpart, s.gcount, s.counter + sd, kp, tile, tl.lo[sd],
                      tl.hi[sd], sm.scratch, sm.sums))
      return;
    // (a settled pack's part2 holds zeros: its reference stays)
    for (int c = g.tid; c < kp; c += g.nth)
      if (sm.sums[2 * kp + c] > 0.0) s.oaa[sd * kp + c] = sm.sums[2 * kp + c];
  } else {
    const double* const parts[2] = {s.part, s.part3};
    if (!tile_sums<2>(g, parts, s.gpart, s.gcount, s.counter + sd, kp, tile, tl.lo[sd],
                      tl.hi[sd], sm.scratch, sm.sums))
      return;
  }
  for (int c = g.tid; c < kp; c += g.nth) s.xx[sd * kp + c] = sm.sums[kp + c];
  __shared__ int cnt, nfl, nnear;
  if (g.tid == 0) cnt = nfl = nnear = 0;
  __syncthreads();
  // attainable accuracy: the rounding error of the binary64 residual of a binary64 x is
  // about u || |A| |x| + |b| ||_2 (u = 2^-53); a residual below kResidualFloor times that
  // is rounding noise, so the column stops there even if rtol is not reached.  The
  // reference (oaa, squared) is refreshed only by the kFloor sweeps; it is a scale,
  // and zero (no floor test) until the first of them
  const double fl2 = (kResidualFloor * 0x1p-53) * (kResidualFloor * 0x1p-53);
  for (int c = g.tid; c < kp; c += g.nth) {
    int i = sd * kp + c;
    double rr = sm.sums[c];
    s.orr[i] = rr;
    bool by_rtol = rr <= rtol2 * s.obb[i];
    bool by_floor = rr <= fl2 * s.oaa[i];
    bool done = (c >= nc) || !(s.obb[i] > 0.0) || by_rtol || by_floor;
    s.scale[i] = done ? 0.0 : 1.0 / sqrt(rr);
    if (!done) atomicAdd(&cnt, 1);
    if (c < nc && s.obb[i] > 0.0 && !by_rtol && by_floor) atomicAdd(&nfl, 1);
    // || |A| |x| + |b| || <= ||A||_inf ||x|| + ||b|| (A symmetric): a column above
    // that bound's rounding level cannot stop on the floor test, so the reference
    // needs refreshing only when some open column is below it
    if (!done) {
      double bnd = anorm[sd] * sqrt(s.xx[i]) + sqrt(s.obb[i]);
      if (rr <= fl2 * bnd * bnd) atomicAdd(&nnear, 1);
    }
  }
  __syncthreads();
  if (g.tid == 0) {
    s.active[sd] = cnt;
    s.nfloor[sd] = nfl;
    s.nnear[sd] = nnear;
  }
}

// ---------------------------------------------------------------------------------
// Restriction r_c = Z^T r on a row tile.  Aggregates are contiguous runs of rows, so the
// tile's rows go to shared memory (SB rows at a time) and one thread per (aggregate, pack)
// adds the run in row order: a fixed order, and no atomics.  (Every thread adding its
// rows to the aggregates' slots by shared-memory atomics, one flush per row as the threads'
// rows lie 23 apart, made the x/r update of the 64^3 workload 217 us a launch, now 203.)
constexpr size_t kRestrictWhole = 32 * 1024;  // a whole tile of r up to this, else equal
constexpr size_t kRestrictBytes = 24 * 1024;  // parts of at most this (or RB rows)
__host__ __device__ constexpr __forceinline__ int restrict_rows(int rb, int kp, size_t tsz) {
  const size_t tile = (size_t)kTileRows * kp * tsz;
  if (tile <= kRestrictWhole) return kTileRows;
  const int parts = (int)((tile + kRestrictBytes - 1) / kRestrictBytes);
  const int rows = ((kTileRows + parts - 1) / parts + rb - 1) / rb * rb;
  return rows < kTileRows ? rows : kTileRows;
}
template <typename T>
struct TileRestrict {
  static constexpr int N = Pack<T>::N;
  T* buf;    // SB rows x kp
  T* cs;     // kMaxSlots x kp: sums of the aggregates (tiles of more than SB rows)
  int* run;  // kMaxSlots + 1: first row (in the tile) of each aggregate
  int a0, nsl, SB;
  __device__ __forceinline__ void begin(const Geo& g, int kp, size_t base, int r0, int nrows,
                                        const int32_t* aloc) {
    extern __shared__ __align__(16) unsigned char raw[];
    SB = restrict_rows(g.rb, kp, sizeof(T));
    size_t o = align16(base);
    buf = reinterpret_cast<T*>(raw + o);
    o += align16(sizeof(T) * (size_t)SB * kp);
    cs = reinterpret_cast<T*>(raw + o);
    if (SB < nrows) o += align16(sizeof(T) * (size_t)kMaxSlots * kp);
    run = reinterpret_cast<int*>(raw + o);
    a0 = aloc[r0];
    nsl = aloc[r0 + nrows - 1] - a0 + 1;
    for (int rr = g.tid; rr < nrows; rr += g.nth) {
      const int a = aloc[r0 + rr];
      if (rr == 0 || a != aloc[r0 + rr - 1]) run[a - a0] = rr;
    }
    if (g.tid == 0) run[nsl] = nrows;
  }
  __device__ __forceinline__ void put(int rr, int kp, int tx, const Pack<T>& v) {
    st(buf + rr * kp + tx * N, v);
  }
  // rows [s0, s0 + SB) are in buf (and visible): add them; the last step stores to dst.
  // S threads share an (aggregate, pack) where there are more threads than pairs, each a
  // stretch of the run, their sums meeting in red (one pack per thread)
  __device__ __forceinline__ void add(const Geo& g, int kp, int s0, int nrows, T* red, T* dst) {
    const int s1 = min(nrows, s0 + SB);
    const int items = nsl * g.nch, S = max(1, g.nth / items);
    for (int idx = g.tid; idx < items * S; idx += g.nth) {
      const int it = idx % items, sg = idx / items;
      const int sl = it / g.nch, pk = it - sl * g.nch;
      const int r0 = max(run[sl], s0), len = max(0, min(run[sl + 1], s1) - r0);
      const int lo = r0 + len * sg / S, hi = r0 + len * (sg + 1) / S;
      Pack<T> acc;
#pragma unroll
      for (int e = 0; e < N; ++e) acc.v[e] = T(0);
#pragma unroll 4
      for (int rr = lo; rr < hi; ++rr) {
        const Pack<T> v = ld(buf + (rr - s0) * kp + pk * N);
#pragma unroll
        for (int e = 0; e < N; ++e) acc.v[e] += v.v[e];
      }
      if (S == 1)
        finish(kp, s0, s1 == nrows, sl, pk, acc, dst);
      else
        st(red + g.tid * N, acc);
    }
    if (S == 1) return;
    __syncthreads();
    if (g.tid < items) {
      Pack<T> acc = ld(red + g.tid * N);
      for (int sg = 1; sg < S; ++sg) {
        const Pack<T> v = ld(red + (sg * items + g.tid) * N);
#pragma unroll
        for (int e = 0; e < N; ++e) acc.v[e] += v.v[e];
      }
      const int sl = g.tid / g.nch;
      finish(kp, s0, s1 == nrows, sl, g.tid - sl * g.nch, acc, dst);
    }
    __syncthreads();
  }
  __device__ __forceinline__ void finish(int kp, int s0, bool last, int sl, int pk, Pack<T> acc,
                                         T* dst) {
    if (s0 > 0) {
      const Pack<T> v = ld(cs + sl * kp + pk * N);
#pragma unroll
      for (int e = 0; e < N; ++e) acc.v[e] = v.v[e] + acc.v[e];
    }
    st((last ? dst + (int64_t)sl * kp : cs + sl * kp) + pk * N, acc);
  }
};
// k_cg_start has a binary64 column-sum area behind the usual layout
template <typename T>
__host__ __device__ constexpr __forceinline__ size_t start_smem_base(int nch, int rb, int kp) {
  return align16(smem_bytes<T>(nch, rb, kp, 0)) +
         sizeof(double) * Pack<T>::N * (size_t)nch * rb;
}
template <typename T>
constexpr size_t restrict_smem_bytes(int rb, int kp) {
  const int SB = restrict_rows(rb, kp, sizeof(T));
  return align16(sizeof(T) * (size_t)SB * kp) +
         (SB < kTileRows ? align16(sizeof(T) * (size_t)kMaxSlots * kp) : 0) +
         align16(sizeof(int) * (kMaxSlots + 1));
}

// Start of a solve with x = 0, in one pass over b: x64 = 0, xT = 0, rT = (T) b, the binary64
// norms that fix the references of the convergence test (RefineState, as k_residual64 leaves
// it for a residual b), the fine r.z = b.D^{-1}b, ||b||^2 and the restriction of b; the
// coarse kernel (INIT) then sets rz and the p update forms p = M^{-1} b.  One read of b and
// three writes instead of a zero fill, a residual sweep A 0, a cast and an init pass: the
// sweep alone was a full binary64 product: 2.35 ms of the 64^3 workload's solve, 0.32 now.
template <typename T>
__global__ void k_cg_start(DTiles tl, const double* __restrict__ b64, double* x64, T* x, T* r,
                           const T* __restrict__ dinv, int kp, int nc, int ncn, double rtol2,
                           CgState s, RefineState rs, Coarse<T> co) {
  constexpr int N = Pack<T>::N;
  Geo g = geo();
  Smem<T> sm = smem_layout<T>(g, kp, 0);
  int tile = blockIdx.x, sd = tl.sd[tile];
  int r0 = tl.r0[tile], r1 = tl.r1[tile];
  const bool coarse = co.aloc != nullptr;
  const int nrows = r1 - r0;
  TileRestrict<T> tr;
  if (coarse) tr.begin(g, kp, start_smem_base<T>(g.nch, g.rb, kp), r0, nrows, co.aloc);
  const int step = coarse ? tr.SB : nrows;
  T arz[N], arr[N];
  double ab[N];
#pragma unroll
  for (int e = 0; e < N; ++e) {
    arz[e] = arr[e] = T(0);
    ab[e] = 0.0;
  }
  Pack<T> zero;
#pragma unroll
  for (int e = 0; e < N; ++e) zero.v[e] = T(0);
  const Pack<double> zero64{{0.0, 0.0}};
  for (int s0 = 0; s0 < nrows; s0 += step) {
    for (int rr = s0 + g.ty; rr < min(nrows, s0 + step); rr += g.rb) {
      const int64_t row = r0 + rr;
      const int64_t o = row * kp + g.tx * N;
      Pack<T> bv;
      const T d = dinv[row];
#pragma unroll
      for (int h = 0; h < N; h += 2) {
        const Pack<double> v = ld(b64 + o + h);
        st(x64 + o + h, zero64);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          ab[h + e] += v.v[e] * v.v[e];
          bv.v[h + e] = (T)v.v[e];
        }
      }
#pragma unroll
      for (int e = 0; e < N; ++e) {
        arz[e] += bv.v[e] * (d * bv.v[e]);
        arr[e] += bv.v[e] * bv.v[e];
      }
      if (coarse) tr.put(rr - s0, kp, g.tx, bv);
      st(x + o, zero);
      st(r + o, bv);
    }
    if (coarse) {
      __syncthreads();
      tr.add(g, kp, s0, nrows, sm.red, co.cpart + co.toff[tile] * kp);
      if (s0 + step < nrows) __syncthreads();
    }
  }
  block_colsum<T, N>(g, arz, sm.red, s.part1 + (int64_t)tile * kp);
  __syncthreads();
  block_colsum<T, N>(g, arr, sm.red, s.part2 + (int64_t)tile * kp);
  __syncthreads();
  double* red64;
  {
    extern __shared__ __align__(16) unsigned char raw[];
    red64 = reinterpret_cast<double*>(raw + align16(smem_bytes<T>(g.nch, g.rb, kp, 0)));
  }
  block_colsum<double, N>(g, ab, red64, rs.part + (int64_t)tile * kp);
  const double* const parts[3] = {rs.part, s.part1, s.part2};
  if (!tile_sums<3>(g, parts, s.gpart, s.gcount, s.counter + sd, kp, tile, tl.lo[sd], tl.hi[sd],
                    sm.scratch, sm.sums))
    return;
  __shared__ double bref, bref64;
  __shared__ int open64;
  if (g.tid == 0) {
    double m = 0.0, m64 = 0.0;
    for (int c = 0; c < ncn; ++c) {
      m = fmax(m, sm.sums[2 * kp + c]);
      m64 = fmax(m64, sm.sums[c]);
    }
    bref = m;
    bref64 = m64;
    open64 = 0;
  }
  __syncthreads();
  for (int c = g.tid; c < kp; c += g.nth) {
    int i = sd * kp + c;
    const double rr = sm.sums[c], obb = c < ncn ? bref64 : rr;
    const bool done = c >= nc || !(obb > 0.0) || rr <= rtol2 * obb || rr <= 0.0;
    rs.obb[i] = obb;
    rs.oaa[i] = 0.0;
    rs.orr[i] = rr;
    rs.xx[i] = 0.0;
    rs.scale[i] = done ? 0.0 : 1.0 / sqrt(rr);
    if (!done) atomicAdd(&open64, 1);
    const double bb = sm.sums[2 * kp + c];
    s.rzf[i] = sm.sums[kp + c];
    s.bb[i] = (c < ncn) ? bref : bb;
    s.rr[i] = bb;
    s.done[i] = (c >= nc || !(bb > 0.0)) ? 1 : 0;
    set_coef(s.alpha, s.alpha32, i, 0.0);
    set_coef(s.beta, s.beta32, i, 0.0);
    set_coef(s.gam, s.gam32, i, 1.0);
  }
  __syncthreads();
  if (g.tid == 0) {
    s.iters[sd] = 0;
    rs.active[sd] = open64;
    rs.nfloor[sd] = rs.nnear[sd] = 0;
  }
  count_active(g, s.done, sd, kp, s.active);
}

// x += alpha p, r -= alpha q; ||r||^2, the fine r.z = r.D^{-1}r and the restriction of
// the new r; the coarse kernel (STEP) completes r.M^{-1}r, beta and the done flags.
// TH = 256: 48 registers (binary32) leave room for five blocks per SM; six cost spills.
// TH = 1024: light loads (light_threads).  R rows in flight per thread (wide_rows)
template <typename T, int TH, int R = 1>
__global__ void __launch_bounds__(TH, TH == 256 ? (R == 2 ? 3 : sizeof(T) == 4 ? 5 : 4) : 1)
    k_cg_update_xr(DTiles tl, T* x, T* r, const T* __restrict__ p, const T* __restrict__ q,
                   const T* __restrict__ dinv, int kp, CgState s, Coarse<T> co) {
  constexpr int N = Pack<T>::N;
  Geo g = geo();
  Smem<T> sm = smem_layout<T>(g, kp, 0);
  int tile = blockIdx.x, sd = tl.sd[tile];
  if (s.active[sd] == 0) return;
  const int r0 = tl.r0[tile], nrows = tl.r1[tile] - r0;
  const bool coarse = co.aloc != nullptr;
  TileRestrict<T> tr;
  if (coarse) tr.begin(g, kp, smem_bytes<T>(g.nch, g.rb, kp, 0), r0, nrows, co.aloc);
  const int step = coarse ? tr.SB : nrows;
  const bool skip = pack_done<T>(s, sd, kp, g.tx);
  const Pack<T> alp = coef_pack<T>(s.alpha, s.alpha32, sd, kp, g.tx);
  T al[N];
#pragma unroll
  for (int e = 0; e < N; ++e) al[e] = alp.v[e];
  T arr[N], arz[N];
#pragma unroll
  for (int e = 0; e < N; ++e) arr[e] = arz[e] = T(0);
  for (int s0 = 0; s0 < nrows; s0 += step) {
    const int send = min(nrows, s0 + step);
    for (int rb = s0 + g.ty; rb < send; rb += R * g.rb) {
      Pack<T> xv[R], pv[R], qv[R], rv[R];
      T d[R];
#pragma unroll
      for (int u = 0; u < R; ++u) {
        const int64_t row = r0 + rb + u * g.rb, o = row * kp + g.tx * N;
        if (skip || rb + u * g.rb >= send) {
#pragma unroll
          for (int e = 0; e < N; ++e) rv[u].v[e] = T(0);
          continue;
        }
        xv[u] = ld(x + o), pv[u] = ld(p + o), qv[u] = ld(q + o);
        rv[u] = ld(r + o);
        d[u] = dinv[row];
      }
#pragma unroll
      for (int u = 0; u < R; ++u) {
        const int rr = rb + u * g.rb;
        if (rr >= send) continue;
        const int64_t o = (int64_t)(r0 + rr) * kp + g.tx * N;
        if (!skip) {
#pragma unroll
          for (int e = 0; e < N; ++e) {
            xv[u].v[e] += al[e] * pv[u].v[e];
            rv[u].v[e] -= al[e] * qv[u].v[e];
            arr[e] += rv[u].v[e] * rv[u].v[e];
            arz[e] += rv[u].v[e] * (d[u] * rv[u].v[e]);
          }
          st(x + o, xv[u]);
          st(r + o, rv[u]);
        }
        if (coarse) tr.put(rr - s0, kp, g.tx, rv[u]);
      }
    }
    if (coarse) {
      __syncthreads();
      tr.add(g, kp, s0, nrows, sm.red, co.cpart + co.toff[tile] * kp);
      if (s0 + step < nrows) __syncthreads();
    }
  }
  block_colsum<T, N>(g, arr, sm.red, s.part1 + (int64_t)tile * kp);
  __syncthreads();
  block_colsum<T, N>(g, arz, sm.red, s.part2 + (int64_t)tile * kp);
  const double* const parts[2] = {s.part1, s.part2};
  if (!tile_sums<2>(g, parts, s.gpart, s.gcount, s.counter + sd, kp, tile, tl.lo[sd], tl.hi[sd],
                    sm.scratch, sm.sums))
    return;
  for (int c = g.tid; c < kp; c += g.nth) {
    int i = sd * kp + c;
    s.rr[i] = sm.sums[c];
    s.rzf[i] = sm.sums[kp + c];
  }
}

constexpr int kCoarseCols = 16;
enum { kCoarseInit = 0, kCoarseStep = 1, kCoarseReplace = 2 };

// The last block of a subdomain in the coarse kernels: r.M^{-1}r = fine part + the
// nrb row blocks' parts of r_c.y_c (in order); mode STEP: the convergence test on the
// recursive residual, beta and gam, the work counts (cw: columns per chunk, each open
// chunk reads E^{-1} once) and the active count; INIT / REPLACE: rz only.
template <typename T>
__device__ void coarse_finish(const Geo& g, const DTiles& tl, int sd, int kp, int cw, int nrb,
                              double tol2, int mode, CgState& s, const Coarse<T>& co) {
  constexpr int PN = Pack<T>::N;
  const int nchunk = (kp + cw - 1) / cw;
  // the subdomain's columns: open packs before the update (the sparse product and the
  // x/r update of this step worked on them), the test and beta, open packs after
  __shared__ int open_pre, open_post, chunks_open, open_cols;
  const bool count = s.work && mode == kCoarseStep;
  if (g.tid == 0) open_pre = open_post = chunks_open = open_cols = 0;
  __syncthreads();
  if (count) {
    for (int pk = g.tid; pk * PN < kp; pk += g.nth) {
      bool open = false;
      for (int e = 0; e < PN; ++e) open = open || !s.done[sd * kp + pk * PN + e];
      if (open) atomicAdd(&open_pre, 1);
    }
    for (int ch = g.tid; ch < nchunk; ch += g.nth) {
      bool open = false;
      for (int j = 0; j < cw && ch * cw + j < kp; ++j) open = open || !s.done[sd * kp + ch * cw + j];
      if (open) atomicAdd(&chunks_open, 1);
    }
    __syncthreads();
  }
  int open = 0;
  for (int c = g.tid; c < kp; c += g.nth) {
    const int i = sd * kp + c;
    const double rzf = s.rzf[i], rr = s.rr[i], bb = s.bb[i], rz = s.rz[i];
    int done = s.done[i];
    double cd = 0.0;
    if (co.dpart)
      for (int r0 = 0; r0 < nrb; r0 += 4) {
        double v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          v[u] = r0 + u < nrb ? __ldcg(co.dpart + ((int64_t)sd * nrb + r0 + u) * kp + c) : 0.0;
#pragma unroll
        for (int u = 0; u < 4; ++u) cd += v[u];
      }
    const double rzn = rzf + cd;
    if (mode == kCoarseStep) {
      double be = 0.0;
      if (!done) {
        if (rr <= tol2 * bb || !(rz > 0.0)) {
          s.done[i] = done = 1;
        } else {
          be = rzn / rz;
          s.rz[i] = rzn;
        }
      }
      set_coef(s.beta, s.beta32, i, be);
      set_coef(s.gam, s.gam32, i, 1.0);
      open += !done;
    } else {
      s.rz[i] = rzn;
    }
  }
  if (mode != kCoarseStep) return;
  if (open) atomicAdd(&open_cols, open);
  __syncthreads();
  if (count) {
    for (int pk = g.tid; pk * PN < kp; pk += g.nth) {
      bool op = false;
      for (int e = 0; e < PN; ++e) op = op || !s.done[sd * kp + pk * PN + e];
      if (op) atomicAdd(&open_post, 1);
    }
    __syncthreads();
    if (g.tid == 0) {
      // work counts of the algorithmic-bytes model
      const int nsd = tl.n_sd;
      const unsigned long long rows = (unsigned long long)s.sd_rows[sd];
      const unsigned long long nc = co.tbase ? (unsigned long long)co.nca[sd] : 0ull;
      atomicAdd(s.work + sd, (unsigned long long)s.sd_nnz[sd]);
      atomicAdd(s.work + nsd + sd, (unsigned long long)open_pre * rows);
      atomicAdd(s.work + 2 * nsd + sd, (unsigned long long)open_post * rows);
      if (nc) atomicAdd(s.work + 3 * nsd + sd, (unsigned long long)chunks_open * nc * nc);
    }
  }
  if (g.tid == 0) {
    s.active[sd] = open_cols;
    if (open_cols > 0) s.iters[sd] += 1;
  }
}

// r_c pack (aggregate ga, N columns from column c): the partials of an aggregate are
// consecutive rows of cpart, one per tile that holds some of its rows
template <typename T>
__device__ __forceinline__ Pack<T> restrict_pack(const Coarse<T>& co, int ga, int kp, int c) {
  const int64_t b0 = co.tbase[ga];
  const int tn = co.tcount[ga];
  Pack<T> v = ld(co.cpart + b0 * kp + c);
  for (int t = 1; t < tn; ++t) {
    const Pack<T> pv = ld(co.cpart + (b0 + t) * kp + c);
#pragma unroll
    for (int e = 0; e < Pack<T>::N; ++e) v.v[e] += pv.v[e];
  }
  return v;
}

// Coarse level of one subdomain in SIMT arithmetic, up to kCoarseSmallMax aggregates
// (block (column chunk, sd), CW columns): r_c = Z^T r for the chunk, y_c = E^{-1} r_c, the
// chunk's part of r_c.y_c; the last chunk of the subdomain (atomic ticket) finishes.
//  - Binary64: one thread per (row, column).  A multiply-add occupies its quarter of the SM
//    for 64 clocks per warp, so the products are spread over as many warps and blocks as
//    there are: 16 columns per thread took 69 us a launch for 27 subdomains of 52
//    aggregates and 32 columns, 20 us now.
//  - Binary32: one thread per row and all CW columns.  Bound by the loads: an element of
//    E^{-1}, read coalesced, feeds CW multiply-adds, and a block of 8 columns reads E^{-1}
//    half as often as one of 4.  14 subdomains of up to 200
//    aggregates, 264 columns: 34 -> 23 us against one thread per (row, column).
constexpr int kCoarseSmallMax = 256;
constexpr int kCoarseThreads = 256;
template <typename T, int CW>
__global__ void __launch_bounds__(kCoarseThreads)
    k_cg_coarse_small(DTiles tl, int kp, double tol2, int mode, CgState s, Coarse<T> co) {
  constexpr int PN = Pack<T>::N;
  __shared__ __align__(16) T rc[kCoarseSmallMax * CW];
  __shared__ double red[(kCoarseThreads / 32) * CW];
  Geo g = geo();
  const int sd = blockIdx.y, c0 = blockIdx.x * CW, ncol = min(CW, kp - c0);
  if (s.active[sd] == 0) return;
  bool open = false;  // a chunk whose columns have all converged needs no coarse product
#pragma unroll
  for (int j = 0; j < CW; ++j) open = (j < ncol && !s.done[sd * kp + c0 + j]) || open;
  const int n = co.tbase && open ? co.nca[sd] : 0;
  const int j = g.tid % CW, lane = g.tid & 31;
  const int a0 = n > 0 ? co.aoff[sd] : 0;
  const T* Eb = n > 0 ? co.einv + co.eoff[sd] : nullptr;
  if (n > 0) {
    for (int idx = g.tid; idx < n * (CW / PN); idx += g.nth) {
      const int a = idx / (CW / PN), pk = idx - a * (CW / PN);
      Pack<T> v;
#pragma unroll
      for (int e = 0; e < PN; ++e) v.v[e] = T(0);
      if (pk * PN < ncol) v = restrict_pack(co, a0 + a, kp, c0 + pk * PN);
      st(rc + a * CW + pk * PN, v);
    }
    __syncthreads();
  }
  if constexpr (sizeof(T) == 4) {
    double dl[CW];
#pragma unroll
    for (int c = 0; c < CW; ++c) dl[c] = 0.0;
    const int a = g.tid;
    if (a < n) {
      T y[CW];
#pragma unroll
      for (int c = 0; c < CW; ++c) y[c] = T(0);
#pragma unroll 8
      for (int b = 0; b < n; ++b) {
        const T e = Eb[(int64_t)b * n + a];  // symmetric: column a as row a
#pragma unroll
        for (int pk = 0; pk < CW / PN; ++pk) {
          const Pack<T> v = ld(rc + b * CW + pk * PN);
#pragma unroll
          for (int c = 0; c < PN; ++c) y[pk * PN + c] += e * v.v[c];
        }
      }
#pragma unroll
      for (int pk = 0; pk < CW / PN; ++pk) {
        Pack<T> yv;
#pragma unroll
        for (int c = 0; c < PN; ++c) {
          yv.v[c] = y[pk * PN + c];
          dl[pk * PN + c] = (double)yv.v[c] * (double)rc[a * CW + pk * PN + c];
        }
        if (pk * PN < ncol) st(co.yc + (int64_t)(a0 + a) * kp + c0 + pk * PN, yv);
      }
    }
    // the warp's CW sums: halves of the columns change sides until a lane holds one
    int c = 0, o = 16;
#pragma unroll
    for (int h = CW / 2; h >= 1; h /= 2, o /= 2) {
      const bool up = (lane & o) != 0;
      c += up ? h : 0;
#pragma unroll
      for (int i = 0; i < h; ++i) {
        const double give = up ? dl[i] : dl[i + h], keep = up ? dl[i + h] : dl[i];
        dl[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
      }
    }
    for (; o >= 1; o /= 2) dl[0] += __shfl_xor_sync(0xffffffffu, dl[0], o);
    if ((lane & (32 / CW - 1)) == 0) red[(g.tid >> 5) * CW + c] = dl[0];
  } else {
    double dl = 0.0;
    for (int a = g.tid / CW; a < n; a += kCoarseThreads / CW) {
      // E^{-1} is symmetric: row a is read as column a (eight rows per warp: one sector or two)
      T acc0 = T(0), acc1 = T(0);
      int b = 0;
      for (; b + 8 <= n; b += 8) {
        T e[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) e[u] = Eb[(int64_t)(b + u) * n + a];
#pragma unroll
        for (int u = 0; u < 8; u += 2) {
          acc0 += e[u] * rc[(b + u) * CW + j];
          acc1 += e[u + 1] * rc[(b + u + 1) * CW + j];
        }
      }
      for (; b < n; ++b) acc0 += Eb[(int64_t)b * n + a] * rc[b * CW + j];
      const T y = acc0 + acc1;
      co.yc[(int64_t)(a0 + a) * kp + c0 + j] = y;
      dl += (double)y * (double)rc[a * CW + j];
    }
    for (int o = CW; o < 32; o <<= 1) dl += __shfl_xor_sync(0xffffffffu, dl, o);
    if (lane < CW) red[(g.tid >> 5) * CW + lane] = dl;
  }
  __syncthreads();
  if (g.tid < ncol && co.dpart) {
    double t = 0.0;
    for (int w = 0; w < kCoarseThreads / 32; ++w) t += red[w * CW + g.tid];
    __stcg(co.dpart + (int64_t)sd * kp + c0 + g.tid, t);
  }
  if (!take_ticket(g, s.counter + sd, gridDim.x)) return;
  coarse_finish<T>(g, tl, sd, kp, CW, 1, tol2, mode, s, co);
}

// Coarse level of one subdomain in SIMT arithmetic, above kCoarseSmallMax aggregates
// (grid: x = row block x column chunk, y = subdomain).  Block (rb, chunk) forms r_c = Z^T r
// for the chunk's kCoarseCols columns from the tile partials, then rows [rb R, (rb + 1) R) of
// y_c = E^{-1} r_c (stored for the p update), R = kCoarseThreads kCoarseRpt with kCoarseRpt
// rows per thread, and their part of r_c.y_c.  The last block of the subdomain (atomic
// ticket) adds the parts in row-block order and finishes.  The blocks of one row block are
// adjacent in the grid, so the chunks read its E^{-1} rows from L2 after the first.
constexpr int kCoarseRpt = 2;  // rows of y_c per thread
constexpr size_t kCoarseRedBytes = sizeof(double) * (kCoarseThreads / 32) * kCoarseCols;
template <typename T>
__global__ void __launch_bounds__(kCoarseThreads)
    k_cg_coarse(DTiles tl, int kp, double tol2, int mode, CgState s, Coarse<T> co) {
  constexpr int kCoarseRows = kCoarseThreads * kCoarseRpt;
  constexpr int CW = kCoarseCols;
  constexpr int PN = Pack<T>::N;
  Geo g = geo();
  extern __shared__ __align__(16) unsigned char raw[];
  T* rc = reinterpret_cast<T*>(raw);  // round_up(n, 8) x CW
  // rc holds round_up(n_max, 8) rows (the product reads whole groups of 8)
  const int n_max8 = (co.n_max + 7) & ~7;
  double* red = reinterpret_cast<double*>(raw + align16(sizeof(T) * n_max8 * CW));
  const int sd = blockIdx.y;
  const int nchunk = (kp + CW - 1) / CW;
  const int chunk = blockIdx.x % nchunk, rbk = blockIdx.x / nchunk;
  const int nrb = gridDim.x / nchunk;
  const int c0 = chunk * CW, ncol = min(CW, kp - c0);
  if (s.active[sd] == 0) return;
  // a chunk whose columns have all converged needs no coarse product
  bool chunk_open = false;
  for (int j = 0; j < ncol; ++j) chunk_open = !s.done[sd * kp + c0 + j] || chunk_open;
  const int n = chunk_open ? co.nca[sd] : 0;
  const int a_lo = rbk * kCoarseRows, a_hi = min(n, a_lo + kCoarseRows);
  double dl[CW];
#pragma unroll
  for (int j = 0; j < CW; ++j) dl[j] = 0.0;
  if (a_lo < n) {
    const int a0 = co.aoff[sd];
    // r_c = Z^T r: one (aggregate, pack) pair per thread step (kp and c0 are multiples of
    // the pack width).  Rows n .. round_up(n, 8) are zero: the product runs in steps of 8.
    const int n8 = (n + 7) & ~7, cwp = CW / PN;
    for (int idx = g.tid; idx < n8 * cwp; idx += g.nth) {
      const int a = idx / cwp, pk = idx - a * cwp;
      Pack<T> v;
#pragma unroll
      for (int e = 0; e < PN; ++e) v.v[e] = T(0);
      if (a < n && pk * PN < ncol) v = restrict_pack(co, a0 + a, kp, c0 + pk * PN);
      st(rc + a * CW + pk * PN, v);
    }
    __syncthreads();
    // rows a_lo + tid + kCoarseThreads i, i < kCoarseRpt, one thread each
    if (a_lo + g.tid < a_hi) {
      // E^{-1} is symmetric: row a is read as column a, coalesced across the block;
      // each element feeds the CW multiply-adds of the chunk, the r_c pieces (broadcast
      // shared loads) feed the kCoarseRpt rows of the thread, and eight columns of
      // loads are issued before their multiply-adds
      const T* Eb = co.einv + co.eoff[sd];
      int ra[kCoarseRpt];
      bool rv[kCoarseRpt];
#pragma unroll
      for (int i = 0; i < kCoarseRpt; ++i) {
        ra[i] = a_lo + g.tid + kCoarseThreads * i;
        rv[i] = ra[i] < a_hi;
      }
      T acc[kCoarseRpt][CW];
#pragma unroll
      for (int i = 0; i < kCoarseRpt; ++i)
#pragma unroll
        for (int j = 0; j < CW; ++j) acc[i][j] = T(0);
      for (int b0 = 0; b0 < n; b0 += 8) {
        T e[8][kCoarseRpt];
#pragma unroll
        for (int u = 0; u < 8; ++u)
#pragma unroll
          for (int i = 0; i < kCoarseRpt; ++i)
            e[u][i] = (b0 + u < n && rv[i]) ? Eb[(int64_t)(b0 + u) * n + ra[i]] : T(0);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const T* rb = rc + (b0 + u) * CW;
#pragma unroll
          for (int h = 0; h < CW; h += PN) {
            Pack<T> xv = ld(rb + h);
#pragma unroll
            for (int i = 0; i < kCoarseRpt; ++i)
#pragma unroll
              for (int e2 = 0; e2 < PN; ++e2) acc[i][h + e2] += e[u][i] * xv.v[e2];
          }
        }
      }
#pragma unroll
      for (int i = 0; i < kCoarseRpt; ++i) {
        if (!rv[i]) continue;
        T* yo = co.yc + (int64_t)(a0 + ra[i]) * kp + c0;
#pragma unroll
        for (int j = 0; j < CW; ++j) {
          if (j < ncol) yo[j] = acc[i][j];
          dl[j] += (double)acc[i][j] * (double)rc[ra[i] * CW + j];
        }
      }
    }
  }
  // this block's part of r_c.y_c per column: rows summed within each warp (fixed
  // shuffle tree), then the warps in order
  {
    const int lane = g.tid & 31, wid = g.tid >> 5;
#pragma unroll
    for (int j = 0; j < CW; ++j) {
      double v = dl[j];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
      if (lane == 0) red[wid * CW + j] = v;
    }
    __syncthreads();
    if (g.tid < ncol) {
      double t = 0.0;
      for (int w = 0; w < g.nth / 32; ++w) t += red[w * CW + g.tid];
      co.dpart[((int64_t)sd * nrb + rbk) * kp + c0 + g.tid] = t;
    }
  }
  if (!take_ticket(g, s.counter + sd, gridDim.x)) return;
  coarse_finish<T>(g, tl, sd, kp, CW, nrb, tol2, mode, s, co);
}

// The coarse product of the binary32 path on the tensor cores, y_c = E^{-1} r_c for
// every column (NP = kp rounded up to 16, at most 128), in two kernels.
// k_coarse_rc_pack forms r_c = Z^T r per 32-aggregate block from the tile partials, keeps
// it in binary32 and as bf16 high and low planes in the K-major operand layout (row =
// column of r_c).  k_cg_coarse_tc then runs a cluster of KS CTAs per 128 rows of y_c: CTA
// k takes every KS-th part of the aggregates and accumulates its products in TMEM
// (tcgen05, A = E^{-1} from launch_coarse_tc_pack, B = r_c, three products hi.hi + hi.lo +
// lo.hi per block: about 16 significant bits of each factor; the dropped lo.lo term is
// below 2^-16 of a product, under the binary32 accumulation error of a 1,000-term sum).
// One thread streams the operand blocks (whole and contiguous) through kTcStages stages
// with bulk copies, another issues the MMAs; stages are handed over by mbarriers alone.
// The CTAs' accumulators then go to shared memory, and every CTA adds the cluster's for its
// share of the columns (distributed shared memory, in order), stores y_c and forms r_c.y_c
// in binary64; the last block of the subdomain finishes.  Every wait is bounded (a timeout
// sets co.tc_err; the CTA still waits for its own copies and MMAs, keeps to the cluster's
// barriers and leaves).
// What bounds it: latency.  One CTA over all of K with cp.async, two block barriers and one
// wait per 32 aggregates took 1.2 us per block, and r_c.y_c 10 us of shuffled binary64
// additions: 53 us a step (with the packing) however few subdomains, 26 us now; 64 subdomains
// of up to 1,000 aggregates 76 -> 51 us.
constexpr int kTcThreads = 128;  // one thread per accumulator row (TMEM lane)
constexpr int kTcStages = 4;
constexpr int kTcTileLd = kCoarseTcM + 1;  // padded row of the accumulator tile
__device__ __forceinline__ void split_bf16(float v, __nv_bfloat16& h, __nv_bfloat16& l) {
  h = __float2bfloat16_rn(v);
  l = __float2bfloat16_rn(v - __bfloat162float(h));
}

// block (kb, sd): r_c of aggregates 32 kb .. 32 kb + 31 into co.rcf and co.rcb, one thread
// per (aggregate, 4 columns)
constexpr int kRcThreads = 128;
__global__ void __launch_bounds__(kRcThreads)
    k_coarse_rc_pack(int kp, int NP, CgState s, Coarse<float> co) {
  const int sd = blockIdx.y, kb = blockIdx.x;
  if (s.active[sd] == 0) return;
  const int n = co.nca[sd];
  if (kb * tc::kKB >= n) return;
  const int npk = NP / 4;
  const int idx = blockIdx.z * kRcThreads + threadIdx.x;
  if (idx >= tc::kKB * npk) return;
  const int a0 = co.aoff[sd];
  __nv_bfloat16* bh = co.rcb + (co.rcb_off[sd] + kb) * (int64_t)(2 * NP * tc::kKB);
  __nv_bfloat16* bl = bh + NP * tc::kKB;
  const int k = idx / npk, pk = idx - k * npk;
  const int a = kb * tc::kKB + k;
  Pack<float> v;
#pragma unroll
  for (int e = 0; e < 4; ++e) v.v[e] = 0.0f;
  if (a < n && 4 * pk < kp) {
    v = restrict_pack(co, a0 + a, kp, 4 * pk);
    st(co.rcf + (int64_t)(a0 + a) * kp + 4 * pk, v);
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    __nv_bfloat16 h, l;
    split_bf16(v.v[e], h, l);
    const uint32_t o = tc::kmajor(4 * pk + e, k) >> 1;
    bh[o] = h;
    bl[o] = l;
  }
}

__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, uint32_t bytes,
                                          uint32_t mbar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(dst),
      "l"(src), "r"(bytes), "r"(mbar)
      : "memory");
}

__global__ void __launch_bounds__(kTcThreads)
    k_cg_coarse_tc(DTiles tl, int kp, int NP, double tol2, int mode, CgState s,
                   Coarse<float> co) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  constexpr int KB = tc::kKB;
  constexpr int A_PLANE = kCoarseTcM * KB * 2;  // bytes
  extern __shared__ __align__(128) unsigned char smem[];
  const int B_PLANE = NP * KB * 2;
  const int STAGE = 2 * A_PLANE + 2 * B_PLANE;  // A hi, A lo, B hi, B lo
  float* tile = reinterpret_cast<float*>(smem);  // after the MMAs: NP x kTcTileLd
  __shared__ uint32_t tmem_base;
  __shared__ __align__(8) uint64_t full[kTcStages], empty[kTcStages], ready;
  __shared__ double red[kTcThreads * 4];
  Geo g = geo();
  const int tid = threadIdx.x, warp = tid >> 5;
  const int KS = (int)cl.num_blocks(), ks = (int)cl.block_rank();
  const int sd = blockIdx.y, mt = blockIdx.x / KS, nmt = gridDim.x / KS;
  if (s.active[sd] == 0) return;  // the whole cluster
  const int n = co.nca[sd];
  const int a_lo = mt * kCoarseTcM;
  const int npk = NP / 4 / KS;  // packs of this CTA's share of the columns
  const int c_lo = ks * npk * 4;
  if (a_lo < n) {
    const int a0 = co.aoff[sd];
    const int nkb = (n + KB - 1) / KB;
    const int kb0 = nkb * ks / KS, nblk = nkb * (ks + 1) / KS - kb0;
    const unsigned char* Ag = reinterpret_cast<const unsigned char*>(
        co.etc + (co.etc_off[sd] + (int64_t)mt * nkb + kb0) * 1024);
    const unsigned char* Bg = reinterpret_cast<const unsigned char*>(
        co.rcb + (co.rcb_off[sd] + kb0) * (int64_t)(2 * NP * KB));
    const uint32_t s0 = (uint32_t)__cvta_generic_to_shared(smem);
    const uint32_t mfull = (uint32_t)__cvta_generic_to_shared(full);
    const uint32_t mempty = (uint32_t)__cvta_generic_to_shared(empty);
    const uint32_t mready = (uint32_t)__cvta_generic_to_shared(&ready);
    uint32_t ncols = 32;
    while (ncols < (uint32_t)NP) ncols <<= 1;
    if (warp == 0) {
      const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&tmem_base);
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                   ::"r"(dst), "r"(ncols));
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
      for (int q = 0; q < kTcStages; ++q) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mfull + 8 * q));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mempty + 8 * q));
      }
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mready));
      asm volatile("fence.mbarrier_init.release.cluster;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tbase = tmem_base;
    bool ok = true;
    if (tid == 32) {
      // operand blocks kb0 .. kb0 + nblk - 1 into the stages in turn
      int i = 0;
      for (; i < nblk && ok; ++i) {
        const int q = i % kTcStages;
        if (i >= kTcStages)
          ok = tc::mbar_wait(mempty + 8 * q, (uint32_t)(i / kTcStages - 1) & 1u, co.tc_budget);
        if (!ok) break;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mfull + 8 * q),
                     "r"((uint32_t)STAGE)
                     : "memory");
        bulk_copy(s0 + q * STAGE, Ag + (int64_t)i * (2 * A_PLANE), 2 * A_PLANE, mfull + 8 * q);
        bulk_copy(s0 + q * STAGE + 2 * A_PLANE, Bg + (int64_t)i * (2 * B_PLANE), 2 * B_PLANE,
                  mfull + 8 * q);
      }
      // after a timeout: the copies in flight still land in this CTA's shared memory
      if (!ok)
        for (int j = i > kTcStages ? i - kTcStages : 0; j < i; ++j)
          tc::mbar_wait(mfull + 8 * (j % kTcStages), (uint32_t)(j / kTcStages) & 1u,
                        co.tc_budget);
    } else if (tid == 0) {
      const uint32_t idesc = tc::instr_desc(kCoarseTcM, NP);
      for (int i = 0; i < nblk; ++i) {
        const int q = i % kTcStages;
        ok = tc::mbar_wait(mfull + 8 * q, (uint32_t)(i / kTcStages) & 1u, co.tc_budget);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;");
        const uint32_t sa = s0 + (uint32_t)(q * STAGE);
        const int pa[3] = {0, 0, 1}, pb[3] = {0, 1, 0};  // hi.hi, hi.lo, lo.hi
#pragma unroll
        for (int x = 0; x < 3; ++x)
#pragma unroll
          for (int k = 0; k < KB / 16; ++k) {
            const uint64_t ad =
                tc::smem_desc(sa + (uint32_t)(pa[x] * A_PLANE + k * 256), 128, (KB / 8) * 128);
            const uint64_t bd = tc::smem_desc(
                sa + (uint32_t)(2 * A_PLANE + pb[x] * B_PLANE + k * 256), 128, (KB / 8) * 128);
            const uint32_t en = (i == 0 && x == 0 && k == 0) ? 0u : 1u;
            asm volatile(
                "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tbase),
                "l"(ad), "l"(bd), "r"(idesc), "r"(en));
          }
        asm volatile(
            "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                mempty + 8 * q));
      }
      // every MMA issued so far (none where the aggregates are fewer than the CTAs)
      if (nblk > 0)
        asm volatile(
            "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                mready));
      else
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mready) : "memory");
    }
    __syncwarp();
    // the MMAs are done: their stages may be overwritten
    if (!tc::mbar_wait(mready, 0, co.tc_budget)) {
      ok = false;
      tc::mbar_wait(mready, 0, co.tc_budget);
    }
    if (!ok) atomicExch(co.tc_err, 1);
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    // row a of the accumulator is TMEM lane a = thread tid; eight columns per load
    for (int c = 0; c < NP; c += 8) {
      uint32_t r[8];
      const uint32_t ta = tbase + ((uint32_t)(warp * 32) << 16) + (uint32_t)c;
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
          : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
            "=r"(r[7])
          : "r"(ta));
      asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
      for (int e = 0; e < 8; ++e)
        tile[(c + e) * kTcTileLd + tid] = nblk > 0 ? __uint_as_float(r[e]) : 0.0f;
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    if (KS > 1)
      cl.sync();
    else
      __syncthreads();
    if (warp == 0)
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase),
                   "r"(ncols));
    // y_c and r_c.y_c for this CTA's columns: thread (pack tx, rows ty, ty + RB, ...)
    const int RB = kTcThreads / npk, tx = tid % npk, ty = tid / npk;
    const int c = c_lo + 4 * tx;
    double dl[4] = {0.0, 0.0, 0.0, 0.0};
    if (ty < RB && c < kp)
      for (int r = ty; r < kCoarseTcM && a_lo + r < n; r += RB) {
        const int64_t at = (int64_t)(a0 + a_lo + r) * kp + c;
        const Pack<float> rv = ld(co.rcf + at);
        Pack<float> y;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          y.v[e] = 0.0f;
          for (int k = 0; k < KS; ++k)
            y.v[e] += *(KS > 1 ? cl.map_shared_rank(tile + (c + e) * kTcTileLd + r, k)
                               : tile + (c + e) * kTcTileLd + r);
          dl[e] += (double)y.v[e] * (double)rv.v[e];
        }
        st(co.yc + at, y);
      }
#pragma unroll
    for (int e = 0; e < 4; ++e) red[tid * 4 + e] = dl[e];
    __syncthreads();
    for (int x = tid; x < 4 * npk && c_lo + x < kp; x += kTcThreads) {
      double t = 0.0;
      for (int q = 0; q < RB; ++q) t += red[(q * npk + x / 4) * 4 + (x & 3)];
      __stcg(co.dpart + ((int64_t)sd * nmt + mt) * kp + c_lo + x, t);
    }
    if (KS > 1) cl.sync();  // no CTA leaves while another reads its accumulators
  } else {
    for (int x = tid; x < 4 * npk && c_lo + x < kp; x += kTcThreads)
      __stcg(co.dpart + ((int64_t)sd * nmt + mt) * kp + c_lo + x, 0.0);
  }
  if (!take_ticket(g, s.counter + sd, gridDim.x)) return;
  coarse_finish<float>(g, tl, sd, kp, kp, nmt, tol2, mode, s, co);
}

// p = gam (D^{-1} r + Z y_c) + beta p (p is not read where beta = 0), and p.r of the
// new direction for the next step length
template <typename T, int TH, int R = 1>
__global__ void __launch_bounds__(TH, TH == 256 ? (sizeof(T) == 4 && R == 1 ? 6 : 4) : 1)
    k_cg_update_p(DTiles tl, const T* __restrict__ r, T* p, const T* __restrict__ dinv, int kp,
                  CgState s, Coarse<T> co) {
  constexpr int N = Pack<T>::N;
  Geo g = geo();
  Smem<T> sm = smem_layout<T>(g, kp, 0);
  int tile = blockIdx.x, sd = tl.sd[tile];
  if (s.active[sd] == 0) return;
  int r0 = tl.r0[tile], r1 = tl.r1[tile];
  const int64_t rend = pack_done<T>(s, sd, kp, g.tx) ? r0 : r1;
  const bool coarse = co.aloc != nullptr;
  const int64_t a0 = coarse ? co.aoff[sd] : 0;
  const Pack<T> bep = coef_pack<T>(s.beta, s.beta32, sd, kp, g.tx);
  const Pack<T> gap = coef_pack<T>(s.gam, s.gam32, sd, kp, g.tx);
  T be[N];
  bool hasp[N], hasz[N];  // beta != 0; gam is 0 or 1
  bool needp = false;
#pragma unroll
  for (int e = 0; e < N; ++e) {
    be[e] = bep.v[e];
    hasp[e] = nonzero(be[e]);
    hasz[e] = nonzero(gap.v[e]);
    needp = needp || hasp[e];
  }
  T apr[N];
#pragma unroll
  for (int e = 0; e < N; ++e) apr[e] = T(0);
  for (int64_t rowb = r0 + g.ty; rowb < rend; rowb += R * g.rb) {
    Pack<T> rv[R], pv[R], yv[R];
    T d[R];
#pragma unroll
    for (int u = 0; u < R; ++u) {
      const int64_t row = rowb + u * g.rb, o = row * kp + g.tx * N;
      if (row >= rend) continue;
      rv[u] = ld(r + o);
      if (needp) pv[u] = ld(p + o);
      if (coarse) yv[u] = ld(co.yc + (a0 + co.aloc[row]) * kp + g.tx * N);
      d[u] = dinv[row];
    }
    // three multiply-adds per element: choices of 0 by select, not by a product (a binary64
    // operation or compare holds its quarter of the SM for 64 clocks per warp)
#pragma unroll
    for (int u = 0; u < R; ++u) {
      const int64_t row = rowb + u * g.rb;
      if (row >= rend) continue;
#pragma unroll
      for (int e = 0; e < N; ++e) {
        T z = coarse ? fma_t(d[u], rv[u].v[e], yv[u].v[e]) : d[u] * rv[u].v[e];
        z = hasz[e] ? z : T(0);
        const T v = fma_t(be[e], hasp[e] ? pv[u].v[e] : T(0), z);
        pv[u].v[e] = v;
        apr[e] = fma_t(v, rv[u].v[e], apr[e]);
      }
      st(p + row * kp + g.tx * N, pv[u]);
    }
  }
  block_colsum<T, N>(g, apr, sm.red, s.part1 + (int64_t)tile * kp);
  const double* const parts[1] = {s.part1};
  if (!tile_sums<1>(g, parts, s.gpart, s.gcount, s.counter + sd, kp, tile, tl.lo[sd], tl.hi[sd],
                    sm.scratch, sm.sums))
    return;
  for (int c = g.tid; c < kp; c += g.nth) s.pr[sd * kp + c] = sm.sums[c];
}

// out[0] = sum of active, out[1] = sum of second (if not null), out[2] = row tiles of the
// subdomains with active > 0
__global__ void k_count_active(DTiles tl, const int* active, const int* second, int* out) {
  __shared__ int tot[3];
  if (threadIdx.x < 3) tot[threadIdx.x] = 0;
  __syncthreads();
  int a = 0, b = 0, t = 0;
  for (int i = threadIdx.x; i < tl.n_sd; i += blockDim.x) {
    const int ac = active[i];
    a += ac;
    if (second) b += second[i];
    if (ac > 0) t += tl.hi[i] - tl.lo[i];
  }
  atomicAdd(&tot[0], a);
  atomicAdd(&tot[1], b);
  atomicAdd(&tot[2], t);
  __syncthreads();
  if (threadIdx.x < 3) out[threadIdx.x] = tot[threadIdx.x];
}

// residual replacement: rT = (T) r64 (the true residual), the fine r.z and the
// restriction of it, each column's done flag from the binary64 convergence test
// (scale == 0).  Columns the recursion had declared converged but the binary64 test
// reopens, and columns whose true residual norm exceeds drift x the recursive one,
// restart from p = M^{-1} r (their stored direction belongs to a much smaller
// residual: gam = 1, beta = 0); the others keep p (gam = 0, beta = 1).  The coarse
// kernel (REPLACE) then sets rz and the p update applies gam and beta.
template <typename T>
__global__ void k_cg_replace(DTiles tl, const double* __restrict__ r64, T* __restrict__ rT,
                             const T* __restrict__ dinv, int kp, double drift2, CgState s,
                             RefineState rs, Coarse<T> co) {
  constexpr int N = Pack<T>::N;
  Geo g = geo();
  Smem<T> sm = smem_layout<T>(g, kp, 0);
  int tile = blockIdx.x, sd = tl.sd[tile];
  // closed in both tests: nothing of this subdomain is read again
  if (s.active[sd] == 0 && rs.active[sd] == 0) return;
  int r0 = tl.r0[tile], r1 = tl.r1[tile];
  const bool coarse = co.aloc != nullptr;
  const int nrows = r1 - r0;
  TileRestrict<T> tr;
  if (coarse) tr.begin(g, kp, smem_bytes<T>(g.nch, g.rb, kp, 0), r0, nrows, co.aloc);
  const int step = coarse ? tr.SB : nrows;
  const bool settled = pack_settled<N>(rs, sd, kp, g.tx, 1);
  T arz[N];
#pragma unroll
  for (int e = 0; e < N; ++e) arz[e] = T(0);
  for (int s0 = 0; s0 < nrows; s0 += step) {
    for (int rr = s0 + g.ty; rr < min(nrows, s0 + step); rr += g.rb) {
      const int64_t row = r0 + rr;
      int64_t o = row * kp + g.tx * N;
      Pack<T> rv;
      if (settled) {
#pragma unroll
        for (int e = 0; e < N; ++e) rv.v[e] = T(0);
      } else {
        T d = dinv[row];
#pragma unroll
        for (int h = 0; h < N; h += 2) {
          const Pack<double> v = ld(r64 + o + h);
          rv.v[h] = (T)v.v[0];
          rv.v[h + 1] = (T)v.v[1];
        }
#pragma unroll
        for (int e = 0; e < N; ++e) arz[e] += rv.v[e] * (d * rv.v[e]);
        st(rT + o, rv);
      }
      if (coarse) tr.put(rr - s0, kp, g.tx, rv);
    }
    if (coarse) {
      __syncthreads();
      tr.add(g, kp, s0, nrows, sm.red, co.cpart + co.toff[tile] * kp);
      if (s0 + step < nrows) __syncthreads();
    }
  }
  block_colsum<T, N>(g, arz, sm.red, s.part1 + (int64_t)tile * kp);
  const double* const parts[1] = {s.part1};
  if (!tile_sums<1>(g, parts, s.gpart, s.gcount, s.counter + sd, kp, tile, tl.lo[sd], tl.hi[sd],
                    sm.scratch, sm.sums))
    return;
  for (int c = g.tid; c < kp; c += g.nth) {
    int i = sd * kp + c;
    // reopened, or the recursion drifted from the true residual (a stale direction
    // would make the next step length meaningless)
    bool restart = rs.scale[i] != 0.0 && (s.done[i] || rs.orr[i] > drift2 * s.rr[i]);
    bool done = rs.scale[i] == 0.0;
    s.rzf[i] = sm.sums[c];
    s.bb[i] = rs.obb[i];
    s.done[i] = done ? 1 : 0;
    set_coef(s.alpha, s.alpha32, i, 0.0);
    set_coef(s.beta, s.beta32, i, (done || restart) ? 0.0 : 1.0);
    set_coef(s.gam, s.gam32, i, (done || restart) ? 1.0 : 0.0);
  }
  __syncthreads();
  count_active(g, s.done, sd, kp, s.active);
}

// x64 += xT; xT = 0 (settled packs: xT is zero)
template <typename T>
__global__ void __launch_bounds__(256)
    k_accum_reset(DTiles tl, T* __restrict__ xT, double* __restrict__ x64, int kp, int seen,
                  RefineState rs) {
  constexpr int N = Pack<T>::N;
  Geo g = geo();
  const int tile = blockIdx.x, sd = tl.sd[tile];
  if (seen && rs.active[sd] == 0) return;
  if (pack_settled<N>(rs, sd, kp, g.tx, seen)) return;
  Pack<T> zero;
#pragma unroll
  for (int e = 0; e < N; ++e) zero.v[e] = T(0);
  const int r1 = tl.r1[tile];
  for (int row = tl.r0[tile] + g.ty; row < r1; row += 2 * g.rb) {
    // both rows' loads before the first store
    Pack<T> v[2];
    Pack<double> y[2][N / 2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int64_t o = (int64_t)(row + u * g.rb) * kp + g.tx * N;
      if (row + u * g.rb >= r1) continue;
      v[u] = ld(xT + o);
#pragma unroll
      for (int h = 0; h < N / 2; ++h) y[u][h] = ld(x64 + o + 2 * h);
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int64_t o = (int64_t)(row + u * g.rb) * kp + g.tx * N;
      if (row + u * g.rb >= r1) continue;
#pragma unroll
      for (int h = 0; h < N / 2; ++h) {
        y[u][h].v[0] += (double)v[u].v[2 * h];
        y[u][h].v[1] += (double)v[u].v[2 * h + 1];
        st(x64 + o + 2 * h, y[u][h]);
      }
      st(xT + o, zero);
    }
  }
}

// per subdomain: max over its rows of sum_j |a_ij| (nonnegative doubles order like
// their bit patterns, so an integer atomicMax is exact); out zeroed by the caller
__global__ void k_row_abs_max(DTiles tl, EllView<double> A, unsigned long long* out) {
  const int tile = blockIdx.x, sd = tl.sd[tile];
  const int64_t row = tl.r0[tile] + (int64_t)threadIdx.x;
  double sum = 0.0;
  if (row < tl.r1[tile]) {
    const int w = A.width[row >> 5];
    for (int j = 0; j < w; ++j) {
      int64_t at = ell_at(row, j, A.W);
      if (A.col[at] >= 0) sum += fabs(A.val[at]);
    }
  }
  for (int o = 16; o > 0; o >>= 1) sum = fmax(sum, __shfl_xor_sync(0xFFFFFFFFu, sum, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out + sd, (unsigned long long)__double_as_longlong(sum));
}

// rows per pass of a tile kernel's block of about `threads` threads, a pack of columns each
template <typename T>
constexpr int block_rows(int kp, int threads) {
  const int rb = threads / (kp / Pack<T>::N);
  return rb < 1 ? 1 : rb < kTileRows ? rb : kTileRows;
}
template <typename T>
dim3 block_of(int kp, int threads = 256) {
  return dim3(kp / Pack<T>::N, block_rows<T>(kp, threads));
}

// Threads per block of a step's tile kernels by the row tiles of the subdomains still
// open.  A full chip wants blocks of 256 (registers, several blocks per SM).  With no more
// tiles than SMs a step is as long as one block, whose threads take their rows one after
// the other: blocks of 1024 shorten that chain (16^3 workload, 113 tiles: 18.4 -> 17.6 ms;
// blocks of 512 up to 456 tiles: no change).  Binary64 steps are bound by their arithmetic,
// of which larger blocks have more (block_colsum; 21 -> 27 ms): 256 always.
template <typename T>
int light_threads(int open_tiles) {
  if (sizeof(T) == 8) return 256;
  return open_tiles <= 152 ? 1024 : 256;
}

}  // namespace

constexpr size_t kSmemSlots = 160 * 1024;  // kernels that stage a tile's slots
constexpr size_t kSmemRows = 180 * 1024;   // kernels that stage a tile's rows of r
template <typename T>
void set_smem_attr(const void* fn, size_t bytes = kSmemSlots) {
  cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <typename T>
void launch_spmm(const DTiles& tiles, const EllView<T>& A, const T* X, T* Y, int kp,
                 cudaStream_t st) {
  if (tiles.n <= 0) return;
  static bool attr = false;
  if (!attr) {
    set_smem_attr<T>((const void*)k_spmm<T>);
    attr = true;
  }
  dim3 bl = block_of<T>(kp);
  count_launch();
  k_spmm<T><<<tiles.n, bl, smem_bytes<T>(bl.x, bl.y, kp, A.W), st>>>(tiles, A, X, Y, kp);
}

// Two rows in flight per thread in the updates where a block holds up to eight (more than 28
// packs of columns): its threads walk 16 or more rows one after another (wide sketches on
// 25^3: x/r update 47 -> 40 us, p update 26 -> 22).
bool wide_rows(dim3 bl) { return bl.y <= 8; }  // (binary32)

template <typename T>
constexpr size_t slot_kernel_smem(int nch, int rb, int kp) {
  return align16(smem_bytes<T>(nch, rb, kp, 0)) + restrict_smem_bytes<T>(rb, kp);
}
template <typename T>
constexpr size_t start_kernel_smem(int nch, int rb, int kp) {
  return align16(start_smem_base<T>(nch, rb, kp)) + restrict_smem_bytes<T>(rb, kp);
}
// every column count a build can have stays within the kernels' limit (the most: 179,712
// bytes, k_cg_start in binary64 at 512 columns)
template <typename T>
constexpr bool rows_smem_fits() {
  for (int kp = 4; kp <= kMaxCols; kp += 4) {
    const int nch = kp / Pack<T>::N;
    for (int threads = 256; threads <= (sizeof(T) == 4 ? 1024 : 256); threads *= 4)
      if (slot_kernel_smem<T>(nch, block_rows<T>(kp, threads), kp) > kSmemRows) return false;
    if (start_kernel_smem<T>(nch, block_rows<T>(kp, 256), kp) > kSmemRows) return false;
  }
  return true;
}
static_assert(rows_smem_fits<float>() && rows_smem_fits<double>(), "shared-memory limit");

template <typename T>
void launch_coarse_then_p(const DTiles& tiles, int n_sd, const T* r, T* p, const T* dinv,
                          int kp, double tol2, int mode, int open_tiles, const CgState& s,
                          const Coarse<T>& co, cudaStream_t st, const cudaEvent_t* ev_mid) {
  static bool attr = false;
  if (!attr) {
    const int mx = (int)(align16(sizeof(T) * kMaxAgg * kCoarseCols) + kCoarseRedBytes);
    cudaFuncSetAttribute((const void*)k_cg_coarse<T>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
    attr = true;
  }
  const int n_max = co.tbase ? co.n_max : 0;
  bool done = false;
  if constexpr (sizeof(T) == 4) {
    if (co.etc) {
      // tensor-core product: a cluster per 128 rows of y_c and subdomain, every column
      const int NP = (kp + 15) & ~15;
      const int nmt = std::max(1, (n_max + kCoarseTcM - 1) / kCoarseTcM);
      const int nkb = std::max(1, (n_max + tc::kKB - 1) / tc::kKB);
      // split the aggregates over 2 or 4 CTAs while the grid stays within two blocks per SM
      int KS = 1;
      while (KS < 4 && 2 * KS * nmt * n_sd <= 2 * 152 && 4 * KS <= nkb) KS *= 2;
      const size_t smt = std::max((size_t)kTcStages * (2 * (kCoarseTcM * tc::kKB * 2) +
                                                       2 * NP * tc::kKB * 2),
                                  sizeof(float) * kTcTileLd * (size_t)NP);
      static bool attr_tc = false;
      if (!attr_tc) {
        cudaFuncSetAttribute((const void*)k_cg_coarse_tc,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        attr_tc = true;
      }
      count_launch(2);
      const int per = tc::kKB * (NP / 4);
      k_coarse_rc_pack<<<dim3(nkb, n_sd, (per + kRcThreads - 1) / kRcThreads), kRcThreads, 0,
                         st>>>(kp, NP, s, co);
      cudaLaunchAttribute at{};
      at.id = cudaLaunchAttributeClusterDimension;
      at.val.clusterDim.x = (unsigned)KS;
      at.val.clusterDim.y = at.val.clusterDim.z = 1;
      cudaLaunchConfig_t cfg{};
      cfg.gridDim = dim3(nmt * KS, n_sd);
      cfg.blockDim = dim3(kTcThreads);
      cfg.dynamicSmemBytes = smt;
      cfg.stream = st;
      cfg.attrs = &at;
      cfg.numAttrs = 1;
      cudaLaunchKernelEx(&cfg, k_cg_coarse_tc, tiles, kp, NP, tol2, mode, s, co);
      done = true;
    }
  }
  if (!done) {
    count_launch();
    if (n_max <= kCoarseSmallMax) {
      // 8 columns a block while that leaves two blocks per SM
      const bool wide = sizeof(T) == 4 && (kp + 7) / 8 * n_sd >= 2 * 152;
      const int cw = wide ? 8 : 4;
      auto fn = wide ? k_cg_coarse_small<T, sizeof(T) == 4 ? 8 : 4> : k_cg_coarse_small<T, 4>;
      fn<<<dim3((kp + cw - 1) / cw, n_sd), kCoarseThreads, 0, st>>>(tiles, kp, tol2, mode, s, co);
    } else {
      const size_t sm = align16(sizeof(T) * ((n_max + 7) & ~7) * kCoarseCols) + kCoarseRedBytes;
      const int rows = kCoarseRpt * kCoarseThreads;
      const int nrb = (n_max + rows - 1) / rows;
      const int nchunk = (kp + kCoarseCols - 1) / kCoarseCols;
      k_cg_coarse<T><<<dim3(nrb * nchunk, n_sd), kCoarseThreads, sm, st>>>(tiles, kp, tol2, mode,
                                                                          s, co);
    }
  }
  if (ev_mid) cudaEventRecord(*ev_mid, st);
  count_launch();
  const int th = light_threads<T>(open_tiles);
  const dim3 bl = block_of<T>(kp, th);
  const size_t sm = smem_bytes<T>(bl.x, bl.y, kp, 0);
  auto fn = k_cg_update_p<T, 256>;
  if constexpr (sizeof(T) == 4)
    fn = th == 1024 ? k_cg_update_p<T, 1024> : wide_rows(bl) ? k_cg_update_p<T, 256, 2> : fn;
  fn<<<tiles.n, bl, sm, st>>>(tiles, r, p, dinv, kp, s, co);
}

template <typename T>
void launch_cg_start(const DTiles& tiles, const double* b64, double* x64, T* x, T* r, T* p,
                     const T* dinv, int kp, int nc, int ncn, double rtol2, const CgState& s,
                     const RefineState& rs, const Coarse<T>& co, cudaStream_t st) {
  if (tiles.n <= 0) return;
  static bool attr = false;
  if (!attr) {
    set_smem_attr<T>((const void*)k_cg_start<T>, kSmemRows);
    attr = true;
  }
  dim3 bl = block_of<T>(kp);
  const size_t sm = start_kernel_smem<T>(bl.x, bl.y, kp);
  count_launch();
  k_cg_start<T><<<tiles.n, bl, sm, st>>>(tiles, b64, x64, x, r, dinv, kp, nc, ncn, rtol2, s, rs,
                                         co);
  launch_coarse_then_p<T>(tiles, tiles.n_sd, r, p, dinv, kp, 0.0, kCoarseInit, tiles.n, s, co, st,
                          nullptr);
}

// ---- autotuner of the sparse product: four launch configurations of k_cg_spmm_pq
// (1 or 2 records per gather batch, blocks of 256 or 128 threads), timed on the first
// product of each (precision, column count, slot width) the process meets, the fastest
// kept for the rest of the process.  The product is a pure function of p (q, its
// column sums and the step length are rewritten), so timing it on live data changes
// no result.
constexpr int kSpmmVariants = 4;
template <typename T>
void launch_spmm_pq_variant(int v, const DTiles& tiles, const EllView<T>& A, const T* p, T* q,
                            int kp, const CgState& s, cudaStream_t st) {
  const int th = (v & 2) ? 128 : 256;
  dim3 bl = block_of<T>(kp, th);
  const size_t sm = smem_bytes<T>(bl.x, bl.y, kp, A.W);
  switch (v) {
    case 0: k_cg_spmm_pq<T, 1, 256><<<tiles.n, bl, sm, st>>>(tiles, A, p, q, kp, s); break;
    case 1: k_cg_spmm_pq<T, 2, 256><<<tiles.n, bl, sm, st>>>(tiles, A, p, q, kp, s); break;
    case 2: k_cg_spmm_pq<T, 1, 128><<<tiles.n, bl, sm, st>>>(tiles, A, p, q, kp, s); break;
    default: k_cg_spmm_pq<T, 2, 128><<<tiles.n, bl, sm, st>>>(tiles, A, p, q, kp, s); break;
  }
}

struct TuneEntry {
  int wide, kp, W, variant;
  float ms[kSpmmVariants];
};
std::mutex g_tune_mu;
std::vector<TuneEntry> g_tune;
bool g_tune_on = true;

template <typename T>
int spmm_variant(const DTiles& tiles, const EllView<T>& A, const T* p, T* q, int kp,
                 const CgState& s, cudaStream_t st) {
  const int wide = sizeof(T) == 8 ? 1 : 0;
  std::lock_guard<std::mutex> lock(g_tune_mu);
  for (const auto& e : g_tune)
    if (e.wide == wide && e.kp == kp && e.W == A.W) return e.variant;
  if (!g_tune_on || kp / Pack<T>::N > 128) return 0;
  static bool attr = false;
  if (!attr) {
    set_smem_attr<T>((const void*)k_cg_spmm_pq<T, 1, 256>);
    set_smem_attr<T>((const void*)k_cg_spmm_pq<T, 2, 256>);
    set_smem_attr<T>((const void*)k_cg_spmm_pq<T, 1, 128>);
    set_smem_attr<T>((const void*)k_cg_spmm_pq<T, 2, 128>);
    attr = true;
  }
  TuneEntry e{wide, kp, A.W, 0, {0, 0, 0, 0}};
  cudaEvent_t a, b;
  cudaEventCreate(&a);
  cudaEventCreate(&b);
  for (int v = 0; v < kSpmmVariants; ++v) {
    launch_spmm_pq_variant<T>(v, tiles, A, p, q, kp, s, st);  // warm-up
    cudaEventRecord(a, st);
    for (int rep = 0; rep < 3; ++rep) launch_spmm_pq_variant<T>(v, tiles, A, p, q, kp, s, st);
    cudaEventRecord(b, st);
    cudaEventSynchronize(b);
    float t = 0.f;
    cudaEventElapsedTime(&t, a, b);
    e.ms[v] = t / 3.0f;
    count_launch(4);
  }
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  for (int v = 1; v < kSpmmVariants; ++v)
    if (e.ms[v] < e.ms[e.variant]) e.variant = v;
  g_tune.push_back(e);
  return e.variant;
}

template <typename T>
void tune_spmm(const DTiles& tiles, const EllView<T>& A, const T* p, T* q, int kp,
               const CgState& s, cudaStream_t st) {
  if (tiles.n > 0) spmm_variant<T>(tiles, A, p, q, kp, s, st);
}
template void tune_spmm<float>(const DTiles&, const EllView<float>&, const float*, float*, int,
                               const CgState&, cudaStream_t);
template void tune_spmm<double>(const DTiles&, const EllView<double>&, const double*, double*,
                                int, const CgState&, cudaStream_t);

template <typename T>
void launch_cg_step(const DTiles& tiles, const EllView<T>& A, T* x, T* r, T* p, T* q,
                    const T* dinv, int kp, double tol2, int open_tiles, const CgState& s,
                    const Coarse<T>& co, cudaStream_t st, const cudaEvent_t* ev) {
  if (tiles.n <= 0) return;
  static bool attr = false;
  if (!attr) {
    set_smem_attr<T>((const void*)k_cg_spmm_pq<T, 1, 256>);
    set_smem_attr<T>((const void*)k_cg_spmm_pq<T, 2, 256>);
    set_smem_attr<T>((const void*)k_cg_spmm_pq<T, 1, 128>);
    set_smem_attr<T>((const void*)k_cg_spmm_pq<T, 2, 128>);
    set_smem_attr<T>((const void*)k_cg_update_xr<T, 256>, kSmemRows);
    if constexpr (sizeof(T) == 4) {
      set_smem_attr<T>((const void*)k_cg_spmm_pq<T, 2, 1024>);
      set_smem_attr<T>((const void*)k_cg_update_xr<T, 256, 2>, kSmemRows);
      set_smem_attr<T>((const void*)k_cg_update_xr<T, 1024>, kSmemRows);
    }
    attr = true;
  }
  const int th = light_threads<T>(open_tiles);
  const dim3 bl = block_of<T>(kp, th);
  const int variant = spmm_variant<T>(tiles, A, p, q, kp, s, st);
  count_launch(2);
  if (ev) cudaEventRecord(ev[0], st);
  if (th == 256)
    launch_spmm_pq_variant<T>(variant, tiles, A, p, q, kp, s, st);
  else if constexpr (sizeof(T) == 4)
    k_cg_spmm_pq<T, 2, 1024><<<tiles.n, bl, smem_bytes<T>(bl.x, bl.y, kp, A.W), st>>>(
        tiles, A, p, q, kp, s);
  if (ev) cudaEventRecord(ev[1], st);
  auto fn = k_cg_update_xr<T, 256>;
  if constexpr (sizeof(T) == 4)
    fn = th == 1024 ? k_cg_update_xr<T, 1024> : wide_rows(bl) ? k_cg_update_xr<T, 256, 2> : fn;
  fn<<<tiles.n, bl, slot_kernel_smem<T>(bl.x, bl.y, kp), st>>>(tiles, x, r, p, q, dinv, kp, s, co);
  if (ev) cudaEventRecord(ev[2], st);
  launch_coarse_then_p<T>(tiles, tiles.n_sd, r, p, dinv, kp, tol2, kCoarseStep, open_tiles, s, co,
                          st, ev ? &ev[3] : nullptr);
  if (ev) cudaEventRecord(ev[4], st);
}

void launch_count_active(const DTiles& tiles, const int* active, int* out, cudaStream_t st,
                         const int* second) {
  count_launch();
  k_count_active<<<1, 256, 0, st>>>(tiles, active, second, out);
}

void launch_residual64(const DTiles& tiles, const EllView<double>& A, const double* b64,
                       const double* x64, double* r64, int kp, int nc, double rtol2, bool seen,
                       bool floor_ref, const double* anorm, const RefineState& s,
                       cudaStream_t st) {
  if (tiles.n <= 0) return;
  static bool attr = false;
  if (!attr) {
    set_smem_attr<double>((const void*)k_residual64<false>);
    set_smem_attr<double>((const void*)k_residual64<true>);
    attr = true;
  }
  dim3 bl = block_of<double>(kp);
  size_t sm = smem_bytes<double>(bl.x, bl.y, kp, A.W);
  count_launch();
  auto fn = floor_ref ? k_residual64<true> : k_residual64<false>;
  fn<<<tiles.n, bl, sm, st>>>(tiles, A, b64, x64, r64, kp, nc, rtol2, seen ? 1 : 0, s, anorm);
}

template <typename T>
void launch_cg_replace(const DTiles& tiles, const double* r64, T* rT, T* pT, const T* dinv,
                       int kp, double drift, const CgState& s, const RefineState& rs,
                       const Coarse<T>& co, cudaStream_t st) {
  if (tiles.n <= 0) return;
  static bool attr = false;
  if (!attr) {
    set_smem_attr<T>((const void*)k_cg_replace<T>, kSmemRows);
    attr = true;
  }
  dim3 bl = block_of<T>(kp);
  count_launch();
  k_cg_replace<T><<<tiles.n, bl, slot_kernel_smem<T>(bl.x, bl.y, kp), st>>>(
      tiles, r64, rT, dinv, kp, drift * drift, s, rs, co);
  launch_coarse_then_p<T>(tiles, tiles.n_sd, rT, pT, dinv, kp, 0.0, kCoarseReplace,
                          tiles.n, s, co, st, nullptr);
}

template <typename T>
void launch_accum_reset(const DTiles& tiles, T* xT, double* x64, int kp, bool seen,
                        const RefineState& rs, cudaStream_t st) {
  if (tiles.n <= 0) return;
  count_launch();
  k_accum_reset<T><<<tiles.n, block_of<T>(kp), 0, st>>>(tiles, xT, x64, kp, seen ? 1 : 0, rs);
}

// out[sd] += stored entries of the rows of each tile of sd (one thread per row)
__global__ void k_count_sd_nnz(DTiles tl, EllView<double> A, unsigned long long* out) {
  const int tile = blockIdx.x, sd = tl.sd[tile];
  const int64_t row = tl.r0[tile] + (int64_t)threadIdx.x;
  unsigned long long c = 0;
  if (row < tl.r1[tile]) {
    const int w = A.width[row >> 5];
    for (int j = 0; j < w; ++j) c += A.col[ell_at(row, j, A.W)] >= 0;
  }
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xFFFFFFFFu, c, o);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(out + sd, c);
}

void launch_count_sd_nnz(const DTiles& tiles, const EllView<double>& A, int64_t* out,
                         cudaStream_t st) {
  if (tiles.n <= 0) return;
  count_launch();
  k_count_sd_nnz<<<tiles.n, kTileRows, 0, st>>>(tiles, A, (unsigned long long*)out);
}

void launch_row_abs_max(const DTiles& tiles, const EllView<double>& A, double* out,
                        cudaStream_t st) {
  if (tiles.n <= 0) return;
  count_launch();
  k_row_abs_max<<<tiles.n, kTileRows, 0, st>>>(tiles, A, (unsigned long long*)out);
}

template void launch_cg_replace<float>(const DTiles&, const double*, float*, float*,
                                       const float*, int, double, const CgState&,
                                       const RefineState&, const Coarse<float>&, cudaStream_t);
template void launch_cg_replace<double>(const DTiles&, const double*, double*, double*,
                                        const double*, int, double, const CgState&,
                                        const RefineState&, const Coarse<double>&,
                                        cudaStream_t);
template void launch_accum_reset<float>(const DTiles&, float*, double*, int, bool,
                                        const RefineState&, cudaStream_t);
template void launch_accum_reset<double>(const DTiles&, double*, double*, int, bool,
                                         const RefineState&, cudaStream_t);
template void launch_spmm<float>(const DTiles&, const EllView<float>&, const float*, float*,
                                 int, cudaStream_t);
template void launch_spmm<double>(const DTiles&, const EllView<double>&, const double*,
                                  double*, int, cudaStream_t);
template void launch_cg_start<float>(const DTiles&, const double*, double*, float*, float*,
                                     float*, const float*, int, int, int, double,
                                     const CgState&, const RefineState&, const Coarse<float>&,
                                     cudaStream_t);
template void launch_cg_start<double>(const DTiles&, const double*, double*, double*, double*,
                                      double*, const double*, int, int, int, double,
                                      const CgState&, const RefineState&, const Coarse<double>&,
                                      cudaStream_t);
template void launch_cg_step<float>(const DTiles&, const EllView<float>&, float*, float*,
                                    float*, float*, const float*, int, double, int,
                                    const CgState&, const Coarse<float>&, cudaStream_t,
                                    const cudaEvent_t*);
template void launch_cg_step<double>(const DTiles&, const EllView<double>&, double*, double*,
                                     double*, double*, const double*, int, double, int,
                                     const CgState&, const Coarse<double>&, cudaStream_t,
                                     const cudaEvent_t*);
void autotune_enable(bool on) {
  std::lock_guard<std::mutex> lock(g_tune_mu);
  g_tune_on = on;
}

void autotune_reset() {
  std::lock_guard<std::mutex> lock(g_tune_mu);
  g_tune.clear();
}

int autotune_entries(int64_t* out, int max_entries) {
  std::lock_guard<std::mutex> lock(g_tune_mu);
  const int n = (int)g_tune.size();
  for (int i = 0; i < n && i < max_entries; ++i) {
    const TuneEntry& e = g_tune[i];
    int64_t* o = out + 8 * (int64_t)i;
    o[0] = e.wide;
    o[1] = e.kp;
    o[2] = e.W;
    o[3] = e.variant;
    for (int v = 0; v < kSpmmVariants; ++v) o[4 + v] = (int64_t)(1e3 * e.ms[v]);  // us
  }
  return n;
}

}  // namespace mor
