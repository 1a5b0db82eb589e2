// Step 3 (Eq. (23), Sec. 6 step 3): the off-diagonal blocks of Q^T A Q from the
// interface couplings of neighbouring subdomains, the reduced CG solve (diagonal
// preconditioner = identity because every diagonal block is I after the step-2
// update), and the lift u~ = sum_i S_i Q_i x_i.
#include "mor_dev.cuh"
#include "mor_kernels.h"

#include <cooperative_groups.h>

#include <algorithm>

namespace mor {
namespace {

// K~_ij = sum over the entries (u, v) of pair (i, j) of a_uv Q[u]^T Q[v].  The entries come
// sorted by u, so a row of Q_i meets the few rows of Q_j it is coupled with first: w_u =
// sum_v a_uv Q[v], then K~_ij = sum_u Q[u]^T w_u.  Bound by binary64 issue; that takes
// kq + kq^2 / (entries per u, three to four) multiply-adds per entry where the plain sum
// took 2 kq^2 operations.  A block takes `rows` of the kq rows of one pair's block: enough
// blocks for every SM where the pairs are few.  56^3 in 343 subdomains (28 columns) 700 -> 141
// us, 48^3 in 40 (68 columns) 6.2 -> 0.39 ms, 16^3 in 8 (12 columns) 39 -> 11 us.
constexpr int kPairThreads = 256;
constexpr int kPairOut = 16;      // outputs per thread: rows * kq <= 256 * 16
constexpr int kPairEntries = 128;  // entries per chunk
constexpr int kPairGroups = 32;    // rows u per pass
__global__ void __launch_bounds__(kPairThreads)
    k_pair_blocks(const int64_t* __restrict__ pair_ptr, const int32_t* __restrict__ urow,
                  const int32_t* __restrict__ vrow, const double* __restrict__ aval,
                  const double* __restrict__ Q, int kq, int rows, double* blocks) {
  extern __shared__ double sh[];
  double* Wv = sh;                      // [kPairGroups][kq]
  double* Qu = Wv + kPairGroups * kq;   // [kPairGroups][rows]
  __shared__ double av[kPairEntries];
  __shared__ int32_t vr[kPairEntries], gu[kPairEntries];
  __shared__ int gs[kPairEntries + 1], wcnt[kPairEntries / 32];
  const int p = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  const int i0 = blockIdx.y * rows, ni = min(rows, kq - i0);
  const int64_t e0 = pair_ptr[p], e1 = pair_ptr[p + 1];
  const int nout = ni * kq;
  double acc[kPairOut];
#pragma unroll
  for (int m = 0; m < kPairOut; ++m) acc[m] = 0.0;
  for (int64_t base = e0; base < e1; base += kPairEntries) {
    const int ne = (int)min((int64_t)kPairEntries, e1 - base);
    // rows u of the chunk: gu[g], entries gs[g] to gs[g + 1]
    bool head = false;
    int32_t u = 0;
    if (tid < ne) {
      u = urow[base + tid];
      head = tid == 0 || urow[base + tid - 1] != u;
      vr[tid] = vrow[base + tid];
      av[tid] = aval[base + tid];
    }
    const unsigned hb = __ballot_sync(0xFFFFFFFFu, head);
    if (lane == 0 && wp < kPairEntries / 32) wcnt[wp] = __popc(hb);
    __syncthreads();
    int ng = 0, before = 0;
#pragma unroll
    for (int w = 0; w < kPairEntries / 32; ++w) {
      if (w < wp) before += wcnt[w];
      ng += wcnt[w];
    }
    if (head) {
      const int g = before + __popc(hb & ((1u << lane) - 1u));
      gu[g] = u;
      gs[g] = tid;
    }
    if (tid == 0) gs[ng] = ne;
    __syncthreads();
    for (int g0 = 0; g0 < ng; g0 += kPairGroups) {
      const int nb = min(kPairGroups, ng - g0);
      for (int idx = tid; idx < nb * kq; idx += kPairThreads) {
        const int g = idx / kq, j = idx - g * kq;
        double w = 0.0;
        for (int e = gs[g0 + g]; e < gs[g0 + g + 1]; ++e) w += av[e] * Q[(int64_t)vr[e] * kq + j];
        Wv[idx] = w;
      }
      for (int idx = tid; idx < nb * ni; idx += kPairThreads) {
        const int g = idx / ni, i = idx - g * ni;
        Qu[idx] = Q[(int64_t)gu[g0 + g] * kq + i0 + i];
      }
      __syncthreads();
#pragma unroll
      for (int m = 0; m < kPairOut; ++m) {
        const int o = tid + m * kPairThreads;
        if (o < nout) {
          const int i = o / kq, j = o - i * kq;
          double s0 = 0.0, s1 = 0.0;
          int g = 0;
          for (; g + 1 < nb; g += 2) {
            s0 += Qu[g * ni + i] * Wv[g * kq + j];
            s1 += Qu[(g + 1) * ni + i] * Wv[(g + 1) * kq + j];
          }
          if (g < nb) s0 += Qu[g * ni + i] * Wv[g * kq + j];
          acc[m] += s0 + s1;
        }
      }
      __syncthreads();
    }
  }
  double* Bij = blocks + (int64_t)(2 * p) * kq * kq;
  double* Bji = blocks + (int64_t)(2 * p + 1) * kq * kq;
#pragma unroll
  for (int m = 0; m < kPairOut; ++m) {
    const int o = tid + m * kPairThreads;
    if (o < nout) {
      const int i = o / kq, j = o - i * kq;
      Bij[(i0 + i) * kq + j] = acc[m];
      Bji[j * kq + i0 + i] = acc[m];
    }
  }
}

// ---- reduced CG: one block per block row (subdomain), global last-block reductions
__device__ __forceinline__ double block_sum128(double x, double* red) {
  red[threadIdx.x] = x;
  __syncthreads();
  for (int s = 64; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  double r = red[0];
  __syncthreads();
  return r;
}

__device__ __forceinline__ bool last_global(int* counter, int nblk) {
  __shared__ int is_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    int prev = atomicAdd(counter, 1);
    is_last = (prev == nblk - 1);
    if (is_last) *counter = 0;
  }
  __syncthreads();
  if (is_last) __threadfence();
  return is_last;
}

__device__ double sum_parts(const double* part, int n, int stride, int off, double* red) {
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) s += __ldcg(part + (int64_t)i * stride + off);
  return block_sum128(s, red);
}

__global__ void k_rcg_init(int n_sd, int kq, const double* __restrict__ bt, RcgState s) {
  __shared__ double red[128];
  int sd = blockIdx.x;
  double loc = 0.0;
  for (int i = threadIdx.x; i < kq; i += blockDim.x) {
    int64_t g = (int64_t)sd * kq + i;
    double b = bt[g];
    s.x[g] = 0.0;
    s.r[g] = b;
    s.p[g] = b;
    loc += b * b;
  }
  double t = block_sum128(loc, red);
  if (threadIdx.x == 0) s.part[2 * sd] = t;
  if (!last_global(s.counter, n_sd)) return;
  double bb = sum_parts(s.part, n_sd, 2, 0, red);
  if (threadIdx.x == 0) {
    s.scal[0] = bb;
    s.scal[1] = bb;
    s.scal[2] = 0.0;
    s.scal[3] = 0.0;
    s.scal[4] = bb;
    s.flag[0] = (bb > 0.0) ? 0 : 1;
    s.flag[1] = 0;
  }
}

__global__ void k_rcg_spmv(int n_sd, int kq, const int32_t* __restrict__ nbr_ptr,
                           const int32_t* __restrict__ nbr_sd, const int32_t* __restrict__ nbr_blk,
                           const double* __restrict__ blocks, RcgState s) {
  __shared__ double red[128];
  int sd = blockIdx.x;
  double loc = 0.0;
  for (int i = threadIdx.x; i < kq; i += blockDim.x) {
    int64_t g = (int64_t)sd * kq + i;
    double acc = s.p[g];
    for (int q = nbr_ptr[sd]; q < nbr_ptr[sd + 1]; ++q) {
      const double* B = blocks + (int64_t)nbr_blk[q] * kq * kq + (int64_t)i * kq;
      const double* pj = s.p + (int64_t)nbr_sd[q] * kq;
      for (int l = 0; l < kq; ++l) acc += B[l] * pj[l];
    }
    s.q[g] = acc;
    loc += s.p[g] * acc;
  }
  double t = block_sum128(loc, red);
  if (threadIdx.x == 0) s.part[2 * sd] = t;
  if (!last_global(s.counter, n_sd)) return;
  double pq = sum_parts(s.part, n_sd, 2, 0, red);
  if (threadIdx.x == 0) s.scal[2] = (s.flag[0] || !(pq > 0.0)) ? 0.0 : s.scal[0] / pq;
}

__global__ void k_rcg_update_xr(int n_sd, int kq, double tol2, RcgState s) {
  __shared__ double red[128];
  int sd = blockIdx.x;
  double al = s.scal[2];
  double loc = 0.0;
  for (int i = threadIdx.x; i < kq; i += blockDim.x) {
    int64_t g = (int64_t)sd * kq + i;
    s.x[g] += al * s.p[g];
    double r = s.r[g] - al * s.q[g];
    s.r[g] = r;
    loc += r * r;
  }
  double t = block_sum128(loc, red);
  if (threadIdx.x == 0) s.part[2 * sd + 1] = t;
  if (!last_global(s.counter, n_sd)) return;
  double rr = sum_parts(s.part, n_sd, 2, 1, red);
  if (threadIdx.x == 0) {
    double be = 0.0;
    if (!s.flag[0]) {
      s.flag[1] += 1;
      s.scal[4] = rr;
      if (rr <= tol2 * s.scal[1] || !(s.scal[0] > 0.0)) {
        s.flag[0] = 1;
      } else {
        be = rr / s.scal[0];
        s.scal[0] = rr;
      }
    }
    s.scal[3] = be;
  }
}

__global__ void k_rcg_update_p(int kq, RcgState s) {
  int sd = blockIdx.x;
  double be = s.scal[3];
  for (int i = threadIdx.x; i < kq; i += blockDim.x) {
    int64_t g = (int64_t)sd * kq + i;
    s.p[g] = s.r[g] + be * s.p[g];
  }
}

// ---- the whole reduced CG in one launch ----
// What bounds it: GB300 does 2 binary64 multiply-adds per SM and clock (a warp
// instruction keeps its quarter of the SM busy for 64 clocks, and dependent steps are
// about 100 clocks apart), and every iteration needs two sums over all rows.  So the
// matrix is spread as far as the sums allow: up to kRcgClusterFma multiply-adds and
// kRcgClusterDim rows one cluster of 8 CTAs keeps matrix and vectors in shared memory
// and sums through distributed shared memory (k_rcg_cluster, 0.9 to 1.5 us a sum by the
// cluster's threads, 64 to 512 a CTA); above,
// every SM takes part and sums through global memory (k_rcg_grid, 3.5 us).  Whole calls
// measured on both, cluster | every SM: 5 k multiply-adds 137 | 248 us, 28 k 221 | 346,
// 50 k 267 | 370, 78 k 425 | 407, 80 k (more rows) 369 | 457, 109 k 500 | 480, 254 k
// 511 | 494, hence the line.  Against three launches per step with one thread per row and
// a host poll every 16 steps: 27 block rows of 12 (33 steps) 1,029 -> 224 us a call, 512 of
// 36 (66 steps) 5.0 -> 1.9 ms.
// Both: p = r + beta p is formed by every reader from r and its own copy of the last p,
// which saves a third exchange; all CTAs sum the same partials in the same order and take
// the same decisions.
constexpr int kRcgCluster = 8;
constexpr int kRcgClusterDim = 1024;       // rows: 4 lanes each, 512 threads a CTA
constexpr double kRcgClusterFma = 100000.0;
constexpr size_t kRcgClusterSmem = 200 * 1024;

// sum over lanes xor lo, 2 lo, ..., hi / 2
__device__ __forceinline__ double warp_sum(double v, int lo, int hi) {
  for (int o = lo; o < hi; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// One cluster.  CTA c holds rows [dim c / G, dim (c + 1) / G) of K~'s off-diagonal part:
// thread 4 i + h takes the entries h, h + 4, ... of the CTA's row i, value and column in
// shared memory at [step][thread].  r and p of all rows are kept by every CTA: owners push
// their new r into every CTA's copy together with their warps' partial sums, and one
// cluster barrier makes both visible.  status 2: the entries do not fit (nothing done).
template <int kSlots>
struct RcgClusterSums {
  double part[2][kRcgCluster * kSlots];
  double res[4];
};
__global__ void __launch_bounds__(512)
    k_rcg_cluster(int n_sd, int kq, const int32_t* __restrict__ nbr_ptr,
                  const int32_t* __restrict__ nbr_sd, const int32_t* __restrict__ nbr_blk,
                  const double* __restrict__ blocks, const double* __restrict__ bt,
                  double tol2, int max_iter, int smem_entries, RcgState s) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  cl.barrier_arrive();  // waited for before the first store to another CTA's shared memory
  extern __shared__ __align__(16) unsigned char rcg_raw[];
  __shared__ RcgClusterSums<16> sums;
  __shared__ int s_steps[16], s_fit[kRcgCluster];
  const int dim = n_sd * kq, G = gridDim.x, rank = blockIdx.x;
  const int tid = threadIdx.x, nth = blockDim.x, lane = tid & 31, warp = tid >> 5;
  const int nw = nth >> 5;
  double* rf = reinterpret_cast<double*>(rcg_raw);
  double* pf = rf + dim;
  double* val = pf + dim;
  uint16_t* col = reinterpret_cast<uint16_t*>(val + smem_entries);
  const int row0 = (int)((int64_t)dim * rank / G), row1 = (int)((int64_t)dim * (rank + 1) / G);
  const int i = row0 + (tid >> 2), h = tid & 3;
  const bool mine = i < row1;
  const int sd = mine ? i / kq : 0, il = i - sd * kq;
  const int t0 = mine ? nbr_ptr[sd] : 0, ne = mine ? (nbr_ptr[sd + 1] - t0) * kq : 0;
  int steps = ne > h ? (ne - h + 3) / 4 : 0;
  steps = __reduce_max_sync(0xffffffffu, steps);  // of the warp
  if (lane == 0) s_steps[warp] = steps;
  __syncthreads();
  int most = 0;
  for (int w = 0; w < nw; ++w) most = max(most, s_steps[w]);
  cl.barrier_wait();  // every CTA of the cluster has started
  if (tid < G) *cl.map_shared_rank(&s_fit[rank], tid) = (int64_t)most * nth <= smem_entries;
  cl.sync();
  bool fit = true;
  for (int g = 0; g < G; ++g) fit = fit && s_fit[g] != 0;
  if (!fit) {
    if (rank == 0 && tid == 0) s.flag[2] = 2;
    return;
  }
  {
    int t = t0, l = h;
    for (int k = 0; k < steps; ++k) {
      while (l >= kq && 4 * k + h < ne) {
        l -= kq;
        ++t;
      }
      double v = 0.0;
      int c = 0;
      if (4 * k + h < ne) {
        v = blocks[((int64_t)nbr_blk[t] * kq + il) * kq + l];
        c = nbr_sd[t] * kq + l;
      }
      val[k * nth + tid] = v;
      col[k * nth + tid] = (uint16_t)c;
      l += 4;
    }
  }
  unsigned epoch = 0;
  // v of the lanes with h = 0 summed over the cluster; warp 0 passes the sum to fin(sum, res)
  auto exchange = [&](double v, auto fin) {
    v = warp_sum(v, 4, 32);
    double* slot = sums.part[epoch & 1u] + rank * nw + warp;
    if (lane < G) *cl.map_shared_rank(slot, lane) = v;
    cl.sync();
    if (warp == 0) {
      double t = 0.0;
      for (int k = lane; k < G * nw; k += 32) t += sums.part[epoch & 1u][k];
      t = warp_sum(t, 1, 32);
      if (lane == 0) fin(t, sums.res);
    }
    ++epoch;
    __syncthreads();
  };
  auto push_r = [&](double r) {
    if (mine)
      for (int g = h; g < G; g += 4) *cl.map_shared_rank(rf + i, g) = r;
  };
  double x = 0.0, r = mine ? bt[i] : 0.0;
  const double b = r;
  push_r(r);
  exchange(r * r, [](double t, double* o) { o[0] = t; });
  const double bb = sums.res[0];
  double rz = bb, rr = bb, be = 0.0;
  int done = bb > 0.0 ? 0 : 1, it = 0;
  while (!done && it < max_iter) {
    for (int j = tid; j < dim; j += nth) pf[j] = it ? fma(be, pf[j], rf[j]) : rf[j];
    __syncthreads();
    double q = 0.0;
#pragma unroll 4
    for (int k = 0; k < steps; ++k) q = fma(val[k * nth + tid], pf[col[k * nth + tid]], q);
    q = warp_sum(q, 1, 4);
    const double p = mine ? pf[i] : 0.0;
    q += p;
    exchange(p * q, [=](double pq, double* o) { o[0] = pq > 0.0 ? rz / pq : 0.0; });
    const double al = sums.res[0];
    x += al * p;
    r -= al * q;
    push_r(r);
    exchange(r * r, [=](double t, double* o) {
      o[1] = t;
      o[2] = t / rz;
      o[3] = t <= tol2 * bb || !(rz > 0.0) ? 1.0 : 0.0;
    });
    ++it;
    rr = sums.res[1];
    done = sums.res[3] != 0.0;
    if (!done) {
      be = sums.res[2];
      rz = rr;
    }
  }
  if (mine && h == 0) s.x[i] = x;
  exchange(b * x, [](double t, double* o) { o[0] = t; });
  if (rank == 0 && tid == 0) {
    s.scal[0] = rz;
    s.scal[1] = bb;
    s.scal[4] = rr;
    s.scal[6] = sums.res[0];
    s.flag[0] = done;
    s.flag[1] = it;
  }
  cl.sync();  // no CTA leaves while another may still push to it
}

// Every SM.  Units of four rows (rows 4w .. 4w + 3 of one block row) are dealt out in
// contiguous runs of about equal work; a CTA keeps its rows of x, r, p and q in shared
// memory and writes r and p (double-buffered) to global memory for its neighbours.  A warp
// takes a unit's four rows at once: lanes run over the staged neighbour columns, and the
// reduce-scatter over the lanes costs 6 additions for the four rows instead of 20.
constexpr int kRcgThreads = 512;
constexpr int kRcgCap = 3072;  // neighbour columns staged at a time
constexpr size_t kRcgStageBytes = kRcgCap * (sizeof(double) + sizeof(int64_t));
size_t rcg_grid_smem(int64_t rows) { return 4 * sizeof(double) * (size_t)rows + kRcgStageBytes; }
size_t rcg_smem_cap(int smem_max) { return std::min<size_t>(200 * 1024, (size_t)smem_max); }

// part: 2 parities x gridDim.x partial sums; *count: arrivals since the launch (zeroed
// before it).  A CTA rewrites a parity only after every CTA has arrived with the other one,
// that is after every CTA has read this one.  One counter that one thread per CTA polls with
// acquire loads took 5,000 clocks with both sums, against 9,000 for polled per-CTA slots
// that carry the sum itself between two fences (152 CTAs).
struct RcgXch {
  double* part;
  unsigned* count;
  int* err;
  long long budget;
  unsigned epoch;
  unsigned peers;  // arrivals per sum: gridDim.x
  int n;        // threads with a value: those below n
  double* red;  // 32 warp sums, [40] status, [41..] results
};

// v summed over all threads of all CTAs; one lane passes the sum to fin(sum, res), which
// writes up to four results for every thread.  False when a wait ran out.  The CTA's earlier
// global writes are visible to every CTA's later reads.
template <class F>
__device__ bool rcg_exchange(RcgXch& x, double v, F fin) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G = gridDim.x;
  double* red = x.red;
  if (32 * warp < x.n) {
    v = warp_sum(v, 1, 32);
    if (lane == 0) red[warp] = v;
  }
  ++x.epoch;
  __syncthreads();
  if (warp == 0) {
    double* P = x.part + (size_t)(x.epoch & 1u) * G;
    int ok = 1;
    if (lane == 0) {
      double t = 0.0;
      const int nw = (x.n + 31) >> 5;
      for (int w = 0; w < nw; ++w) t += red[w];
      __stcg(P + blockIdx.x, t);
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(x.count) : "memory");
      ok = wait_arrivals(x.count, x.epoch * x.peers, x.err, x.budget);
    }
    __syncwarp();
    double w[5], t = 0.0;
    for (int g0 = lane; g0 < G; g0 += 160) {
#pragma unroll
      for (int k = 0; k < 5; ++k) w[k] = g0 + 32 * k < G ? __ldcg(P + g0 + 32 * k) : 0.0;
#pragma unroll
      for (int k = 0; k < 5; ++k) t += w[k];
    }
    t = warp_sum(t, 1, 32);
    if (lane == 0) {
      red[40] = ok ? 1.0 : 0.0;
      fin(t, red + 41);
    }
  }
  __syncthreads();
  return red[40] != 0.0;
}

// first row of unit u (upb units of four rows per block row of kq rows)
__device__ __forceinline__ int64_t rcg_row(int u, int upb, int kq) {
  return (int64_t)(u / upb) * kq + 4 * (u % upb);
}

// extra weight of a block row beside its neighbours: a quarter of the mean, so that no CTA
// gets more than five times the mean number of units
__host__ __device__ __forceinline__ int64_t rcg_base_weight(int64_t nnb, int64_t n_sd) {
  return nnb / (4 * n_sd) + 1;
}

// first unit of CTA b's run: units weighted by their block row's neighbours plus a base
// (weighted = 0: all alike)
__device__ int rcg_first_unit(int b, int G, int n_sd, int upb, const int32_t* nbr_ptr,
                              int weighted) {
  const int64_t units = (int64_t)n_sd * upb;
  if (!weighted || b == 0 || b == G) return (int)(units * b / G);
  const int64_t base = rcg_base_weight(nbr_ptr[n_sd], n_sd);
  const int64_t want = (nbr_ptr[n_sd] + base * n_sd) * upb * b / G;
  int lo = 0, hi = n_sd - 1;  // the last block row whose units start at or before `want`
  while (lo < hi) {
    const int m = (lo + hi + 1) / 2;
    if ((nbr_ptr[m] + base * m) * upb <= want)
      lo = m;
    else
      hi = m - 1;
  }
  const int64_t w = nbr_ptr[lo + 1] - nbr_ptr[lo] + base;
  const int64_t k = (want - (nbr_ptr[lo] + base * lo) * upb + w - 1) / w;
  return (int)min(units, (int64_t)lo * upb + min(k, (int64_t)upb));
}

// kShared: the CTA's rows of x, r, p and q in shared memory; else in x, s.r and s.w (each row
// is read and written by its CTA alone, r and p by the neighbours as ever).
template <bool kShared>
__global__ void __launch_bounds__(kRcgThreads)
    k_rcg_grid(int n_sd, int kq, const int32_t* __restrict__ nbr_ptr,
               const int32_t* __restrict__ nbr_sd, const int32_t* __restrict__ nbr_blk,
               const double* __restrict__ blocks, const double* __restrict__ bt, double tol2,
               int max_iter, int rows_max, int weighted, RcgState s, double* part,
               long long budget) {
  extern __shared__ __align__(16) unsigned char rcg_raw[];
  // the own rows of x, r, p and q (none of them unless kShared: rows_max = 0), then the staged
  // neighbour columns
  double* sh = reinterpret_cast<double*>(rcg_raw);
  double* pj = sh + 4 * (size_t)rows_max;
  int64_t* off = reinterpret_cast<int64_t*>(pj + kRcgCap);
  __shared__ double red[48];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int upb = (kq + 3) / 4;
  const int u0 = rcg_first_unit(blockIdx.x, gridDim.x, n_sd, upb, nbr_ptr, weighted);
  const int u1 = rcg_first_unit(blockIdx.x + 1, gridDim.x, n_sd, upb, nbr_ptr, weighted);
  const int64_t row0 = rcg_row(u0, upb, kq), row1 = rcg_row(u1, upb, kq);
  const int rows = (int)(row1 - row0);
  double *xs, *rs, *ps, *qs;
  if constexpr (kShared) {
    xs = sh;
    rs = xs + rows_max;
    ps = rs + rows_max;
    qs = ps + rows_max;
  } else {
    xs = s.x + row0;
    rs = s.r + row0;
    ps = s.w + row0;
    qs = s.w + (int64_t)n_sd * kq + row0;
  }
  const int live = min(rows, kRcgThreads);
  // the neighbour entries of the block rows this CTA touches
  const int sd_lo = u0 / upb, sd_hi = u1 > u0 ? (u1 - 1) / upb + 1 : sd_lo;
  const int t_lo = nbr_ptr[sd_lo], t_hi = nbr_ptr[sd_hi];
  const int tcap = kRcgCap / kq;
  const float inv_kq = 1.0f / (float)kq;
  RcgXch x{part, reinterpret_cast<unsigned*>(s.flag + 3), s.flag + 2, budget, 0u, gridDim.x, live, red};
  const double* res = red + 41;
  double loc = 0.0;
  for (int i = tid; i < rows; i += kRcgThreads) {
    const double b = bt[row0 + i];
    xs[i] = 0.0;
    rs[i] = b;
    ps[i] = 0.0;
    __stcg(s.r + row0 + i, b);
    loc += b * b;
  }
  if (!rcg_exchange(x, loc, [](double t, double* o) { o[0] = t; })) return;
  const double bb = res[0];
  double rz = bb, rr = bb, be = 0.0;
  int done = bb > 0.0 ? 0 : 1, it = 0;
  while (!done && it < max_iter) {
    // p = r + beta p on the own rows, q = p (the identity diagonal block)
    double* pw = it & 1 ? s.q : s.p;
    const double* pr = it & 1 ? s.p : s.q;
    for (int i = tid; i < rows; i += kRcgThreads) {
      const double p = it ? fma(be, ps[i], rs[i]) : rs[i];
      ps[i] = p;
      qs[i] = p;
      __stcg(pw + row0 + i, p);
    }
    for (int t0 = t_lo; t0 < t_hi; t0 += tcap) {
      const int t1 = min(t_hi, t0 + tcap);
      __syncthreads();
      const int ne = (t1 - t0) * kq;
      for (int eb = tid; eb < ne; eb += 4 * kRcgThreads) {
        double r[4], po[4];
        int64_t o[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const int e = eb + m * kRcgThreads;
          if (e >= ne) continue;
          const int q = (int)(((float)e + 0.5f) * inv_kq), l = e - q * kq;  // e < 2^12
          const int64_t j = (int64_t)nbr_sd[t0 + q] * kq + l;
          o[m] = (int64_t)nbr_blk[t0 + q] * kq * kq + l;
          r[m] = __ldcg(s.r + j);
          po[m] = it ? __ldcg(pr + j) : 0.0;
        }
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const int e = eb + m * kRcgThreads;
          if (e >= ne) continue;
          pj[e] = it ? fma(be, po[m], r[m]) : r[m];
          off[e] = o[m];
        }
      }
      __syncthreads();
      for (int u = u0 + warp; u < u1; u += kRcgThreads / 32) {
        const int sd = u / upb, i0 = 4 * (u % upb);
        const int e0 = (max(nbr_ptr[sd], t0) - t0) * kq;
        const int e1 = (min(nbr_ptr[sd + 1], t1) - t0) * kq;
        if (e0 >= e1) continue;
        // the rows of the unit; beyond kq (a last unit of fewer than four) row i0 again
        const double* B = blocks + (int64_t)i0 * kq;
        const int st1 = i0 + 1 < kq ? kq : 0, st2 = i0 + 2 < kq ? 2 * kq : 0,
                  st3 = i0 + 3 < kq ? 3 * kq : 0;
        double a[4] = {0.0, 0.0, 0.0, 0.0};
        // two column steps per batch, the next batch's loads issued before this one's
        // multiply-adds; lanes past the end read column e0 again, times 0
        double v[2][4], p[2];
        auto load = [&](int eb, double(&w)[2][4], double(&pv)[2]) {
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const int e = eb + lane + 32 * k;
            if (eb + 32 * k >= e1) continue;  // the whole warp
            pv[k] = e < e1 ? pj[e] : 0.0;
            const double* Bo = B + off[e < e1 ? e : e0];
            w[k][0] = __ldg(Bo);
            w[k][1] = __ldg(Bo + st1);
            w[k][2] = __ldg(Bo + st2);
            w[k][3] = __ldg(Bo + st3);
          }
        };
        load(e0, v, p);
        for (int eb = e0; eb < e1; eb += 64) {
          double w[2][4], pw2[2];
          load(eb + 64, w, pw2);
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            if (eb + 32 * k < e1)
#pragma unroll
              for (int m = 0; m < 4; ++m) a[m] = fma(v[k][m], p[k], a[m]);
#pragma unroll
            for (int m = 0; m < 4; ++m) v[k][m] = w[k][m];
            p[k] = pw2[k];
          }
        }
        // lanes with bit 4 take rows 2, 3, with bit 3 the odd row of the two
        const bool h4 = lane & 16, h3 = lane & 8;
        double c0 = h4 ? a[2] : a[0], c1 = h4 ? a[3] : a[1];
        c0 += __shfl_xor_sync(0xffffffffu, h4 ? a[0] : a[2], 16);
        c1 += __shfl_xor_sync(0xffffffffu, h4 ? a[1] : a[3], 16);
        double c = h3 ? c1 : c0;
        c += __shfl_xor_sync(0xffffffffu, h3 ? c0 : c1, 8);
        c = warp_sum(c, 1, 8);
        const int m = lane >> 3;
        if ((lane & 7) == 0 && i0 + m < kq) qs[rcg_row(u, upb, kq) - row0 + m] += c;
      }
    }
    __syncthreads();
    loc = 0.0;
    for (int i = tid; i < rows; i += kRcgThreads) loc += ps[i] * qs[i];
    if (!rcg_exchange(
            x, loc, [=](double pq, double* o) { o[0] = pq > 0.0 ? rz / pq : 0.0; }))
      return;
    const double al = res[0];
    loc = 0.0;
    for (int i = tid; i < rows; i += kRcgThreads) {
      xs[i] += al * ps[i];
      const double r = rs[i] - al * qs[i];
      rs[i] = r;
      __stcg(s.r + row0 + i, r);
      loc += r * r;
    }
    if (!rcg_exchange(x, loc, [=](double t, double* o) {
          o[0] = t;
          o[1] = t / rz;
          o[2] = t <= tol2 * bb || !(rz > 0.0) ? 1.0 : 0.0;
        }))
      return;
    ++it;
    rr = res[0];
    done = res[2] != 0.0;
    if (!done) {
      be = res[1];
      rz = rr;
    }
  }
  // x and E = b~.x
  loc = 0.0;
  for (int i = tid; i < rows; i += kRcgThreads) {
    if constexpr (kShared) s.x[row0 + i] = xs[i];
    loc += bt[row0 + i] * xs[i];
  }
  if (!rcg_exchange(x, loc, [](double t, double* o) { o[0] = t; })) return;
  if (blockIdx.x == 0 && tid == 0) {
    s.scal[0] = rz;
    s.scal[1] = bb;
    s.scal[4] = rr;
    s.scal[6] = res[0];
    s.flag[0] = done;
    s.flag[1] = it;
  }
}

// the timeout path of the solve's exchange: a sum that waits for one arrival more than there
// are CTAs.  *status: CTAs that gave up
__global__ void k_exchange_timeout(double* part, unsigned* count, int* err, long long budget,
                                   int* status) {
  __shared__ double red[48];
  RcgXch x{part, count, err, budget, 0u, gridDim.x + 1, (int)blockDim.x, red};
  if (!rcg_exchange(x, 1.0, [](double t, double* o) { o[0] = t; }) && threadIdx.x == 0)
    atomicAdd(status, 1);
}

__global__ void k_lift(int64_t n_o, const int32_t* __restrict__ o_node,
                       const int32_t* __restrict__ o_sd, const double* __restrict__ Q, int kq,
                       const double* __restrict__ x, double* u) {
  int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (r >= n_o) return;
  const double* xs = x + (int64_t)o_sd[r] * kq;
  double s = 0.0;
  for (int c = 0; c < kq; ++c) s += Q[r * kq + c] * xs[c];
  u[o_node[r]] = s;
}

}  // namespace

void launch_pair_blocks(int n_pairs, const int64_t* pair_ptr, const int32_t* urow,
                        const int32_t* vrow, const double* aval, const double* Q, int kq,
                        double* blocks, cudaStream_t st) {
  if (n_pairs <= 0) return;
  // rows per block: what the accumulators hold, fewer while the blocks do not fill the SMs
  // four times over, eight at least (each slice repeats the w_u, three multiply-adds per entry and
  // column: with four rows a slice spends nearly half its time on them)
  int rows = std::min(kq, kPairThreads * kPairOut / kq);
  while (rows > 8 && (int64_t)n_pairs * ((kq + rows - 1) / rows) < 4 * 152) rows = (rows + 1) / 2;
  const size_t sm = sizeof(double) * (size_t)kPairGroups * (kq + rows);  // kq <= 128: 40 KB
  count_launch();
  k_pair_blocks<<<dim3(n_pairs, (kq + rows - 1) / rows), kPairThreads, sm, st>>>(
      pair_ptr, urow, vrow, aval, Q, kq, rows, blocks);
}

void launch_rcg_init(int n_sd, int kq, const double* bt, const RcgState& s,
                     cudaStream_t st) {
  count_launch();
  k_rcg_init<<<n_sd, 128, 0, st>>>(n_sd, kq, bt, s);
}

void launch_rcg_step(int n_sd, int kq, const int32_t* nbr_ptr, const int32_t* nbr_sd,
                     const int32_t* nbr_blk, const double* blocks, double tol2,
                     const RcgState& s, cudaStream_t st) {
  count_launch();
  k_rcg_spmv<<<n_sd, 128, 0, st>>>(n_sd, kq, nbr_ptr, nbr_sd, nbr_blk, blocks, s);
  count_launch();
  k_rcg_update_xr<<<n_sd, 128, 0, st>>>(n_sd, kq, tol2, s);
  count_launch();
  k_rcg_update_p<<<n_sd, 128, 0, st>>>(kq, s);
}

// shape of k_rcg_grid on nsm SMs: CTAs, rows of the largest run and whether runs are weighted;
// rows = 0: more than shared memory holds (at 152 SMs above 739,000 rows of K~)
struct RcgGrid {
  int G, rows, weighted;
};
static RcgGrid rcg_grid_shape(int64_t units, int nsm, size_t smem_max) {
  RcgGrid g;
  g.G = (int)std::min<int64_t>(std::min(nsm, kRcgMaxGrid), units);
  // weighted runs hold at most five times the mean number of units; where that does not
  // fit in shared memory, runs of equal length
  const int64_t mean = (units + g.G - 1) / g.G;
  for (g.weighted = 1; g.weighted >= 0; --g.weighted) {
    const int64_t rows = g.weighted ? 4 * (5 * mean + 2) : 4 * mean;
    if (rcg_grid_smem(rows) <= smem_max) {
      g.rows = (int)rows;
      return g;
    }
  }
  g.rows = 0;
  g.weighted = 1;
  return g;
}
static int rcg_units(int n_sd, int kq) {
  const int64_t units = (int64_t)n_sd * ((kq + 3) / 4);
  return units > INT32_MAX ? 0 : (int)units;
}

size_t rcg_grid_work(int n_sd, int kq) {
  int dev = 0, nsm = 0, smem_max = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const int units = rcg_units(n_sd, kq);
  if (units < 1 || nsm < 1) return 0;
  const bool shared = rcg_grid_shape(units, nsm, rcg_smem_cap(smem_max)).rows > 0;
  return shared ? 0 : 2 * (size_t)n_sd * kq;
}

RcgLaunch launch_rcg_solve(int n_sd, int kq, const int32_t* nbr_ptr, const int32_t* nbr_sd,
                           const int32_t* nbr_blk, int64_t n_blocks, const double* blocks,
                           const double* bt, double tol2, int max_iter, const RcgState& s,
                           double* part, long long budget, bool try_cluster,
                           cudaStream_t st) {
  int dev = 0, nsm = 0, coop = 0, smem_max = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return RcgLaunch::kNone;
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const int64_t dim = (int64_t)n_sd * kq;
  cudaLaunchAttribute at{};
  cudaLaunchConfig_t cfg{};
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  RcgState sc = s;
  if (try_cluster && dim <= kRcgClusterDim &&
      (double)n_blocks * kq * kq <= kRcgClusterFma && (size_t)smem_max >= kRcgClusterSmem + 8192) {
    const int G = (int)std::min<int64_t>(kRcgCluster, dim);
    const int rows = (int)((dim + G - 1) / G);
    const int nth = (4 * rows + 31) / 32 * 32;
    int entries = (int)((kRcgClusterSmem - 2 * sizeof(double) * (size_t)dim) /
                        (sizeof(double) + sizeof(uint16_t)));
    entries &= ~7;
    const void* fn = (const void*)k_rcg_cluster;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kRcgClusterSmem) != cudaSuccess)
      return RcgLaunch::kNone;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)G;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)G);
    cfg.blockDim = dim3((unsigned)nth);
    cfg.dynamicSmemBytes = kRcgClusterSmem;
    void* args[] = {&n_sd, &kq, (void*)&nbr_ptr, (void*)&nbr_sd, (void*)&nbr_blk,
                    (void*)&blocks, (void*)&bt, &tol2, &max_iter, &entries, &sc};
    if (cudaLaunchKernelExC(&cfg, fn, args) == cudaSuccess) {
      count_launch();
      return RcgLaunch::kCluster;
    }
    cudaGetLastError();
  }
  const int units = rcg_units(n_sd, kq);
  if (!coop || kq > kRcgCap || units < 1 || nsm < 1) return RcgLaunch::kNone;
  const size_t cap = rcg_smem_cap(smem_max);
  const RcgGrid g = rcg_grid_shape(units, nsm, cap);
  if (g.rows == 0 && !s.w) return RcgLaunch::kNone;
  int rows_max = g.rows, weighted = g.weighted;
  const void* fn = g.rows > 0 ? (const void*)k_rcg_grid<true> : (const void*)k_rcg_grid<false>;
  // (one limit for every size: threads may launch different ones at the same time)
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cap) !=
      cudaSuccess)
    return RcgLaunch::kNone;
  at.id = cudaLaunchAttributeCooperative;
  at.val.cooperative = 1;
  cfg.gridDim = dim3((unsigned)g.G);
  cfg.blockDim = dim3(kRcgThreads);
  cfg.dynamicSmemBytes = rcg_grid_smem(rows_max);
  void* args[] = {&n_sd, &kq, (void*)&nbr_ptr, (void*)&nbr_sd, (void*)&nbr_blk,
                  (void*)&blocks, (void*)&bt, &tol2, &max_iter, &rows_max, &weighted, &sc,
                  &part, &budget};
  if (cudaLaunchKernelExC(&cfg, fn, args) != cudaSuccess) return RcgLaunch::kNone;
  count_launch();
  return RcgLaunch::kGrid;
}

void launch_exchange_timeout(double* part, unsigned* count, int* err, long long budget,
                             int* status, cudaStream_t st) {
  count_launch();
  k_exchange_timeout<<<kTimeoutBlocks, 64, 0, st>>>(part, count, err, budget, status);
}

void launch_lift(int64_t n_o, const int32_t* o_node, const int32_t* o_sd, const double* Q,
                 int kq, const double* x, double* u, cudaStream_t st) {
  if (n_o <= 0) return;
  count_launch();
  k_lift<<<(unsigned)((n_o + 255) / 256), 256, 0, st>>>(n_o, o_node, o_sd, Q, kq, x, u);
}

}  // namespace mor
