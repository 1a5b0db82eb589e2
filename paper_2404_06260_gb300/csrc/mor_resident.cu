// The local CG of small subdomains with everything on chip: up to a replacement interval
// of steps in one launch.
//
// A cluster of S CTAs owns one 16-byte column pack of one subdomain.  CTA c holds the rows
// [c R, (c + 1) R): their matrix slots (value and 16-bit local column) in shared memory,
// their x and r in registers; every CTA has the whole p of the pack in shared memory (the
// owners push their rows into all copies), so the product's gathers are local, and the
// whole aggregate inverse E^{-1}, so every CTA forms the coarse correction y_c = E^{-1} r_c
// itself from r_c parts that the owners push.  The recursion, its tests and their
// precisions are those of the kernels in mor_sparse.cu: sums run in the working precision
// over at most 128 rows (a warp's rows), in binary64 beyond.  A step has three cluster
// barriers: after p.q, after the restriction with r.r and r.D^{-1}r, after p with p.r.
//
// What bounds it: the chain of a step (six short phases between barriers), no longer
// five launches of latency-bound kernels with their tile sums.  16^3 workload: 40 us a step
// there, 7 here with the launch (binary64: 46 and 20, bound by binary64 issue).  Larger
// subdomains do not fit; they have work enough to hide the launches.
#include <cooperative_groups.h>

#include <algorithm>
#include <utility>

#include "mor_kernels.h"

namespace mor {
namespace {

constexpr int kResCluster = 8;    // largest cluster (portable size)
constexpr int kResRows = 4;       // rows per thread
constexpr int kResAggMax = 128;   // aggregates: E^{-1} whole in shared memory
template <typename T>
struct ResThreads {
  static constexpr int n = sizeof(T) == 4 ? 512 : 320;  // binary64 sums cost per warp
  // dynamic shared memory: what 227 KB leave beside the slots of the sums (17 and 5 KB)
  static constexpr size_t smem = sizeof(T) == 4 ? 209 * 1024 : 220 * 1024;
};

template <typename T>
struct alignas(16) RPack {
  static constexpr int N = 16 / sizeof(T);
  T v[N];
};

// M values per lane (M a power of two), summed over the warp: lane l returns the sum of value
// l / (32 / M).  Halving exchanges: M - 1 + log2(32 / M) additions instead of 5 M.
template <int M, typename T>
__device__ __forceinline__ T warp_sums(T (&v)[M]) {
  const int lane = threadIdx.x & 31;
  int o = 16;
#pragma unroll
  for (int h = M / 2; h >= 1; h >>= 1, o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int k = 0; k < h; ++k) {
      const T keep = up ? v[k + h] : v[k], send = up ? v[k] : v[k + h];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  T t = v[0];
  for (; o >= 1; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}

__host__ __device__ __forceinline__ size_t up16(size_t x) { return (x + 15) & ~(size_t)15; }

// shared memory of a CTA: p of n rows; r of R rows; W x R slots; E^{-1}; r_c parts, r_c, y_c;
// first own row of each own aggregate
template <typename T>
__host__ __device__ __forceinline__ size_t res_smem(int n, int R, int W, int nc, int S) {
  return up16(16 * (size_t)n) + up16(16 * (size_t)R) + up16((size_t)W * R * sizeof(T)) +
         up16((size_t)W * R * sizeof(uint16_t)) + up16((size_t)nc * nc * sizeof(T)) +
         16 * (size_t)nc * (S + 2) + up16(sizeof(int) * (size_t)(nc + 2));
}

template <typename T>
__global__ void __launch_bounds__(ResThreads<T>::n, 1)
    k_cg_resident(DTiles tl, EllView<T> A, T* __restrict__ xg, const T* __restrict__ rg,
                  T* __restrict__ pg, const T* __restrict__ dinv, int kp, double tol2, int steps,
                  CgState s, Coarse<T> co, int* steps_run) {
  namespace cg = cooperative_groups;
  constexpr int N = RPack<T>::N, KR = kResRows, NT = ResThreads<T>::n, NW = NT / 32;
  using P = RPack<T>;
  cg::cluster_group cl = cg::this_cluster();
  extern __shared__ __align__(16) unsigned char res_raw[];
  // per warp and CTA: p.q (0), r.r (1), r.D^{-1}r (2), p.r (3) of every column
  __shared__ double slot[4][kResCluster][NW][N];
  __shared__ double res[3][N];                  // sums for the step's scalars
  __shared__ double c_rz[N], c_bb[N], c_pr[N];  // column state
  __shared__ T c_al[N], c_be[N];
  __shared__ int c_done[N], s_open;
  const int S = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int sd = blockIdx.y, pk = blockIdx.x / S;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int c0 = pk * N;
  bool any = false;
#pragma unroll
  for (int e = 0; e < N; ++e) any = !s.done[sd * kp + c0 + e] || any;
  if (!any || tl.lo[sd] >= tl.hi[sd]) return;  // the whole cluster
  const int first = tl.r0[tl.lo[sd]];
  const int n = tl.r1[tl.hi[sd] - 1] - first;
  const int nc = co.tbase ? co.nca[sd] : 0;
  const int W = A.W;
  const int R = (n + S - 1) / S;
  const int own0 = min(n, rank * R), own = min(n, own0 + R) - own0;
  unsigned char* at = res_raw;
  auto take = [&](size_t b) {
    unsigned char* q = at;
    at += up16(b);
    return q;
  };
  P* pf = reinterpret_cast<P*>(take(16 * (size_t)n));
  P* rb = reinterpret_cast<P*>(take(16 * (size_t)R));
  T* val = reinterpret_cast<T*>(take((size_t)W * R * sizeof(T)));
  uint16_t* col = reinterpret_cast<uint16_t*>(take((size_t)W * R * sizeof(uint16_t)));
  T* E = reinterpret_cast<T*>(take((size_t)nc * nc * sizeof(T)));
  P* rcp = reinterpret_cast<P*>(take(16 * (size_t)nc * S));
  P* rc = reinterpret_cast<P*>(take(16 * (size_t)nc));
  P* yc = reinterpret_cast<P*>(take(16 * (size_t)nc));
  int* run = reinterpret_cast<int*>(take(sizeof(int) * (size_t)(nc + 2)));
  // ---- load ----
  P x[KR], r[KR];
  T d[KR];
  int w[KR], ag[KR];
#pragma unroll
  for (int k = 0; k < KR; ++k) {
    const int i = tid + k * NT;
    w[k] = 0;
    ag[k] = 0;
    d[k] = T(0);
#pragma unroll
    for (int e = 0; e < N; ++e) x[k].v[e] = r[k].v[e] = T(0);
    if (i >= own) continue;
    const int64_t row = first + own0 + i;
    x[k] = *reinterpret_cast<const P*>(xg + row * kp + c0);
    r[k] = *reinterpret_cast<const P*>(rg + row * kp + c0);
    d[k] = dinv[row];
    w[k] = A.width[row >> 5];
    if (nc) ag[k] = co.aloc[row];
    for (int j = 0; j < w[k]; ++j) {
      const int64_t a = ell_at(row, j, W);
      const int c = A.col[a];
      // padding: the row's own p times zero
      col[j * R + i] = (uint16_t)(c < 0 ? own0 + i : c - first);
      val[j * R + i] = c < 0 ? T(0) : A.val[a];
    }
  }
  for (int i = tid; i < n; i += NT)
    pf[i] = *reinterpret_cast<const P*>(pg + (int64_t)(first + i) * kp + c0);
  for (int i = tid; i < nc * nc; i += NT) E[i] = co.einv[co.eoff[sd] + i];
  for (int i = tid; i < nc * S; i += NT)
#pragma unroll
    for (int e = 0; e < N; ++e) rcp[i].v[e] = T(0);
  const int a_lo = nc && own > 0 ? co.aloc[first + own0] : 0;
  const int a_n = nc && own > 0 ? co.aloc[first + own0 + own - 1] - a_lo + 1 : 0;
  for (int i = tid; i < own; i += NT)
    if (nc) {
      const int a = co.aloc[first + own0 + i];
      if (i == 0 || a != co.aloc[first + own0 + i - 1]) run[a - a_lo] = i;
    }
  if (tid == 0) run[a_n] = own;
  if (tid < N) {
    const int i = sd * kp + c0 + tid;
    c_rz[tid] = s.rz[i];
    c_bb[tid] = s.bb[i];
    c_pr[tid] = s.pr[i];
    c_done[tid] = s.done[i];
  }
  // a warp's sums of N values into every CTA's slots
  auto push = [&](int which, T (&v)[N]) {
    const double t = (double)warp_sums<N>(v);
#pragma unroll
    for (int e = 0; e < N; ++e) {
      const double te = __shfl_sync(0xffffffffu, t, e * (32 / N));
      if (lane < S) *cl.map_shared_rank(&slot[which][rank][warp][e], lane) = te;
    }
  };
  // quantity `which` of column e added over CTAs and warps by 16 lanes of this thread's half
  // warp (every lane of a full warp must come)
  auto total = [&](int which, int e, int l) {
    double t = 0.0;
    for (int g = 0; g < S; ++g)
      for (int u = l; u < NW; u += 16) t += slot[which][g][u][e];
    for (int o = 8; o >= 1; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
  };
  cl.sync();
  int it = 0;
  for (; it < steps; ++it) {
    // q = A p and p.q
    P q[KR];
    T pq[N];
#pragma unroll
    for (int e = 0; e < N; ++e) pq[e] = T(0);
#pragma unroll
    for (int k = 0; k < KR; ++k) {
      const int i = tid + k * NT;
#pragma unroll
      for (int e = 0; e < N; ++e) q[k].v[e] = T(0);
      if (i >= own) continue;
#pragma unroll 4
      for (int j = 0; j < w[k]; ++j) {
        const T a = val[j * R + i];
        const P g = pf[col[j * R + i]];
#pragma unroll
        for (int e = 0; e < N; ++e) q[k].v[e] += a * g.v[e];
      }
      const P p = pf[own0 + i];
#pragma unroll
      for (int e = 0; e < N; ++e) pq[e] += p.v[e] * q[k].v[e];
    }
    push(0, pq);
    cl.sync();
    if (tid < 16 * N) {
      const int e = tid / 16;
      const double t = total(0, e, tid & 15);
      double pr = c_pr[e];
      if (it > 0) pr = total(3, e, tid & 15);
      if ((tid & 15) == 0) {
        double a = 0.0;
        if (!c_done[e]) {
          if (t > 0.0)
            a = pr / t;
          else
            c_done[e] = 1;  // breakdown, as in k_cg_spmm_pq
        }
        c_al[e] = (T)a;
      }
    }
    __syncthreads();
    // x += alpha p, r -= alpha q, r.r, r.D^{-1}r
    T sm2[2][N];
#pragma unroll
    for (int e = 0; e < N; ++e) sm2[0][e] = sm2[1][e] = T(0);
#pragma unroll
    for (int k = 0; k < KR; ++k) {
      const int i = tid + k * NT;
      if (i >= own) continue;
      const P p = pf[own0 + i];
#pragma unroll
      for (int e = 0; e < N; ++e) {
        const T a = c_al[e];
        x[k].v[e] += a * p.v[e];
        r[k].v[e] -= a * q[k].v[e];
        sm2[0][e] += r[k].v[e] * r[k].v[e];
        sm2[1][e] += r[k].v[e] * (d[k] * r[k].v[e]);
      }
      rb[i] = r[k];
    }
    push(1, sm2[0]);
    push(2, sm2[1]);
    if (nc) {
      __syncthreads();
      // r_c parts of the own aggregates: 16 lanes each, rows in stride order
      for (int a0 = 0; a0 < a_n; a0 += NT / 16) {
        const int a = a0 + tid / 16, l = tid & 15;
        P acc;
#pragma unroll
        for (int e = 0; e < N; ++e) acc.v[e] = T(0);
        if (a < a_n)
          for (int i = run[a] + l; i < run[a + 1]; i += 16) {
            const P v = rb[i];
#pragma unroll
            for (int e = 0; e < N; ++e) acc.v[e] += v.v[e];
          }
#pragma unroll
        for (int e = 0; e < N; ++e)
          for (int o = 8; o >= 1; o >>= 1)
            acc.v[e] += __shfl_xor_sync(0xffffffffu, acc.v[e], o);
        if (a < a_n && l < S) *cl.map_shared_rank(rcp + rank * nc + a_lo + a, l) = acc;
      }
    }
    cl.sync();
    if (nc) {
      for (int i = tid; i < nc; i += NT) {
        P t = rcp[i];
        for (int g = 1; g < S; ++g)
#pragma unroll
          for (int e = 0; e < N; ++e) t.v[e] += rcp[g * nc + i].v[e];
        rc[i] = t;
      }
      __syncthreads();
      // y_c = E^{-1} r_c, eight lanes per aggregate
      for (int a0 = 0; a0 < nc; a0 += NT / 8) {
        const int a = a0 + tid / 8, l = tid & 7;
        P acc;
#pragma unroll
        for (int e = 0; e < N; ++e) acc.v[e] = T(0);
        if (a < nc)
          for (int b = l; b < nc; b += 8) {
            const T ev = E[a * nc + b];
            const P v = rc[b];
#pragma unroll
            for (int e = 0; e < N; ++e) acc.v[e] += ev * v.v[e];
          }
#pragma unroll
        for (int e = 0; e < N; ++e)
          for (int o = 4; o >= 1; o >>= 1)
            acc.v[e] += __shfl_xor_sync(0xffffffffu, acc.v[e], o);
        if (a < nc && l == 0) yc[a] = acc;
      }
      __syncthreads();
    }
    // r.r, the fine and the coarse part of r.M^{-1}r: 16 lanes per quantity and column
    if (tid < 16 * 3 * N) {
      const int qn = tid / (16 * N), e = tid / 16 % N, l = tid & 15;
      double t = 0.0;
      if (qn < 2) {
        for (int g = 0; g < S; ++g)
          for (int u = l; u < NW; u += 16) t += slot[1 + qn][g][u][e];
      } else {
        for (int a = l; a < nc; a += 16) t += (double)yc[a].v[e] * (double)rc[a].v[e];
      }
      for (int o = 8; o >= 1; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if (l == 0) res[qn][e] = t;
    }
    __syncthreads();
    if (warp == 0) {
      int open = 0;
      if (lane < N) {
        const double rzn = res[1][lane] + res[2][lane];
        double be = 0.0;
        if (!c_done[lane]) {
          if (res[0][lane] <= tol2 * c_bb[lane] || !(c_rz[lane] > 0.0)) {
            c_done[lane] = 1;
          } else {
            be = rzn / c_rz[lane];
            c_rz[lane] = rzn;
          }
        }
        c_be[lane] = (T)be;
        open = !c_done[lane];
      }
      open = __any_sync(0xffffffffu, open);
      if (lane == 0) s_open = open;
    }
    __syncthreads();
    if (!s_open) {  // every CTA of the cluster takes the same decision
      ++it;
      break;
    }
    // p = D^{-1} r + Z y_c + beta p (p is not read where beta = 0), p.r
    T prs[N];
#pragma unroll
    for (int e = 0; e < N; ++e) prs[e] = T(0);
#pragma unroll
    for (int k = 0; k < KR; ++k) {
      const int i = tid + k * NT;
      if (i >= own) continue;
      P p = pf[own0 + i];
#pragma unroll
      for (int e = 0; e < N; ++e) {
        T z = d[k] * r[k].v[e];
        if (nc) z += yc[ag[k]].v[e];
        if (c_be[e] != T(0)) z += c_be[e] * p.v[e];
        p.v[e] = z;
        prs[e] += z * r[k].v[e];
      }
      for (int g = 0; g < S; ++g) *cl.map_shared_rank(pf + own0 + i, g) = p;
    }
    push(3, prs);
    cl.sync();
  }
  // ---- store: x, p, the residual norm and the flags (r and rz are formed anew at the
  // replacement) ----
#pragma unroll
  for (int k = 0; k < KR; ++k) {
    const int i = tid + k * NT;
    if (i >= own) continue;
    const int64_t o = (int64_t)(first + own0 + i) * kp + c0;
    *reinterpret_cast<P*>(xg + o) = x[k];
    *reinterpret_cast<P*>(pg + o) = pf[own0 + i];
  }
  if (rank == 0 && tid < N) {
    const int i = sd * kp + c0 + tid;
    s.rr[i] = res[0][tid];
    s.done[i] = c_done[tid];
    if (!c_done[tid]) atomicAdd(s.active_next + sd, 1);
    if (tid == 0) {
      atomicMax(s.iters + sd, it);
      atomicMax(steps_run, it);
    }
  }
  cl.sync();  // no CTA leaves while another may still push to it
}

}  // namespace

template <typename T>
ResidentPlan resident_plan(int n_sd, int n_max, int W, int nc_max, int kp) {
  ResidentPlan rp;
  if (n_sd <= 0 || n_max <= 0 || n_max > 65535 || nc_max > kResAggMax) return rp;
  constexpr int NT = ResThreads<T>::n;
  const int tasks = n_sd * (kp / RPack<T>::N);
  int S = 1;
  auto fits = [&](int S_) {
    const int R = (n_max + S_ - 1) / S_;
    return R <= kResRows * NT && res_smem<T>(n_max, R, W, nc_max, S_) <= ResThreads<T>::smem;
  };
  while (S <= kResCluster && !fits(S)) S *= 2;
  if (S > kResCluster) return rp;
  // more CTAs per subdomain while the chip is not full and a CTA keeps a warp's worth of rows
  // per warp
  while (2 * S <= kResCluster && 2 * S * tasks <= 152 && n_max / (2 * S) >= NT / 2) S *= 2;
  // Clusters beyond what the chip holds at once run in waves, each with its own chain of
  // steps, while a streaming step has one fixed cost for all subdomains.  Builds, streaming
  // against on chip: binary64 at S = 8 and 5.7 waves 35.4 and 29.2 ms, 11.4 waves 42.1 and
  // 47.6; S = 4, 6.7 waves 47.6 and 43.0, 13.5 waves 61.5 and 70.5; S = 2, 13.5 waves 39.9
  // and 38.6, 22 waves 61.9 and 67.9.  Binary32 at S = 8 and 5.7 waves 21.5 and 16.8 ms, 11.4
  // waves 26.6 and 28.2; S = 4, 13.5 waves 35.2 and 29.1, 22 waves 51.5 and 51.6; S = 2, 23
  // waves 57.8 and 45.9, 37 waves 89.3 and 86.7.  One CTA each (398 and 724 rows): binary64
  // 11.4 waves 35.7 and 34.2, 13.2 waves 37.4 and 37.9, 18 waves 29.0 and 34.2, 27 waves 39.1
  // and 51.1; binary32 10.7 waves 28.3 and 25.2, 13.5 waves 24.0 and 21.3, 18 waves 26.3
  // and 27.1, 29 waves 44.7 and 55.8, 44 waves 61.5 and 81.6
  const double waves = (double)S * tasks / 152.0;
  const double most = sizeof(T) == 8 ? (S == 1 ? 12.0 : S == 2 ? 15.0 : S == 4 ? 7.5 : 6.0)
                                     : (S == 1 ? 16.0 : 48.0 / S);
  if (waves > most) return rp;
  rp.S = S;
  rp.smem = res_smem<T>(n_max, (n_max + S - 1) / S, W, nc_max, S);
  return rp;
}

template <typename T>
bool launch_cg_resident(const ResidentPlan& rp, const DTiles& tiles, const EllView<T>& A, T* x,
                        const T* r, T* p, const T* dinv, int kp, double tol2, int steps,
                        CgState& s, const Coarse<T>& co, int* steps_run, cudaStream_t st) {
  cudaMemsetAsync(s.active_next, 0, sizeof(int) * (size_t)tiles.n_sd, st);
  // (one limit for every shape: threads may launch different ones at the same time)
  cudaError_t e = cudaFuncSetAttribute((const void*)k_cg_resident<T>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)ResThreads<T>::smem);
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)rp.S;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(kp / RPack<T>::N * rp.S), (unsigned)tiles.n_sd);
  cfg.blockDim = dim3(ResThreads<T>::n);
  cfg.dynamicSmemBytes = rp.smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  if (e == cudaSuccess)
    e = cudaLaunchKernelEx(&cfg, k_cg_resident<T>, tiles, A, x, r, p, dinv, kp, tol2, steps, s,
                           co, steps_run);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  count_launch();
  std::swap(s.active, s.active_next);
  return true;
}

template ResidentPlan resident_plan<float>(int, int, int, int, int);
template ResidentPlan resident_plan<double>(int, int, int, int, int);
template bool launch_cg_resident<float>(const ResidentPlan&, const DTiles&, const EllView<float>&,
                                        float*, const float*, float*, const float*, int, double,
                                        int, CgState&, const Coarse<float>&, int*, cudaStream_t);
template bool launch_cg_resident<double>(const ResidentPlan&, const DTiles&,
                                         const EllView<double>&, double*, const double*, double*,
                                         const double*, int, double, int, CgState&,
                                         const Coarse<double>&, int*, cudaStream_t);

}  // namespace mor
