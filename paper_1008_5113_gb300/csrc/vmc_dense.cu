// vmc_dense.cu -- the standard algorithm (Sec. 1) on the GPU, FP64: an explicit
// inverse B = A^{-1} per walker, the ratio 1 + u^T B e_i, and the Sherman-Morrison
// update B <- B - (B e_i)(u^T B) / ratio on acceptance, with a fresh inverse (Gauss-
// Jordan elimination with partial pivoting) every sm_refresh sweeps.  The reference
// point the sparse engines are compared with; one CTA per walker.
//
// B is row-major over (orbital, particle): the ratio reads the entries B[j][i] of the
// support of u only; the update reads the rows B[j][.] of that support and then
// streams all of B once (coalesced).  On GB300 the n^2 FP64 multiply-adds of an update
// run at the FP64 rate (about 2 per clock per SM), not at the memory rate: 0.15 ms at n = 729
// on one SM.  So the rows of B are split over a cluster of CTAs, as many as the walkers leave
// SMs for (2 for 64 walkers, up to 8): every CTA computes the move and the vectors for
// itself, in the same order, updates its own rows, and meets the others after an accepted
// move only.  A warp takes a row at a time with the other vector in shared memory.  (One CTA
// a walker over a flat index, with a 64-bit division per element, took 1.3 ms an update and
// 1.3 ms a step of the inversion at n = 729; set-up and a sweep of 64 walkers 1535 ms, now
// 262 ms, with the same results bit for bit.)  Systems
// whose vectors do not fit shared memory keep that form.
#include <algorithm>

#include "vmc_internal.h"
#include "vmc_geom.cuh"

namespace vmc {

// Dense A (orbital columns, particle rows) from the sparse slots into B, then
// B <- A^{-1} in place (Gauss-Jordan, partial pivoting, column swaps undone at the end).
// Returns false if a pivot is exactly zero.
__device__ __noinline__ bool dense_invert_flat(const Walker& w, Shared& sh) {
  const int n = w.n, tid = threadIdx.x, nt = blockDim.x, cap = w.cap;
  double* B = w.Bd;
  for (size_t idx = tid; idx < (size_t)n * n; idx += nt) B[idx] = 0.0;
  __syncthreads();
  for (int p = tid; p < n; p += nt)
    for (int t = 0; t < w.a_len[p]; ++t) B[(size_t)p * n + w.a_col[(size_t)p * cap + t]] = w.a_val[(size_t)p * cap + t];
  __syncthreads();
  bool ok = true;
  for (int k = 0; k < n; ++k) {
    double bd = -1.0;
    int bi = k;
    for (int i = k + tid; i < n; i += nt) {
      const double v = fabs(B[(size_t)i * n + k]);
      if (v > bd) { bd = v; bi = i; }
    }
    double neg = -bd;
    block_argmin(neg, bi, sh);  // largest |B[i][k]|, lowest index on ties
    const int p = bi;
    if (-neg == 0.0) { ok = false; break; }
    if (p != k)
      for (int j = tid; j < n; j += nt) {
        const double t = B[(size_t)k * n + j];
        B[(size_t)k * n + j] = B[(size_t)p * n + j];
        B[(size_t)p * n + j] = t;
      }
    if (tid == 0) w.dpiv[k] = p;
    __syncthreads();
    const double inv = 1.0 / B[(size_t)k * n + k];
    __syncthreads();
    for (int j = tid; j < n; j += nt) {
      const double v = (j == k) ? inv : B[(size_t)k * n + j] * inv;
      B[(size_t)k * n + j] = v;
    }
    for (int i = tid; i < n; i += nt) w.dcol[i] = B[(size_t)i * n + k];
    __syncthreads();
    // rows i != k: B[i][j] -= f_i B[k][j] (j != k), B[i][k] = -f_i B[k][k]
    for (size_t idx = tid; idx < (size_t)n * n; idx += nt) {
      const int i = (int)(idx / n), j = (int)(idx - (size_t)i * n);
      if (i == k) continue;
      const double f = w.dcol[i];
      if (j == k) B[idx] = -f * B[(size_t)k * n + k];
      else B[idx] = fma(-f, B[(size_t)k * n + j], B[idx]);
    }
    __syncthreads();
  }
  // undo the row interchanges as column interchanges, last first
  for (int k = n - 1; k >= 0 && ok; --k) {
    const int p = w.dpiv[k];
    if (p != k)
      for (int i = tid; i < n; i += nt) {
        const double t = B[(size_t)i * n + k];
        B[(size_t)i * n + k] = B[(size_t)i * n + p];
        B[(size_t)i * n + p] = t;
      }
    __syncthreads();
  }
  return ok;
}

// One Metropolis step of particle k with the explicit inverse.
__device__ __noinline__ void dense_step_flat(const Walker& w, int k, uint64_t seed, uint32_t sweep, double sigma, uint8_t* acc_log,
                           double* ratio_log, Shared& sh) {
  const int n = w.n, tid = threadIdx.x, nt = blockDim.x, cap = w.cap;
  Ctl* c = w.ctl;
  if (tid == 0) {
    double z[3];
    normal3(seed, sweep, (uint32_t)k, 1u, z);
    for (int d = 0; d < 3; ++d) sh.rnew[d] = wrap_box(__dadd_rn(w.R[3 * k + d], __dmul_rn(sigma, z[d])), w.L);
  }
  __syncthreads();
  if (tid < 32) {
    const int alen = build_row_warp(w, sh.rnew, sh.acol, sh.aval, cap);
    int ulen = 0;
    if (alen >= 0) ulen = build_u_warp(w, k, sh.acol, sh.aval, alen, sh.ucol, sh.uval);
    if (tid == 0) { sh.alen = alen; sh.ulen = ulen; }
  }
  __syncthreads();
  if (sh.alen < 0) {
    if (tid == 0) c->status = ST_CAPACITY;
    return;
  }
  const double* B = w.Bd;
  double part = 0.0;
  for (int t = tid; t < sh.ulen; t += nt) part += sh.uval[t] * B[(size_t)sh.ucol[t] * n + k];
  const double ratio = 1.0 + block_sum(part, sh);
  const double U = accept_uniform(seed, sweep, (uint32_t)k);
  const bool acc = __dmul_rn(ratio, ratio) > U;
  if (tid == 0) {
    if (acc_log) *acc_log = acc ? 1 : 0;
    if (ratio_log) *ratio_log = ratio;
    c->proposals += 1;
    c->accepts += acc ? 1 : 0;
  }
  if (!acc) return;
  // Sherman-Morrison: col = B e_k, row = u^T B, B -= col row^T / ratio
  for (int a = tid; a < n; a += nt) w.dcol[a] = B[(size_t)a * n + k] / ratio;
  for (int b = tid; b < n; b += nt) {
    double s = 0.0;
    for (int t = 0; t < sh.ulen; ++t) s = fma(sh.uval[t], B[(size_t)sh.ucol[t] * n + b], s);
    w.drow[b] = s;
  }
  for (int t = tid; t < sh.alen; t += nt) {
    w.a_col[(size_t)k * cap + t] = sh.acol[t];
    w.a_val[(size_t)k * cap + t] = sh.aval[t];
  }
  if (tid == 0) {
    w.a_len[k] = sh.alen;
    for (int d = 0; d < 3; ++d) w.R[3 * k + d] = sh.rnew[d];
  }
  __syncthreads();
  double* Bw = w.Bd;
  for (size_t idx = tid; idx < (size_t)n * n; idx += nt) {
    const int a = (int)(idx / n), b = (int)(idx - (size_t)a * n);
    Bw[idx] = fma(-w.dcol[a], w.drow[b], Bw[idx]);
  }
  __syncthreads();
}

// ---- rows split over a cluster -----------------------------------------------------
__device__ __forceinline__ int cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return (int)r;
}
// Barrier of the cluster's CTAs; their global writes before it are visible after it (to loads
// that bypass L1).
__device__ __forceinline__ void cluster_sync(int size) {
  if (size > 1) {
    asm volatile("fence.acq_rel.gpu;" ::: "memory");
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  } else {
    __syncthreads();
  }
}
// A load of what another CTA of the cluster may have written; a walker's only CTA reads its own
// writes through L1.
template <bool kSplit>
__device__ __forceinline__ double ld_other(const double* p) {
  return kSplit ? __ldcg(p) : *p;
}
struct DenseRows {
  int rank, size, lo, hi;  // this CTA's rows of B
};
__device__ __forceinline__ DenseRows dense_rows(int n, int size) {
  const int rank = size > 1 ? cluster_rank() : 0;
  return DenseRows{rank, size, (int)((long long)n * rank / size), (int)((long long)n * (rank + 1) / size)};
}
// Elements of a row that a lane has in flight: 12, or 4 in the kernels that are compiled for four
// CTAs an SM (64 registers a thread).  Those serve walkers that would otherwise queue for an SM
// (a sweep is a chain of short steps, which only other walkers fill) and rows of up to 128
// elements, for which 12 batches of 32 are mostly loads past the row's end.  A sweep, ms, the
// flat form before the split, 12 elements, 4: n = 64 x 250 walkers 1.58, 1.93, 1.54; x 600 3.16,
// 3.80, 2.09; n = 125 x 250 4.82, 5.09, 3.93; n = 216 x 400 34.6, 23.3, 14.9.
template <int kPerSm>
constexpr int kBatchOf = kPerSm > 1 ? 4 : 12;
// Shared memory of the split form: two rows, a column, the column permutation.
__host__ __device__ __forceinline__ size_t dense_smem(int n) { return (size_t)n * (3 * 8 + 4); }

// As dense_invert_flat, the CTA's rows of it.  Every CTA finds the pivot itself.
template <int kPerSm, bool kSplit>
__device__ __noinline__ bool dense_invert(const Walker& w, const DenseRows d, Shared& sh) {
  constexpr int kBatch = kBatchOf<kPerSm>;
  const int n = w.n, tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5, nw = nt >> 5, cap = w.cap;
  double* B = w.Bd;
  double* rk = (double*)dyn_smem();  // old row k
  double* rp = rk + n;               // the pivot row, scaled: the new row k
  int* piv = (int*)(rp + 2 * (size_t)n);
  for (int i = d.lo + wid; i < d.hi; i += nw) {
    for (int j = lane; j < n; j += 32) B[(size_t)i * n + j] = 0.0;
    __syncwarp();
    const int len = w.a_len[i];
    for (int t = lane; t < len; t += 32) B[(size_t)i * n + w.a_col[(size_t)i * cap + t]] = w.a_val[(size_t)i * cap + t];
  }
  cluster_sync(d.size);
  bool ok = true;
  for (int k = 0; k < n; ++k) {
    double bd = -1.0;
    int bi = k;
    for (int i = k + tid; i < n; i += nt) {
      const double v = fabs(ld_other<kSplit>(B + (size_t)i * n + k));
      if (v > bd) { bd = v; bi = i; }
    }
    double neg = -bd;
    block_argmin(neg, bi, sh);  // largest |B[i][k]|, lowest index on ties
    const int p = bi;
    if (-neg == 0.0) { ok = false; break; }
#pragma unroll 4
    for (int j = tid; j < n; j += nt) {
      rk[j] = ld_other<kSplit>(B + (size_t)k * n + j);
      rp[j] = ld_other<kSplit>(B + (size_t)p * n + j);
    }
    if (tid == 0) piv[k] = p;
    __syncthreads();
    const double pv = rp[k];
    __syncthreads();
    if (tid == 0) sh.dflag[0] = 1.0 / pv;
    __syncthreads();
    const double inv = sh.dflag[0];
    for (int j = tid; j < n; j += nt) rp[j] = j == k ? inv : rp[j] * inv;
    cluster_sync(d.size);  // rows k and p and column k have been read
    // rows i != k: B[i][j] -= f_i B[k][j] (j != k), B[i][k] = -f_i B[k][k]; row p starts from
    // the old row k
    for (int i = d.lo + wid; i < d.hi; i += nw) {
      double* Bi = B + (size_t)i * n;
      if (i == k) {
        for (int j = lane; j < n; j += 32) Bi[j] = rp[j];
        continue;
      }
      // kBatch loads in flight, then the stores (a load after a store that may alias it would
      // wait for the load before: one DRAM latency per 32 elements)
      if (i == p) {
        const double f = rk[k];
        for (int j = lane; j < n; j += 32) Bi[j] = j == k ? -f * inv : fma(-f, rp[j], rk[j]);
      } else {
        const double f = Bi[k];
        __syncwarp();
        for (int j0 = lane; j0 < n; j0 += 32 * kBatch) {
          double x[kBatch];
#pragma unroll
          for (int u = 0; u < kBatch; ++u) x[u] = Bi[min(j0 + 32 * u, n - 1)];
#pragma unroll
          for (int u = 0; u < kBatch; ++u) {
            const int j = j0 + 32 * u;
            if (j < n) Bi[j] = j == k ? -f * inv : fma(-f, rp[j], x[u]);
          }
        }
      }
    }
    cluster_sync(d.size);
  }
  // undo the row interchanges as column interchanges, last first
  int* from = (int*)rp;
  for (int j = tid; j < n; j += nt) from[j] = j;
  __syncthreads();
  if (tid == 0 && ok)
    for (int k = n - 1; k >= 0; --k) {
      const int p = piv[k], t = from[k];
      from[k] = from[p];
      from[p] = t;
    }
  __syncthreads();
  if (ok)
    for (int i = d.lo; i < d.hi; ++i) {
      double* Bi = B + (size_t)i * n;
#pragma unroll 4
      for (int j = tid; j < n; j += nt) rk[j] = Bi[j];
      __syncthreads();
#pragma unroll 4
      for (int j = tid; j < n; j += nt) Bi[j] = rk[from[j]];
      __syncthreads();
    }
  cluster_sync(d.size);
  return ok;
}

// One Metropolis step of particle k, the CTA's rows of it; st: the walker's status, which
// every CTA keeps alike.  The CTAs write the same matrix row and position.
template <int kPerSm, bool kSplit>
__device__ __forceinline__ void dense_step(const Walker& w, const DenseRows d, int k, uint64_t seed, uint32_t sweep,
                                           double sigma, uint8_t* acc_log, double* ratio_log, int& st, Shared& sh) {
  constexpr int kBatch = kBatchOf<kPerSm>;
  const int n = w.n, tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5, nw = nt >> 5, cap = w.cap;
  Ctl* c = w.ctl;
  if (tid == 0) {
    double z[3];
    normal3(seed, sweep, (uint32_t)k, 1u, z);
    for (int q = 0; q < 3; ++q) sh.rnew[q] = wrap_box(__dadd_rn(w.R[3 * k + q], __dmul_rn(sigma, z[q])), w.L);
  }
  __syncthreads();
  if (tid < 32) {
    const int alen = build_row_warp(w, sh.rnew, sh.acol, sh.aval, cap);
    int ulen = 0;
    if (alen >= 0) ulen = build_u_warp(w, k, sh.acol, sh.aval, alen, sh.ucol, sh.uval);
    if (tid == 0) { sh.alen = alen; sh.ulen = ulen; }
  }
  __syncthreads();
  if (sh.alen < 0) {
    if (tid == 0 && d.rank == 0) c->status = ST_CAPACITY;
    st = ST_CAPACITY;
    return;
  }
  double* B = w.Bd;
  double part = 0.0;
  for (int t = tid; t < sh.ulen; t += nt) part += sh.uval[t] * ld_other<kSplit>(B + (size_t)sh.ucol[t] * n + k);
  const double ratio = 1.0 + block_sum(part, sh);
  const double U = accept_uniform(seed, sweep, (uint32_t)k);
  const bool acc = __dmul_rn(ratio, ratio) > U;
  if (tid == 0 && d.rank == 0) {
    if (acc_log) *acc_log = acc ? 1 : 0;
    if (ratio_log) *ratio_log = ratio;
    c->proposals += 1;
    c->accepts += acc ? 1 : 0;
  }
  if (!acc) return;
  // Sherman-Morrison: col = B e_k, row = u^T B, B -= col row^T / ratio
  double* row = (double*)dyn_smem();
  double* col = row + n;
  for (int a = d.lo + tid; a < d.hi; a += nt) col[a] = B[(size_t)a * n + k] / ratio;
  const int ulen = sh.ulen;
  for (int b = tid; b < n; b += nt) {
    double s = 0.0;
#pragma unroll 8
    for (int t = 0; t < ulen; ++t) s = fma(sh.uval[t], ld_other<kSplit>(B + (size_t)sh.ucol[t] * n + b), s);
    row[b] = s;
  }
  // every CTA has formed u from the old row and read the rows of u's support (a CTA may be
  // several rejected moves ahead of another): only now may the row, the position and B change
  cluster_sync(d.size);
  for (int t = tid; t < sh.alen; t += nt) {
    w.a_col[(size_t)k * cap + t] = sh.acol[t];
    w.a_val[(size_t)k * cap + t] = sh.aval[t];
  }
  if (tid == 0) {
    w.a_len[k] = sh.alen;
    for (int q = 0; q < 3; ++q) w.R[3 * k + q] = sh.rnew[q];
  }
  for (int a = d.lo + wid; a < d.hi; a += nw) {
    double* Ba = B + (size_t)a * n;
    const double f = -col[a];
    for (int b0 = lane; b0 < n; b0 += 32 * kBatch) {
      double x[kBatch];
#pragma unroll
      for (int u = 0; u < kBatch; ++u) x[u] = Ba[min(b0 + 32 * u, n - 1)];
#pragma unroll
      for (int u = 0; u < kBatch; ++u)
        if (b0 + 32 * u < n) Ba[b0 + 32 * u] = fma(f, row[b0 + 32 * u], x[u]);
    }
  }
  cluster_sync(d.size);
}

// split: rows over a cluster of `size` CTAs; else (size 0) one CTA in the flat form.
template <int kPerSm, bool kSplit>
__global__ void __launch_bounds__(kMaxThreads, kPerSm) k_dense_setup(const Walker* __restrict__ W, int size) {
  __shared__ Shared sh;
  const Walker& w = stage_walker(sh, W[blockIdx.x / max(size, 1)]);
  const DenseRows d = size ? dense_rows(w.n, size) : DenseRows{0, 1, 0, w.n};
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int bad = 0;
  for (int p = wid; p < w.n; p += nw) {  // every CTA the whole matrix: the same values
    const int len = build_row_warp(w, w.R + 3 * p, w.a_col + (size_t)p * w.cap, w.a_val + (size_t)p * w.cap, w.cap);
    if (lane == 0) {
      if (len < 0) bad = 1;
      w.a_len[p] = len < 0 ? 0 : len;
    }
  }
  bad = __syncthreads_or(bad);
  const bool ok = size ? dense_invert<kPerSm, kSplit>(w, d, sh) : dense_invert_flat(w, sh);
  if (threadIdx.x == 0 && d.rank == 0) {
    if (bad) w.ctl->status = ST_CAPACITY;
    else if (!ok) w.ctl->status = ST_BREAKDOWN;
    w.ctl->factorizations += 1;
  }
}

template <int kPerSm, bool kSplit>
__global__ void __launch_bounds__(kMaxThreads, kPerSm) k_dense_sweep(const Walker* __restrict__ W, int n_sweeps,
                                                             long long sweep0, double sigma,
                                                             const uint64_t* __restrict__ seeds, uint8_t* acc_log,
                                                             double* ratio_log, int refresh, int size) {
  __shared__ Shared sh;
  const int wi = blockIdx.x / max(size, 1);
  const Walker& w = stage_walker(sh, W[wi]);
  const DenseRows d = size ? dense_rows(w.n, size) : DenseRows{0, 1, 0, w.n};
  const uint64_t seed = seeds[wi];
  const int n = w.n;
  int st = w.ctl->status;  // the CTAs of a cluster keep their own, alike: they meet at barriers
  cluster_sync(size);      // read by all before the first can write it
  for (int s = 0; s < n_sweeps; ++s) {
    if (refresh > 0 && s > 0 && (sweep0 + s) % refresh == 0) {
      const bool ok = size ? dense_invert<kPerSm, kSplit>(w, d, sh) : dense_invert_flat(w, sh);
      if (!ok) st = ST_BREAKDOWN;
      if (threadIdx.x == 0 && d.rank == 0) {
        w.ctl->factorizations += 1;
        if (!ok) w.ctl->status = ST_BREAKDOWN;
      }
      __syncthreads();
    }
    for (int k = 0; k < n; ++k) {
      const long long idx = (long long)n_sweeps * w.log_base + (long long)s * n + k;
      if (!size) st = w.ctl->status;
      __syncthreads();
      if (st != ST_OK) {
        if (threadIdx.x == 0 && d.rank == 0) {
          if (acc_log) acc_log[idx] = 0;
          if (ratio_log) ratio_log[idx] = 0.0;
        }
        continue;
      }
      uint8_t* al = acc_log ? acc_log + idx : nullptr;
      double* rl = ratio_log ? ratio_log + idx : nullptr;
      if (size) dense_step<kPerSm, kSplit>(w, d, k, seed, (uint32_t)(sweep0 + s), sigma, al, rl, st, sh);
      else dense_step_flat(w, k, seed, (uint32_t)(sweep0 + s), sigma, al, rl, sh);
      __syncthreads();
    }
  }
}

// CTAs a walker: the largest power of two (at most 8) that keeps every CTA on an SM of its
// own; 0 (the flat form) when the vectors do not fit shared memory.
static int dense_cluster(int nwalk, int max_n, int static_smem) {
  int dev = 0, nsm = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (dense_smem(max_n) + (size_t)static_smem > (size_t)optin) return 0;
  int cs = 1;
  while (cs < 8 && 2 * cs * nwalk <= nsm) cs *= 2;
  return cs;
}
// kernels: for long rows and for many walkers or short rows (kBatchOf), each with rows split over
// a cluster and with one CTA a walker.
template <typename K, typename... A>
static cudaError_t dense_launch(const K (&kernels)[4], const LaunchCfg& L, int nwalk, int max_n, A... args) {
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaFuncAttributes fa{};
  cudaError_t e = cudaFuncGetAttributes(&fa, kernels[0]);
  if (e != cudaSuccess) return e;
  const int cs = dense_cluster(nwalk, max_n, (int)fa.sharedSizeBytes);
  const K kernel = kernels[2 * (nwalk > 2 * nsm || max_n <= 128) + (cs <= 1)];
  e = allow_dynamic_smem(kernel);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(std::max(cs, 1) * nwalk);
  lc.blockDim = dim3(L.threads);
  lc.dynamicSmemBytes = cs ? dense_smem(max_n) : 0;
  lc.stream = L.stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = std::max(cs, 1);
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  lc.attrs = at;
  lc.numAttrs = cs > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&lc, kernel, args..., cs);
}

cudaError_t launch_dense_setup(const LaunchCfg& L, const Walker* W, int nwalk, int max_n) {
  static constexpr decltype(&k_dense_setup<1, true>) kernels[] = {k_dense_setup<1, true>, k_dense_setup<1, false>,
                                                                  k_dense_setup<4, true>, k_dense_setup<4, false>};
  return dense_launch(kernels, L, nwalk, max_n, W);
}
cudaError_t launch_dense_sweep(const LaunchCfg& L, const Walker* W, int nwalk, int max_n, int n_sweeps, long long sweep0,
                               double sigma, const uint64_t* seeds, uint8_t* acc, double* ratio, int refresh) {
  static constexpr decltype(&k_dense_sweep<1, true>) kernels[] = {k_dense_sweep<1, true>, k_dense_sweep<1, false>,
                                                                  k_dense_sweep<4, true>, k_dense_sweep<4, false>};
  return dense_launch(kernels, L, nwalk, max_n, W, n_sweeps, sweep0, sigma, seeds, acc, ratio, refresh);
}

}  // namespace vmc
