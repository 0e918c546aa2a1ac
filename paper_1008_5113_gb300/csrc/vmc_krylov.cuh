// vmc_krylov.cuh -- the per-move solve A_p z = e_r and the determinant ratio.
//
//   * M v = prod_s (I - z_hat_s u_s^T) Q (L U)^{-1} v                (Sec. 3.2 Eq. 18)
//     the triangular solves from task streams (vmc_blocks.cuh) or, from chunk streams, level
//     by level, then the column permutation Q, then the update chain:
//     c = (I + G)^{-1} (u_s^T w_0)_s,  w = w_0 - sum_s z_hat_s c_s.
//   * right-preconditioned GMRES(m) on A_p M (Sec. 3.2 Eq. 15) with classical
//     Gram-Schmidt (reorthogonalised when it cancels), Givens rotations, and the effective stability
//     N = max_j ||v_j - A_p M v_j||_2 over the Arnoldi vectors (Sec. 3.1 Eq. 10),
//     computed in the same pass as the first projections.
//   * FP64 iterative refinement: r = e_r - A_p x in FP64, inner GMRES in the working
//     precision T on r, x += d; the ratio 1 + u^T x (Sec. 3 Eq. 13) in FP64.
#pragma once
#include "vmc_precond.cuh"

namespace vmc {

// 16-byte vector views of the Slater slots (slot starts are 16-byte aligned: cap % 4 == 0)
template <typename T> struct Vec4;
template <> struct Vec4<float> {
  float v[4];
  __device__ __forceinline__ void load(const float* p) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  }
};
template <> struct Vec4<double> {
  double v[4];
  __device__ __forceinline__ void load(const double* p) {
    const double2 a = *reinterpret_cast<const double2*>(p);
    const double2 b = *reinterpret_cast<const double2*>(p + 2);
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
  }
};

// Rows of V, Z or the update chain that a thread has in flight at once (the loads of a batch
// are issued together, the last batch's under a predicate: an unrolled loop's remainder would
// pay an L2 round trip a row).
constexpr int kRows = 8;
// Elements of a vector that a thread holds at once: 16 bytes.  (With 32 bytes of FP64 a vector
// of 216 elements is on two warps, whose DFMAs queue on two of the SM's four schedulers.)
template <typename T>
constexpr int kWide = 16 / (int)sizeof(T);
// The loads are volatile assembly: the compiler would otherwise sink a load that is under the
// same predicate as its use down to the use, and a batch would become a chain of round trips.
template <typename T> struct Wide;
template <> struct Wide<float> {
  float v[4];
  __device__ __forceinline__ void load(const float* p) {  // any address space
    asm volatile("ld.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "l"(p));
  }
  // streaming load (evict first): data read once per apply
  __device__ __forceinline__ void load_cs(const float* p) {
    asm volatile("ld.global.cs.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "l"(p));
  }
};
template <> struct Wide<double> {
  double v[2];
  __device__ __forceinline__ void load(const double* p) {
    asm volatile("ld.v2.f64 {%0, %1}, [%2];" : "=d"(v[0]), "=d"(v[1]) : "l"(p));
  }
  __device__ __forceinline__ void load_cs(const double* p) {
    asm volatile("ld.global.cs.v2.f64 {%0, %1}, [%2];" : "=d"(v[0]), "=d"(v[1]) : "l"(p));
  }
};

// Dot product of Slater slot p (len entries, capacity cap) with x: 16-byte loads of
// four column indices and four values at a time (cap is a multiple of 4).  Up to 16
// entries at a time have their index and value loads issued together -- bounded by the
// slot's capacity, not its length, so the first ones need not wait for len -- then
// their gathers (entries < len only), then the products are summed in entry order.
template <typename T, typename X>
__device__ __forceinline__ X slot_dot(const int* __restrict__ cols, const T* __restrict__ vals, int len, int cap,
                                      const X* __restrict__ x) {
  constexpr int U = 4;
  X acc = 0;
  int q0 = 0;
  do {
    int4 c[U];
    Vec4<T> v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      c[u] = make_int4(0, 0, 0, 0);
      if (q0 + 4 * u < cap) {
        c[u] = *reinterpret_cast<const int4*>(cols + q0 + 4 * u);
        v[u].load(vals + q0 + 4 * u);
      }
    }
    X xv[4 * U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int q = q0 + 4 * u;
      xv[4 * u + 0] = q + 0 < len ? x[c[u].x] : (X)0;
      xv[4 * u + 1] = q + 1 < len ? x[c[u].y] : (X)0;
      xv[4 * u + 2] = q + 2 < len ? x[c[u].z] : (X)0;
      xv[4 * u + 3] = q + 3 < len ? x[c[u].w] : (X)0;
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (q0 + 4 * u + k < len) acc += (X)v[u].v[k] * xv[4 * u + k];
    q0 += 4 * U;
  } while (q0 < len);
  return acc;
}

template <typename T>
__device__ __forceinline__ const T* ell_vals(const Walker& w);
template <>
__device__ __forceinline__ const float* ell_vals<float>(const Walker& w) { return w.ell_val32; }
template <>
__device__ __forceinline__ const double* ell_vals<double>(const Walker& w) { return w.ell_val; }

// Loads that are issued where they stand (see Wide).
__device__ __forceinline__ int load_now(const int* p) {
  int v;
  asm volatile("ld.global.b32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ float load_now(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ double load_now(const double* p) {
  double v;
  asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
  return v;
}

// 16-bit columns and values of four entries of a row in the transposed copy.
template <typename T>
struct EllQuad {
  unsigned c0, c1;  // two columns each
  Wide<T> v[sizeof(T) / 4];
  __device__ __forceinline__ void load(const unsigned short* col, const T* val) {
    asm volatile("ld.global.v2.u32 {%0, %1}, [%2];" : "=r"(c0), "=r"(c1) : "l"(col));
#pragma unroll
    for (int k = 0; k < (int)sizeof(T) / 4; ++k) v[k].load(val + kWide<T> * k);
  }
  __device__ __forceinline__ T value(int u) const { return v[u / kWide<T>].v[u % kWide<T>]; }
};

// Dot product of particle p's row (len entries) with x.  From the transposed copy of the slots (quads of
// entries, quad q of every particle side by side, zeros past the row's end): coalesced
// 8- and 16-byte loads, all of a row of up to 24 entries in flight, summed in entry order;
// else from the slot itself.  Two running pointers: as twelve precomputed addresses they made
// the solve spill around the loads (in an iteration of 256 walkers of n = 4096, two an SM, FP32:
// product 63.9 us, FP64 residual 53.7; so 55.2 and 43.1; with five quads in flight 41.2 and 55.0,
// but a second trip for the rows beyond 20 entries: one walker of n = 4096 14.3 us, 12.0 so).
template <typename T, typename X>
__device__ __forceinline__ X row_dot(const Walker& w, int p, int len, const X* x) {
  const int cap = w.cap;
  if (w.ell_col == nullptr) {
    const T* v = sizeof(T) == 4 ? (const T*)w.a_val32 : (const T*)w.a_val;
    return slot_dot<T, X>(w.a_col + (size_t)p * cap, v + (size_t)p * cap, len, cap, x);
  }
  const size_t step = 4 * (size_t)w.ld;
  const unsigned short* col = w.ell_col + 4 * (size_t)p;
  const T* val = ell_vals<T>(w) + 4 * (size_t)p;
  constexpr int U = 6;
  X acc = 0;
#pragma unroll 1
  for (int left = len; left > 0; left -= 4 * U) {
    EllQuad<T> e[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (4 * u < left) e[u].load(col, val);
      col += step;
      val += step;
      asm volatile("" : "+l"(col), "+l"(val));
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (4 * u < left) {
        acc += (X)e[u].value(0) * x[e[u].c0 & 0xffffu];
        acc += (X)e[u].value(1) * x[e[u].c0 >> 16];
        acc += (X)e[u].value(2) * x[e[u].c1 & 0xffffu];
        acc += (X)e[u].value(3) * x[e[u].c1 >> 16];
      }
  }
  return acc;
}

// The length and the row of A_p of the thread's particles, read one particle ahead: a row's
// entries and v's element then start without a memory round trip before them.
struct NextRow {
  int len, row;
  __device__ __forceinline__ NextRow(const Walker& w, int p) : len(0), row(0) {
    if (p < w.n) {
      len = load_now(w.a_len + p);
      row = load_now(w.row_of_part + p);
    }
  }
};

// y = A_p x - v (v may be null): a particle's row per thread in slot order, the result
// scattered to its row of A_p.  Bound by memory round trips: with a row's length, then its
// entries, and v's place, then v, one after the other, an apply of 152 walkers of n = 32768 took
// 283 us in FP32, 64 of n = 8000 88, 64 of n = 1000 10.0 (FP64 14.0); so 216, 43, 4.4 (7.3).
// (v subtracted in a pass of its own, without the gather: 64 of n = 8000 89 us an iteration's
// product, 55 with it; n = 216 FP64 3.7 and 3.2.)
template <typename T>
__device__ __forceinline__ void spmv(const Walker& w, const T* x, const T* v, T* y) {
  const int n = w.n;
  NextRow at(w, threadIdx.x);
#pragma unroll 1
  for (int p = threadIdx.x; p < n; p += blockDim.x) {
    const NextRow next(w, p + blockDim.x);
    const T vr = v ? load_now(v + at.row) : (T)0;
    y[at.row] = row_dot<T, T>(w, p, at.len, x) - vr;
    at = next;
  }
}

// The product's input vector copied into the solve area where that is in shared memory (idle
// between preconditioner applies): the gathers then read shared memory instead of scattered
// global lines.  For walkers whose vectors the task ring does not hold (FP32 from n = 24 000 or
// so, FP64 from 12 000) and for the chunk streams.  n = 32768 x 152 walkers FP32: an apply 449 us
// gathering from global memory, 283 us so (kappa 1, r_c 2: 644, 406).
// Block-wide, ends synchronised; returns the vector to read.
template <typename T>
__device__ __forceinline__ const T* stage_x(const Walker& w, const Params& P, const T* x) {
  if (!P.y_smem) return x;
  T* xs = (T*)dyn_smem();
  block_copy(xs, x, w.n);
  __syncthreads();
  return xs;
}

// Shared-memory ring of the stream chunks: one mbarrier per slot, initialised once
// per kernel launch; chunk g of the launch lives in slot g % S, phase (g / S) & 1.
__device__ __forceinline__ void ring_init(Shared& sh, const Params& P) {
  if (threadIdx.x == 0) {
    // a slot is released by every consumer warp once it is done with the chunk
    const unsigned rel = (unsigned)((blockDim.x >> 5) - 1);
#pragma unroll 1
    for (int s = 0; s < P.ring_slots; ++s) {
      mbar_init(&sh.bar[s], 1);
      mbar_init(&sh.ebar[s], rel);
    }
    sh.ring_seq = 0;
    sh.iflag[3] = 0;
#pragma unroll 1
    for (int i = 0; i < 16; ++i) sh.cyc[i] = 0;
    sh.cnt = SolveCounts{};
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
}

// Producer of the chunk streams (lane 0 of the last warp): streams the factor's chunks
// into the ring with bulk copies, refilling a slot once the consumers have released it
// (the slot's "empty" barrier).  Returns the cycles spent waiting for free slots.
__device__ __forceinline__ long long stream_chunks(const unsigned char* stream, const int2* tab, int nch,
                                                   const Params& P, unsigned char* ring, int seq0, Shared& sh) {
  const int S = P.ring_slots;
  const int SB = P.slot_bytes;
  long long twait = 0;
  int2 pre[kMaxSlots];
#pragma unroll 1
  for (int k = 0; k < S && k < nch; ++k) pre[k] = tab[k];
  int slot = seq0 % S;
  int g = seq0;
  const unsigned long long pol = l2_policy_evict_last();
#pragma unroll 1
  for (int c = 0; c < nch; ++c, ++g) {
    unsigned char* dst = ring + (size_t)slot * SB;
    if (g >= S) {  // the consumers must have released the slot's previous use
      const long long tw = clock64();
      if (!mbar_wait(&sh.ebar[slot], (unsigned)(((g / S) - 1) & 1))) sh.iflag[3] = 1;
      twait += clock64() - tw;
    }
    // chunk c's descriptor: from the table for the first S chunks, else from the
    // header of chunk c - S, still in this slot
    const int2 tc = c < S ? pre[c] : ((const int2*)(dst + 16))[S - 1];
    mbar_expect_tx(&sh.bar[slot], (unsigned)tc.y);
    bulk_g2s_hint(dst, stream + tc.x, (unsigned)tc.y, &sh.bar[slot], pol);
    if (++slot == S) slot = 0;
  }
  return twait;
}

// One triangular solve in place on y (shared or global), level-synchronous.  The last
// warp produces (stream_chunks); the other warps solve: per chunk they wait for it to
// land, solve its segments (levels) one after the other with a barrier among the
// consumer warps between segments, and release the slot.  A segment marked for one
// warp (few rows) is solved by the first consumer warp alone, with only a warp
// synchronisation after it; the other consumer warps skip it and meet that warp at the
// barrier before the next segment solved by all.
// Lower: y_r -= sum_t L_rt y_t.  Upper: y_r = (y_r - sum_t U_rt y_t) / U_rr.
// Every wait gives up after ~1 s (status VMC_ERR_TIMEOUT).
template <typename T>
__device__ __forceinline__ void tri_staged(const Walker& w, const Params& P, bool upper, T* y, Shared& sh) {
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5, nwarp = nt >> 5;
  const unsigned char* stream = upper ? w.ustream : w.lstream;
  const int2* tab = upper ? w.uchunk : w.lchunk;
  const int nch = upper ? w.ctl->nchunk_u : w.ctl->nchunk_l;
  const int S = P.ring_slots;
  const int SB = P.slot_bytes;
  unsigned char* ring = dyn_smem() + P.y_bytes;
  const int seq0 = sh.ring_seq;
  const int nct = nt - 32;
  long long twait = 0;
  if (wid == nwarp - 1) {
    if (lane == 0) twait = stream_chunks(stream, tab, nch, P, ring, seq0, sh);
  } else {
    int slot = seq0 % S;
    unsigned parity = (unsigned)((seq0 / S) & 1);
    long long tdata = 0;
    bool pend = false;  // the first warp solved rows the others have not synchronised with
#pragma unroll 1
    for (int c = 0; c < nch; ++c) {
      const long long tw0 = clock64();
      if (!mbar_wait(&sh.bar[slot], parity)) sh.iflag[3] = 1;
      tdata += clock64() - tw0;
      const unsigned char* ch = ring + (size_t)slot * SB;
      const int4 hd = *(const int4*)ch;
      const int nseg = hd.x, nr = hd.y, ne = hd.z;
      const int4* seg = (const int4*)(ch + kChunkHdr);
      const int* rws = (const int*)(ch + kChunkHdr + 16 * nseg);
      const int* st = rws + pad4(nr);
      const int* cl = st + pad4(nr + 1);
      const T* vl = (const T*)(cl + pad4(ne));
      const T* dv = (const T*)((const unsigned char*)vl + pad16((int)sizeof(T) * ne));
#pragma unroll 1
      for (int sgi = 0; sgi < nseg; ++sgi) {
        const int4 sm = seg[sgi];
        const int r0 = sm.x, sr = sm.y;
        if (sm.w) {  // one warp
          if (wid == 0) {
            const int gs = sm.w - 1, G = 1 << gs, gl = lane & (G - 1);
            const int i = r0 + (lane >> gs);
            const bool on = (lane >> gs) < sr;
            T part = 0;
            int r = 0;
            if (on) {
              r = rws[i];
              T part2 = 0;
              const int e = st[i + 1];
              int t = st[i] + gl;
#pragma unroll 1
              for (; t + G < e; t += 2 * G) {
                part += vl[t] * y[cl[t]];
                part2 += vl[t + G] * y[cl[t + G]];
              }
              if (t < e) part += vl[t] * y[cl[t]];
              part += part2;
            }
#pragma unroll 1
            for (int o = G >> 1; o; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o, G);
            if (on && gl == 0) {
              T acc = y[r] - part;
              if (upper) acc *= dv[i];
              y[r] = acc;
            }
            __syncwarp();
          }
          pend = true;
          continue;
        }
        if (pend) {  // publish the first warp's rows before a segment solved by all
          asm volatile("bar.sync 1, %0;" ::"r"(nct) : "memory");
          pend = false;
        }
        const int gs = sm.z;
        const int G = 1 << gs;
        const int gl = tid & (G - 1);
        const int ng = nct >> gs;
#pragma unroll 1
        for (int base = 0; base < sr; base += ng) {  // same trip count in every lane
          const int i = r0 + base + (tid >> gs);
          const bool on = base + (tid >> gs) < sr;
          T part = 0;
          int r = 0;
          if (on) {
            r = rws[i];
            T part2 = 0;
            const int e = st[i + 1];
            int t = st[i] + gl;
#pragma unroll 1
            for (; t + G < e; t += 2 * G) {  // two entries in flight per lane
              part += vl[t] * y[cl[t]];
              part2 += vl[t + G] * y[cl[t + G]];
            }
            if (t < e) part += vl[t] * y[cl[t]];
            part += part2;
          }
#pragma unroll 1
          for (int o = G >> 1; o; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o, G);
          if (on && gl == 0) {
            T acc = y[r] - part;
            if (upper) acc *= dv[i];
            y[r] = acc;
          }
        }
        asm volatile("bar.sync 1, %0;" ::"r"(nct) : "memory");  // level barrier (consumers)
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.ebar[slot]);  // this warp is done with the chunk
      if (++slot == S) { slot = 0; parity ^= 1u; }
    }
    if (tid == 0) sh.cyc[PH_TRIDATA] += tdata;
  }
  if (wid == nwarp - 1 && lane == 0) sh.cyc[PH_TRIWAIT] += twait;
  __syncthreads();
  if (tid == 0) sh.ring_seq = seq0 + nch;
  __syncthreads();
}

// "Not yet solved" marker for the synchronisation-free solves: a quiet NaN with a
// payload that arithmetic never produces (GPU arithmetic returns the canonical NaN).
template <typename T>
struct Pending;
template <>
struct Pending<float> {
  static __device__ __forceinline__ float value() { return __int_as_float(0x7fc5a5a5); }
  static __device__ __forceinline__ bool is(float v) { return __float_as_int(v) == 0x7fc5a5a5; }
};
template <>
struct Pending<double> {
  static __device__ __forceinline__ double value() { return __longlong_as_double(0x7ff8a5a5a5a5a5a5ll); }
  static __device__ __forceinline__ bool is(double v) { return __double_as_longlong(v) == 0x7ff8a5a5a5a5a5a5ll; }
};
// Most retries of one row group's operands before giving up (status VMC_ERR_TIMEOUT).
constexpr int kSpinMax = 1 << 22;

// One triangular solve without level barriers: x = L^{-1} rhs (lower) or
// x = U^{-1} rhs (upper), x in shared memory pre-filled with Pending.  Rows are taken
// in the stream's level order, each by a group of G lanes (the level's group size),
// a warp's groups holding consecutive rows of one level.  A warp waits only until the
// operands of its own rows have been solved -- by whichever warp owns them -- instead
// of for the whole previous level; it retries as a unit, so its lanes stay converged.
// Rows only depend on earlier rows of the order, and every warp takes its rows in that
// order, so the waits always end.  Each row's sum is taken in the same order as the
// level-synchronous solve.
template <typename T>
__device__ __forceinline__ void tri_syncfree(const Walker& w, const Params& P, bool upper, const T* rhs, T* x,
                                             Shared& sh) {
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5, nwarp = nt >> 5;
  const unsigned char* stream = upper ? w.ustream : w.lstream;
  const int2* tab = upper ? w.uchunk : w.lchunk;
  const int nch = upper ? w.ctl->nchunk_u : w.ctl->nchunk_l;
  const int S = P.ring_slots;
  const int SB = P.slot_bytes;
  unsigned char* ring = dyn_smem() + P.y_bytes;
  const int seq0 = sh.ring_seq;
  const int nct = nt - 32;
  const volatile T* xv = x;
  long long twait = 0;
  if (wid == nwarp - 1) {
    if (lane == 0) twait = stream_chunks(stream, tab, nch, P, ring, seq0, sh);
  } else {
    int slot = seq0 % S;
    unsigned parity = (unsigned)((seq0 / S) & 1);
    long long tdata = 0;
#pragma unroll 1
    for (int c = 0; c < nch; ++c) {
      const long long tw0 = clock64();
      if (!mbar_wait(&sh.bar[slot], parity)) sh.iflag[3] = 1;
      tdata += clock64() - tw0;
      const unsigned char* ch = ring + (size_t)slot * SB;
      const int4 hd = *(const int4*)ch;
      const int nseg = hd.x, nr = hd.y, ne = hd.z;
      const int4* seg = (const int4*)(ch + kChunkHdr);
      const int* rws = (const int*)(ch + kChunkHdr + 16 * nseg);
      const int* st = rws + pad4(nr);
      const int* cl = st + pad4(nr + 1);
      const T* vl = (const T*)(cl + pad4(ne));
      const T* dv = (const T*)((const unsigned char*)vl + pad16((int)sizeof(T) * ne));
#pragma unroll 1
      for (int sgi = 0; sgi < nseg; ++sgi) {
        const int4 sm = seg[sgi];
        const int r0 = sm.x, sr = sm.y, gs = sm.z;
        const int G = 1 << gs;
        const int gl = tid & (G - 1);
        const int ng = nct >> gs;
#pragma unroll 1
        for (int base = 0; base < sr; base += ng) {  // warp-uniform trip count
          const int i = base + (tid >> gs);
          const bool on = i < sr;
          int r = 0, t0 = 0, e = 0;
          if (on) {
            r = rws[r0 + i];
            t0 = st[r0 + i] + gl;
            e = st[r0 + i + 1];
          }
          // sum and readiness in one pass; the warp retries together until every lane's
          // operands were solved (so its lanes never diverge on a wait)
          T part = 0;
#pragma unroll 1
          for (int it = 0;; ++it) {
            T p1 = 0, p2 = 0;
            bool rdy = true;
            int t = t0;
#pragma unroll 1
            for (; t + G < e; t += 2 * G) {  // two entries in flight per lane
              const T a = xv[cl[t]], b = xv[cl[t + G]];
              rdy &= !Pending<T>::is(a) && !Pending<T>::is(b);
              p1 += vl[t] * a;
              p2 += vl[t + G] * b;
            }
            if (t < e) {
              const T a = xv[cl[t]];
              rdy &= !Pending<T>::is(a);
              p1 += vl[t] * a;
            }
            if (__all_sync(0xffffffffu, rdy)) { part = p1 + p2; break; }
            if (it >= kSpinMax || *(volatile int*)&sh.iflag[3]) { sh.iflag[3] = 1; break; }  // one give-up ends all waits
          }
#pragma unroll 1
          for (int o = G >> 1; o; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o, G);
          if (on && gl == 0) {
            T acc = rhs[r] - part;
            if (upper) acc *= dv[r0 + i];
            ((volatile T*)x)[r] = acc;
          }
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.ebar[slot]);  // one arrival per consumer warp
      if (++slot == S) { slot = 0; parity ^= 1u; }
    }
    if (tid == 0) sh.cyc[PH_TRIDATA] += tdata;
  }
  if (wid == nwarp - 1 && lane == 0) sh.cyc[PH_TRIWAIT] += twait;
  __syncthreads();
  if (tid == 0) sh.ring_seq = seq0 + nch;
  __syncthreads();
}

// Both triangular solves on v (indexed by rows): returns the result L^{-1} then U^{-1}
// applied, in factor-label order (shared or global memory).  Block-wide.
template <typename T>
__device__ __forceinline__ const T* tri_both(const Walker& w, const Params& P, const T* v, Shared& sh) {
  const int n = w.n, tid = threadIdx.x, nt = blockDim.x;
  if (w.ctl->tri_tasks) return tri_tasks<T>(w, P, v);
  T* y = P.y_smem ? (T*)dyn_smem() : (T*)w.tv;
  if (P.tri_sf) {
    T* x2 = (T*)(dyn_smem() + P.y_half);
#pragma unroll 1
    for (int i = tid; i < n; i += nt) { y[i] = Pending<T>::value(); x2[i] = Pending<T>::value(); }
    __syncthreads();
    tri_syncfree<T>(w, P, false, v, y, sh);
    tri_syncfree<T>(w, P, true, y, x2, sh);
    return x2;
  }
  block_copy(y, v, n);
  __syncthreads();
  tri_staged<T>(w, P, false, y, sh);
  tri_staged<T>(w, P, true, y, sh);
  return y;
}

// The update chain: zs <- zs - sum_s z_hat_s c_s with c the solution of the unit lower
// system (I + G) c = d, d_s = u_s^T zs, and a copy of the result in zout (may be zs).  The
// inverse of I + G is kept (commit_move), so c is a product.  Everything a thread repeats is
// in the working precision: a conversion from FP64 holds the warp's FP64 unit like an FP64
// multiply, and one per element and update was 17 us of a 64-update FP32 apply at n = 1000
// (substitution by one warp: 27 us at 128 updates).  Block-wide, starts and ends synchronised.
template <typename T>
__device__ __forceinline__ void update_chain(const Walker& w, T* zs, T* zout, Shared& sh) {
  const int n = w.n, tid = threadIdx.x, nt = blockDim.x, mu = w.ctl->n_upd;
  const int ld = w.ld, lu = w.mu;
  if (mu == 0) {
    if (zout != zs) {
#pragma unroll 1
      for (int i = tid; i < n; i += nt) zout[i] = zs[i];
      __syncthreads();
    }
    return;
  }
  // d and c: thread (s, g) sums every G-th term of update s; the lists and the inverse are
  // stored with s fastest, so that a warp reads 32 updates side by side
  const int S = min(mu, nt), G = nt / S, sl = tid % S, g = tid / S;
  T* cT = reinterpret_cast<T*>(sh.ccoef);
  for (int step = 0; step < 2; ++step)  // d, then c
    for (int sb = 0; sb < mu; sb += S) {
      const int s = sb + sl;
      if (g < G && s < mu) {
        double acc = 0.0;
        if (step == 0) {
          const int ul = w.upd_ulen[s];
          const T* uu = (const T*)w.upd_uval + s;
          const int* uc = w.upd_ucol + s;
#pragma unroll 4
          for (int t = g; t < ul; t += G) acc += (double)uu[t * lu] * (double)zs[uc[t * lu]];
        } else {
          const double* gi = w.upd_G + s;
          if (g == 0) acc = sh.cupd[s];
#pragma unroll 4
          for (int t = g; t < s; t += G) acc += gi[(size_t)t * kMaxUpd] * sh.cupd[t];
        }
        sh.cpart[tid] = acc;
      }
      __syncthreads();
      if (tid < S && s < mu) {
        double v = 0.0;
#pragma unroll 1
        for (int q = 0; q < G; ++q) v += sh.cpart[q * S + tid];
        if (step == 0) sh.cupd[s] = v;
        else cT[s] = (T)v;
      }
      __syncthreads();
    }
  // streaming loads: the chain is read once per apply and should not push the task streams
  // out of L2
  const T* Z = (const T*)w.upd_z;
#pragma unroll 1
  for (int i = kWide<T> * tid; i < n; i += kWide<T> * nt) {
    T a[kWide<T>];
#pragma unroll
    for (int u = 0; u < kWide<T>; ++u) a[u] = zs[i + u];
#pragma unroll 1
    for (int s0 = 0; s0 < mu; s0 += kRows) {
      Wide<T> v[kRows];
#pragma unroll
      for (int q = 0; q < kRows; ++q)
        if (s0 + q < mu) v[q].load_cs(Z + (size_t)(s0 + q) * ld + i);
#pragma unroll
      for (int q = 0; q < kRows; ++q)
        if (s0 + q < mu) {
          const T c = cT[s0 + q];
#pragma unroll
          for (int u = 0; u < kWide<T>; ++u) a[u] -= v[q].v[u] * c;
        }
    }
#pragma unroll
    for (int u = 0; u < kWide<T>; ++u)
      if (i + u < n) {
        zs[i + u] = a[u];
        if (zout != zs) zout[i + u] = a[u];
      }
  }
  __syncthreads();
}

// z = M v  (v indexed by rows, z by columns of A_p).  Block-wide, ends synchronised.
// SM: v is the solve vector in shared memory (tri_vec) and the result is left in the idle
// task ring too (z_ring), so that the SpMV gathers from shared memory.
template <typename T>
__device__ __forceinline__ T* z_ring(const Params& P) { return (T*)(dyn_smem() + P.y_bytes); }
template <typename T>
__device__ __forceinline__ bool krylov_in_smem(const Walker& w, const Params& P) {
  return w.ctl->tri_tasks && (size_t)w.ld * sizeof(T) <= (size_t)P.ring_bytes;
}
template <typename T, bool SM>
__device__ __forceinline__ void precond_apply(const Walker& w, const Params& P, const T* v, T* z, Shared& sh) {
  const long long t0 = clock64();
  const T* y = SM ? tri_tasks<T>(w, P, (const T*)nullptr) : tri_both<T>(w, P, v, sh);
  const long long t1 = clock64();
  T* zs = SM ? z_ring<T>(P) : z;
  block_scatter(zs, w.perm, y, w.n);
  if (SM && threadIdx.x < w.ld - w.n) zs[w.n + threadIdx.x] = (T)0;
  __syncthreads();
  update_chain<T>(w, zs, z, sh);
  if (threadIdx.x == 0) {
    sh.cyc[PH_TRI] += t1 - t0;
    sh.cyc[PH_CHAIN] += clock64() - t1;
    sh.cnt.applies += 1;
  }
}

// Dot products <V_k, wv> for k = 0..nk-1 into out[k] and ||wv||^2 into out[nk].  A warp takes
// up to four dots at a time (one read of wv, four rows of V in flight) and reduces them
// together.  V has row stride ld; its rows and wv are zero from n to ld.  Ends synchronised.
template <typename T>
__device__ __forceinline__ void multi_dot(const T* V, int ld, int nk, const T* wv, double* out) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll 1
  for (int k0 = wid; k0 <= nk; k0 += 4 * nw) {
    T a[4] = {0, 0, 0, 0}, b[4] = {0, 0, 0, 0};
    const T* row[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) row[q] = k0 + q * nw < nk ? V + (size_t)(k0 + q * nw) * ld : wv;
    const int live = min(4, (nk - k0) / nw + 1);
#pragma unroll 4
    for (int i = kWide<T> * lane; i < ld; i += 32 * kWide<T>) {
      Wide<T> x, v[4];
      x.load(wv + i);
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (q < live) v[q].load(row[q] + i);
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (q < live)
#pragma unroll
          for (int u = 0; u < kWide<T>; u += 2) {
            a[q] += v[q].v[u] * x.v[u];
            b[q] += v[q].v[u + 1] * x.v[u + 1];
          }
    }
    double s[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) s[q] = (double)a[q] + (double)b[q];
#pragma unroll 1
    for (int o = 16; o; o >>= 1)
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (q < live) s[q] += __shfl_xor_sync(0xffffffffu, s[q], o);
    if (lane == 0)
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (q < live) out[k0 + q * nw] = s[q];
  }
  __syncthreads();
}

// wv -= sum_{k <= j} h_k V_k; returns the thread's part of ||wv||^2 (its elements are the
// chunks of kWide of every pass over the vector).
template <typename T>
__device__ __forceinline__ T subtract_basis(const T* __restrict__ V, int ld, int j, T* wv, const T* h) {
  T nrm = 0;
#pragma unroll 1
  for (int i = kWide<T> * threadIdx.x; i < ld; i += kWide<T> * blockDim.x) {
    Wide<T> w0;
    w0.load(wv + i);
    T a[kWide<T>];
#pragma unroll
    for (int u = 0; u < kWide<T>; ++u) a[u] = w0.v[u];
#pragma unroll 1
    for (int k0 = 0; k0 <= j; k0 += kRows) {
      Wide<T> v[kRows];
#pragma unroll
      for (int q = 0; q < kRows; ++q)
        if (k0 + q <= j) v[q].load(V + (size_t)(k0 + q) * ld + i);
#pragma unroll
      for (int q = 0; q < kRows; ++q)
        if (k0 + q <= j) {
          const T hk = h[k0 + q];
#pragma unroll
          for (int u = 0; u < kWide<T>; ++u) a[u] -= hk * v[q].v[u];
        }
    }
#pragma unroll
    for (int u = 0; u < kWide<T>; ++u) {
      wv[i + u] = a[u];
      nrm += a[u] * a[u];
    }
  }
  return nrm;
}

// Sum over the block of one double into *out (shared memory); thread 0's warp forms it.
// The caller synchronises before reading.
__device__ __forceinline__ void block_sum_to(double v, double* out, Shared& sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  v = warp_sum(v);
  if (lane == 0) sh.redv[wid] = v;
  __syncthreads();
  if (wid == 0) {
    double t = lane < nw ? sh.redv[lane] : 0.0;
#pragma unroll 1
    for (int o = 1; o < nw; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) *out = t;
  }
}

// Right-preconditioned GMRES(m) on A_p M d = rhs (FP64 rhs, norm beta); adds the
// correction M V y into x64.  Returns the iteration count; conv (reached rtol), the
// monitor N and the iteration at which the residual estimate first reached trig * beta (-1:
// not in this cycle; the controller's convergence test).
//
// SM: the vector that is worked on never leaves shared memory between the steps of an
// iteration -- v in the solve area, L and U in place, Q and the update chain into the idle
// task ring, the SpMV back into the solve area, Gram-Schmidt in place; V and Z are written
// once each.  Scalars (norms, rotations) are formed by one warp: FP64 instructions of the
// other warps would only queue for the SM's FP64 unit.
template <typename T, bool SM>
__device__ __forceinline__ int gmres_cycle(const Walker& w, const Params& P, double beta, double rtol, bool& conv,
                                        double& Nmon, Shared& sh, double trig, int& its_trig) {
  const int n = w.n, ld = w.ld, tid = threadIdx.x, nt = blockDim.x, m = P.m;
  T* V = (T*)w.V;
  T* Zk = (T*)w.Zk;
  T* hT = reinterpret_cast<T*>(sh.ccoef);
  if (tid == 0) {
    sh.dflag[3] = 1.0 / beta;
    sh.dflag[7] = 0.0;  // the monitor
    sh.g[0] = beta;
    sh.iflag[1] = 0;
    sh.iflag[8] = -1;
  }
  __syncthreads();
  {
    const double inv = sh.dflag[3];
    T* vec = (T*)dyn_smem();
#pragma unroll 1
    for (int i = tid; i < n; i += nt) {
      const T v = (T)(w.r64[i] * inv);
      V[i] = v;
      if (SM) vec[i] = v;
    }
  }
  __syncthreads();
  int j = 0;
#pragma unroll 1
  for (; j < m;) {
    T* vj = V + (size_t)j * ld;
    T* zj = Zk + (size_t)j * ld;
    T* vn = V + (size_t)(j + 1) * ld;
    precond_apply<T, SM>(w, P, vj, zj, sh);
    const long long ts = clock64();
    T* wv = SM ? (T*)dyn_smem() : vn;  // the solve area is free again
    // the vector that joins the basis is A M v - v: the same Krylov space, and with a good
    // preconditioner A M v is mostly v, whose removal by projection alone would cancel nearly
    // all of w and need the second Gram-Schmidt pass every time; ||A M v - v|| is the monitor
    spmv<T>(w, SM ? z_ring<T>(P) : stage_x<T>(w, P, zj), vj, wv);
    if (tid < ld - n) wv[n + tid] = (T)0;
    __syncthreads();
    const long long to = clock64();
#pragma unroll 1
    for (int pass = 0;; ++pass) {
      double* h = pass ? sh.h2 : sh.h1;
      multi_dot<T>(V, ld, j + 1, wv, h);  // projections, ||w||^2
      if (tid <= j) {
        hT[tid] = (T)h[tid];
        if (pass == 0) sh.h2[tid] = 0.0;
      }
      __syncthreads();
      block_sum_to((double)subtract_basis<T>(V, ld, j, wv, hT), &sh.dflag[0], sh);
      if (tid == 0) {
        const double nrm2 = sh.dflag[0];
        const double r = nrm2 > 0.0 ? rsqrt(nrm2) : 0.0;
        sh.dflag[1] = r;
        reinterpret_cast<T*>(&sh.dflag[2])[0] = (T)r;
        // a second pass only when the first cancelled much of w: ||w'|| < ||w|| / sqrt(2)
        // (Daniel, Gragg, Kaufman, Stewart 1976); else its coefficients are taken as zero
        sh.iflag[11] = pass == 0 && 2.0 * nrm2 < sh.h1[j + 1];
        if (pass) {
          sh.cnt.its2 += 1;
          sh.cnt.sumj2 += j + 1;
        }
      }
      __syncthreads();
      if (!sh.iflag[11]) break;
    }
    const T sc = reinterpret_cast<T*>(&sh.dflag[2])[0];
#pragma unroll 1
    for (int i = kWide<T> * tid; i < ld; i += kWide<T> * nt)
#pragma unroll
      for (int u = 0; u < kWide<T>; ++u) {
        const T x = wv[i + u] * sc;
        wv[i + u] = x;
        if (SM) vn[i + u] = x;
      }
    if (tid == 0) {
      // the new column of the Hessenberg matrix, the rotations so far, and the next one
      double* H = sh.H;
      double a0 = sh.h1[0] + sh.h2[0] + (j == 0 ? 1.0 : 0.0);  // v_j comes back on the diagonal
#pragma unroll 1
      for (int k = 0; k < j; ++k) {
        const double a1 = sh.h1[k + 1] + sh.h2[k + 1] + (k + 1 == j ? 1.0 : 0.0), c = sh.cs[k], s = sh.sn[k];
        H[k * kMaxM + j] = c * a0 + s * a1;
        a0 = c * a1 - s * a0;
      }
      const double nrm2 = sh.dflag[0], nrm = nrm2 * sh.dflag[1];
      const double q2 = a0 * a0 + nrm2;
      const double ri = q2 > 0.0 ? rsqrt(q2) : 0.0;
      const double c = q2 > 0.0 ? a0 * ri : 1.0, s = nrm * ri, g = sh.g[j];
      sh.cs[j] = c;
      sh.sn[j] = s;
      H[j * kMaxM + j] = q2 * ri;
      sh.y[j] = ri;  // 1 / H_jj
      const double gn = -s * g;
      sh.g[j + 1] = gn;
      sh.g[j] = c * g;
      sh.iflag[1] = (fabs(gn) <= rtol * beta) || nrm2 == 0.0;
      if (sh.iflag[8] < 0 && fabs(gn) <= trig * beta) sh.iflag[8] = j + 1;
      sh.dflag[7] = fmax(sh.dflag[7], sh.h1[j + 1]);
      sh.cyc[PH_SPMV] += to - ts;
      sh.cyc[PH_ORTH] += clock64() - to;
      sh.cnt.its += 1;
      sh.cnt.sumj += j + 1;
    }
    __syncthreads();
    ++j;
    if (sh.iflag[1]) break;
  }
  conv = sh.iflag[1] != 0;
  its_trig = sh.iflag[8];
  if (tid < 32) {  // H y = g, from the last column back; lane l holds rows l and l + 32
    const double* H = sh.H;
    double g0 = tid < j ? sh.g[tid] : 0.0, g1 = tid + 32 < j ? sh.g[tid + 32] : 0.0;
#pragma unroll 1
    for (int k = j - 1; k >= 0; --k) {
      const double yk = __shfl_sync(0xffffffffu, k < 32 ? g0 : g1, k & 31) * sh.y[k];
      if (tid < k) g0 -= H[tid * kMaxM + k] * yk;
      if (tid + 32 < k) g1 -= H[(tid + 32) * kMaxM + k] * yk;
      if (tid == 0) hT[k] = (T)yk;
    }
    if (tid == 0) sh.dflag[3] = sqrt(sh.dflag[7]);
  }
  __syncthreads();
  Nmon = sh.dflag[3];
#pragma unroll 1
  for (int i = kWide<T> * tid; i < n; i += kWide<T> * nt) {
    T a[kWide<T>] = {};
#pragma unroll 1
    for (int k0 = 0; k0 < j; k0 += kRows) {
      Wide<T> v[kRows];
#pragma unroll
      for (int q = 0; q < kRows; ++q)
        if (k0 + q < j) v[q].load(Zk + (size_t)(k0 + q) * ld + i);
#pragma unroll
      for (int q = 0; q < kRows; ++q)
        if (k0 + q < j) {
          const T yk = hT[k0 + q];
#pragma unroll
          for (int u = 0; u < kWide<T>; ++u) a[u] += yk * v[q].v[u];
        }
    }
#pragma unroll
    for (int u = 0; u < kWide<T>; ++u)
      if (i + u < n) w.x64[i + u] += (double)a[u];
  }
  if (tid == 0) { sh.cnt.cycles += 1; sh.cnt.sumx += j; }
  __syncthreads();
  return j;
}
// Thread 0: the phase cycles and algorithmic bytes gathered in shared memory into the
// walker's statistics (one read-modify-write of global memory per phase and iteration
// cost about 3 us an iteration).  Before anything that changes the counts' factors.
template <typename T>
__device__ __forceinline__ void flush_counts(const Walker& w, Shared& sh) {
  if (threadIdx.x != 0) return;
  Ctl* c = w.ctl;
  const SolveCounts k = sh.cnt;
  const double n = w.n, b = sizeof(T);
  double by = 0.0;
  // triangular solves: factor values + indices, diagonal, v read, z write, the row records;
  // update chain: z_hat vectors, sparse u vectors, z read + write
  by += k.applies * (c->nnz_LU * (b + 4.0) + n * (3.0 * b + 8.0));
  if (c->n_upd > 0) by += k.applies * (c->n_upd * n * b + c->upd_nnz * (b + 4.0) + 2.0 * n * b);
  // SpMV: values + indices, x read, y write; the first Gram-Schmidt pass: projections
  // (V_0..V_j and w read) and update (V_0..V_j and w read, w written), normalisation
  by += k.its * (c->nnz_A * (b + 4.0) + n * (2.0 * b + 4.0)) + n * b * (2.0 * k.sumj + 6.0 * k.its);
  by += n * b * (2.0 * k.sumj2 + 3.0 * k.its2);       // second passes
  by += n * (k.sumx * b + 16.0 * k.cycles);            // Zk y, x read + write
  by += k.resid * (c->nnz_A * 12.0 + n * 24.0);        // FP64 A, x read, r write, row lengths
  c->alg_bytes += by;
#pragma unroll 1
  for (int i = 0; i < 16; ++i) {
    c->cyc[i] += sh.cyc[i];
    sh.cyc[i] = 0;
  }
  sh.cnt = SolveCounts{};
}

// r64 = e_brow - A_p x64 (FP64), and into sh.dflag: [4] ||r64||_2, [5] ||x64||_2, [6] the
// ratio 1 + u^T x64 over the u list in shared memory.  The three sums are reduced together
// and the scalars formed by one thread.  Ends synchronised.
__device__ __forceinline__ void residual64(const Walker& w, int brow, Shared& sh) {
  const int n = w.n, nt = blockDim.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
  const long long t0 = clock64();
  double s[3] = {0.0, 0.0, 0.0};
  NextRow at(w, tid);
#pragma unroll 1
  for (int p = tid; p < n; p += nt) {  // slots in order (see spmv)
    const NextRow next(w, p + nt);
    const double xp = load_now(w.x64 + p);
    const double acc = row_dot<double, double>(w, p, at.len, w.x64);
    const double rr = (at.row == brow ? 1.0 : 0.0) - acc;
    w.r64[at.row] = rr;
    s[0] += rr * rr;
    s[1] += xp * xp;
    at = next;
  }
#pragma unroll 1
  for (int t = tid; t < sh.ulen; t += nt) s[2] += sh.uval[t] * w.x64[sh.ucol[t]];
#pragma unroll
  for (int o = 16; o; o >>= 1)
#pragma unroll
    for (int q = 0; q < 3; ++q) s[q] += __shfl_xor_sync(0xffffffffu, s[q], o);
  if (lane == 0)
#pragma unroll
    for (int q = 0; q < 3; ++q) sh.red[8 * q + wid] = s[q];
  __syncthreads();
  if (wid == 0) {
    double v = (lane & 7) < nw && lane < 24 ? sh.red[lane] : 0.0;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) sh.dflag[4] = sqrt(v);
    if (lane == 8) sh.dflag[5] = sqrt(v);
    if (lane == 16) sh.dflag[6] = 1.0 + v;
    if (lane == 0) {
      sh.cyc[PH_RESID] += clock64() - t0;
      sh.cnt.resid += 1;
    }
  }
  __syncthreads();
}

struct SolveOut {
  double ratio;
  int its1;          // iterations of the first cycle
  bool conv1;        // the first cycle reached its tolerance
  int its_trig;      // iterations (all cycles) until the residual reached Params::trig_rtol; -1: never
  double N;
  int passes;
  int total_its;
  int status;
};

// The solve of a move: a first pass from x = 0 (whose iterations, convergence and monitor the
// controller reads), then refinement.  The ratio error after a pass is u^T A^{-1} r.  It is
// predicted as the larger of |u^T d_j| ||r_j|| / ||r_{j-1}|| (the last correction scaled by
// the last residual reduction) and ||u|| ||x|| ||r_j|| (||x|| ~ ||A^{-1} e_r|| as a norm
// estimate), and passes continue until it is <= ratio_tol max(|ratio|, 1e-3).  Each
// pass asks the inner GMRES for only the reduction the goal needs (never below rtol).
// One call site of everything it inlines: calls would keep the loops' registers in local
// memory, which the full shared memory leaves no L1 for.
template <typename T, bool SM>
__device__ __noinline__ void solve_passes(const Walker& w, const Params& P, int brow, double rtol, int max_passes,
                                          SolveOut& out, Shared& sh) {
  const int tid = threadIdx.x;
  SolveOut o;
  {
    const int n = w.n;
#pragma unroll 1
    for (int i = tid; i < n; i += blockDim.x) {
      w.x64[i] = 0.0;
      w.r64[i] = i == brow ? 1.0 : 0.0;
    }
    double usq = 0.0;
#pragma unroll 1
    for (int t = tid; t < sh.ulen; t += blockDim.x) usq += sh.uval[t] * sh.uval[t];
    block_sum_to(usq, &sh.red[24], sh);
    if (tid == 0) {  // sh.red[24]: ||u||, [25]: previous ratio, [26]: previous ||r||
      sh.red[24] = sqrt(sh.red[24]);
      sh.red[25] = 1.0;
      sh.red[26] = 1.0;
    }
    __syncthreads();
  }
  o.status = ST_OK;
  o.passes = 0;
  o.total_its = 0;
  o.its_trig = -1;
  double beta = 1.0, tol = rtol, trig = P.trig_rtol;
  const long long t0 = clock64();
  long long t1 = t0;
  for (;;) {
    bool conv = false;
    double N = 0.0;
    int at = -1;
    const int its = gmres_cycle<T, SM>(w, P, beta, tol, conv, N, sh, trig, at);
    if (o.its_trig < 0 && at > 0) o.its_trig = o.total_its + at;
    if (o.passes == 0) {
      o.its1 = its;
      o.conv1 = conv;
      o.N = N;
      t1 = clock64();
    }
    o.total_its += its;
    o.passes += 1;
    residual64(w, brow, sh);
    // ||e_r|| = 1: the FP64 residual norm is also the relative residual
    const double rn = sh.dflag[4];
    if (o.its_trig < 0 && rn <= P.trig_rtol) o.its_trig = o.total_its;
    if (tid == 0) {
      const double ratio = sh.dflag[6];
      const double delta = fabs(ratio - sh.red[25]);
      const double pred = fmax(delta * rn / sh.red[26], sh.red[24] * sh.dflag[5] * rn);
      const double goal = P.ratio_tol * fmax(fabs(ratio), 1e-3);
      sh.iflag[10] = pred <= goal || rn == 0.0;
      sh.red[27] = fmin(fmax(0.1 * goal / pred, rtol), 0.1);  // the reduction to ask for
      sh.red[28] = P.trig_rtol / rn;
      sh.red[25] = ratio;
      sh.red[26] = rn;
    }
    __syncthreads();
    if (sh.iflag[10]) break;
    if (o.passes >= max_passes) {
      if (rn > 1e-6) o.status = ST_NOCONV;
      break;
    }
    beta = rn;
    tol = sh.red[27];
    trig = sh.red[28];
  }
  o.ratio = sh.dflag[6];
  out = o;
  if (tid == 0) {
    sh.cyc[PH_FIRST] += t1 - t0;
    sh.cyc[PH_REFINE] += clock64() - t1;
  }
  __syncthreads();
}
template <typename T>
__device__ __forceinline__ void solve_move(const Walker& w, const Params& P, int brow, double rtol, int max_passes,
                                           SolveOut& o, Shared& sh) {
  if (krylov_in_smem<T>(w, P)) solve_passes<T, true>(w, P, brow, rtol, max_passes, o, sh);
  else solve_passes<T, false>(w, P, brow, rtol, max_passes, o, sh);
}

}  // namespace vmc
