// vmc_blocks.cuh -- blocked triangular solves (a partitioned inverse of each factor).
//
// The rows of L (of U, from the last row up) are taken in blocks of B consecutive factor
// labels.  With O_b the entries of block b outside its diagonal block D_b, a block is
// solved in two steps whose rows are independent:
//   A:  s_i = v_r - sum_{c outside} O_rc y_c            (sparse rows of the factor)
//   B:  y_r = sum_i (D_b^{-1})_{ri} s_i                 (sparse rows of the inverse)
// The inverse of a diagonal block is formed once per factorisation in FP64 and rounded
// once to the working precision; the operator is that of row-by-row substitution in exact
// arithmetic.  A block without entries inside D_b needs step A alone.
//
// What bounds it, and the split.  Substitution is a chain: measured on GB300, a CTA barrier
// costs 22-46 cycles, a shared-memory load 30, a lane-group reduction step 30 (FP32) or 105
// (FP64), and an FP64 instruction of a warp holds its scheduler's FP64 unit for 64 cycles.
// The number of steps decides in FP32, the number of FP64 instructions in FP64.  Blocks of
// 64 rows at n = 1000 (20 sweeps from the start, fill limit 32) take 2 x 32 steps over
// 78 k entries; merging levels into groups with every row expanded to earlier groups took
// 114 steps over 98 k entries, level by level 405 steps over 57 k.
//
// Layout.  Every warp has a stream of its own: its tasks of every step, L then U.  A task
// holds 8 entries for each of the warp's lanes -- a word a lane {destination, lanes of the
// row, barriers after the task}, 8 16-bit sources, 8 values -- and a row takes as many
// neighbouring lanes as its entries need, up to 32, widest rows first.  Every task has the same size and every lane
// copies its own 16 bytes of it (cp.async) up to four tasks ahead into shared memory, and
// from there into registers one task ahead: no barrier, no release and no other warp
// between a warp and its data.  (A ring of 1 KB bulk copies per warp took 62 us FP32 and
// 112 us FP64 for L and U at that state, 950 cycles a step waiting for, releasing and
// refilling pages; loading two tasks ahead into registers 28 and 99 us, four ahead 48 us:
// the loads share too few scoreboards.)
#pragma once
#include "vmc_device.cuh"

namespace vmc {

// 16-byte asynchronous copy to shared memory that bypasses L1 (the factor CTA rewrites the
// streams) and asks to stay in L2, where the next apply finds it.
__device__ __forceinline__ void cp16(unsigned dst, const void* src, unsigned long long pol) {
  asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "l"(pol) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ void values_from(const unsigned char* p, float* q) {
#pragma unroll
  for (int k = 0; k < kLaneEntries / 4; ++k) {
    const float4 v = *reinterpret_cast<const float4*>(p + 512 * k);
    q[4 * k] = v.x; q[4 * k + 1] = v.y; q[4 * k + 2] = v.z; q[4 * k + 3] = v.w;
  }
}
__device__ __forceinline__ void values_from(const unsigned char* p, double* q) {
#pragma unroll
  for (int k = 0; k < kLaneEntries / 2; ++k) {
    const double2 v = *reinterpret_cast<const double2*>(p + 512 * k);
    q[2 * k] = v.x; q[2 * k + 1] = v.y;
  }
}

__device__ __forceinline__ void bar_all() { asm volatile("bar.sync 0;" ::: "memory"); }

template <typename T>
__device__ __forceinline__ void run_tasks(const Walker& w, const Params& P, const T* v, T* vec) {
  const int D = tasks_ahead<T>(P) >= 4 ? 4 : 2;  // tasks in flight
  constexpr int TB = task_bytes((int)sizeof(T));
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int2 tl = w.lchunk[wid], tu = w.uchunk[wid];
  const unsigned char* src = w.lstream + tl.x + 16 * lane;
  const int nl = tl.y & 0xffffff, lead_l = tl.y >> 24, lead_u = tu.y >> 24;
  const int nt = nl + (tu.y & 0xffffff);
  const unsigned long long pol = l2_policy_evict_last();
  const unsigned char* ring = dyn_smem() + P.y_bytes + (size_t)wid * D * TB;
  const unsigned ring32 = smem_u32(ring) + 16 * lane;
  auto issue = [&](int t, int slot, int lanes) {  // only the lanes that hold a row
    if (t < nt) {
      const unsigned char* p = src + (size_t)t * TB;
      const unsigned d = ring32 + slot * TB;
      if (lane < 8) cp16(d, p, pol);
      if (lane < lanes) {
#pragma unroll
        for (int k = 0; k < (TB - 128) / 512; ++k) cp16(d + 128 + 512 * k, p + 128 + 512 * k, pol);
      }
    }
    cp_commit();
  };
#pragma unroll 1
  for (int d = 0; d < D; ++d) issue(d, d, 32);
  if (v) block_copy(vec, v, w.n);  // else v is in the solve vector already
  unsigned word = 0;
  uint4 c = make_uint4(0u, 0u, 0u, 0u);
  T q[kLaneEntries];
  auto fetch = [&](int slot) {  // the task that has landed in slot, into registers
    if (D == 4) cp_wait<3>();
    else cp_wait<1>();
    __syncwarp();
    const unsigned char* p = ring + slot * TB;
    word = *reinterpret_cast<const unsigned*>(p + 4 * lane);
    c = *reinterpret_cast<const uint4*>(p + 128 + 16 * lane);
    if (!(word >> 31)) c = make_uint4(0u, 0u, 0u, 0u);  // a lane without a row: nothing was copied for it
    values_from(p + 640 + 16 * lane, q);
  };
  if (nt > 0) fetch(0);
  __syncthreads();
#pragma unroll 1
  for (int i = 0; i < lead_l; ++i) bar_all();
  int slot = 0;
#pragma unroll 1
  for (int t = 0; t < nt; ++t) {
    if (t == nl)
#pragma unroll 1
      for (int i = 0; i < lead_u; ++i) bar_all();
    const int after = (int)((word >> 16) & 31u), nb = (int)((word >> 22) & 15u), dst = (int)(word & 0xffffu);
    const bool first = (word & (1u << 21)) != 0;
    const int widest = __shfl_sync(0xffffffffu, after, 0);
    T a = q[0] * vec[c.x & 0xffffu], b = q[1] * vec[c.x >> 16];
    a += q[2] * vec[c.y & 0xffffu]; b += q[3] * vec[c.y >> 16];
    a += q[4] * vec[c.z & 0xffffu]; b += q[5] * vec[c.z >> 16];
    a += q[6] * vec[c.w & 0xffffu]; b += q[7] * vec[c.w >> 16];
    T part = a + b;
    issue(t + D, slot, (int)((word >> 26) & 31u) + 1);  // every lane has read the slot: its own part above, the words at the shuffle
    slot = slot + 1 == D ? 0 : slot + 1;
    fetch(slot);
#pragma unroll 1
    for (int o = 1; o <= widest; o <<= 1) {  // sum over the row's lanes into its first
      const T p2 = __shfl_down_sync(0xffffffffu, part, o);
      if (o <= after) part += p2;
    }
    if (first) vec[dst] = part;
#pragma unroll 1
    for (int i = 0; i < nb; ++i) bar_all();
  }
  if (nl == nt)  // no task in U's steps
#pragma unroll 1
    for (int i = 0; i < lead_u; ++i) bar_all();
  __syncthreads();
}

// x := U^{-1} L^{-1} v on the walker's block streams: returns the solve vector (shared
// memory, factor-label order).  Block-wide, ends synchronised.  Every warp passes the same
// number of barriers: one per step, counted in the tasks.
template <typename T>
__device__ __forceinline__ T* tri_tasks(const Walker& w, const Params& P, const T* v) {
  T* vec = (T*)dyn_smem();
  run_tasks<T>(w, P, v, vec);
  return vec;
}

// ---------------------------------------------------------------------------
// Building the streams, once per factorisation (block-wide).
// ---------------------------------------------------------------------------

// Lanes of a row of len entries.
__device__ __forceinline__ int row_lanes(int len) { return max(1, (len + kLaneEntries - 1) / kLaneEntries); }

// One warp: the lanes of the m <= 128 rows of one step, lens in len[0..3] (row i = lane + 32 q):
// first fit, widest rows first, into tasks of 32 lanes; pos = first lane | 32 x task.  Returns
// the number of tasks, or -1 when a row needs more than 32 lanes or the step more than 128
// tasks.
__device__ __forceinline__ int plan_step(const int (&len)[4], int m, int (&pos)[4]) {
  const int lane = threadIdx.x & 31;
  int room[4], tasks = 0, most = 0;  // task lane + 32 q: free lanes
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    room[q] = 32;
    if (lane + 32 * q < m) most = max(most, row_lanes(len[q]));
  }
  most = warp_max_int(most);
  if (most > 32) return -1;
#pragma unroll 1
  for (int g = most; g > 0; --g) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      unsigned rows = __ballot_sync(0xffffffffu, lane + 32 * q < m && row_lanes(len[q]) == g);
      while (rows) {
        const int src = __ffs(rows) - 1;
        rows &= rows - 1;
        int at = -1;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const unsigned f = __ballot_sync(0xffffffffu, room[k] >= g);
          if (at < 0 && f) {
            const int t = __ffs(f) - 1;
            at = 32 * (t + 32 * k) + 32 - __shfl_sync(0xffffffffu, room[k], t);
            if (lane == t) room[k] -= g;
          }
        }
        if (at < 0) return -1;
        tasks = max(tasks, (at >> 5) + 1);
        if (lane == src) pos[q] = at;
      }
    }
  }
  return tasks;
}

// Builds the task streams of both factors into w.lstream (a region of 2 x w.sbytes that
// w.ustream ends): steps of blocks, or with trisolve_group <= 1 a step per level (its rows
// are independent and read only earlier levels; w.l/u_lvl_ptr and _rows hold them), in
// parts of at most 128 rows.  w.lchunk[warp] = {offset, L tasks | barriers before the first << 24},
// w.uchunk[warp].y the same for U; the step counts go to ctl->nchunk_l / nchunk_u.  Returns
// false (block-uniform) when a row needs more than a warp's lanes or a warp's stream would
// not fit its share of the region: the caller then builds the level-by-level streams.
template <typename T>
__device__ __noinline__ bool build_tasks(const Walker& w, const Params& P, Shared& sh) {
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
  const int n = w.n, capLU = w.capLU, EX = w.exmax, B = block_rows(w, P), nb = (n + B - 1) / B;
  const bool by_level = P.tri_group <= 1;
  constexpr int tsz = (int)sizeof(T);
  constexpr int TB = task_bytes(tsz);
  const int share = (int)min((2 * w.sbytes / nw) & ~(size_t)127, (size_t)0x7fffff80 / 8);
  // scratch: first task of (step, warp) in the warp's stream; first task and barriers after
  // it per step and warp
  int* tbase = (int*)w.seg_meta;
  int* posA = w.gP;  // lanes of every row in step A (or its level's), in step B
  int* posB = w.gQ;
  int* stepof = w.wpos;  // by level: the step of every row
  const int room = 4 * n + 4;  // entries of tbase and of tbar
  int* tbar = tbase + 4 * (size_t)n + 4;
  int ntask = 0;  // thread w < nw: warp w's tasks so far
  // task t of step s goes to warp (t + s) % nw: no warp waits for more than nw steps
  auto warp_tasks = [&](int s, int wq) {
    const int t0 = (wq - s % nw + nw) % nw, T_ = w.chunk_meta[s].w;
    return t0 < T_ ? (T_ - 1 - t0) / nw + 1 : 0;
  };
  if (tid == 0) sh.iflag[10] = 0;
#pragma unroll 1
  for (int upper = 0; upper < 2; ++upper) {
    const int* flen = upper ? w.u_len : w.l_len;
    const int* fcol = upper ? w.u_col : w.l_col;
    const double* fval = upper ? w.u_val64 : w.l_val64;
    const int* lptr = upper ? w.u_lvl_ptr : w.l_lvl_ptr;
    const int* lrows = upper ? w.u_lvl_rows : w.l_lvl_rows;
    const int nlev = upper ? w.ctl->nlev_u : w.ctl->nlev_l;
    int nst;
    // rows of block b are [lo, hi); local index i in solve order
    auto lo_of = [&](int b) { return upper ? max(0, n - (b + 1) * B) : b * B; };
    auto hi_of = [&](int b) { return upper ? n - b * B : min(n, (b + 1) * B); };
    if (by_level) {
#pragma unroll 1
      for (int l = tid; l < nlev; l += nt) w.lvl_cur[l] = (lptr[l + 1] - lptr[l] + kMaxBlk - 1) / kMaxBlk;
      __syncthreads();
      nst = block_scan_inplace(w.lvl_cur, nlev, sh);  // first step of every level
      if ((size_t)nst * nw > (size_t)room || nst > n) return false;
#pragma unroll 1
      for (int l = wid; l < nlev; l += nw)
#pragma unroll 1
        for (int q0 = lptr[l], s = w.lvl_cur[l]; q0 < lptr[l + 1]; q0 += kMaxBlk, ++s) {
          const int m = min(kMaxBlk, lptr[l + 1] - q0);
          int len[4], pos[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int i = lane + 32 * q;
            len[q] = i < m ? 1 + flen[lrows[q0 + i]] : 0;
            pos[q] = 0;
          }
          const int tasks = plan_step(len, m, pos);
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (lane + 32 * q < m) {
              const int r = lrows[q0 + lane + 32 * q];
              posA[r] = pos[q];
              stepof[r] = s;
            }
          if (lane == 0) {
            w.chunk_meta[s] = make_int4(q0, m, 0, max(tasks, 0));
            if (tasks < 0) sh.iflag[10] = 1;
          }
        }
    } else {
      // 1. entries of every row inside its diagonal block: {entry, local column}, and the counts
#pragma unroll 1
      for (int r = wid; r < n; r += nw) {
        const int b = upper ? (n - 1 - r) / B : r / B;
        const int lo = lo_of(b), hi = hi_of(b), L = flen[r];
        int nin = 0;
#pragma unroll 1
        for (int t0 = 0; t0 < L; t0 += 32) {
          const int t = t0 + lane;
          const int c = t < L ? fcol[(size_t)r * capLU + t] : -1;
          const bool in = c >= lo && c < hi;
          const unsigned m = __ballot_sync(0xffffffffu, in);
          if (in) w.ex_col[(size_t)r * EX + nin + __popc(m & lanemask_lt())] = t | ((upper ? hi - 1 - c : c - lo) << 16);
          nin += __popc(m);
        }
        if (lane == 0) w.ex_len[r] = nin;
      }
      __syncthreads();
      // 2. inverses of the diagonal blocks, a thread per column: X(i, j) of block b at
      //    ex_val[row of i][j]
#pragma unroll 1
      for (int idx = tid; idx < nb * B; idx += nt) {
        const int b = idx / B, j = idx - b * B;
        const int lo = lo_of(b), hi = hi_of(b), m = hi - lo;
        if (j >= m) continue;
#pragma unroll 1
        for (int i = 0; i < m; ++i) {
          const int r = upper ? hi - 1 - i : lo + i;
          const double d = upper ? w.u_dinv64[r] : 1.0;
          double xv = 0.0;
          if (i == j) {
            xv = d;
          } else if (i > j) {
            const int k = w.ex_len[r];
            double acc = 0.0;
#pragma unroll 1
            for (int t = 0; t < k; ++t) {
              const int e = w.ex_col[(size_t)r * EX + t], li = e >> 16;
              if (li >= j)
                acc += fval[(size_t)r * capLU + (e & 0xffff)] * w.ex_val[(size_t)(upper ? hi - 1 - li : lo + li) * EX + j];
            }
            xv = acc != 0.0 ? -d * acc : 0.0;
          }
          w.ex_val[(size_t)r * EX + j] = xv;
        }
      }
      __syncthreads();
      // 3. steps of every block: 2, or 1 when no row has an entry inside its diagonal block (0
      //    for L when there is none outside either)
#pragma unroll 1
      for (int b = wid; b < nb; b += nw) {
        int in = 0, out = 0;
#pragma unroll 1
        for (int r = lo_of(b) + lane; r < hi_of(b); r += 32) {
          in |= w.ex_len[r];
          out |= flen[r] - w.ex_len[r];
        }
        const bool any_in = __any_sync(0xffffffffu, in != 0), any_out = __any_sync(0xffffffffu, out != 0);
        if (lane == 0) w.lvl_nchunk[b] = any_in ? 2 : (any_out || upper ? 1 : 0);
      }
      __syncthreads();
#pragma unroll 1
      for (int b = tid; b < nb; b += nt) w.lvl_cur[b] = w.lvl_nchunk[b];
      __syncthreads();
      nst = block_scan_inplace(w.lvl_cur, nb, sh);  // first step of every block
      // 4. lanes of every row
#pragma unroll 1
      for (int b = wid; b < nb; b += nw) {
        const int lo = lo_of(b), m = hi_of(b) - lo, ns = w.lvl_nchunk[b];
#pragma unroll 1
        for (int ph = 0; ph < ns; ++ph) {
          int len[4], pos[4];
  #pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int i = lane + 32 * q;
            len[q] = 0;
            pos[q] = 0;
            if (i < m) {
              const int r = lo + i;
              if (ph == 0) {
                len[q] = 1 + flen[r] - w.ex_len[r];
              } else {
                int k = 0;
#pragma unroll 1
                for (int j = 0; j < m; ++j) k += w.ex_val[(size_t)r * EX + j] != 0.0;
                len[q] = k;
              }
            }
          }
          const int tasks = plan_step(len, m, pos);
  #pragma unroll
          for (int q = 0; q < 4; ++q)
            if (lane + 32 * q < m) (ph == 0 ? posA : posB)[lo + lane + 32 * q] = pos[q];
          if (lane == 0) {
            w.chunk_meta[w.lvl_cur[b] + ph] = make_int4(lo, m, ph, max(tasks, 0));
            if (tasks < 0) sh.iflag[10] = 1;
          }
        }
      }
    }
    __syncthreads();
    if (sh.iflag[10]) return false;
    // 5. thread w: the places of warp w's tasks in its stream and the barriers after them
    const int before = ntask;
    int lead = nst;
    if (tid < nw) {
#pragma unroll 1
      for (int s = 0; s < nst; ++s) {
        tbase[(size_t)s * nw + tid] = ntask;
        ntask += warp_tasks(s, tid);
      }
#pragma unroll 1
      for (int s = nst - 1; s >= 0; --s) {
        tbar[(size_t)s * nw + tid] = lead - s;
        if (warp_tasks(s, tid) > 0) lead = s;
      }
      (upper ? w.uchunk : w.lchunk)[tid] = make_int2(tid * share, (ntask - before) | (lead << 24));
    }
    if (block_max_int(tid < nw ? ntask : 0, sh) > share / TB) return false;
    // 6. fill: empty lanes, then the rows
    auto task_at = [&](int s, int t) {
      const int wq = (t + s) % nw;
      return w.lstream + (size_t)wq * share + (size_t)(tbase[(size_t)s * nw + wq] + t / nw) * TB;
    };
    // a lane's word: destination (16 bits), lanes of the row after it (5), first lane of the row
    // (1), barriers after the task -- only after the warp's last one of the step -- (4), lanes
    // in use of the task to be copied next, less one (5), lane in use (1)
    auto bars_after = [&](int s, int t) {
      return (unsigned)(t + nw >= w.chunk_meta[s].w ? tbar[(size_t)s * nw + (t + s) % nw] : 0) << 22;
    };
#pragma unroll 1
    for (int s = 0; s < nst; ++s)
#pragma unroll 1
      for (int t = wid; t < w.chunk_meta[s].w; t += nw) {
        unsigned char* base = task_at(s, t);
        ((unsigned*)base)[lane] = bars_after(s, t);
        ((uint4*)(base + 128))[lane] = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll 1
        for (int k = 0; k < kLaneEntries * tsz / 16; ++k) ((uint4*)(base + 640 + 512 * k))[lane] = make_uint4(0u, 0u, 0u, 0u);
      }
    __syncthreads();
#pragma unroll 1
    for (int r = wid; r < n; r += nw) {
      const int b = upper ? (n - 1 - r) / B : r / B;
      const int lo = by_level ? r : lo_of(b), hi = by_level ? r + 1 : hi_of(b), m = hi - lo;
      const int ns = by_level ? 1 : w.lvl_nchunk[b], s0 = by_level ? stepof[r] : w.lvl_cur[b];
      const int li = upper ? hi - 1 - r : r - lo;
#pragma unroll 1
      for (int ph = 0; ph < ns; ++ph) {
        const int s = s0 + ph;
        const int p = (ph == 0 ? posA : posB)[r], l0 = p & 31;
        unsigned char* base = task_at(s, p >> 5);
        int k = 0, G = 0;
        auto put = [&](int i, int col, double val) {  // entry i of the row: lane i % G, place i / G
          const int e = i / G, ln = l0 + (i - e * G), o = e * tsz;
          ((unsigned short*)(base + 128 + 16 * ln))[e] = (unsigned short)col;
          *(T*)(base + 640 + 512 * (o >> 4) + 16 * ln + (o & 15)) = (T)val;
        };
        // step A of a block with a step B writes s_i (after the solve vector), else y_r
        const int dst = ph == 0 && ns == 2 ? n + li : r;
        const int self = ph == 0 ? r : n + li;
        if (ph == 0) {
          G = row_lanes(1 + flen[r] - (by_level ? 0 : w.ex_len[r]));
          const double d = ns == 1 && upper ? w.u_dinv64[r] : 1.0;
          if (lane == 0) put(0, r, d);
          k = 1;
          const int L = flen[r];
#pragma unroll 1
          for (int t0 = 0; t0 < L; t0 += 32) {
            const int t = t0 + lane;
            const int c = t < L ? fcol[(size_t)r * capLU + t] : -1;
            const bool outside = c >= 0 && (c < lo || c >= hi);
            const unsigned mk = __ballot_sync(0xffffffffu, outside);
            if (outside) put(k + __popc(mk & lanemask_lt()), c, -d * fval[(size_t)r * capLU + t]);
            k += __popc(mk);
          }
        } else {
          int cnt = 0;
#pragma unroll 1
          for (int j0 = 0; j0 < m; j0 += 32)
            cnt += __popc(__ballot_sync(0xffffffffu, j0 + lane < m && w.ex_val[(size_t)r * EX + j0 + lane] != 0.0));
          G = row_lanes(cnt);
#pragma unroll 1
          for (int j0 = 0; j0 < m; j0 += 32) {
            const int j = j0 + lane;
            const double xv = j < m ? w.ex_val[(size_t)r * EX + j] : 0.0;
            const unsigned mk = __ballot_sync(0xffffffffu, xv != 0.0);
            if (xv != 0.0) put(k + __popc(mk & lanemask_lt()), n + j, xv);
            k += __popc(mk);
          }
        }
#pragma unroll 1
        for (int i = k + lane; i < kLaneEntries * G; i += 32) put(i, self, 0.0);  // padding reads the row's own value
        if (lane < G)
          ((unsigned*)base)[l0 + lane] = (unsigned)dst | ((unsigned)(G - 1 - lane) << 16) | (lane == 0 ? 1u << 21 : 0u) |
                                         bars_after(s, p >> 5) | (1u << 31);
      }
    }
    __syncthreads();
    if (tid == 0) (upper ? w.ctl->nchunk_u : w.ctl->nchunk_l) = nst;
  }
  // the copy of the task `ahead` places on is issued with a task: its lanes in use
  const int ahead = tasks_ahead<T>(P) >= 4 ? 4 : 2;
  int used = 0;  // lanes in use of this warp's tasks
  {
    const int mine = (w.lchunk[wid].y & 0xffffff) + (w.uchunk[wid].y & 0xffffff);
    unsigned* base = (unsigned*)(w.lstream + (size_t)wid * share);
#pragma unroll 1
    for (int t = 0; t < mine; ++t) {
      const int lanes = __popc(__ballot_sync(0xffffffffu, base[(size_t)t * (TB / 4) + lane] >> 31));
      used += lanes;
      if (t >= ahead) base[(size_t)(t - ahead) * (TB / 4) + lane] |= (unsigned)(lanes - 1) << 26;
    }
    used = 128 * mine + used * (16 + kLaneEntries * tsz);
  }
  const double bytes = block_sum(lane == 0 ? (double)used : 0.0, sh);
  if (tid == 0) w.ctl->stream_bytes = (long long)bytes;
  __syncthreads();
  return true;
}

}  // namespace vmc
