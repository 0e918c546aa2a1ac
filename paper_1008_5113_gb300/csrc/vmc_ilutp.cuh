// vmc_ilutp.cuh -- ILUTP with the rows in flight on several warps.
//
// The factorisation of ilutp_warp (same elimination, drop, fill and pivot rules, in the same
// order for every entry, so the same factors bit for bit) with row r on warp r mod W.  Rows
// only wait for the labels they need: a pivot of row k permutes labels >= k, so while rows
// d, d + 1, ... are unfinished the labels below d are final.  A row is kept by original
// column, eliminates its entries with final labels in increasing order, and, when it has
// none left, waits for the next row to finish and looks whether it holds that row's pivot
// column.  A row is published -- U part, pivot -- as soon as its last predecessor's
// contribution is in; its L part is selected and written after that, off the chain.
//
// What bounds it: one warp spends about 150 k cycles a row at n = 1000 (157 eliminations, a
// U row, the drop and fill rules) almost all of it latency: shared-memory and L2 round trips
// and FP64 instructions of 64 cycles.  Rows in flight overlap these; the chain that remains
// is, per row, the predecessor's elimination, the U selection and the pivot.  Measured, one
// walker's ILUTP: n = 216 9.3 -> 1.6 ms, n = 1000 (fill limit 32, 20 sweeps from the start)
// 120 -> 17 ms, n = 4096 316 -> 53 ms (380 ms where two CTAs shared an SM).
//
// Shared memory: the permutation and its inverse in 16 bits (4 n bytes), and per warp a map
// from column to slot (2 n), a bitmap of pending labels, and the slots: column, value (the
// first kPipeVals in shared memory, the rest in global scratch), selection scratch.  n = 1000
// fits 8 warps, n = 4096 seven of a walker alone on its SM and two of walkers that share it.
#pragma once
#include "vmc_select.cuh"

namespace vmc {

constexpr int kPipeVals = 1024;  // slots of a row whose values are in shared memory

struct PipePlan {
  int warps;
  unsigned o_perm, o_ip, o_warp, per_warp;                          // bytes
  unsigned o_bits, o_sum, o_wpos, o_nz, o_val, o_sel, o_selk, o_hist, o_bnd;  // within a warp's part
};
template <typename W>
__device__ __forceinline__ PipePlan ilu_pipe_plan(int n, size_t dbytes, int nwarps) {
  PipePlan pl{};
  pl.warps = 0;
  if (n >= 0xffff) return pl;
  const unsigned nwords = (n + 31) >> 5, nsum = (nwords + 31) >> 5;
  pl.o_perm = 0;
  pl.o_ip = pad16(2 * n);
  pl.o_warp = 2 * pad16(2 * n);
  unsigned o = 0;
  pl.o_val = o; o += (unsigned)sizeof(W) * min(kPipeVals, pad16(n));
  pl.o_bits = o; o += 4u * pad4(nwords);
  pl.o_sum = o; o += 4u * pad4(nsum);
  pl.o_hist = o; o += 4u * 64;
  pl.o_wpos = o; o += pad16(2 * n);
  pl.o_nz = o; o += 2u * min(kMaxRowNZ, pad16(n));
  pl.o_sel = o; o += 2u * min(kMaxSel, pad16(n));
  pl.o_bnd = o; o += 2u * 256;
  pl.o_selk = o; o += pad16(min(kMaxSel, n));
  pl.per_warp = (unsigned)pad16((int)o);
  if (pl.o_warp + pl.per_warp > dbytes) return pl;
  pl.warps = min(nwarps, (int)((dbytes - pl.o_warp) / pl.per_warp));
  return pl;
}

// Block-wide; the first pl.warps warps factor.  over: global scratch for the values beyond
// kPipeVals, kMaxRowNZ - kPipeVals per warp (needed when n > kPipeVals).  Results as
// ilutp_warp (thread 0 has them), except the L levels, which the caller computes.  Bit 2 of the
// result: a wait ran out (P.ilu_wait_ns) and the rows are incomplete -- the column permutation
// is one, but unfinished rows hold the entries of an older factorisation, in its labels, so
// nothing may be built from them.
template <typename W>
__device__ __noinline__ int ilutp_pipe(const Walker& w, const Params& P, Shared& sh, const PipePlan& pl, W* over_all,
                                       int* npiv_out, double* nnz_out, int* p_out) {
  const int n = w.n, lane = threadIdx.x & 31, wid = threadIdx.x >> 5, cap = w.cap, capLU = w.capLU, NW = pl.warps;
  using K = decltype(mag_key(W(0)));
  unsigned char* dsm = dyn_smem();
  unsigned short* perm = (unsigned short*)(dsm + pl.o_perm);
  unsigned short* ip = (unsigned short*)(dsm + pl.o_ip);
  volatile int* done = &sh.ilu_done;
  volatile int* lost = &sh.ilu_lost;
#pragma unroll 1
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    perm[i] = (unsigned short)i;
    ip[i] = (unsigned short)i;
  }
  if (threadIdx.x == 0) {
    *done = 0;
    *lost = 0;
    sh.ilu_flags = 0;
    sh.ilu_npiv = 0;
    sh.ilu_nnz = 0;
  }
  // the fill limit, as ilutp_warp
  int p = P.lfil_extra;
  if (p < 0) {
    long long tot = 0;
#pragma unroll 1
    for (int i = lane; i < n; i += 32) tot += w.a_len[i];
    tot = warp_sum_ll(tot);
    p = (int)((tot + 2LL * n - 1) / (2LL * n));  // ceil(avg nnz per row / 2)
  }
  p = min(p, (capLU - 2) / 2);
  const int pk = max(0, min(p, capLU - 2 - cap));  // never exceeds the row capacity
  __syncthreads();
  if (wid < NW) {
    unsigned char* mine = dsm + pl.o_warp + (size_t)wid * pl.per_warp;
    unsigned* lbits = (unsigned*)(mine + pl.o_bits);
    unsigned* lsum = (unsigned*)(mine + pl.o_sum);
    unsigned short* wpos = (unsigned short*)(mine + pl.o_wpos);  // slot of a column, 0xffff: none
    unsigned short* nz = (unsigned short*)(mine + pl.o_nz);      // column of a slot
    W* val = (W*)(mine + pl.o_val);
    W* over = over_all + (size_t)wid * (kMaxRowNZ - kPipeVals) - kPipeVals;
    unsigned short* sel = (unsigned short*)(mine + pl.o_sel);    // slots of the candidates
    unsigned char* selk = mine + pl.o_selk;
    int* hist = (int*)(mine + pl.o_hist);
    unsigned short* bnd = (unsigned short*)(mine + pl.o_bnd);
    auto at = [&](int s) -> W& { return s < kPipeVals ? val[s] : over[s]; };
    const int nwords = (n + 31) >> 5, nsum = (nwords + 31) >> 5;
#pragma unroll 1
    for (int i = lane; i < nwords; i += 32) lbits[i] = 0u;
#pragma unroll 1
    for (int i = lane; i < nsum; i += 32) lsum[i] = 0u;
#pragma unroll 1
    for (int i = lane; i < n; i += 32) wpos[i] = 0xffffu;
    __syncwarp();
    auto mark = [&](int f) {
      atomicOr(&lbits[f >> 5], 1u << (f & 31));
      atomicOr(&lsum[f >> 10], 1u << ((f >> 5) & 31));
    };
    int flags = 0, npiv = 0;
    long long n_elim = 0, n_cand = 0, nnz = 0;
#pragma unroll 1
    for (int r = wid; r < n; r += NW) {
      const int part = w.part_of_row[r];
      const int len = w.a_len[part];
      const int* ac = w.a_col + (size_t)part * cap;
      const double* av = w.a_val + (size_t)part * cap;
      int d = __shfl_sync(0xffffffffu, *done, 0);  // labels below d are final
      __threadfence_block();
      double ss = 0.0;
#pragma unroll 1
      for (int t = lane; t < len; t += 32) {
        const int c = ac[t];
        const double v = av[t];
        nz[t] = (unsigned short)c;
        wpos[c] = (unsigned short)t;
        at(t) = (W)v;
        ss += v * v;
        const int f = ip[c];
        if (f < d) mark(f);
      }
      ss = warp_sum(ss);
      const double norm = sqrt(ss);
      const W thr = (W)(P.drop_tol * norm);
      const K kthr = mag_key(thr);
      int cnt = len, last = -1;
      // --- elimination with the previous U rows, in increasing label order ---
      for (;;) {
        __syncwarp();
        int best = 0x7fffffff;
        {
          // next pending label > last: first the rest of last's word, then the summary
          const int w0 = (last + 1) >> 5;
          const unsigned cur = w0 < nwords ? lbits[w0] & (0xffffffffu << ((last + 1) & 31)) : 0u;
          if (cur) {
            best = (w0 << 5) + __ffs(cur) - 1;
          } else {
            const int s0 = (w0 + 1) >> 5;  // summary word holding bitmap word w0 + 1
#pragma unroll 1
            for (int sb = s0; sb < nsum && best == 0x7fffffff; sb += 32) {
              const int si = sb + lane;
              unsigned sv = si < nsum ? lsum[si] : 0u;
              if (si == s0) sv &= 0xffffffffu << ((w0 + 1) & 31);
              const unsigned any = __ballot_sync(0xffffffffu, sv != 0u);
              if (any) {
                const int src = __ffs(any) - 1;
                const unsigned svs = __shfl_sync(0xffffffffu, sv, src);
                const int word = ((sb + src) << 5) + __ffs(svs) - 1;
                best = (word << 5) + __ffs(lbits[word]) - 1;
              }
            }
          }
        }
        if (best == 0x7fffffff) {
          if (d == r) break;
          // nothing left below d: wait for the next row (bounded), then look for the pivot
          // columns of the rows finished since
          int d2 = *done;
          if (d2 == d) {
            const unsigned long long t0 = global_ns();
            while ((d2 = *done) == d && !*lost) {
              __nanosleep(20);
              if (global_ns() - t0 > P.ilu_wait_ns) *lost = 1;
            }
          }
          d2 = __shfl_sync(0xffffffffu, d2, 0);
          if (d2 == d) break;  // gave up
          __threadfence_block();
          d2 = min(d2, r);
#pragma unroll 1
          for (int k = d + lane; k < d2; k += 32)
            if (wpos[perm[k]] != 0xffffu) mark(k);
          d = d2;
          continue;
        }
        last = best;
        ++n_elim;
        const double2 hd = w.u_head[best];
        const size_t rb = (size_t)best * capLU;
        int c0 = 0, c1 = 0;
        W v0 = 0, v1 = 0;
        if (lane < capLU) { c0 = w.u_col[rb + lane]; v0 = (W)w.u_val64[rb + lane]; }
        if (lane + 32 < capLU) { c1 = w.u_col[rb + lane + 32]; v1 = (W)w.u_val64[rb + lane + 32]; }
        const int tb = wpos[perm[best]];
        const W wk = at(tb) * (W)hd.x;
        const int ul = (int)hd.y;
        __syncwarp();
        if (mag_key(wk) < kthr) {
          if (lane == 0) at(tb) = (W)0;  // dropped multiplier
          continue;
        }
        if (lane == 0) at(tb) = wk;
#pragma unroll 1
        for (int base = 0; base < ul; base += 32) {
          const int t = base + lane;
          const bool valid = t < ul;
          int c = 0, s = 0xffff;
          W v = 0;
          if (valid) {
            if (base == 0) { c = c0; v = v0; }
            else if (base == 32) { c = c1; v = v1; }
            else { c = w.u_col[rb + t]; v = (W)w.u_val64[rb + t]; }
            s = wpos[c];
          }
          const bool fresh = valid && s == 0xffff;
          const unsigned nm = __ballot_sync(0xffffffffu, fresh);
          if (fresh) {
            const int slot = cnt + __popc(nm & lanemask_lt());
            if (slot < kMaxRowNZ) {
              nz[slot] = (unsigned short)c;
              wpos[c] = (unsigned short)slot;
              at(slot) = -wk * v;
              const int f = ip[c];
              if (f < d) mark(f);
            }
          } else if (valid) {
            at(s) = fma(-wk, v, at(s));  // (the product above is not shared: one rounding, as ilutp_warp)
          }
          cnt += __popc(nm);
          __syncwarp();
        }
        if (cnt > kMaxRowNZ) { flags |= 2; cnt = kMaxRowNZ; }
      }
      if (__any_sync(0xffffffffu, *lost)) break;
      n_cand += cnt;
      // entries of the original row on either side (labels below r are final now)
      int nl = 0, nu = 0;
#pragma unroll 1
      for (int t = lane; t < len; t += 32) {
        const int f = ip[nz[t]];
        nl += f < r;
        nu += f > r;
      }
      nl = warp_sum_int(nl);
      nu = warp_sum_int(nu);
      // candidates on one side: L keeps every nonzero multiplier, U the entries above threshold
      auto compact = [&](bool upper) {
        int c = 0;
#pragma unroll 1
        for (int base = 0; base < cnt; base += 32) {
          const int t = base + lane;
          bool k = false;
          if (t < cnt) {
            const int f = ip[nz[t]];
            const K m = mag_key(at(t));
            k = m != 0 && (upper ? f > r && m >= kthr : f < r);
          }
          const unsigned mk = __ballot_sync(0xffffffffu, k);
          const int slot = c + __popc(mk & lanemask_lt());
          if (k && slot < kMaxSel) sel[slot] = (unsigned short)t;
          c += __popc(mk);
        }
        if (c > kMaxSel) { flags |= 2; c = kMaxSel; }
        __syncwarp();
        return c;
      };
      auto key = [&](int e) { return mag_key(at(sel[e])); };
      auto label = [&](int e) { return (int)ip[nz[sel[e]]]; };
      // --- U part and pivot: the largest kept U entry (ties: smaller label) ---
      const int td = wpos[perm[r]];
      const W dval = td != 0xffff ? at(td) : (W)0;
      const int cU = compact(true);
      select_topk<K>(hist, bnd, selk, cU, nu + pk, key, label);
      K bk = 0;
      int bf = 0x7fffffff, be = 0;
#pragma unroll 1
      for (int e = lane; e < cU; e += 32)
        if (selk[e]) {
          const K m = key(e);
          const int f = label(e);
          if (m > bk || (m == bk && f < bf)) { bk = m; bf = f; be = e; }
        }
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        const K k2 = __shfl_xor_sync(0xffffffffu, bk, o);
        const int f2 = __shfl_xor_sync(0xffffffffu, bf, o);
        const int e2 = __shfl_xor_sync(0xffffffffu, be, o);
        if (k2 > bk || (k2 == bk && f2 < bf)) { bk = k2; bf = f2; be = e2; }
      }
      W newdiag = dval;
      int jm = -1;
      const int cr = perm[r];
      if (bf != 0x7fffffff) {
        const W v = at(sel[be]);
        if ((W)P.permtol * fabs(v) > fabs(dval)) { jm = be; newdiag = v; }
      }
      if (jm >= 0) {
        // the column labelled bf becomes the diagonal; the old diagonal value moves to
        // label bf (a U-part entry, or nothing if it was zero)
        if (lane == 0) {
          const int cj = perm[bf];
          perm[r] = (unsigned short)cj; perm[bf] = (unsigned short)cr;
          ip[cj] = (unsigned short)r; ip[cr] = (unsigned short)bf;
        }
        ++npiv;
      }
      int nU = 0;
#pragma unroll 1
      for (int base = 0; base < cU; base += 32) {
        const int e = base + lane;
        bool k = e < cU && selk[e];
        W v = 0;
        int c = 0;
        if (k) {
          c = nz[sel[e]];
          v = at(sel[e]);
          if (e == jm) { c = cr; v = dval; k = dval != (W)0; }
        }
        const unsigned mk = __ballot_sync(0xffffffffu, k);
        const int slot = nU + __popc(mk & lanemask_lt());
        if (k && slot < capLU) {
          w.u_col[(size_t)r * capLU + slot] = c;  // original column label
          w.u_val64[(size_t)r * capLU + slot] = (double)v;
        }
        nU += __popc(mk);
      }
      if (nU > capLU) { flags |= 2; nU = capLU; }
      if (newdiag == (W)0) {
        newdiag = (W)((1e-4 + P.drop_tol) * (norm > 0.0 ? norm : 1.0));
        flags |= 1;
      }
      if (lane == 0) {
        const W di = (W)(1.0 / newdiag);
        w.u_len[r] = nU;
        w.u_dinv64[r] = (double)di;
        w.u_head[r] = make_double2((double)di, (double)nU);
      }
      __threadfence_block();
      __syncwarp();
      if (lane == 0) *done = r + 1;  // publish the row
      // --- L part: keep the nl + p largest multipliers ---
      const int cL = compact(false);
      select_topk<K>(hist, bnd, selk, cL, nl + pk, key, label);
      int nL = 0;
#pragma unroll 1
      for (int base = 0; base < cL; base += 32) {
        const int e = base + lane;
        const bool k = e < cL && selk[e];
        const unsigned mk = __ballot_sync(0xffffffffu, k);
        const int slot = nL + __popc(mk & lanemask_lt());
        if (k && slot < capLU) {
          w.l_col[(size_t)r * capLU + slot] = label(e);
          w.l_val64[(size_t)r * capLU + slot] = (double)at(sel[e]);
        }
        nL += __popc(mk);
      }
      if (nL > capLU) { flags |= 2; nL = capLU; }
      if (lane == 0) w.l_len[r] = nL;
      nnz += nL + nU + 1;
      // clear the working row (and the pending-label bitmaps)
#pragma unroll 1
      for (int t = lane; t < cnt; t += 32) {
        const int c = nz[t];
        const int f = ip[c];
        wpos[c] = 0xffffu;
        if (f < r) { lbits[f >> 5] = 0u; lsum[f >> 10] = 0u; }
      }
      __syncwarp();
    }
    if (lane == 0) {
      atomicOr(&sh.ilu_flags, flags);
      atomicAdd(&sh.ilu_npiv, npiv);
      atomicAdd((unsigned long long*)&sh.ilu_nnz, (unsigned long long)nnz);
      atomicAdd((unsigned long long*)&w.ctl->ilu_elims, (unsigned long long)n_elim);
      atomicAdd((unsigned long long*)&w.ctl->ilu_cand, (unsigned long long)n_cand);
    }
  }
  __syncthreads();
#pragma unroll 1
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    w.perm[i] = perm[i];
    w.iperm[i] = ip[i];
  }
  if (threadIdx.x == 0) w.ctl->ilu_rows += n;
  __syncthreads();
  *npiv_out = sh.ilu_npiv;
  *nnz_out = (double)sh.ilu_nnz;
  *p_out = p;
  return sh.ilu_flags | (sh.ilu_lost ? 4 : 0);
}

}  // namespace vmc
