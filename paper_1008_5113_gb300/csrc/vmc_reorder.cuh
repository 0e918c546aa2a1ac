// vmc_reorder.cuh -- the greedy particle/orbital reordering of Sec. 3.1.
//
// For i = 0..n-2: find the orbital nearest to the particle at position i among positions
// >= i and swap it into column i; if the nearest is already at i, find the particle nearest
// to orbital i among positions >= i and swap it into row i.  Minimum-image distances in
// plainly rounded FP64, ties to the lowest position.  Positions are the current columns;
// afterwards orbitals return to their fixed columns carrying their new partner particle, so
// only part_of_row / row_of_part change.
//
// The rule is a chain of up to 2 (n - 1) nearest-neighbour searches.  Scanning all positions
// with the CTA took 12 ms at n = 1000 and 214 ms at n = 4096: n^2 distances with three FP64
// divisions each, on a chip that issues about two FP64 operations a clock per SM.  Here one
// warp searches the lattice cells around the particle (orbitals are sites; particles are
// kept in a list per cell) out to a radius that holds the nearest one for certain, and scans
// the positions only when few are left or nothing near is free.  Distances are compared in
// FP32 first, in units of the lattice constant, from a copy of the coordinates made for it (any
// constant gives the same comparisons, and a search converts nothing); FP64 decides between
// those that FP32 cannot tell apart, so the result is the rule's.  Positions outside the box,
// which the FP32 minimum image and the cells do not cover, are scanned in FP64.  Measured, one walker's reordering: n = 1000 12.4 -> 2.1 ms, n = 4096
// 214 -> 13 ms (397 ms where two CTAs shared an SM) with the coordinates converted in every
// search; the copy takes n = 1000 from 3.05 to 2.37 ms and n = 4096 from 13.9 to 11.0 ms
// (electrons 0.2 a from their sites).
#pragma once
#include "vmc_geom.cuh"

namespace vmc {

// A candidate's position and FP64 distance, in the rule's order.
struct Nearest {
  double d;
  int pos;
};

// Nearest candidate of a warp's search: each(f) calls f(position, FP32 distance^2, id) for
// the lane's candidates, exact(id) is the FP64 distance^2.  limit: FP32 distances^2 at or
// beyond it do not count as found (a candidate outside the searched cells may be nearer);
// kScan: every candidate is among those searched.  margin(d): twice the error of FP32
// distances^2 around d (infinite: FP64 decides alone).  Returns the position, or -1 (in a scan
// only when no distance is a number).
constexpr float kScan = 3e38f;
template <typename Each, typename Exact, typename Margin>
__device__ __forceinline__ int nearest_warp(float limit, Each each, Exact exact, Margin margin) {
  float m = 3e38f, thr = 0.0f;
  int cnt = 0, pos = 0x7fffffff;
  Nearest b{__longlong_as_double(0x7ff0000000000000ll), 0x7fffffff};
#pragma unroll 1
  for (int pass = 0; pass < 3; ++pass) {  // the least FP32 distance; who is near it; FP64 among those
    each([&](int p, float d, int id) {
      if (pass == 0) {
        m = fminf(m, d);
      } else if (d <= thr) {
        if (pass == 1) {
          ++cnt;
          pos = p;
        } else {
          const double x = exact(id);
          if (x < b.d || (x == b.d && p < b.pos)) { b.d = x; b.pos = p; }
        }
      }
    });
    if (pass == 0) {
      m = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(m)));  // d >= 0
      thr = m + margin(m);
      if (limit < kScan && !(thr < limit)) return -1;
    } else if (pass == 1) {
      if (__reduce_add_sync(0xffffffffu, cnt) == 1) return __reduce_min_sync(0xffffffffu, pos);
    }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    const double d2 = __shfl_xor_sync(0xffffffffu, b.d, o);
    const int p2 = __shfl_xor_sync(0xffffffffu, b.pos, o);
    if (d2 < b.d || (d2 == b.d && p2 < b.pos)) { b.d = d2; b.pos = p2; }
  }
  return b.pos == 0x7fffffff ? -1 : b.pos;
}

// I: index type of the position tables (16 bits in shared memory, int in global memory).
template <typename I>
__device__ __noinline__ void reorder_search(const Walker& w, I* pos_orb, I* pos_part, I* orb_at, I* part_at, I* next,
                                            int* head) {
  const int n = w.n, K = w.K, per = w.per, tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
  constexpr int kNone = sizeof(I) == 2 ? 0xffff : -1;
  // lengths in units of the lattice constant, FP32: a particle within 3e-5 of a face may be taken
  // for its neighbour cell's, which the factor 0.9999 on the search limits covers (K <= 64)
  float* xs = (float*)w.ex_val;  // scratch of at least 8 n doubles, free until the factorisation
  auto cell_axis = [&](float x) { return min(K - 1, max(0, (int)floorf(x))); };
  int inside = 1;
  {
    const double inva = 1.0 / w.a, L = w.L;
#pragma unroll 1
    for (int i = tid; i < 3 * n; i += nt) {
      const double r = w.R[i];
      xs[i] = (float)(r * inva);
      inside &= r >= 0.0 && r < L;
    }
  }
#pragma unroll 1
  for (int c = tid; c < n; c += nt) {
    const int p = w.part_of_row[c], o = w.orb_of_col[c];
    part_at[c] = (I)p;
    orb_at[c] = (I)o;
    pos_part[p] = (I)c;
    pos_orb[o] = (I)c;
  }
#pragma unroll 1
  for (int c = tid; c < K * K * K; c += nt) head[c] = kNone;
  inside = __syncthreads_and(inside);
#pragma unroll 1
  for (int p = tid; p < n; p += nt) {
    const float* r = xs + 3 * p;
    const int c = cell_axis(r[0]) + K * (cell_axis(r[1]) + K * cell_axis(r[2]));
    next[p] = (I)atomicExch(&head[c], p);
  }
  __syncthreads();
  if (tid < 32) {
    const float L = (float)K, hL = 0.5f * L;
    // coordinates up to L, their differences and the image shift: below 4 x 2^-24 L each,
    // 7 x 2^-24 L on the distance; twice that, times two distances, with room
    const float eps = inside ? 32.0f * 5.9604645e-8f * L : __int_as_float(0x7f800000);
    auto margin = [&](float d2) { return eps * (1.0f + d2); };  // 2 d <= 1 + d^2
    auto dist32 = [&](float x, float y, float z) {
      x = fabsf(x); y = fabsf(y); z = fabsf(z);
      x = x > hL ? L - x : x;
      y = y > hL ? L - y : y;
      z = z > hL ? L - z : z;
      return x * x + y * y + z * z;
    };
    auto site32 = [&](int o, float& x, float& y, float& z) {
      const int b = per == 2 ? (o & 1) : 0;
      int c = per == 2 ? o >> 1 : o;
      const float off = 0.5f * (float)b;
      const int cx = c % K;
      c /= K;
      x = (float)cx + off;
      y = (float)(c % K) + off;
      z = (float)(c / K) + off;
    };
    auto wrap_cell = [&](int c) { return c < 0 ? c + K : (c >= K ? c - K : c); };
#pragma unroll 1
    for (int i = 0; i < n - 1; ++i) {
      const int p = part_at[i];
      const double rp[3] = {w.R[3 * p], w.R[3 * p + 1], w.R[3 * p + 2]};
      const float px = xs[3 * p], py = xs[3 * p + 1], pz = xs[3 * p + 2];
      const bool few = n - i <= 64 || !inside;
      int bj = -1;
      if (!few) {
        const int cx = cell_axis(px), cy = cell_axis(py), cz = cell_axis(pz);
#pragma unroll 1
        for (int rad = 1; rad <= 3 && 2 * rad + 1 <= K && bj < 0; ++rad) {
          const int s = 2 * rad + 1, tot = s * s * s * per;
          auto each = [&](auto f) {
#pragma unroll 1
            for (int q = lane; q < tot; q += 32) {
              const int b = per == 2 ? (q & 1) : 0;
              int t = per == 2 ? q >> 1 : q;
              const int x = wrap_cell(cx - rad + t % s);
              t /= s;
              const int y = wrap_cell(cy - rad + t % s), z = wrap_cell(cz - rad + t / s);
              const int o = (x + K * (y + K * z)) * per + b;
              const int j = (int)pos_orb[o];
              if (j < i) continue;
              const float off = 0.5f * (float)b;
              f(j, dist32(px - ((float)x + off), py - ((float)y + off), pz - ((float)z + off)), o);
            }
          };
          // every site outside the searched cells is at least rad away along one axis
          bj = nearest_warp((float)(rad * rad) * 0.9999f, each,
                            [&](int o) { return dist2(rp, w.Z + 3 * o, w.L); }, margin);
        }
      }
      if (bj < 0) {
        auto each = [&](auto f) {
#pragma unroll 1
          for (int j = i + lane; j < n; j += 32) {
            const int o = orb_at[j];
            float x, y, z;
            site32(o, x, y, z);
            f(j, dist32(px - x, py - y, pz - z), o);
          }
        };
        bj = nearest_warp(kScan, each, [&](int o) { return dist2(rp, w.Z + 3 * o, w.L); }, margin);
        if (bj < 0) bj = i;
      }
      if (bj != i) {
        __syncwarp();
        if (lane == 0) {
          const I oi = orb_at[i], oj = orb_at[bj];
          orb_at[i] = oj; orb_at[bj] = oi;
          pos_orb[oj] = (I)i; pos_orb[oi] = (I)bj;
        }
        __syncwarp();
        continue;
      }
      const int o = orb_at[i];
      const double* zo = w.Z + 3 * o;
      float ox, oy, oz;
      site32(o, ox, oy, oz);
      auto part_dist = [&](int q) {
        const float* r = xs + 3 * q;
        return dist32(r[0] - ox, r[1] - oy, r[2] - oz);
      };
      auto exact = [&](int q) { return dist2(w.R + 3 * q, zo, w.L); };
      int bk = -1;
      if (!few) {
        int c = per == 2 ? o >> 1 : o;
        const int cx = c % K;
        c /= K;
        const int cy = c % K, cz = c / K;
#pragma unroll 1
        for (int rad = 1; rad <= 3 && 2 * rad + 1 <= K && bk < 0; ++rad) {
          const int s = 2 * rad + 1, tot = s * s * s;
          auto each = [&](auto f) {
#pragma unroll 1
            for (int q = lane; q < tot; q += 32) {
              int t = q;
              const int x = wrap_cell(cx - rad + t % s);
              t /= s;
              const int y = wrap_cell(cy - rad + t % s), z = wrap_cell(cz - rad + t / s);
#pragma unroll 1
              for (int k = head[x + K * (y + K * z)]; k != kNone; k = (int)next[k]) {
                const int g = (int)pos_part[k];
                if (g >= i) f(g, part_dist(k), k);
              }
            }
          };
          // a site lies in [0, 1) of its cell on each axis: cells out to rad hold everything
          // nearer than rad
          bk = nearest_warp((float)(rad * rad) * 0.9999f, each, exact, margin);
        }
      }
      if (bk < 0) {
        auto each = [&](auto f) {
#pragma unroll 1
          for (int k = i + lane; k < n; k += 32) {
            const int q = part_at[k];
            f(k, part_dist(q), q);
          }
        };
        bk = nearest_warp(kScan, each, exact, margin);
        if (bk < 0) bk = i;
      }
      __syncwarp();
      if (bk != i && lane == 0) {
        const I pi = part_at[i], pk = part_at[bk];
        part_at[i] = pk; part_at[bk] = pi;
        pos_part[pk] = (I)i; pos_part[pi] = (I)bk;
      }
      __syncwarp();
    }
  }
  __syncthreads();
#pragma unroll 1
  for (int g = tid; g < n; g += nt) {
    const int c = w.col_of_orb[orb_at[g]];
    const int p = part_at[g];
    w.part_of_row[c] = p;
    w.row_of_part[p] = c;
  }
  __syncthreads();
}

// Block-wide.  The tables in shared memory as 16-bit positions where they fit (5 n of them
// and a list head per cell), else in the factorisation's global scratch.
static __device__ __noinline__ void reorder_block(const Walker& w, const Params& P) {
  const int n = w.n, ncell = w.K * w.K * w.K;
  if (n < 0xffff && (size_t)10 * n + 16 + 4 * (size_t)ncell <= (size_t)P.dsm_bytes) {
    int* head = (int*)dyn_smem();
    unsigned short* t = (unsigned short*)(head + ncell);
    reorder_search<unsigned short>(w, t, t + n, t + 2 * n, t + 3 * n, t + 4 * n, head);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // scratch is reused by bulk copies
    __syncthreads();
  } else {
    reorder_search<int>(w, w.iperm, w.wpos, w.gQ, w.gP, w.lvl_cur, w.lvl_nchunk);
  }
}

}  // namespace vmc
