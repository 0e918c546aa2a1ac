// vmc_select.cuh -- the fill rule's selection: the k largest of a row's candidates, by one warp.
#pragma once
#include "vmc_device.cuh"

namespace vmc {

// Magnitude of a value as an ordered integer (integer compares: an FP64 compare holds the
// warp's FP64 unit for 64 cycles) and its binary exponent.
__device__ __forceinline__ unsigned long long mag_key(double v) {
  return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
}
__device__ __forceinline__ unsigned mag_key(float v) { return (unsigned)__float_as_int(v) & 0x7fffffffu; }
__device__ __forceinline__ int key_exp(unsigned long long k) { return (int)(k >> 52); }
__device__ __forceinline__ int key_exp(unsigned k) { return (int)(k >> 23); }

// Top-k of c candidates by magnitude (ties: smaller label), by one warp: a histogram of
// binary exponents below the largest one (bins of one octave, the last bin collecting
// everything smaller) finds the octave that holds the k-th largest; entries in higher
// octaves are kept, entries in that octave are ranked among themselves.  key(e): magnitude
// key of candidate e, label(e): its label.  Result in selK[0..c); hist (64) and bnd (256)
// are scratch.
template <typename K, typename Key, typename Label, typename B>
__device__ __forceinline__ void select_topk(int* hist, B* bnd, unsigned char* selK, int c, int keep, Key key,
                                            Label label) {
  const int lane = threadIdx.x & 31;
  if (c <= keep) {
#pragma unroll 1
    for (int e = lane; e < c; e += 32) selK[e] = 1;
    __syncwarp();
    return;
  }
  int emax = 0;
#pragma unroll 1
  for (int e = lane; e < c; e += 32) emax = max(emax, key_exp(key(e)));
  emax = __reduce_max_sync(0xffffffffu, emax);
  auto bin = [&](K k) { return min(63, emax - key_exp(k)); };
#pragma unroll 1
  for (int b = lane; b < 64; b += 32) hist[b] = 0;
  __syncwarp();
#pragma unroll 1
  for (int e = lane; e < c; e += 32) atomicAdd(&hist[bin(key(e))], 1);
  __syncwarp();
  // boundary bin bb: count(bins < bb) < keep <= count(bins <= bb)
  int h0 = hist[lane], h1 = hist[lane + 32];
  int inc0 = h0;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) { const int v = __shfl_up_sync(0xffffffffu, inc0, o); if (lane >= o) inc0 += v; }
  const int tot0 = __shfl_sync(0xffffffffu, inc0, 31);
  int inc1 = h1;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) { const int v = __shfl_up_sync(0xffffffffu, inc1, o); if (lane >= o) inc1 += v; }
  inc1 += tot0;
  const unsigned m0 = __ballot_sync(0xffffffffu, inc0 >= keep);
  const unsigned m1 = __ballot_sync(0xffffffffu, inc1 >= keep);
  const int bb = m0 ? __ffs(m0) - 1 : 32 + __ffs(m1) - 1;
  const int below = (bb < 32 ? __shfl_sync(0xffffffffu, inc0 - h0, bb & 31)
                             : __shfl_sync(0xffffffffu, inc1 - h1, bb & 31));
  const int need = keep - below;  // entries to keep from the boundary bin
  // compact the boundary octave, decide the others
  int cb = 0;
#pragma unroll 1
  for (int base = 0; base < c; base += 32) {
    const int e = base + lane;
    int b = 64;
    if (e < c) {
      b = bin(key(e));
      selK[e] = b < bb ? 1 : 0;
    }
    const unsigned m = __ballot_sync(0xffffffffu, b == bb);
    const int slot = cb + __popc(m & lanemask_lt());
    if (b == bb && slot < 256) bnd[slot] = (B)e;
    cb += __popc(m);
  }
  __syncwarp();
  if (cb <= 256) {
#pragma unroll 1
    for (int q = lane; q < cb; q += 32) {
      const int e = bnd[q];
      const K me = key(e);
      const int fe = label(e);
      int rank = 0;
#pragma unroll 1
      for (int o = 0; o < cb; ++o) {
        const int eo = bnd[o];
        const K mo = key(eo);
        rank += (mo > me) || (mo == me && label(eo) < fe);
      }
      selK[e] = rank < need ? 1 : 0;
    }
  } else {
#pragma unroll 1
    for (int e = lane; e < c; e += 32) {
      const K me = key(e);
      if (bin(me) != bb) continue;
      const int fe = label(e);
      int rank = 0;
#pragma unroll 1
      for (int o = 0; o < c; ++o) {
        const K mo = key(o);
        if (bin(mo) != bb) continue;
        rank += (mo > me) || (mo == me && label(o) < fe);
      }
      selK[e] = rank < need ? 1 : 0;
    }
  }
  __syncwarp();
}
}  // namespace vmc
