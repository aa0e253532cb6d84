// Sums of doubles over warps and blocks.
//
// What a sum costs on this part is a chain of dependent FP64 operations: one takes 64 clocks, and a warp issues one
// every 64 clocks whatever its lanes do (measured; an FP64 division 560, a shuffle tree over a warp 546). So the sums
// here run on the integer pipes. A warp's values are aligned to their largest exponent 2^e as 64-bit integers (what lies
// below 2^(e - 63) is cut off) and added without rounding in three limbs by warp-wide integer reductions (236 clocks for a
// value), with no order dependence at all; the sum keeps the bits from 2^(e - 57) up (M > 1: 2^(e - 54)). A block's warps
// are aligned and added the same way, and the one rounding is the last conversion. Worst error of 512 values over sum |v|,
// 2,400 draws of six distributions: 1.2e-16, where the tree of shuffles and warp sums had 3.9e-16. Values no such window
// holds (subnormal sums, infinities, NaN, sums next to overflow) go through the floating-point tree, so they mean what they
// meant there. A warp of zeros is an ordinary sum: the solvers' server warp holds none, and with the mark of a special value
// on its zero every grid sum took the tree (an iteration of the level-0 CG on 48^3 cells 5.9 us instead of 5.5, of the
// BiCGStab 19.9 instead of 18.7).
#pragma once
#include <cuda_runtime.h>

#include "fp64.cuh"

namespace nlmg {

// A sum in integer form: t 2^(mx - 1077), or, with mx < 0, the double whose bits t are (special values, see above).
struct ISum {
  long long t;
  int mx;
};
__device__ __forceinline__ double isum_value(const ISum& s) {
  if (s.mx < 0) return __longlong_as_double(s.t);
  const long long d = __double_as_longlong((double)s.t);
  return s.t == 0 ? 0.0 : __longlong_as_double(d + ((long long)(s.mx - 1077) << 52));
}

// s[k] = the sum over the warp of v[k][0..M) (see above), in every lane; all 32 lanes take part.
template <int NV, int M>
__device__ __forceinline__ void warp_sums(const double (&v)[NV][M], ISum (&s)[NV]) {
  int mx[NV];
  bool odd = false;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    unsigned m = 0u;   // the high word, its last bit set where only the low one holds a value
#pragma unroll
    for (int j = 0; j < M; ++j)
      m = max(m, ((unsigned)__double2hiint(v[k][j]) & 0x7fffffffu) | min((unsigned)__double2loint(v[k][j]), 1u));
    m = __reduce_max_sync(0xffffffffu, m);
    mx[k] = (int)(m >> 20);
    // not zeros (an idle warp), but values next to the subnormals or to overflow
    odd = odd || m - 1u < (64u << 20) - 1u || mx[k] > 2032;
  }
  if (odd) {   // the same in every lane
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      double a = v[k][0];
#pragma unroll
      for (int j = 1; j < M; ++j) a += v[k][j];
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
      s[k].t = __double_as_longlong(a);
      s[k].mx = -1;
    }
    return;
  }
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    int lo = 0, mi = 0, hi = 0;   // limbs of 22, 21 and 21 bits: at most 32 M <= 224 terms, no limb overflows
#pragma unroll
    for (int j = 0; j < M; ++j) {
      const unsigned long long b = (unsigned long long)__double_as_longlong(v[k][j]);
      const int ex = (int)((b >> 52) & 0x7ffu), sh = mx[k] - ex;
      unsigned long long x = (b << 11) | 0x8000000000000000ull;
      x = ex != 0 && sh < 64 ? x >> sh : 0ull;   // (a subnormal is far below the window)
      const int sg = (int)((long long)b >> 63);
      lo += ((int)(x & 0x3fffffu) ^ sg) - sg;
      mi += ((int)((x >> 22) & 0x1fffffu) ^ sg) - sg;
      hi += ((int)(x >> 43) ^ sg) - sg;
    }
    static_assert(M <= 7, "limbs sized for 224 terms");
    lo = __reduce_add_sync(0xffffffffu, lo);
    mi = __reduce_add_sync(0xffffffffu, mi);
    hi = __reduce_add_sync(0xffffffffu, hi);
    // the window's bits from 2^SH up, as many as leave |t| < 2^63: the error is below 2^-54 (M = 1: 2^-57) of the largest
    // value
    constexpr int SH = M == 1 ? 6 : 9;
    s[k].t = ((long long)hi << (43 - SH)) + ((long long)mi << (22 - SH)) + (long long)(lo >> SH);
    s[k].mx = max(mx[k] + SH - 9, 0);   // (a zero's window: a negative one marks special values, other sums have 61 at least)
  }
}

// The sum over the warp of one integer sum per lane, as a double in every lane; all 32 lanes take part.
template <int NV>
__device__ __forceinline__ void warp_sums_i(const ISum (&v)[NV], double (&s)[NV]) {
  bool odd = false;
#pragma unroll
  for (int k = 0; k < NV; ++k) odd = odd || v[k].mx < 0;
  if (__any_sync(0xffffffffu, odd)) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      double a = isum_value(v[k]);
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
      s[k] = a;
    }
    return;
  }
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    const int mx = (int)__reduce_max_sync(0xffffffffu, (unsigned)v[k].mx), sh = mx - v[k].mx;
    const long long x = sh < 63 ? v[k].t >> sh : 0ll;
    const int lo = __reduce_add_sync(0xffffffffu, (int)(x & 0x3fffff));
    const int mi = __reduce_add_sync(0xffffffffu, (int)((x >> 22) & 0x1fffff));
    const int hi = __reduce_add_sync(0xffffffffu, (int)(x >> 43));
    // the sum in 63 bits: all of it, or, from 2^62 up, without its last six (an eighth of its rounding at most)
    const long long up = ((long long)hi << 21) + (long long)mi + (long long)(lo >> 22);
    const int sh6 = (up >> 40) == (up >> 63) ? 0 : 6;
    ISum r;
    r.t = (up << (22 - sh6)) + (long long)((lo & 0x3fffff) >> sh6);
    r.mx = mx + sh6;
    s[k] = isum_value(r);
  }
}

// s[k] = the sums over the block of v[k][0..M), in every lane of warp 0 (nw warps, at most 32; sm: NV * 32 entries of shared
// memory, free again after the next __syncthreads).
template <int NV, int M>
__device__ __forceinline__ void block_sums(const double (&v)[NV][M], double (&s)[NV], ISum* sm, int nw) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  ISum w[NV];
  warp_sums<NV, M>(v, w);
  if (lane < NV) {
    ISum mine = w[0];
#pragma unroll
    for (int k = 1; k < NV; ++k)
      if (lane == k) mine = w[k];
    sm[lane * 32 + warp] = mine;
  }
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) w[k] = lane < nw ? sm[k * 32 + lane] : ISum{0ll, 0};
    warp_sums_i<NV>(w, s);
  }
}

}  // namespace nlmg
