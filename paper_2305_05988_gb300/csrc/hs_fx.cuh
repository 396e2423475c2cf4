// hs_fx.cuh -- sums of FP64 values on the integer pipes.
//
// The FP64 pipe of this GPU retires 2 lanes per clock and SM (one warp
// instruction every 64 cycles of a sub-partition); integer additions run at
// 126 lanes, shifts and logic at 64.  A sum of several doubles is therefore
// cheaper as a fixed-point sum: each term is split once into a signed 60-bit
// significand and its exponent (fx_make), the terms are shifted to the largest
// exponent of the sum, added as 64-bit integers and rounded once to binary64
// (fx_total).  Six terms take about 42 cycles per warp and sub-partition, a split 8
// (measured at full occupancy); five FP64 additions take 320.
//
// Accuracy: a term loses less than 2^-59 of the largest term's power of two
// when it is shifted, so n <= 7 terms are summed to within 7 x 2^-59 of it
// before the one rounding (weighted sums: 6 x 2^-57 of the largest weighted
// one); a chain of FP64 additions rounds n - 1 times at
// 2^-53 of its partial sums.  Sums that cancel below 2^-16 of the largest
// term, terms outside 2^-943 .. 2^1006 and non-finite terms take the FP64
// additions themselves (fx_value restores every double exactly, zeros,
// subnormals, infinities and NaNs included).
#pragma once
#include <cuda_runtime.h>

#include "hs_common.cuh"

namespace hs {

// hi:lo = (-1)^s (1.f) 2^59, e = the biased exponent.  A zero or subnormal (e = 0) carries the implicit
// bit too; it only matters next to terms of that size, which are summed in FP64.
struct Fx {
  unsigned lo;
  int hi;
  unsigned e;
};

__device__ __forceinline__ Fx fx_make(double v) {
  const int vh = __double2hiint(v);
  const unsigned vl = (unsigned)__double2loint(v);
  const int s = vh >> 31;
  const unsigned m = ((unsigned)vh & 0xfffffu) | 0x100000u;
  Fx r;
  r.e = ((unsigned)vh >> 20) & 0x7ffu;
  const unsigned long long w =
      ((((unsigned long long)__funnelshift_l(vl, m, 7) << 32) | (vl << 7)) ^ (unsigned long long)(long long)s) -
      (unsigned long long)(long long)s;
  r.lo = (unsigned)w;
  r.hi = (int)(w >> 32);
  return r;
}

__device__ __forceinline__ double fx_value(const Fx& f) {
  const unsigned s = (unsigned)(f.hi >> 31);
  const long long w = ((long long)f.hi << 32) | f.lo;
  const unsigned long long a = (unsigned long long)(w < 0 ? -w : w);
  const unsigned lo = (unsigned)a, hi = (unsigned)(a >> 32);
  return __hiloint2double((int)(((hi >> 7) & 0xfffffu) | (f.e << 20) | (s & 0x80000000u)),
                          (int)__funnelshift_r(lo, hi, 7));
}

// Rounds acc 2^(top - 1023 - 59) to binary64; false (y untouched) where the
// sum has cancelled or the exponents leave the range this path handles.
__device__ __forceinline__ bool fx_round(long long acc, unsigned top, double& y) {
  const int s = (int)(acc >> 63);
  const unsigned long long a = (unsigned long long)((acc ^ (long long)s) - (long long)s);
  const unsigned ah = (unsigned)(a >> 32), al = (unsigned)a;
  if (!(top - 80u < 1950u && ah >= 0x1000u)) return false;
  int z;                                                       // leading zeros of ah: 1 .. 19
  asm("bfind.shiftamt.u32 %0, %1;" : "=r"(z) : "r"(ah));
  z -= 1;
  // leading bit to 2^62, round to nearest even at 2^10 (a tie is one sum in
  // eight or four when the exponents are close: rounded away from zero it
  // would bias the sums by 2^-57, which a solve's smooth error accumulates)
  const unsigned tl = al << z;
  const unsigned long long t =
      (((unsigned long long)__funnelshift_l(al, ah, z) << 32) | tl) + (511u + ((tl >> 10) & 1u));
  const unsigned lo = (unsigned)(t >> 10);
  const unsigned hi = (unsigned)(t >> 42) + ((top + 2u) << 20) - ((unsigned)z << 20);
  y = __hiloint2double((int)(hi | ((unsigned)s & 0x80000000u)), (int)lo);
  return true;
}

// The significand shifted to the exponent top >= f.e.
__device__ __forceinline__ long long fx_align(const Fx& f, unsigned top) {
  long long m = ((long long)f.hi << 32) | f.lo;
  asm("shr.s64 %0, %0, %1;" : "+l"(m) : "r"(top - f.e));   // amounts above 63 leave the sign
  return m;
}

template <int n>
__device__ __forceinline__ unsigned fx_top(const Fx (&v)[n]) {
  unsigned top = v[0].e;
#pragma unroll
  for (int q = 1; q < n; q++) top = max(top, v[q].e);
  return top;
}

// v[0] + ... + v[n-1]
template <int n>
__device__ __forceinline__ double fx_total(const Fx (&v)[n]) {
  static_assert(n >= 2 && n <= 7, "three bits of headroom above 2^60");
  const unsigned top = fx_top(v);
  long long acc = 0;
#pragma unroll
  for (int q = 0; q < n; q++) acc += fx_align(v[q], top);
  double y;
  if (fx_round(acc, top, y)) return y;
  y = fx_value(v[0]);
#pragma unroll
  for (int q = 1; q < n; q++) y += fx_value(v[q]);
  return y;
}

// m c / 2^63 rounded to nearest, |m| < 2^61, c = ch 2^31 + cl < 2^61 (every
// partial sum below 2^63):
//   (mh 2^32 + ml)(ch 2^31 + cl) / 2^63 = mh ch + (2 mh cl + ml ch + ml cl / 2^31) / 2^32,
// the last term replaced by its mean cl (ml is uniform): rc = 2^31 + cl.
__device__ __forceinline__ long long fx_scale(long long m, const FxW& W, int q) {
  const int mh = (int)(m >> 32);
  const unsigned ml = (unsigned)m;
  long long t, r;
  asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(t) : "r"(ml), "r"(W.ch[q]), "l"((long long)W.rc[q]));
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(t) : "r"(mh + mh), "r"(W.cl[q]));
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(mh), "r"(W.ch[q]), "l"(t >> 32));
  return r;
}

// The sum of a node's neighbours in the order w, e, s, n, b, t, weighted by
// the couplings relative to the upper x one (OP_WSYM, OP_WNON).  Terms are
// aligned first (exact for exponents up to 7 apart), then scaled with
// rounding to 2^-57 of the largest coupling's term.
template <int OPK, int n>
__device__ __forceinline__ double fx_neighbours(const Fx (&v)[n], const FxW& W) {
  if constexpr (OPK == OP_ISO) {
    return fx_total(v);
  } else {
    const unsigned top = fx_top(v);
    long long acc = 0;
    if constexpr (OPK == OP_WSYM) {
#pragma unroll
      for (int q = 0; q < n; q += 2) acc += fx_scale(fx_align(v[q], top) + fx_align(v[q + 1], top), W, q);
    } else {
#pragma unroll
      for (int q = 0; q < n; q++) acc += fx_scale(fx_align(v[q], top), W, q);
    }
    double y;
    if (fx_round(acc, top, y)) return __hiloint2double(__double2hiint(y) + ((W.k + 1) << 20), __double2loint(y));
    y = W.w[0] * fx_value(v[0]);
#pragma unroll
    for (int q = 1; q < n; q++) y = fma(W.w[q], fx_value(v[q]), y);
    return y;
  }
}

}  // namespace hs
