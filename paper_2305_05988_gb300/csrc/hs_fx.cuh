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
// when it is shifted by more than seven places (up to there the shift is
// exact), always towards minus infinity, so n <= 7 terms are summed to within
// 7 x 2^-59 of it before the one rounding.  Weighted terms are aligned by the
// exponent of the weighted term, so their error is relative to the largest
// weighted term too, however far the weights lie apart: 4.5 x 2^-56 of its
// power of two for three pairs, 7.5 x 2^-56 for six single terms
// (fx_neighbours).  A chain of FP64 additions rounds n - 1 times at 2^-53 of
// its partial sums.  Sums that cancel below 2^-16 (weighted: 2^-12) of the
// largest term, terms outside 2^-943 .. 2^1006 and non-finite terms take the
// FP64 additions themselves (fx_value restores every double exactly, zeros,
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

// The significand shifted right.
__device__ __forceinline__ long long fx_align(const Fx& f, unsigned by) {
  long long m = ((long long)f.hi << 32) | f.lo;
  asm("shr.s64 %0, %0, %1;" : "+l"(m) : "r"(by));   // amounts above 63 leave the sign
  return m;
}

template <int n>
__device__ __forceinline__ unsigned fx_top(const Fx (&v)[n]) {
  unsigned top = v[0].e;
#pragma unroll
  for (int q = 1; q < n; q++) top = max(top, v[q].e);
  return top;
}

// Whether every term is a zero; y = their sum (-0 if all of them are).  The
// untouched part of a grid (the first pass from x0 = 0, a local source) has
// such nodes only, which fx_round cannot take: without this exit they paid for
// the additions in both forms (256^3 SpMV of zeros 249 us, so 109; 20 Jacobi
// sweeps from a point source 236 and 120 us each).
template <int n>
__device__ __forceinline__ bool fx_zeros(const Fx (&v)[n], double& y) {
  unsigned any = 0;
  int neg = -1;
#pragma unroll
  for (int q = 0; q < n; q++) {
    any |= v[q].e | v[q].lo | ((unsigned)v[q].hi & 0x07ffffffu);   // a zero's significand is +-2^59
    neg &= v[q].hi;
  }
  y = __hiloint2double(neg & (int)0x80000000, 0);
  return any == 0u;
}

// v[0] + ... + v[n-1]
template <int n>
__device__ __forceinline__ double fx_total(const Fx (&v)[n]) {
  static_assert(n >= 2 && n <= 7, "three bits of headroom above 2^60");
  const unsigned top = fx_top(v);
  long long acc = 0;
#pragma unroll
  for (int q = 0; q < n; q++) acc += fx_align(v[q], top - v[q].e);
  double y;
  if (fx_round(acc, top, y) || fx_zeros(v, y)) return y;
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
// the couplings relative to the upper x one (OP_WSYM, OP_WNON).
//
// Coupling q is (c_q / 2^60) 2^(x_q) with c_q in [2^60, 2^61), so the weighted
// term's exponent is e + x_q, up to the last bit; terms are shifted to the
// largest of those and the products summed in units of 2^-56 of that power of
// two.  A product is off by one unit at most (fx_scale: half for the rounding,
// half for the mean), the shift in front of it by a quarter (a pair: half).
// Aligned by e alone, as in OP_ISO, the unit would be relative to the largest
// value times the largest coupling: at a ratio of 62 a single neighbour on the
// weak axis came out wrong by 5.9 x 2^-53, and large ones next to small
// neighbours on the strong axes by up to 25 x 2^-53 of the terms.  Emulated over
// ratios of 1 to 62 and values of all shapes the present form stays below 1.1 x
// 2^-53 of the terms, FP64 additions below 3.5.
template <int OPK, int n>
__device__ __forceinline__ double fx_neighbours(const Fx (&v)[n], const FxW& W) {
  if constexpr (OPK == OP_ISO) {
    return fx_total(v);
  } else {
    // W.x[1], and in OP_WSYM W.x[0], is zero: the upper x weight is 1.  (The
    // two forms: 250 x 187 x 141 Jacobi, OP_WSYM, 72.0 us per sweep against 73.3
    // in the other; 256^3, OP_WNON, 176.8 against 181.5.)
    int top;
    long long acc = 0;
    if constexpr (OPK == OP_WSYM) {
      top = max((int)v[0].e, (int)v[1].e);
#pragma unroll
      for (int q = 2; q < n; q++) top = __viaddmax_s32((int)v[q].e, W.x[q], top);
#pragma unroll
      for (int q = 0; q < n; q += 2) {
        const unsigned at = (unsigned)(q == 0 ? top : top - W.x[q]);
        acc += fx_scale(fx_align(v[q], at - v[q].e) + fx_align(v[q + 1], at - v[q + 1].e), W, q);
      }
    } else {
      int e[n];
      top = -64;
#pragma unroll
      for (int q = 0; q < n; q++) {
        e[q] = (int)v[q].e + (q == 1 ? 0 : W.x[q]);
        top = max(top, e[q]);
      }
#pragma unroll
      for (int q = 0; q < n; q++) acc += fx_scale(fx_align(v[q], (unsigned)(top - e[q])), W, q);
    }
    double y;
    if (fx_round(acc, (unsigned)top, y)) return __hiloint2double(__double2hiint(y) + (3 << 20), __double2loint(y));
    if (fx_zeros(v, y)) return y;
    y = W.w[0] * fx_value(v[0]);
#pragma unroll
    for (int q = 1; q < n; q++) y = fma(W.w[q], fx_value(v[q]), y);
    return y;
  }
}

}  // namespace hs
