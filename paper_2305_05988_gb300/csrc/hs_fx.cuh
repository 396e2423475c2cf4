// hs_fx.cuh -- sums of FP64 values on the integer pipes.
//
// The FP64 pipe of this GPU retires 2 lanes per clock and SM (one warp
// instruction every 64 cycles of a sub-partition); integer additions run at
// 126 lanes, shifts and logic at 64.  A sum of several doubles is therefore
// cheaper as a fixed-point sum: each term is split once into a signed 60-bit
// significand and its exponent (fx_make), the terms are shifted to the largest
// exponent of the sum, added as 64-bit integers and rounded once to binary64
// (fx_total).  Six terms take 42 cycles per warp and sub-partition, a split 8
// (measured at full occupancy); five FP64 additions take 320.
//
// Accuracy: a term loses less than 2^-59 of the largest term's power of two
// when it is shifted, so n <= 7 terms are summed to within 7 x 2^-59 of it
// before the one rounding; a chain of FP64 additions rounds n - 1 times at
// 2^-53 of its partial sums.  Sums that cancel below 2^-16 of the largest
// term, terms outside 2^-943 .. 2^1016 and non-finite terms take the FP64
// additions themselves (fx_value restores every double exactly, zeros,
// subnormals, infinities and NaNs included).
#pragma once
#include <cuda_runtime.h>

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

// v[0] + ... + v[n-1]
template <int n>
__device__ __forceinline__ double fx_total(const Fx (&v)[n]) {
  static_assert(n >= 2 && n <= 7, "three bits of headroom above 2^60");
  unsigned top = v[0].e;
#pragma unroll
  for (int q = 1; q < n; q++) top = max(top, v[q].e);
  long long acc = 0;
#pragma unroll
  for (int q = 0; q < n; q++) {
    long long m = ((long long)v[q].hi << 32) | v[q].lo;
    asm("shr.s64 %0, %0, %1;" : "+l"(m) : "r"(top - v[q].e));   // amounts above 63 leave the sign
    acc += m;
  }
  const int s = (int)(acc >> 63);
  const unsigned long long a = (unsigned long long)((acc ^ (long long)s) - (long long)s);
  const unsigned ah = (unsigned)(a >> 32), al = (unsigned)a;
  if (top - 80u < 1960u && ah >= 0x1000u) {
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
    return __hiloint2double((int)(hi | ((unsigned)s & 0x80000000u)), (int)lo);
  }
  double y = fx_value(v[0]);
#pragma unroll
  for (int q = 1; q < n; q++) y += fx_value(v[q]);
  return y;
}

}  // namespace hs
