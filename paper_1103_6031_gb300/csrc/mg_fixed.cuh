// Float64 stencil sums on the integer pipe.
//
// GB300 issues about 1.6 FP64 instructions per clock and SM (500-529 G/s measured) but 33
// times as many 64-bit integer additions (16.4 T/s), so the float64 stencils, 15 of whose
// 19 operations are additions of neighbours, are bound by the FP64 pipe although they are
// far from every other limit.  Here the neighbours of ONE cell are aligned to the largest
// exponent among them, as 59-bit two's-complement integers (the mantissa shifted by the
// difference of the exponents), summed exactly, weighted by the small integers of the
// Table 1 operators (multiples of 1/256, by shifts and additions), and converted back
// once: 1 conversion and 1 fma instead of 18-19 operations, and about 13 cheap integer
// operations per neighbour.
//
// Accuracy: an aligned value is off by less than one unit of 2^-59 of the largest
// neighbour (dropped low bits; negative values by one's complement), the shifts of the
// weights by a few such units, the conversion rounds to 53 bits.  A sum in FP64
// arithmetic rounds at every addition, each time by up to 2^-53 of its partial sum, so
// the result here is the more accurate one unless a whole stencil cancels below 2^-6 of
// its largest value, where both are at the rounding level of the values themselves.  In the
// kernels that work cell by cell the alignment depends only on the cell's own neighbours (no
// level-wide scale, no state) and the integer sums do not depend on the order: these kernels
// give the same bits on the same values.  The tile kernels (mg_tile.cuh) align to the largest
// value of a block of cells instead and leave blocks of too wide a range to FP64.
//
// Range: the largest neighbour must be finite and at least 2^-926 in magnitude (biased
// exponent kFxMinExp); otherwise (all zero, denormal, infinite, NaN) the caller uses FP64
// arithmetic.
#pragma once

#include "mg_internal.h"

namespace mgk {

constexpr unsigned kFxMinExp = 96;
// Order-6 half-sweeps of more cells align 4 of the 18 neighbours on the FP64 pipe
// (fx_align_cvt).  One V-cycle, without / with: a base and two nests of 64^3 287 / 301 us (the
// conversions' latency), 80^3 466 / 456, 128^3 1007 / 973; a periodic 192^3 level 988 / 937.
constexpr long long kFxCvtMinCells = 1ll << 18;
// A value is its aligned integer times 2^(e - kFxBias), e the largest biased exponent:
// a mantissa of 53 bits (value = mantissa 2^(e - 1075)) is shifted left by 6.
constexpr int kFxBias = 1081;

// The largest exponent field of the values, in bits 21..31, as the maximum of (high word
// << 1); low bits arbitrary.
__device__ __forceinline__ unsigned fx_key(double v) {
  return (unsigned)__double2hiint(v) << 1;
}

__device__ __forceinline__ bool fx_in_range(unsigned key) {
  return (key >> 21) - kFxMinExp < 0x7ffu - kFxMinExp;
}

// v as an integer in units of 2^(e - kFxBias); key: the maximum of fx_key over the values
// that are summed, with its low 21 bits set.  The shift (PTX clamps amounts above 63) is
// the difference of the exponents; zeros and denormals shift out entirely.
__device__ __forceinline__ long long fx_align(double v, unsigned key) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const unsigned sh = (key - (hi << 1)) >> 21;
  const unsigned xh = __funnelshift_l(lo, (hi & 0xfffffu) | 0x100000u, 6);
  unsigned long long x = ((unsigned long long)xh << 32) | (lo << 6);
  asm("shr.u64 %0, %0, %1;" : "+l"(x) : "r"(sh));
  unsigned s;  // the sign in every bit (prmt's sign replication: 5% of a half-sweep)
  asm("prmt.b32 %0, %1, 0, 0xbbbb;" : "=r"(s) : "r"(hi));
  return (long long)(x ^ (((unsigned long long)s << 32) | s));
}

// The same on the FP64 pipe (rounded down: at most a unit from fx_align): the exponent moved
// by kFxBias - e, then one conversion.  That pipe is idle most of the time while neighbours
// are aligned: 4 of 18 this way are the fastest mix (order 6, 128^3 half-sweep: none 17.2 us,
// 2 16.8, 4 16.0, 6 19.2), on levels large enough that throughput counts (kFxCvtMinCells).  Values that the moved exponent would leave below the normal range
// (only possible with WIDE, e > kFxBias) round to 0 or -1 all the same.
template <bool WIDE>
__device__ __forceinline__ long long fx_align_cvt(double v, unsigned key) {
  const int d = kFxBias - (int)(key >> 21);
  const int hi = __double2hiint(v);
  if (WIDE && ((hi >> 20) & 0x7ff) + d <= 0) return hi >> 31;
  return __double2ll_rd(__hiloint2double(hi + (d << 20), __double2loint(v)));
}

// c * 2^(e - kFxBias) by an addition to the exponent field; c a normal constant whose
// exponent stays in range (checked by fx_scalable for run-time constants).
__device__ __forceinline__ double fx_scale(double c, unsigned key) {
  const int d = (int)(key >> 21) - kFxBias;
  return __hiloint2double(__double2hiint(c) + (d << 20), __double2loint(c));
}

__device__ __forceinline__ bool fx_scalable(double c, unsigned key) {
  const int ec = (__double2hiint(c) >> 20) & 0x7ff;
  const int er = ec + (int)(key >> 21) - kFxBias;
  return ec > 0 && ec < 0x7ff && er > 0 && er < 0x7ff;
}

// Table 1 weights as integers over a common denominator: sum_off w u = T / kFxUnit^-1 with
// order 2: T = s1 - 6 c; order 4 (x 12/16): T = s1 - s2/16 - (90/16) c; order 6 (x 180/256):
// T = (270 s1 - 27 s2 + 2 s3 - 1470 c) / 256.
template <int ORDER>
struct FxUnit;
template <>
struct FxUnit<2> {
  static constexpr double v = 1.0;
};
template <>
struct FxUnit<4> {
  static constexpr double v = 16.0 / 12.0;
};
template <>
struct FxUnit<6> {
  static constexpr double v = 256.0 / 180.0;
};

// The integer formulas below are written over the integer type I, so that a host program can
// run them on a type that records the size of every intermediate.  In units of 2^59, above
// which no aligned value lies, the largest intermediates at orders 2 / 4 / 6 are: Laplacian
// 12 / 12 / 12.75, second difference 4 / 4.13 / 4.34, first derivative 2 / 2.25 / 6, first
// derivative of first derivatives 4 / 5.07 / 10.32.  64 bits hold 16.

// The neighbours' part of T from their sums at distance 1, 2, 3.
template <int ORDER, typename I>
__host__ __device__ __forceinline__ I fx_weighted(const I (&s)[3]) {
  if (ORDER == 2) return s[0];
  if (ORDER == 4) return s[0] - (s[1] >> 4);
  // 270/256 = 1 + 1/16 - 1/128, 27/256 = 1/8 - 1/64 - 1/256, 2/256 = 1/128
  return s[0] + (s[0] >> 4) - (s[1] >> 3) + ((s[1] + (s[1] >> 2)) >> 6) + ((s[2] - s[0]) >> 7);
}

// The same from the neighbours (nb[6 d .. 6 d + 5] at distance d + 1); key as for fx_align.
template <int ORDER, bool CVT, bool WIDE>
__device__ __forceinline__ long long fx_neighbours_by(const double (&nb)[3 * ORDER], unsigned key) {
  long long s[3] = {0, 0, 0};
#pragma unroll
  for (int d = 0; d < ORDER / 2; ++d)
#pragma unroll
    for (int q = 0; q < 6; ++q)
      s[d] += CVT && d == 2 && q < 4 ? fx_align_cvt<WIDE>(nb[6 * d + q], key)
                                     : fx_align(nb[6 * d + q], key);
  return fx_weighted<ORDER>(s);
}

template <int ORDER, bool CVT = false>
__device__ __forceinline__ long long fx_neighbours(const double (&nb)[3 * ORDER], unsigned key) {
  if constexpr (CVT && ORDER == 6) {
    if ((int)(key >> 21) > kFxBias) return fx_neighbours_by<ORDER, true, true>(nb, key);
    return fx_neighbours_by<ORDER, true, false>(nb, key);
  }
  return fx_neighbours_by<ORDER, false, false>(nb, key);
}

// The centre's term of T (weight 3 w0), c its aligned integer.
template <int ORDER, typename I>
__host__ __device__ __forceinline__ I fx_centre(I c) {
  if (ORDER == 2) return -6 * c;
  if (ORDER == 4) return -6 * c + (c >> 2) + (c >> 3);  // 90/16 = 6 - 1/4 - 1/8
  return -6 * c + (c >> 2) + (c >> 7);                  // 1470/256 = 6 - 1/4 - 1/128
}

// One axis: h^2 u'' = T FxUnit 2^(e - kFxBias) from the sums u(+d) + u(-d) and the centre.
template <int ORDER, typename I>
__host__ __device__ __forceinline__ I fx_second(const I (&s)[3], I c) {
  if (ORDER == 2) return s[0] - 2 * c;
  if (ORDER == 4) return fx_weighted<4>(s) - 2 * c + (c >> 3);  // 30/16 = 2 - 1/8
  return fx_weighted<6>(s) - 2 * c + (c >> 4) + (c >> 6) + (c >> 7);  // 490/256 = 2 - 22/256
}

// One axis: h u' = T FxGradUnit 2^(e - kFxBias) from the differences u(+d) - u(-d); order 6:
// T = (45 d1 - 9 d2 + d3) / 64, order 4: (8 d1 - d2) / 8.  |T| <= 2, 9/4, 110/64 max |u|.  The
// operator is applied to its own result for mixed derivatives, whose differences reach 3.44
// max |u| at order 6: every term is shifted before its factor could carry the sum past 64
// bits (45/64 = 1 - 1/4 - 1/32 - 1/64).
template <int ORDER>
struct FxGradUnit {
  static constexpr double v = ORDER == 2 ? 0.5 : (ORDER == 4 ? 8.0 / 12.0 : 64.0 / 60.0);
};

template <int ORDER, typename I>
__host__ __device__ __forceinline__ I fx_first(const I (&d)[3]) {
  if (ORDER == 2) return d[0];
  if (ORDER == 4) return d[0] - (d[1] >> 3);
  return d[0] - (d[0] >> 2) - (d[0] >> 5) - (d[1] >> 3) + ((d[2] - d[1] - d[0]) >> 6);
}

}  // namespace mgk
