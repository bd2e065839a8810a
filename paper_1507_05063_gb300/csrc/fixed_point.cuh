// Block fixed point: the 19-point sums of float64 data on the integer units.
//
// GB300 issues float64 arithmetic -- and every conversion to or from float64 -- at 2 lanes
// per clock and SM (measured), 32-bit integer adds at 119 and shifts, logic and multiplies
// at 64.  The stencils of the scheme are short linear forms, so a tile of float64 values
// is brought to one power-of-two scale (the largest exponent of the tile and its halo),
// held as 64-bit integers, and its second differences and their products with 1/hx^2,
// 1/hy^2, 1/hz^2 are formed there exactly; the sum rounds once (to about 2^-62 of the largest
// possible sum, against float64's 2^-53 of every partial sum).
//
// With c a node's value, S_x, S_y, S_z its neighbour sums and E_xy ... its edge sums, and
// d_x the second difference along x, eq. (compact)'s left-hand side is
//   2 LHS(u) = a X + b Y + c Z,   X = d_x (12 + d_y + d_z) u
//            = 8 S_x + E_xy + E_xz - 16 u - 2 S_y - 2 S_z   (Y, Z likewise),
// with a = 1/hx^2, b = 1/hy^2, c = 1/hz^2: the printed weights, grouped by a, b and c.
#pragma once

#include <stdint.h>

#include "excmg_internal.cuh"

namespace excmg {

// Bits of a fixed-point u: |u| < 2^kFxBits, so |X| <= 48 2^56 < 2^61.6.
constexpr int kFxBits = 56;
// Bits of a fixed-point f: |6 f + six faces| <= 12 2^59 < 2^62.6.
constexpr int kFxBitsF = 59;
// Tiles whose largest biased exponent lies outside [kFxMinExp, kFxMaxExp] (zeros apart)
// take the float64 form: infinities and NaN (2047), and values whose scale or result
// could leave float64's normal range.
constexpr int kFxMinExp = 200, kFxMaxExp = 1800;
// A neighbourhood of nodes may be this many powers of two smaller than the scale it is held at.
// A value is held to 2^-57 of the scale: 2^-50 of the largest value near it then, the bound of
// eight float64 roundings in a row.  Fields that vanish smoothly on a face stay inside (two
// columns and rows and three planes from the boundary against the slab's far end: 2^-6), layers
// and peaks that fall off within a slab do not.  Error of r in 2^-53 of the node's own absolute
// sum, largest and root mean square, in float64 / without this rule / with it: exp(-200 r^2) on
// 64^3 cells 2.1, 0.4 / 6e15, 5e14 / 1.9, 0.4; exp(-100 x) on 128 x 40 x 40 0.6, 0.3 / 2e9, 3e8 /
// 0.6, 0.3; exp(4 (x + y + z)) on 48^3, 2 wide, 0.9, 0.24 / 69, 4.3 / 4.8, 0.33.
constexpr int kFxRange = 6;
// ... of the vectors of CG (p in slabs, r in the shared-memory boxes): held to 2^-46 of the largest
// value near them then, below what a solve that takes integers can ask for (1e-13, kFloat64Eps),
// and in norm the error stays 2^-57 of the largest value.  2^6 sent vectors of ordinary solves to
// float64: they are small where boundary planes or zeros of the data meet, and r after EXP_finite
// in the middle of a cell.  2^6 / 2^10: six solves of 128^3 cells with sums of sines, one batch,
// 27.5 / 21.9 ms (20.0 without a check); 128^3 with u = exp(-100 x) 26.8 / 22.8 ms (16.0; 41.4 in
// float64).  Shared-memory CG, the levels of a 512 x 256 x 128 solve at 1e-12: 3.7 ms with 2^6, 2.40
// with 2^8, 2.31 with 2^10, 2.30 with 2^14.
constexpr int kFxRangeCG = 10;

#ifdef __CUDACC__

// The magnitude bits of x's high word: ordered as |x| is, to 2^-20.
__device__ __forceinline__ unsigned fx_mag(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }

// x as an integer of scale 2^(BITS - (E - 1022)), E >= every biased exponent of the tile,
// to nearest: |result| <= 2^BITS, exact for x within 2^(BITS - 53) of the largest, else off
// by 2^-(BITS + 1) of the tile's largest value at most.  The magnitude is rounded and the sign
// put back: -x gives the negative (zeros of either sign, and denormal x, give 0: E >=
// kFxMinExp).
template <int BITS>
__device__ __forceinline__ long long fx_from_double(double x, int E) {
  static_assert(BITS >= 53 && BITS <= 62, "the significand is shifted left by BITS - 52");
  const int hi = __double2hiint(x);
  const unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u, d = (unsigned)(E - ((hi >> 20) & 0x7ff));
  // one bit below the unit, for rounding
  const unsigned long long m = ((unsigned long long)mh << 32 | (unsigned)__double2loint(x)) << (BITS - 52);
  unsigned long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(m), "r"(d));  // clamps at 64
  return ((long long)(r ^ (unsigned long long)(long long)(hi >> 31)) + 1) >> 1;  // r + 1 or -r, halved
}

// 2^n for |n| <= 1022.
__device__ __forceinline__ double fx_pow2(int n) { return __hiloint2double((1023 + n) << 20, 0); }

// (float)x, to nearest (ties away from zero), by integer instructions where the result is
// a normal number: the conversion instruction runs at the float64 rate.
__device__ __forceinline__ float fx_to_float(double x) {
  const int hi = __double2hiint(x);
  const unsigned lo = (unsigned)__double2loint(x);
  const unsigned e = ((unsigned)hi >> 20) & 0x7ffu;
  if (e - 897u >= 253u) return (float)x;  // zero, denormal or overflowing as a float, Inf, NaN
  const unsigned m = (((unsigned)hi << 3) | (lo >> 29)) & 0x7fffffu;
  const unsigned b = ((e - 896u) << 23 | m) + ((lo >> 28) & 1u);  // a carry moves to the next power of two
  return __uint_as_float(b | ((unsigned)hi & 0x80000000u));
}

// x 2^q by its exponent field, for x = 0 or |x| and |x 2^q| in the normal range.
__device__ __forceinline__ double fx_scale(double x, int q) {
  const int hi = __double2hiint(x);
  return __hiloint2double((hi & 0x7fffffff) ? hi + (q << 20) : hi, __double2loint(x));
}

// -x 2^q, likewise.
__device__ __forceinline__ double fx_scale_neg(double x, int q) {
  const int hi = __double2hiint(x);
  return __hiloint2double((hi & 0x7fffffff) ? hi + (int)(((unsigned)q << 20) ^ 0x80000000u) : hi, __double2loint(x));
}

// The power of two of the sums L (2 LHS = L 2^q) at scale E.
__device__ __forceinline__ int fx_sum_exp(int k, int E) { return 60 - k - (kFxBits - (E - 1022)); }

// PTX multiply-adds: one instruction per product.
__device__ __forceinline__ long long fx_mad_s(int a, int b, long long c) {
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}

// (X W_0 + Y W_1 + Z W_2) / 2^60 for |X|, |Y|, |Z| < 2^61.6 and 0 <= W = h 2^31 + l <= 2^60 (l
// signed, l2 = 2 l); |result| <= 96 2^56 < 2^62.6.  With X = x_h 2^32 + x_l (x_l signed) the sum
// is t 2^63 + m 2^31 + n, every product one 32 x 32 multiply-add: t = sum x_h h, m = sum x_l h +
// x_h l2 (< 2^62.9), n = sum x_l l (< 2^62.6).  The whole sum is formed and rounded once, to
// nearest, ties to even, so that -X, -Y, -Z give the negative and no rounding has a preferred
// side.  (A floor, half a unit the same way at every node, is a smooth right-hand side: the
// solution of the level moved by 1e-14 with it; dropped low products break the symmetry in
// sign; the odd one of the two neighbours is off by up to a unit, which the residual of a smooth
// field on unequal meshsizes shows: root mean square 7.7e-13 against 3.9e-13 for exp(x + y + z)
// on 48 x 100 x 37 cells.)
__device__ __forceinline__ long long fx_weigh(long long X, long long Y, long long Z, const FxWeights& W) {
  const int xl = (int)X, yl = (int)Y, zl = (int)Z;
  const int xh = (int)(X >> 32) - (xl >> 31), yh = (int)(Y >> 32) - (yl >> 31), zh = (int)(Z >> 32) - (zl >> 31);
  const long long n = fx_mad_s(zl, W.l[2], fx_mad_s(yl, W.l[1], (long long)xl * W.l[0]));
  long long m = fx_mad_s(xl, W.h[0], (n >> 31) + (1 << 28));  // half a unit
  m = fx_mad_s(yl, W.h[1], m);
  m = fx_mad_s(zl, W.h[2], m);
  m = fx_mad_s(xh, W.l2[0], m);
  m = fx_mad_s(yh, W.l2[1], m);
  m = fx_mad_s(zh, W.l2[2], m);
  const long long t = fx_mad_s(zh, W.h[2], fx_mad_s(yh, W.h[1], (long long)xh * W.h[0]));
  const unsigned rest = ((unsigned)m & 0x1fffffffu) | ((unsigned)n & 0x7fffffffu);  // 0: a tie
  return ((t << 3) + (m >> 29)) & ~(long long)(rest == 0);
}

#endif  // __CUDACC__

}  // namespace excmg
