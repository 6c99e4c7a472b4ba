// Fixed-point arithmetic of the double-precision path's stencils.
//
// GB300 issues 2 double-precision operations per clock and multiprocessor
// and 64 integer ones (measured per warp instruction and scheduler: 64.5
// clocks for a DFMA, 5 for a 32 x 32 + 64 bit multiply-add, 2 for an
// integer add; the two kinds overlap).  The linear and bilinear parts of
// the right-hand side therefore run on the integer unit, in fixed point of 59
// or 62 bits, more than the 53 of a double.
//
// A value is held as an integer F, cut towards zero, for an exponent E with
// |f| < 2^E: f 2^(59-E) in two limbs F = hi 2^30 + lo with the sign of f on
// both (|lo| < 2^30, |hi| <= 2^29) where fields are multiplied, the 64-bit word
// f 2^(62-E) where they are added up with constant weights.  Values of at
// least 2^-7 (words: 2^-10) of 2^E keep all of their 53 bits.
//
// E is an exponent of the field for the whole grid (its ghosts included), so
// that a value is converted once for all the stencils that it enters, for
// every stencil whose largest value is at least 2^-5 (words: 2^-8; density in
// products: 2^-2) of 2^E.  A value that loses bits there is at least 3/4 of
// that away from the largest, so the cut is below a double's rounding of
// their difference.  A stencil of smaller values only (a field near a zero, a
// quiet region beside a jet) is read from memory again, and taken with the
// exponent of its own largest value or in double.  Both depend on the fields
// alone, so results do not depend on tiles or launch shapes.  With the grid's
// exponent alone a region with velocities of 1e-18 of the largest had no
// correct digit left in its mass flux.
//
// The path is taken when every maximum is zero or from 2^-280 to 2^200 (the
// products of three fields and a grid factor then stay inside the range of a
// double), in the fluxes when besides the density spans at most 2^6;
// otherwise, and for non-finite states, the kernels run their double-precision
// arithmetic.  Stencils of values below 2^-280 are cut at 2^-339; values below
// the normal range count as zero.
#pragma once
#include "s2_internal.cuh"

namespace s2 {

constexpr int FX_LIMB = 30;
constexpr int FX_MASK = (1 << FX_LIMB) - 1;
// Biased exponents of the smallest and largest maxima that the path takes.
// Grid factors are within 2^-100 .. 2^100.
constexpr int FX_EMIN = 1023 - 280, FX_EMAX = 1023 + 200;
constexpr int FX_SPAN = 6;
constexpr int FX_UNIT = 1022 + 62;  // a word's unit is 2^(e - FX_UNIT) for the biased exponent e
// The hi limb of 2^-5 of 2^E, the hi half of a word of 2^-8 of 2^E.
constexpr int FX_LOUD = 1 << 24, FX_LOUD_WORD = 1 << 22;

// The biased exponent field of a double.
__device__ __forceinline__ int fx_exponent(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// Biased exponent of a field's maximum, and the magnitude of a hi limb from
// which a stencil is loud (a field that is zero everywhere has no quiet ones).
struct FxField {
  int e, loud, loud_word;
};

// One of the running exponents of Scal is raised; most calls find it high
// enough already.
__device__ __forceinline__ void fx_raise(unsigned *at, unsigned e) {
  if (__ldcg(at) < e) atomicMax(at, e);
}
__device__ __forceinline__ void fx_clear(Scal *s) {
#pragma unroll
  for (int f = 0; f < FX_NF; ++f) s->fx_e[f] = 0;
  s->fx_m = 0;
}

// The field's exponent; ok is cleared when it is out of range.
__device__ __forceinline__ FxField fx_field(const Dev &d, int f, bool &ok) {
  const int e = (int)__ldcg(&d.scal->fx_e[f]);
  if (e > FX_EMAX || (e && e < FX_EMIN)) ok = false;
  return FxField{e ? e : FX_EMIN, e ? FX_LOUD : 0, e ? FX_LOUD_WORD : 0};
}

// Whether the fixed-point path may be taken, by the fields that are complete
// before the gradient pass; the dilatation, which that pass adds, is checked
// where it is read.
__device__ __forceinline__ bool fx_ok(const Dev &d) {
  bool ok = d.fx != 0;
  for (int f = 0; f < FX_TH; ++f) fx_field(d, f, ok);
  return ok;
}
// The fluxes multiply three fields, each of which may be small in a stencil:
// besides, the density must not span more than 2^6.
__device__ __forceinline__ bool fx_flux_ok(const Dev &d) {
  const int e = (int)__ldcg(&d.scal->fx_e[FX_RHO]), m = 2047 - (int)__ldcg(&d.scal->fx_m);
  return fx_ok(d) && e - m <= FX_SPAN;
}

// x as limbs (.x = lo, .y = hi) for a field of biased exponent ex.
__device__ __forceinline__ int2 fx_split(double x, int ex) {
  const int hx = __double2hiint(x);
  const unsigned lx = (unsigned)__double2loint(x);
  const unsigned mh = ((unsigned)hx & 0xfffffu) | 0x100000u;
  unsigned long long m = ((unsigned long long)__funnelshift_l(lx, mh, 6) << 32) | (lx << 6);
  m >>= min(ex - ((hx >> 20) & 0x7ff), 63);
  const int s = hx >> 31;
  return make_int2((((int)m & FX_MASK) ^ s) - s, ((int)(m >> FX_LIMB) ^ s) - s);
}

// Running largest magnitude of a stencil's values on the hi words, and the
// exponent that it gives them.
__device__ __forceinline__ int fx_mag(double x) { return __double2hiint(x) & 0x7fffffff; }
__device__ __forceinline__ int fx_own_exponent(int mag) { return max(mag >> 20, FX_EMIN); }

// A product of limb pairs / 2^60.
__device__ __forceinline__ long long fx_mul(int al, int ah, int bl, int bh) {
  const long long hl = (long long)ah * bl + (long long)al * bh + (((long long)al * bl) >> FX_LIMB);
  return (long long)ah * bh + (hl >> FX_LIMB);
}

// Central difference weights of order 2 NP over a common denominator:
// first derivative c1(l) / D1 (l = 1..NP), second derivative c2(l) / D2
// (l = 0..NP); W1, W2: bits of the weights' magnitudes added up.
template <int NP>
struct FxStencil;
template <>
struct FxStencil<1> {
  static constexpr int D1 = 2, D2 = 1, W1 = 1, W2 = 2;
  __host__ __device__ static constexpr int c1(int) { return 1; }
  __host__ __device__ static constexpr int c2(int l) { return l == 0 ? -2 : 1; }
};
template <>
struct FxStencil<2> {
  static constexpr int D1 = 12, D2 = 12, W1 = 5, W2 = 6;
  __host__ __device__ static constexpr int c1(int l) { return l == 1 ? 8 : -1; }
  __host__ __device__ static constexpr int c2(int l) { return l == 0 ? -30 : (l == 1 ? 16 : -1); }
};
template <>
struct FxStencil<3> {
  static constexpr int D1 = 60, D2 = 180, W1 = 7, W2 = 11;
  __host__ __device__ static constexpr int c1(int l) { return l == 1 ? 45 : (l == 2 ? -9 : 1); }
  __host__ __device__ static constexpr int c2(int l) { return l == 0 ? -490 : (l == 1 ? 270 : (l == 2 ? -27 : 2)); }
};
template <>
struct FxStencil<4> {
  static constexpr int D1 = 840, D2 = 5040, W1 = 11, W2 = 15;
  __host__ __device__ static constexpr int c1(int l) { return l == 1 ? 672 : (l == 2 ? -168 : (l == 3 ? 32 : -3)); }
  __host__ __device__ static constexpr int c2(int l) {
    return l == 0 ? -14350 : (l == 1 ? 8064 : (l == 2 ? -1008 : (l == 3 ? 128 : -9)));
  }
};

// v 2^n as a double, rounded to nearest (ties away from zero), on the
// integer unit: the conversion instruction occupies the double unit like a
// DFMA.
__device__ __forceinline__ double fx_i2d(long long v, int n = 0) {
  const long long s = v >> 63;
  unsigned long long a = (unsigned long long)((v ^ s) - s);
  const int z = __clzll((long long)a);
  a <<= z & 63;
  const unsigned long long m = (a >> 11) + ((a >> 10) & 1);  // bit 52 set
  const int hi = (int)(m >> 32) + (1023 + 62 - z + n) * (1 << 20);
  return a ? __hiloint2double(hi | ((int)(v >> 32) & (int)0x80000000), (int)m) : 0.0;
}

// Words of the linear stencils: the integer f 2^(62-E) cut towards zero, of
// which two add up in 64 bits.  Values of at least 2^-10 of 2^E keep all of
// their bits.
__device__ __forceinline__ long long fx_word(double x, int ex) {
  const int hx = __double2hiint(x);
  const unsigned lx = (unsigned)__double2loint(x);
  const unsigned mh = ((unsigned)hx & 0xfffffu) | 0x100000u;
  unsigned long long m = ((unsigned long long)__funnelshift_l(lx, mh, 9) << 32) | (lx << 9);
  m >>= min(ex - ((hx >> 20) & 0x7ff), 63);
  const long long s = hx >> 31;
  return ((long long)m ^ s) - s;
}
__device__ __forceinline__ int fx_hi(long long v) { return (int)(v >> 32); }

// Sum of words (or sums of two) with small integer weights: the high and low
// 32 bits apart, the low ones by the sign of their weight.
struct FxSum {
  long long hi = 0;
  unsigned long long pos = 0, neg = 0;
  __device__ __forceinline__ void add(int c, long long v) {
    hi += (long long)c * fx_hi(v);
    if (c > 0) pos += (unsigned long long)(unsigned)c * (unsigned)v;
    else neg += (unsigned long long)(unsigned)-c * (unsigned)v;
  }
  // The sum as an integer times 2^drop, for weights that add up to at most
  // 2^W, each word counted: exact below 2^62; above (differences of the order
  // of the field's maximum) its last W bits are cut towards zero, far below
  // the rounding of a double-precision sum, whose terms are rounded at
  // 2^(W-2-53) of the maximum.
  template <int W>
  __device__ __forceinline__ long long value(int &drop) const {
    const long long lo = (long long)(pos - neg), t = hi + (lo >> 32);
    drop = (unsigned long long)(t + (1ll << 30)) >> 31 ? W : 0;
    const unsigned long long r = (unsigned long long)(unsigned)lo + (t < 0 ? (1ull << drop) - 1 : 0);
    return (t << (32 - drop)) + (long long)(r >> drop);
  }
};

// x 2^n, x and the result being normal.
__device__ __forceinline__ double fx_ldexp(double x, int n) {
  return __hiloint2double(__double2hiint(x) + n * (1 << 20), __double2loint(x));
}

}  // namespace s2
