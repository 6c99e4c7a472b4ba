// Fixed-point arithmetic of the double-precision path's stencils.
//
// GB300 issues 2 double-precision operations per clock and multiprocessor
// and 64 integer ones (measured per warp instruction and scheduler: 64.5
// clocks for a DFMA, 5 for a 32 x 32 + 64 bit multiply-add, 2 for an
// integer add; the two kinds overlap).  The linear and bilinear parts of
// the right-hand side therefore run on the integer unit, in 59-bit fixed
// point, which carries more bits than the 53 of a double.
//
// A field f gets one exponent for the whole grid (its ghosts included):
// |f| < 2^E, and f is held as the integer F = f 2^(59-E) cut towards zero,
// in two limbs F = hi 2^30 + lo with the sign of f on both (|lo| < 2^30,
// |hi| <= 2^29).  Values of at least 2^-7 of 2^E keep all of their 53 bits;
// smaller ones are cut at 2^-59 of 2^E, below the rounding error that a
// double-precision sum with the larger ones makes.  The exponents depend on
// the fields alone, so results do not depend on tiles or launch shapes.
//
// The path is taken when every maximum is finite and below 2^200
// and density, temperature and pressure, which the equations divide by or
// whose small differences drive the flow, span at most 2^6 (all of their
// bits are then kept); otherwise, and for non-finite states, the kernels
// run their double-precision arithmetic.
#pragma once
#include "s2_internal.cuh"

namespace s2 {

constexpr int FX_LIMB = 30;
constexpr int FX_MASK = (1 << FX_LIMB) - 1;
// Biased exponents below the first are raised to it (fields that are zero
// or tiny everywhere), those above the second take the double path.  The
// products of three fields and a grid factor (within 2^-100 .. 2^100, or its
// square) then stay far inside the range of a double.
constexpr int FX_EMIN = 1023 - 200, FX_EMAX = 1023 + 200;
constexpr int FX_SPAN = 6;

// The biased exponent field of a double.
__device__ __forceinline__ int fx_exponent(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// Biased exponents of the fields' maxima (fx_e[FX_*] of Scal, raised to
// FX_EMIN) and whether the fixed-point path may be taken.
struct FxScale {
  int e[FX_NF];
  bool ok;
};

// A value of field f is raised into the running exponents of Scal; most
// calls find them high enough already.
__device__ __forceinline__ void fx_raise(Scal *s, int f, int e) {
  if (__ldcg(&s->fx_e[f]) < (unsigned)e) atomicMax(&s->fx_e[f], (unsigned)e);
  if (f < FX_NMIN && __ldcg(&s->fx_m[f]) < 2047u - (unsigned)e) atomicMax(&s->fx_m[f], 2047u - (unsigned)e);
}
__device__ __forceinline__ void fx_clear(Scal *s) {
#pragma unroll
  for (int f = 0; f < FX_NF; ++f) s->fx_e[f] = 0;
#pragma unroll
  for (int f = 0; f < FX_NMIN; ++f) s->fx_m[f] = 0;
}

__device__ __forceinline__ FxScale fx_scale(const Dev &d) {
  FxScale s;
  s.ok = d.fx != 0;
#pragma unroll
  for (int f = 0; f < FX_NF; ++f) {
    const int e = (int)__ldcg(&d.scal->fx_e[f]);
    if (e > FX_EMAX) s.ok = false;
    if (f < FX_NMIN && e - (2047 - (int)__ldcg(&d.scal->fx_m[f])) > FX_SPAN) s.ok = false;
    s.e[f] = e < FX_EMIN ? FX_EMIN : e;
  }
  return s;
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

// The high part of a product of limb pairs, (a b) / 2^60 up to the dropped
// lo lo product: hh + hl / 2^30.
__device__ __forceinline__ long long fx_mulhi(int al, int ah, int bl, int bh) {
  const long long hl = (long long)ah * bl + (long long)al * bh;
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

// The limb sums hi 2^30 + lo of a stencil whose weights add up to less than
// 2^W in magnitude, as an integer times 2^drop.  Below 2^62 the sum is
// exact; above (differences of the order of the field's maximum) its last
// W - 3 bits are cut, which leaves at least 54 bits for first derivatives
// and for Laplacians at least the accuracy of a double-precision sum, whose
// terms are rounded at 2^(W-2-53) of the field's maximum.
template <int W>
__device__ __forceinline__ long long fx_sum(long long hi, long long lo, int &drop) {
  constexpr int CUT = W > 3 ? W - 3 : 0;
  const long long t = hi + (lo >> FX_LIMB);
  const int r = (int)lo & FX_MASK;
  drop = CUT && ((unsigned long long)(t + (1ll << 32)) >> 33) != 0 ? CUT : 0;
  return (t << (FX_LIMB - drop)) + (r >> drop);
}

// x 2^n, x and the result being normal.
__device__ __forceinline__ double fx_ldexp(double x, int n) {
  return __hiloint2double(__double2hiint(x) + n * (1 << 20), __double2loint(x));
}

}  // namespace s2
