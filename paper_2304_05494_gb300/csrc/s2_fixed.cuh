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
// products of three fields and a grid factor (2^-200 .. 2^200 as well) then
// stay far inside the range of a double.
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

// x 2^n, x and the result being normal.
__device__ __forceinline__ double fx_ldexp(double x, int n) {
  return __hiloint2double(__double2hiint(x) + n * (1 << 20), __double2loint(x));
}

}  // namespace s2
