// Power law and logarithm of the double-precision path on the integer unit.
//
// The double unit of GB300 issues one operation per 64 clocks and scheduler
// (csrc/s2_fixed.cuh); a power through repeated squaring and a Halley step
// cost the primitive pass 24 of its 41 operations per point, a logarithm of
// the thermally perfect gas more.  Both are evaluated in 64-bit fixed point
// instead, with the table-driven method of P. T. P. Tang (ACM TOMS 15
// (1989) and 16 (1990)): x = 2^e m, a table value r near 1/m with 10
// fraction bits makes t = m r - 1 exact and |t| < 2^-7.6, then
//   log2 x = e - log2 r + log2(1 + t),
//   2^E = 2^n 2^(j/128) e^z,  E = n + j/128 + z / ln 2,  0 <= z < 2^-7.5,
// with the series of log(1 + t) and e^z; the factors that enter with t^4 or
// z^3 and higher powers need 32 bits only.  Fraction bits are written Qn.
// The result is within 0.54 ulp of x^omega (the Halley step: 4 ulp).  The
// primitive pass on 420 x 250 x 320 points went from 3.04 to 1.29 ms, with
// the thermally perfect gas on 256 x 128 x 128 from 1.43 to 0.73.
#pragma once
#include <math.h>

#include "s2_fixed.cuh"

namespace s2 {

struct PowTab {
  long long wl[128];  // -omega log2(r / 1024), Q58
  long long ll[128];  // -ln(r / 1024), Q58
  long long b[128];   // 2^(j/128), Q62
  int r[128];         // 1024 / (1 + (i + 1/2) / 128), rounded
};

constexpr long long POW_LN2_Q63 = 0x58b90bfbe8e7bcd6ll;  // ln 2
constexpr long long POW_LN2_Q58 = POW_LN2_Q63 >> 5;

// The part of the table that does not depend on omega, and the logarithms
// (base 2) for the rest: evaluated once per process (128 extended-precision
// logarithms and exponentials take 0.5 ms where they are done in software).
struct PowBase {
  PowTab t;
  long double lg[128];
  PowBase() {
    const long double ln2 = logl(2.0L);
    for (int i = 0; i < 128; ++i) {
      t.r[i] = (int)floorl(1024.0L / (1.0L + (i + 0.5L) / 128.0L) + 0.5L);
      const long double lr = logl(t.r[i] / 1024.0L);
      lg[i] = lr / ln2;
      t.ll[i] = llroundl(ldexpl(-lr, 58));
      t.b[i] = llroundl(ldexpl(expl(ln2 * i / 128.0L), 62));
    }
  }
};

// The table, and omega and the range of its use in d (visc_exp set).
inline void pow_setup(Dev &d, PowTab &t) {
  static const PowBase base;
  const long double ln2 = logl(2.0L), w = d.visc_exp;
  const bool inside = fabs(d.visc_exp) <= 4.0;
  t = base.t;
  for (int i = 0; i < 128; ++i) t.wl[i] = inside ? llroundl(ldexpl(-w * base.lg[i], 58)) : 0;
  d.pow_emax = -1;  // no exponent is in range
  if (inside) {
    d.pow_w = llroundl(ldexpl(w, 58));
    d.pow_w2 = llroundl(ldexpl(w / ln2, 60));
    // (omega is cut at Q58, an error that an exponent multiplies)
    d.pow_emax = d.visc_exp == 0.0 ? 32 : (int)fmin(32.0, floor(30.0 / fabs(d.visc_exp)) - 1.0);
  }
}

// ln(1 + t) in Q67 of the mantissa of a positive normal x, and its table
// index and exponent.
__device__ __forceinline__ long long pow_log1p(double x, const PowTab *tab, int &i, int &e) {
  const int hx = __double2hiint(x);
  e = (hx >> 20) - 1023;
  i = (hx >> 13) & 127;
  const long long m = ((long long)((hx & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(x);
  const long long t = m * __ldg(tab->r + i) - (1ll << 62);  // Q62
  const int t32 = (int)(t >> 24);                           // Q38
  // 1 - t (1/2 - t (1/3 - t (1/4 - t (1/5 - t (1/6 - t/7)))))
  int h = 0x7fffffff / 7;
  h = 0x7fffffff / 6 - (int)(((long long)t32 * h) >> 38);
  h = 0x7fffffff / 5 - (int)(((long long)t32 * h) >> 38);
  h = (1 << 29) - (int)(((long long)t32 * h) >> 38);
  const long long h3 = (1ll << 62) / 3 - (((long long)t32 * h) >> 7);
  const long long ts = t << 7;
  const long long h2 = (1ll << 61) - (__mul64hi(ts, h3) >> 5);
  return __mul64hi(ts, (1ll << 62) - (__mul64hi(ts, h2) >> 5));
}

// x^omega for a positive normal x with |exponent of x| <= Dev::pow_emax
// (omega in Q58 and omega / ln 2 in Q60 from the parameters).
__device__ __forceinline__ double pow_fixed(const Dev &d, double x) {
  int i, e;
  const long long ln = pow_log1p(x, d.powt, i, e);
  const long long E = e * d.pow_w + __ldg(d.powt->wl + i) + ((__mul64hi(ln << 1, d.pow_w2) + 32) >> 6);  // Q58
  const int n = (int)(E >> 58);
  const long long f = E & ((1ll << 58) - 1);
  const long long B = __ldg(d.powt->b + (int)(f >> 51));
  const long long z = __mul64hi((f & ((1ll << 51) - 1)) << 12, POW_LN2_Q63);  // Q69
  const int z32 = (int)(z >> 31);                                            // Q38
  // z (1 + z (1/2 + z (1/6 + z (1/24 + z (1/120 + z/720)))))
  int h = (int)((1ll << 34) / 720);
  h = (int)((1ll << 34) / 120) + (int)(((long long)z32 * h) >> 38);
  h = (int)((1ll << 34) / 24) + (int)(((long long)z32 * h) >> 38);
  const long long h3 = (1ll << 62) / 6 + (((long long)z32 * h) >> 10);
  const long long h2 = (1ll << 61) + (__mul64hi(z, h3) >> 5);
  const long long h1 = (1ll << 62) + (__mul64hi(z, h2) >> 5);
  // Q62, from 1 to 2, which a power just below 2^(n+1) can reach
  const unsigned long long r = (unsigned long long)(B + ((__mul64hi(B, __mul64hi(z, h1)) + 4) >> 3));
  const unsigned long long m = (r + (1 << 9)) >> 10;  // bit 52 set, or 2^53
  return __hiloint2double((int)(m >> 32) + (n + 1022) * (1 << 20), (int)m);
}

// mu = (T/T_ref)^omega / Re; outside the table method's range (an exponent
// omega beyond 4, T many powers of two from T_ref, or not positive) by the
// general function.
__device__ __forceinline__ double viscosity_fixed(const Dev &d, double T) {
  const double x = T * d.inv_t_ref;
  const int e = (__double2hiint(x) >> 20) - 1023;  // the sign bit makes e large
  if (d.powt && e >= -d.pow_emax && e <= d.pow_emax) return pow_fixed(d, x) * d.inv_re;
  return viscosity(d, T);
}

// ln x for a positive x of moderate size, to 2^-57 absolute.
struct FixedLog {
  const PowTab *tab;
  __device__ __forceinline__ double operator()(double x) const {
    const int he = (__double2hiint(x) >> 20) - 1023;
    if (!tab || (unsigned)(he + 40) > 80u) return log(x);
    int i, e;
    const long long ln = pow_log1p(x, tab, i, e);
    return fx_i2d(e * POW_LN2_Q58 + __ldg(tab->ll + i) + ((ln + 256) >> 9), -58);
  }
};

}  // namespace s2
