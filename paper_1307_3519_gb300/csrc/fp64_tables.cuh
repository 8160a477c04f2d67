// fp64_tables.cuh -- FP64 exponential and logarithm from small tables, for the passes that
// FP64 issue bounds (a 64th of the FP32 rate on this part): table reduction as in Tang,
// "Table-driven implementation of the exponential function" (1989) and "... of the
// logarithm function" (1990).  Conversions work on the bits: they issue as slowly as the
// arithmetic.
#pragma once
#include <cmath>

namespace krux {

// exp(-x), 0 <= x <= 700: x = k ln2 / 2^kBits + r, |r| <= ln2 / 2^(kBits + 1), and exp(-r) - 1
// to r^3 (kBits = 12) or r^5 (7): the next term is below 3e-18.  tab holds 2^(-j / 2^kBits)
// as high and low parts.
template <int kBits>
__device__ __forceinline__ double exp_neg(double x, const double *tab) {
  static_assert(kBits == 12 || kBits == 7, "tables of 4096 or 128 entries");
  const double kMagic = 6755399441055744.0;  // 1.5 * 2^52: rounds to whole numbers
  const double t = fma(x, kBits == 12 ? 5909.278887481194 : 184.66496523378730914, kMagic);  // 2^kBits / ln 2
  const double kd = t - kMagic;
  const int k = __double2loint(t);
  // ln2 / 2^kBits in two parts, the first of 30 (35) bits (k has at most 23, 18)
  double r = fma(-kd, kBits == 12 ? 0x1.62e42fe8p-13 : 0x1.62e42fefap-8, x);
  r = fma(-kd, kBits == 12 ? 0x1.e8e7bcd5e4f1ep-43 : 0x1.cf79abc9e3b3ap-47, r);
  double q;
  if (kBits == 12) {
    q = fma(r, -1.0 / 6.0, 0.5);
  } else {
    q = fma(r, -1.0 / 120.0, 1.0 / 24.0);
    q = fma(r, q, -1.0 / 6.0);
    q = fma(r, q, 0.5);
  }
  q = fma(r, q, -1.0);
  q *= r;
  const double2 T = *reinterpret_cast<const double2 *>(tab + 2 * (k & ((1 << kBits) - 1)));
  const double y = T.x + fma(T.x, q, T.y);
  return __hiloint2double(__double2hiint(y) - ((k >> kBits) << 20), __double2loint(y));
}
template <int kBits>
inline void fill_exp_table(double *tab) {
  for (int j = 0; j < (1 << kBits); ++j) {
    const long double v = std::exp2(-(long double)j / (1 << kBits));
    tab[2 * j] = (double)v;
    tab[2 * j + 1] = (double)(v - (long double)tab[2 * j]);
  }
}

// log(u) of a normal u >= 1: u = 2^e m, inv within 2^-12 of the reciprocal of the middle of
// m's 512th of [1, 2), r = m inv - 1 (|r| < 2^-9), and log1p(r) to r^5 (the next term is
// below 1e-17).  tab holds inv, -log(inv) to 40 bits below the point and the rest of it,
// for each 512th; the first has inv = 1.
// The result comes with what its rounding left out, in `low`.
constexpr int kLogTab = 512;
__device__ __forceinline__ double log_ge1(double u, const double *tab, double &low) {
  const int hi = __double2hiint(u);
  const double m = __hiloint2double((hi & 0x000fffff) | 0x3ff00000, __double2loint(u));
  const double *T = tab + 3 * ((hi >> 11) & (kLogTab - 1));
  const double r = fma(m, T[0], -1.0);
  double q = fma(r, 0.2, -0.25);
  q = fma(r, q, 1.0 / 3.0);
  q = fma(r, q, -0.5);
  q = fma(r * r, q, r);
  // e as FP64 on the bits (2^52 + e, less 2^52), ln 2 to 40 bits below the point and the rest
  const double e = __hiloint2double(0x43300000, (hi >> 20) - 1023) - 4503599627370496.0;
  const double high = fma(e, 0x1.62e42fefa2p-1, T[1]);
  const double rest = q + fma(e, 0x1.9ef35793c7673p-41, T[2]);
  const double l = high + rest;
  low = (high - l) + rest;  // (high is 0 or the larger of the two)
  return l;
}
inline void fill_log_table(double *tab) {
  for (int i = 0; i < kLogTab; ++i) {
    const long double inv =
        i ? std::round(4096.0L / (1.0L + (i + 0.5L) / kLogTab)) / 4096.0L : 1.0L;
    const long double l = -std::log(inv), high = std::floor(std::ldexp(l, 40)) / std::ldexp(1.0L, 40);
    tab[3 * i] = (double)inv;
    tab[3 * i + 1] = (double)high;
    tab[3 * i + 2] = (double)(l - high);
  }
}

}  // namespace krux
