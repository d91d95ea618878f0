// Chebyshev coefficients of the small exponential (krylov_impl.cuh), computed by the
// compiler: a __constant__ table with a constant initialiser is part of the module,
// on every device and before the first launch on any stream.  (Filled by a copy on
// the host's first use it would be there for one device only, and ordered with
// the legacy stream, not with a non-blocking one.)
#pragma once

namespace etd {

constexpr int CHEB_TABLES = 19, CHEB_MAX = 1529;

// Coefficients 2 e^-a I_k(a) of e^(a (x - 1)) for a = 2^(i/2), i = 0 ..
// CHEB_TABLES - 1, down to 1e-24: table i at c + at[i] (20 coefficients at a = 1,
// 87 at 64, 233 at 512).
struct ChebTables {
  double c[CHEB_MAX];
  double two_a[CHEB_TABLES];  // 2 / a
  int at[CHEB_TABLES + 1];
};

// I_k(a) up to a factor by Miller's downward recurrence I_{k-1} = I_{k+1} +
// (2k/a) I_k (Abramowitz & Stegun 9.12), normalised by I_0 + 2 sum I_k = e^a.
constexpr ChebTables cheb_tables() {
  ChebTables o{};
  int n = 0;
  double pw = 1.0;  // 2^(i/2) for even i
  for (int i = 0; i < CHEB_TABLES; ++i) {
    const double a = i % 2 ? pw * 1.4142135623730951 : pw;
    if (i % 2) pw *= 2.0;
    o.two_a[i] = 2.0 / a;
    o.at[i] = n;
    double t[512] = {};
    double up = 0.0, sum = 0.0, cur = 1e-200;
    for (int k = 511; k >= 0; --k) {  // cur = I_k, up = I_{k+1}
      t[k] = cur;
      sum += k > 0 ? 2.0 * cur : cur;
      const double down = up + 2.0 * k / a * cur;
      up = cur;
      cur = down;
      if (cur > 1e200) {
        for (int j = k; j < 512; ++j) t[j] = t[j] > 1e-100 ? t[j] * 1e-200 : 0.0;
        cur *= 1e-200;
        up *= 1e-200;
        sum *= 1e-200;
      }
    }
    for (int k = 0; k < 512 && n < CHEB_MAX; ++k) {
      const double c = 2.0 * t[k] / sum;
      if (c < 1e-24) break;
      o.c[n++] = c;
    }
  }
  o.at[CHEB_TABLES] = n;
  return o;
}

}  // namespace etd
