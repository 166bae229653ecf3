// Host construction of the Planck tables as the kernels read them: the FP64 edge table, and the FP32 band
// table's coefficients from its nodes (at the end).
//
// FP64 edge table (PETAB_ROWS rows of 8 coefficients; see planck_edge_tab in fx_device.cuh).  Row n holds the polynomial in t = 16 x - n, |t| <= 1/2, that
// interpolates at the 8 Chebyshev nodes
//   n < PETAB_SPLIT:   R(x) = x^-3 Int_0^x s^3/(e^s - 1) ds   (Q = x^3 R)
//   n >= PETAB_SPLIT:  Q(x) = Int_x^inf s^3/(e^s - 1) ds.
// Interpolation error relative to the value: 2 (1/64)^8 / 8! ~ 2e-19 for the exponential part, less
// below it, so the coefficients are formed in double-double arithmetic (two doubles with error-free
// sums and products; Dekker 1971, Knuth) and rounded once.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "fx_types.h"

namespace fx {
namespace ddp {

struct DD { double h, l; };
inline DD two_sum(double a, double b) {
  const volatile double s = a + b, bv = s - a, av = s - bv;
  const volatile double eb = b - bv, ea = a - av;
  return {s, ea + eb};
}
inline DD quick(double a, double b) {
  const volatile double s = a + b, d = s - a;
  return {s, b - d};
}
inline DD add(DD a, DD b) {
  const DD s = two_sum(a.h, b.h), t = two_sum(a.l, b.l);
  const volatile double c = s.l + t.h;
  const DD u = quick(s.h, c);
  const volatile double e = u.l + t.l;
  return quick(u.h, e);
}
inline DD neg(DD a) { return {-a.h, -a.l}; }
inline DD mul(DD a, DD b) {
  const volatile double p = a.h * b.h;
  const double e = std::fma(a.h, b.h, -p);
  const volatile double x = a.h * b.l, y = a.l * b.h;
  const volatile double c = x + y;
  const volatile double f = e + c;
  return quick(p, f);
}
inline DD div(DD a, DD b) {
  const volatile double q0 = a.h / b.h;
  DD r = add(a, neg(mul({q0, 0.0}, b)));
  const volatile double q1 = r.h / b.h;
  r = add(r, neg(mul({q1, 0.0}, b)));
  const volatile double q2 = r.h / b.h;
  return add(quick(q0, q1), {q2, 0.0});
}
inline DD of(double x) { return {x, 0.0}; }
// e^-x: Taylor series of x / 2^8, squared eight times
inline DD exp_neg(DD x) {
  const DD y = mul(x, of(-1.0 / 256.0));
  DD s = of(1.0), t = of(1.0);
  for (int k = 1; k <= 26; ++k) {
    t = div(mul(t, y), of((double)k));
    s = add(s, t);
  }
  for (int k = 0; k < 8; ++k) s = mul(s, s);
  return s;
}

}  // namespace ddp

// The table, built once per process (universal constants), PETAB_ROWS x 8 doubles.
inline const std::vector<double>& planck_edge_table() {
  static const std::vector<double> table = [] {
    using namespace ddp;
    // b_2m = B_2m / (2m)!: the first Bernoulli numbers as rationals, the others from the even zeta
    // values, 2 (-1)^(m+1) zeta(2m) / (2 pi)^2m
    constexpr int M = 34;
    DD b[M + 1];
    const double num[8] = {1, -1, 1, -1, 5, -691, 7, -3617}, den[8] = {6, 30, 42, 30, 66, 2730, 6, 510};
    const DD pi = {3.14159265358979311600e+00, 1.22464679914735320717e-16};
    const DD tp2 = mul(mul(pi, pi), of(4.0));
    DD fact = of(1.0), pw = of(1.0);
    for (int m = 1; m <= M; ++m) {
      fact = mul(fact, of((2.0 * m - 1.0) * (2.0 * m)));
      pw = mul(pw, tp2);
      if (m <= 8) {
        b[m] = div(div(of(num[m - 1]), of(den[m - 1])), fact);
      } else {
        DD z = of(1.0);
        for (int k = 2; k <= 60; ++k) {
          DD p = of(1.0);
          const DD ik = div(of(1.0), of((double)k * k));
          for (int j = 0; j < m; ++j) p = mul(p, ik);
          z = add(z, p);
        }
        b[m] = div(mul(z, of(m % 2 ? 2.0 : -2.0)), pw);
      }
    }
    DD bq[M + 1], rk[25];  // b_2m / (2m + 3), 1 / k
    for (int m = 1; m <= M; ++m) bq[m] = div(b[m], of(2.0 * m + 3.0));
    for (int k = 1; k <= 24; ++k) rk[k] = div(of(1.0), of((double)k));
    // y = e^-x (upper rows)
    auto value = [&](int n, DD x, DD y) -> DD {
      if (n < PETAB_SPLIT) {
        const DD x2 = mul(x, x);
        DD s = of(0.0);
        for (int m = M; m >= 1; --m) s = add(mul(s, x2), bq[m]);
        return add(add(div(of(1.0), of(3.0)), mul(x, of(-0.125))), mul(s, x2));
      }
      const DD x2 = mul(x, x), x3 = mul(x2, x);
      DD yn = y, s = of(0.0);
      for (int k = 1; k <= 24; ++k) {
        const DD r = rk[k];
        DD p = add(mul(r, of(6.0)), mul(x, of(6.0)));
        p = add(mul(p, r), mul(x2, of(3.0)));
        p = add(mul(p, r), x3);
        const DD t = mul(mul(yn, r), p);
        s = add(s, t);
        if (t.h < 1e-34 * s.h) break;
        yn = mul(yn, y);
      }
      return s;
    };
    // the 8 Chebyshev nodes of [-1/2, 1/2], and the inverse of their Vandermonde matrix (columns:
    // the monomial coefficients of the Lagrange polynomials)
    constexpr int K = 8;
    double node[K];
    for (int j = 0; j < K; ++j) node[j] = 0.5 * std::cos(M_PI * (2 * j + 1) / (2.0 * K));
    DD lag[K][K];
    for (int j = 0; j < K; ++j) {
      DD c[K] = {};
      c[0] = of(1.0);
      int deg = 0;
      DD d = of(1.0);
      for (int i = 0; i < K; ++i) {
        if (i == j) continue;
        for (int q = deg + 1; q >= 0; --q) {
          DD v = q > 0 ? c[q - 1] : of(0.0);
          if (q <= deg) v = add(v, mul(c[q], of(-node[i])));
          c[q] = v;
        }
        ++deg;
        d = mul(d, two_sum(node[j], -node[i]));
      }
      for (int q = 0; q < K; ++q) lag[j][q] = div(c[q], d);
    }
    std::vector<double> t((size_t)PETAB_ROWS * K);
    DD en = of(1.0), ej[K];  // e^-(n/16) by multiplication, e^-(node/16)
    const DD e1 = exp_neg(of(1.0 / 16.0));
    for (int j = 0; j < K; ++j) ej[j] = exp_neg(of(node[j] / 16.0));
    for (int n = 0; n < PETAB_ROWS; ++n, en = mul(en, e1)) {
      DD f[K];
      for (int j = 0; j < K; ++j) f[j] = value(n, mul(two_sum((double)n, node[j]), of(1.0 / 16.0)), mul(en, ej[j]));
      for (int q = 0; q < K; ++q) {
        DD s = of(0.0);
        for (int j = 0; j < K; ++j) s = add(s, mul(lag[j][q], f[j]));
        t[(size_t)n * K + q] = s.h;
      }
    }
    return t;
  }();
  return table;
}

// Coefficients of one interval (see PlanckTable) from its two nodes (L - floor(L), h dL/du, floor(L),
// 2^floor(L)).
inline void planck_interval_entry(const float4& p, const float4& q, float c[4]) {
  const double d = ((double)q.z - (double)p.z) + ((double)q.x - (double)p.x);  // L at the right node less L at the left
  const double m0 = p.y, m1 = q.y;
  c[0] = p.x;
  c[1] = p.y;
  c[2] = (float)(3.0 * d - 2.0 * m0 - m1);
  c[3] = (float)(m0 + m1 - 2.0 * d);
  unsigned sc, b;
  std::memcpy(&sc, &p.w, 4);
  std::memcpy(&b, &c[3], 4);
  b = (b & ~0xffu) | (sc >> 23);
  std::memcpy(&c[3], &b, 4);
}
// The device table: (groups + 1)/2 pairs (an odd count's last pair repeats its group).
inline std::vector<float4> planck_device_table(const std::vector<float4>& tab, int G, int nu, bool node_major) {
  const int NP = (G + 1) / 2;
  std::vector<float4> out((size_t)2 * NP * nu);
  for (int p = 0; p < NP; ++p)
    for (int i = 0; i < nu; ++i) {
      float c[2][4];
      for (int s = 0; s < 2; ++s) {
        const float4* const t = tab.data() + (size_t)std::min(2 * p + s, G - 1) * nu;
        planck_interval_entry(t[i], t[std::min(i + 1, nu - 1)], c[s]);
      }
      float4* const e = out.data() + 2 * (node_major ? (size_t)i * NP + p : (size_t)p * nu + i);
      e[0] = make_float4(c[0][0], c[1][0], c[0][1], c[1][1]);
      e[1] = make_float4(c[0][2], c[1][2], c[0][3], c[1][3]);
    }
  return out;
}

}  // namespace fx
