// Line operators of the tensor-product elements to ~100 bits (host code).
//
// The fixed-point kernels hold operator entries to 60 bits; entries taken
// from the FP64 construction (Vandermonde inverses, a few 1e-15 off) would
// bound their accuracy.  Here the line points are polished by Newton steps
// and the operators formed in double-double arithmetic: a value is hi + lo,
// with Knuth's two-sum and an FMA for the error of a product.
#pragma once
#include <cmath>
#include <vector>

namespace frgb {

struct DD {
  double hi = 0.0, lo = 0.0;
  DD() = default;
  DD(double h) : hi(h) {}
  DD(double h, double l) : hi(h), lo(l) {}
};

inline DD dd_sum(double a, double b) {
  const double s = a + b, t = s - a;
  return DD(s, (a - (s - t)) + (b - t));
}
inline DD operator-(DD a) { return DD(-a.hi, -a.lo); }
inline DD operator+(DD a, DD b) {
  const DD s = dd_sum(a.hi, b.hi), t = dd_sum(a.lo, b.lo);
  const DD u = dd_sum(s.hi, s.lo + t.hi);
  return dd_sum(u.hi, u.lo + t.lo);
}
inline DD operator-(DD a, DD b) { return a + (-b); }
inline DD operator*(DD a, DD b) {
  const double p = a.hi * b.hi;
  const double e = std::fma(a.hi, b.hi, -p) + (a.hi * b.lo + a.lo * b.hi);
  return dd_sum(p, e);
}
inline DD operator/(DD a, DD b) {
  DD q(a.hi / b.hi);
  for (int i = 0; i < 2; ++i) q = q + DD((a - q * b).hi / b.hi);
  return q;
}

// Legendre P_n(x) and P_n'(x)
inline void dd_legendre(int n, DD x, DD* p, DD* d) {
  DD p0(1.0), p1 = x, d0(0.0), d1(1.0);
  if (n == 0) {
    *p = p0;
    *d = d0;
    return;
  }
  for (int k = 2; k <= n; ++k) {
    const DD p2 = (DD(2.0 * k - 1.0) * x * p1 - DD(k - 1.0) * p0) / DD(double(k));
    const DD d2 = d0 + DD(2.0 * k - 1.0) * p1;
    p0 = p1;
    p1 = p2;
    d0 = d1;
    d1 = d2;
  }
  *p = p1;
  *d = d1;
}

// Operators on n Gauss-Legendre (family 0) or Gauss-Lobatto (1) points near
// x: derivative d[a * n + m] = l_m'(x_a), interpolation lm[m] = l_m(-1) to the
// minus face and DG correction weights gr[a] = g_R'(x_a) of the plus face
// (the other face's are their mirror images).
struct DDLine {
  std::vector<DD> d, lm, gr;
};

inline DDLine dd_line_ops(const std::vector<double>& x, int family) {
  const int n = int(x.size());
  std::vector<DD> z(x.begin(), x.end());
  DD p, q;
  for (int a = 0; a < n; ++a) {
    if (family == 1 && (a == 0 || a == n - 1)) {
      z[a] = DD(a == 0 ? -1.0 : 1.0);
      continue;
    }
    if (2 * a + 1 == n) {
      z[a] = DD(0.0);
      continue;
    }
    for (int it = 0; it < 4; ++it) {
      if (family == 0) {
        dd_legendre(n, z[a], &p, &q);
        z[a] = z[a] - p / q;
      } else {  // roots of P_{n-1}': (1 - x^2) P'' = 2 x P' - (n - 1) n P
        dd_legendre(n - 1, z[a], &p, &q);
        const DD w = DD(1.0) - z[a] * z[a];
        z[a] = z[a] - q * w / (DD(2.0) * z[a] * q - DD(double((n - 1) * n)) * p);
      }
    }
  }
  DDLine o;
  std::vector<DD> w(n, DD(1.0));  // prod_k (x_m - x_k)
  for (int m = 0; m < n; ++m)
    for (int k = 0; k < n; ++k)
      if (k != m) w[m] = w[m] * (z[m] - z[k]);
  o.d.assign(size_t(n) * n, DD(0.0));
  for (int a = 0; a < n; ++a) {
    DD diag(0.0);
    for (int m = 0; m < n; ++m)
      if (m != a) {
        const DD v = w[a] / (w[m] * (z[a] - z[m]));
        o.d[size_t(a) * n + m] = v;
        diag = diag - v;
      }
    o.d[size_t(a) * n + a] = diag;
  }
  for (int m = 0; m < n; ++m) {
    DD v(1.0);
    for (int k = 0; k < n; ++k)
      if (k != m) v = v * (DD(-1.0) - z[k]) / (z[m] - z[k]);
    o.lm.push_back(v);
  }
  for (int a = 0; a < n; ++a) {  // g_R = (P_n + P_{n-1}) / 2
    DD d0, d1;
    dd_legendre(n, z[a], &p, &d1);
    dd_legendre(n - 1, z[a], &p, &d0);
    o.gr.push_back(DD(0.5) * (d0 + d1));
  }
  return o;
}

// v 2^(60 - s) to the nearest integer
inline long long dd_fixed(DD v, int s) {
  const double h = std::ldexp(v.hi, 60 - s), l = std::ldexp(v.lo, 60 - s), r = std::rint(h);
  return (long long)r + std::llrint((h - r) + l);
}

}  // namespace frgb
