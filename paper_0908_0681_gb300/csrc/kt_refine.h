// Eigenpairs of the blocks in double-double arithmetic (host, at model setup).
//
// The operator matrices between block eigenbases need their zeros: an element that a symmetry forbids
// but that an eigenvector's rounding fills is amplified by the propagator as exp(dt gap). In FP64 that
// rounding reaches 1e-13 and cannot be told from a small element of the model (a weak pair hopping, a weak
// splitting). In 106 bits it ends below 1e-24, and elements above it are the model's own.
#pragma once

#include <cmath>
#include <vector>

namespace kt {

// An unevaluated sum h + l, |l| <= ulp(h) / 2; operations with a relative error of a few 2^-104 (T. J. Dekker,
// Numer. Math. 18, 1971; the error of a product by a fused multiply-add).
struct dd {
  double h = 0.0, l = 0.0;
  dd() = default;
  dd(double a) : h(a) {}
  dd(double a, double b) : h(a), l(b) {}
};
inline dd dd_sum(double a, double b) {  // exact
  const double s = a + b, bb = s - a;
  return dd(s, (a - (s - bb)) + (b - bb));
}
inline dd dd_fast(double a, double b) {  // exact for |a| >= |b|
  const double s = a + b;
  return dd(s, b - (s - a));
}
inline dd operator+(dd a, dd b) {
  const dd s = dd_sum(a.h, b.h), t = dd_sum(a.l, b.l);
  const dd u = dd_fast(s.h, s.l + t.h);
  return dd_fast(u.h, u.l + t.l);
}
inline dd operator-(dd a) { return dd(-a.h, -a.l); }
inline dd operator-(dd a, dd b) { return a + (-b); }
inline dd operator*(dd a, dd b) {
  const double p = a.h * b.h;
  double e = std::fma(a.h, b.h, -p);
  e = std::fma(a.h, b.l, e);
  e = std::fma(a.l, b.h, e);
  return dd_fast(p, e);
}
inline dd operator/(dd a, dd b) {
  const double q = a.h / b.h;
  const dd r = a - b * dd(q);
  const double q2 = r.h / b.h;
  const dd r2 = r - b * dd(q2);
  return dd_fast(q, q2) + dd(r2.h / b.h);
}
inline dd dd_sqrt(dd a) {  // a > 0: a Newton step from the FP64 root, twice
  const double x = std::sqrt(a.h);
  dd r = dd(x) + (a - dd(x) * dd(x)) / dd(2.0 * x);
  return r + (a - r * r) / (dd(2.0) * r);
}
inline double dd_abs(dd a) { return std::fabs(a.h); }

// What refine_eigh leaves of an off-diagonal element, for a block of d rows with norm (largest absolute column sum)
// nrm: the rounding of sums of d products.
inline double refine_rest(int d, double nrm) { return 4.0 * d * std::ldexp(nrm, -104); }

// Eigenpairs of the symmetric d x d matrix H (row-major) from an FP64 eigenbasis V0 (column j in V0[i d + j]):
// orthonormalised, and H rotated to a diagonal in it by Jacobi rotations, which from an FP64 basis are small
// but between nearly degenerate vectors; pair j stays pair j. The rest off the diagonal is at most
// refine_rest(d, nrm), so degenerate vectors keep the FP64 basis' choice.
inline void refine_eigh(int d, const std::vector<dd> &H, double nrm, const std::vector<double> &V0, std::vector<dd> &w,
                        std::vector<dd> &V) {
  // vector j in V[j d ..]
  V.resize((size_t)d * d);
  for (int j = 0; j < d; ++j) {
    dd *v = &V[(size_t)j * d];
    for (int i = 0; i < d; ++i) v[i] = dd(V0[(size_t)i * d + j]);
    for (int k = 0; k <= j; ++k) {  // modified Gram-Schmidt, then the norm
      const dd *u = &V[(size_t)k * d];
      dd s;
      for (int i = 0; i < d; ++i) s = s + u[i] * v[i];
      if (k < j)
        for (int i = 0; i < d; ++i) v[i] = v[i] - s * u[i];
      else {
        const dd r = dd(1.0) / dd_sqrt(s);
        for (int i = 0; i < d; ++i) v[i] = v[i] * r;
      }
    }
  }
  std::vector<dd> A((size_t)d * d), t(d);
  for (int q = 0; q < d; ++q) {
    const dd *v = &V[(size_t)q * d];
    for (int i = 0; i < d; ++i) {
      dd s;
      for (int k = 0; k < d; ++k)
        if (H[(size_t)i * d + k].h != 0.0) s = s + H[(size_t)i * d + k] * v[k];
      t[i] = s;
    }
    for (int p = 0; p <= q; ++p) {
      const dd *u = &V[(size_t)p * d];
      dd s;
      for (int i = 0; i < d; ++i) s = s + u[i] * t[i];
      A[(size_t)p * d + q] = A[(size_t)q * d + p] = s;
    }
  }
  const double rest = refine_rest(d, nrm);
  for (int sweep = 0; sweep < 50; ++sweep) {
    bool any = false;
    for (int p = 0; p < d; ++p)
      for (int q = p + 1; q < d; ++q) {
        const dd apq = A[(size_t)p * d + q];
        if (!(dd_abs(apq) > rest)) continue;
        any = true;
        const dd theta = (A[(size_t)q * d + q] - A[(size_t)p * d + p]) / (dd(2.0) * apq);
        dd tn;
        if (dd_abs(theta) > 1e100) {
          tn = dd(0.5) / theta;
        } else {
          const dd a = theta.h >= 0.0 ? theta : -theta;
          tn = dd(1.0) / (a + dd_sqrt(a * a + dd(1.0)));
          if (theta.h < 0.0) tn = -tn;
        }
        const dd c = dd(1.0) / dd_sqrt(tn * tn + dd(1.0)), s = tn * c;
        for (int k = 0; k < d; ++k) {
          if (k == p || k == q) continue;
          const dd akp = A[(size_t)k * d + p], akq = A[(size_t)k * d + q];
          A[(size_t)k * d + p] = A[(size_t)p * d + k] = c * akp - s * akq;
          A[(size_t)k * d + q] = A[(size_t)q * d + k] = s * akp + c * akq;
        }
        A[(size_t)p * d + p] = A[(size_t)p * d + p] - tn * apq;
        A[(size_t)q * d + q] = A[(size_t)q * d + q] + tn * apq;
        A[(size_t)p * d + q] = A[(size_t)q * d + p] = dd();
        dd *vp = &V[(size_t)p * d], *vq = &V[(size_t)q * d];
        for (int i = 0; i < d; ++i) {
          const dd a = vp[i], b = vq[i];
          vp[i] = c * a - s * b;
          vq[i] = s * a + c * b;
        }
      }
    if (!any) break;
  }
  w.resize(d);
  for (int j = 0; j < d; ++j) w[j] = A[(size_t)j * d + j];
}

}  // namespace kt
