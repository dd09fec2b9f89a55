// Nodes and weights of the Rys quadrature (Dupuis, Rys, King, J. Chem. Phys. 65, 111 (1976)):
// int_0^1 f(t^2) exp(-T t^2) dt = sum_r w_r f(x_r), exact for polynomials f of degree <= 2n - 1, as
// polynomials in T on unit intervals of [0, 100), and the large-T limit.
//
// For one T: the recurrence coefficients of the polynomials orthogonal under exp(-T t^2) on t in [0, 1] in the
// variable x = t^2 by Stieltjes' procedure on an 80-point Gauss-Legendre rule in t (Gautschi, Orthogonal
// Polynomials, 2004), the nodes by bisection between the nodes of one order less and Newton's method, the
// weights as 1 / sum_k p_k(x_r)^2 over the orthonormal polynomials (a sum of squares: the weights keep their
// relative accuracy down to exp(-T)). Everything in double-double arithmetic (Dekker 1971; about 31 digits),
// whose results do not depend on the machine's long double. The degree-12 Chebyshev fit of an interval is
// below 1e-16 of every node and weight (the fit's error falls off as (1/4)^k / k!).
//
// Above T = 100: x_r = X_r / T, w_r = W_r / (2 sqrt(T)) with the Gauss rule of x^(-1/2) exp(-x) on [0, inf);
// the part of the measure beyond t = 1 is exp(-100).
#include <algorithm>
#include <cmath>
#include <exception>
#include <mutex>
#include <thread>
#include <vector>

#include "mdx_internal.h"

namespace mdx {
namespace {

struct dd {
  double h = 0.0, l = 0.0;
  dd() = default;
  dd(double x) : h(x) {}
  dd(double x, double y) : h(x), l(y) {}
};
inline dd quick(double a, double b) {
  const double s = a + b;
  return dd(s, b - (s - a));
}
inline dd operator+(dd a, dd b) {
  const double s = a.h + b.h, bb = s - a.h;
  const double e = (a.h - (s - bb)) + (b.h - bb);
  const double t = a.l + b.l, tb = t - a.l;
  const double f = (a.l - (t - tb)) + (b.l - tb);
  dd r = quick(s, e + t);
  return quick(r.h, r.l + f);
}
inline dd operator-(dd a) { return dd(-a.h, -a.l); }
inline dd operator-(dd a, dd b) { return a + (-b); }
inline dd operator*(dd a, dd b) {
  const double p = a.h * b.h;
  const double e = std::fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h);
  return quick(p, e);
}
inline dd operator/(dd a, dd b) {
  const double q1 = a.h / b.h;
  dd r = a - b * dd(q1);
  const double q2 = r.h / b.h;
  r = r - b * dd(q2);
  const double q3 = r.h / b.h;
  return quick(q1, q2) + dd(q3);
}
inline dd sqrt_dd(dd a) {
  if (a.h <= 0.0) return dd(0.0);
  dd x(std::sqrt(a.h));
  x = dd(0.5) * (x + a / x);
  return dd(0.5) * (x + a / x);
}
// exp(a) for a <= 0: a = k ln 2 + 64 r, Taylor series of exp(r), six squarings
dd exp_dd(dd a) {
  const dd ln2(0.6931471805599453094, 2.319046813846299558e-17);
  const int k = (int)std::nearbyint(a.h / ln2.h);
  const dd r = (a - dd((double)k) * ln2) * dd(1.0 / 64.0);
  dd term(1.0), sum(1.0);
  for (int i = 1; i < 18; ++i) {
    term = term * r / dd((double)i);
    sum = sum + term;
  }
  for (int i = 0; i < 6; ++i) sum = sum * sum;
  return dd(std::ldexp(sum.h, k), std::ldexp(sum.l, k));
}

constexpr int kQuad = 80;
struct Legendre {
  dd t[kQuad], w[kQuad];   // on [0, 1]
  Legendre() {
    for (int i = 0; i < kQuad; ++i) {
      dd x(std::cos(3.14159265358979323846 * (i + 0.75) / (kQuad + 0.5)));
      dd d;
      for (int it = 0; it < 6; ++it) {
        dd p0(1.0), p1 = x;
        for (int k = 2; k <= kQuad; ++k) {
          const dd p = (dd(2.0 * k - 1.0) * x * p1 - dd(k - 1.0) * p0) / dd((double)k);
          p0 = p1;
          p1 = p;
        }
        d = dd((double)kQuad) * (x * p1 - p0) / (x * x - dd(1.0));
        x = x - p1 / d;
      }
      t[i] = (x + dd(1.0)) * dd(0.5);
      w[i] = dd(1.0) / ((dd(1.0) - x * x) * d * d);
    }
  }
};

constexpr int N = kRysMax;

// Gauss rules of orders 1..N from the recurrence coefficients al, be (be[0]: the measure's integral), the
// nodes in (0, top): x[n], w[n] with n entries each, ascending.
void gauss(const dd* al, const dd* be, double top, std::vector<dd>* x, std::vector<dd>* w) {
  dd rb[N + 1];
  for (int k = 0; k <= N; ++k) rb[k] = sqrt_dd(be[k]);
  x[0].clear();
  for (int n = 1; n <= N; ++n) {
    x[n].assign(n, dd());
    w[n].assign(n, dd());
    auto monic = [&](double z) {
      double p0 = 0.0, p1 = 1.0;
      for (int k = 0; k < n; ++k) {
        const double p = (z - al[k].h) * p1 - (k ? be[k].h * p0 : 0.0);
        p0 = p1;
        p1 = p;
      }
      return p1;
    };
    for (int r = 0; r < n; ++r) {
      double lo = r == 0 ? 0.0 : x[n - 1][r - 1].h, hi = r == n - 1 ? top : x[n - 1][r].h;
      const bool rising = (n - r) % 2 == 1;   // p_n changes sign from - to + at this node
      for (int it = 0; it < 40; ++it) {
        const double mid = 0.5 * (lo + hi);
        if ((monic(mid) > 0.0) == rising) hi = mid; else lo = mid;
      }
      dd z(0.5 * (lo + hi));
      for (int it = 0; it < 4; ++it) {
        dd p0, p1(1.0), q0, q1;   // values and derivatives
        for (int k = 0; k < n; ++k) {
          const dd c = z - al[k];
          dd p = c * p1, q = c * q1 + p1;
          if (k) { p = p - be[k] * p0; q = q - be[k] * q0; }
          p0 = p1; p1 = p;
          q0 = q1; q1 = q;
        }
        z = z - p1 / q1;
      }
      dd s, p0, p1 = dd(1.0) / rb[0];
      for (int k = 0; k < n; ++k) {
        s = s + p1 * p1;
        dd p = (z - al[k]) * p1;
        if (k) p = p - rb[k] * p0;
        p0 = p1;
        p1 = p / rb[k + 1];
      }
      x[n][r] = z;
      w[n][r] = dd(1.0) / s;
    }
  }
}

void rules(const Legendre& gl, double T, std::vector<dd>* x, std::vector<dd>* w) {
  dd X[kQuad], W[kQuad], pm[kQuad], p[kQuad], al[N + 1], be[N + 1], old;
  for (int i = 0; i < kQuad; ++i) {
    X[i] = gl.t[i] * gl.t[i];
    W[i] = gl.w[i] * exp_dd(dd(-T) * X[i]);
    p[i] = dd(1.0);
  }
  for (int k = 0; k <= N; ++k) {
    dd nrm, mom;
    for (int i = 0; i < kQuad; ++i) {
      const dd wpp = W[i] * p[i] * p[i];
      nrm = nrm + wpp;
      mom = mom + wpp * X[i];
    }
    al[k] = mom / nrm;
    be[k] = k ? nrm / old : nrm;
    old = nrm;
    for (int i = 0; i < kQuad; ++i) {
      dd q = (X[i] - al[k]) * p[i];
      if (k) q = q - be[k] * pm[i];
      pm[i] = p[i];
      p[i] = q;
    }
  }
  gauss(al, be, 1.0, x, w);
}

void interval(const Legendre& gl, int iv, double* tab) {
  constexpr int C = kRysTerms;
  std::vector<dd> x[C][N + 1], w[C][N + 1];
  dd node[C];
  for (int j = 0; j < C; ++j) {
    const double z = std::cos(3.14159265358979323846 * (2 * j + 1) / (2.0 * C));
    node[j] = dd(0.5 * z);                       // T - (iv + 1/2); any distinct nodes near Chebyshev's serve
    rules(gl, iv + 0.5 + 0.5 * z, x[j], w[j]);
    node[j] = dd(iv + 0.5 + 0.5 * z) - dd(iv + 0.5);   // as rounded
  }
  for (int n = 1; n <= N; ++n)
    for (int r = 0; r < 2 * n; ++r) {
      // Newton's divided differences, then the power basis in T - (iv + 1/2)
      dd c[C];
      for (int j = 0; j < C; ++j) c[j] = r < n ? x[j][n][r] : w[j][n][r - n];
      for (int k = 1; k < C; ++k)
        for (int j = C - 1; j >= k; --j) c[j] = (c[j] - c[j - 1]) / (node[j] - node[j - k]);
      dd poly[C];
      for (int k = C - 1; k >= 0; --k) {
        for (int j = C - 1; j > 0; --j) poly[j] = poly[j - 1] - poly[j] * node[k];
        poly[0] = c[k] - poly[0] * node[k];
      }
      double* t = tab + rys_offset(n) + (size_t)iv * C * 2 * n + r;
      for (int k = 0; k < C; ++k) t[(size_t)k * 2 * n] = poly[k].h + poly[k].l;
    }
}

std::vector<double> build() {
  std::vector<double> tab((size_t)rys_offset(N + 1), 0.0);
  const Legendre gl;
  const int nt = std::max(1, std::min(16, (int)std::thread::hardware_concurrency()));
  std::exception_ptr failed;   // the first exception (memory) of any thread, for the caller
  std::mutex mu;
  auto work = [&](int t0) noexcept {
    try {
      for (int iv = t0; iv < kRysIntervals; iv += nt) interval(gl, iv, tab.data());
    } catch (...) {
      const std::lock_guard<std::mutex> lock(mu);
      if (!failed) failed = std::current_exception();
    }
  };
  std::vector<std::thread> th;
  try {
    for (int t = 1; t < nt; ++t) th.emplace_back(work, t);
  } catch (...) {
  }
  work(0);
  const int started = (int)th.size() + 1;
  for (auto& t : th) t.join();
  for (int t = started; t < nt; ++t) work(t);   // threads that could not be started
  if (failed) std::rethrow_exception(failed);
  // x^(-1/2) exp(-x): al_k = 2k + 1/2, be_k = k (k - 1/2), be_0 = sqrt(pi)
  dd al[N + 1], be[N + 1];
  for (int k = 0; k <= N; ++k) {
    al[k] = dd(2.0 * k + 0.5);
    be[k] = k ? dd(k * (k - 0.5)) : dd(1.772453850905516027, 4.803764720986022e-17);
  }
  std::vector<dd> x[N + 1], w[N + 1];
  gauss(al, be, 8.0 * N, x, w);
  for (int n = 1; n <= N; ++n) {
    double* t = tab.data() + rys_offset(n) + (size_t)kRysIntervals * kRysTerms * 2 * n;
    for (int r = 0; r < n; ++r) {
      t[r] = x[n][r].h;
      t[n + r] = 0.5 * w[n][r].h;
    }
  }
  return tab;
}

}  // namespace

const std::vector<double>& rys_table() {
  static const std::vector<double> tab = build();   // once per process, on first use (again after an exception)
  return tab;
}

}  // namespace mdx
