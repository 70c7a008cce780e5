// Host check of the block fixed-point reconstruction (csrc/hw_fixed.h) against the scheme's formulas in long
// double. Prints per kind of data the largest error of the weighted value and of the limited value, in units of
// 2^-53 of the stencil's largest entry, then the reciprocal's relative error (as a power of two) and the number
// of wrong conversions.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "hw_fixed.h"

using namespace hw;
typedef long double Q;

static Q side(const Q f[3], const Q p[3], Q eps) {
  const Q d1 = f[0] - f[1], d2 = f[1] - f[2];
  const Q B1 = 2 * d1 + p[0] + p[1], A1 = B1 + d1 + p[1], B2 = 2 * d2 + p[1] + p[2], A2 = B2 + d2 + p[1];
  const Q P = f[1] + p[1] / 2, e = d1 - d2, g = f[0] - f[2] + 2 * p[1], a = Q(13) / 3, b = Q(781) / 20;
  const Q t1 = p[1] * p[1] + eps + a * A1 * A1 + b * B1 * B1, t2 = p[1] * p[1] + eps + a * A2 * A2 + b * B2 * B2,
          t3 = p[1] * p[1] + eps + a / 4 * e * e + b / 4 * g * g;
  const Q w1 = 3 / (t1 * t1), w2 = 3 / (t2 * t2), w3 = 4 / (t3 * t3);
  return P + (w1 * A1 / 6 - w2 * A2 / 6 + w3 * e / 12) / (w1 + w2 + w3);
}
static Q limited(Q dl, Q dr, Q nl, Q nr, Q eps) {
  const Q pl = 2 * dl - nl, pr = 2 * dr - nr, pc = (dl + dr) / 2, a = Q(13) / 3;
  const Q t1 = pl * pl + a * (dl - nl) * (dl - nl) + eps, t2 = pr * pr + a * (dr - nr) * (dr - nr) + eps,
          t3 = pc * pc + a / 4 * (dr - dl) * (dr - dl) + eps;
  const Q w1 = 1 / (t1 * t1), w2 = 1 / (t2 * t2), w3 = 2 / (t3 * t3);
  return (w1 * pl + w2 * pr + w3 * pc) / (w1 + w2 + w3);
}

int main(int argc, char** argv) {
  const int n = argc > 1 ? atoi(argv[1]) : 20000;
  std::mt19937_64 g(argc > 2 ? atoi(argv[2]) : 1);
  std::uniform_real_distribution<double> U(-1, 1);
  bool bad = false;
  for (int kind = 0; kind < 8; ++kind) {
    // smooth | rough | jump in one value | two values | one derivative | flat with a step | tiny against eps | zero
    double worst = 0, worst_l = 0;
    for (int i = 0; i < n; ++i) {
      const double sc = std::pow(2.0, 30 * U(g)), sm = std::pow(10.0, -4 - 4 * U(g));
      double f[3], p[3];
      const double b0 = sc * (1 + 0.5 * U(g)), sl = sm * sc * U(g), cu = sm * sm * sc * U(g);
      for (int t = 0; t < 3; ++t) {
        f[t] = b0 + sl * (t - 1) + cu * (t - 1) * (t - 1);
        p[t] = sl + 2 * cu * (t - 1);
        if (kind == 1) { f[t] = sc * U(g); p[t] = sc * U(g); }
        if (kind == 5) { f[t] = b0; p[t] = 0; }
        if (kind == 7) { f[t] = 0; p[t] = 0; }
      }
      if (kind == 2) f[2] += 0.01 * sc * U(g);
      if (kind == 3) { f[0] += sc * U(g); f[1] += sc * U(g); }
      if (kind == 4) p[2] += 0.1 * sc * U(g);
      if (kind == 5) f[2] *= 1 + 1e-3 * U(g);
      const double eps = std::pow(10.0, -6 - 4 * std::fabs(U(g))) * (kind == 6 ? 1e10 * sc * sc : (i & 1) ? 16 : sc * sc);
      double mx = 1e-300;
      for (int t = 0; t < 3; ++t) mx = std::max({mx, std::fabs(f[t]), std::fabs(p[t])});
      int ex;
      std::frexp(mx, &ex);
      const int u = std::max(ex, -900) - 57;
      int64_t F[3], P[3];
      Q fq[3], pq[3];
      for (int t = 0; t < 3; ++t) {
        F[t] = (int64_t)std::ldexp(f[t], -u);
        P[t] = (int64_t)std::ldexp(p[t], -u);
        fq[t] = std::ldexp((Q)F[t], u);
        pq[t] = std::ldexp((Q)P[t], u);
      }
      const double ulp = mx / 9007199254740992.0;
      int64_t w1, w2;
      // the epsilon each form takes, as the kernels round it
      const double es = eps * (20.0 / 781.0), el = eps * (3.0 / 13.0);
      const int64_t v = fx_hweno_side(F[0], F[1], F[2], P[0], P[1], P[2], fx_eps(es, bad), u, w1, w2);
      worst = std::max(worst, (double)(std::fabs(std::ldexp((Q)v / 6, u) - side(fq, pq, (Q)es * 781 / 20)) / ulp));
      const int64_t l = fx_limiter_field(F[1] - F[0], F[2] - F[1], P[0], P[2], fx_eps(el, bad), u);
      const Q lq = limited(fq[1] - fq[0], fq[2] - fq[1], pq[0], pq[2], (Q)el * 13 / 3);
      worst_l = std::max(worst_l, (double)(std::fabs(std::ldexp((Q)l / 2, u) - lq) / ulp));
      if (kind == 7 && (v != 0 || l != 0)) worst = 1e9;
    }
    printf("%g %g\n", worst, worst_l);
  }
  double rel = 0;
  long wrong = 0;
  for (int i = 0; i < n; ++i) {
    uint64_t d = (g() >> 2) | (1ull << 62);
    if (i < 64) d = (1ull << 62) + i;
    if (i >= 64 && i < 128) d = (1ull << 63) - 1 - (i - 64);
    rel = std::max(rel, (double)std::fabs(std::ldexp((Q)fx_rcp(d), -62) * std::ldexp((Q)d, -63) - 1));
    // doubles to fixed point (towards zero) and back (to nearest)
    const double x = std::ldexp(U(g), (int)(g() % 90) - 45);
    const int em = 1023 + 46;
    const double trunc = std::ldexp(std::trunc(std::ldexp(x, 1082 - em)), em - 1082);
    if (std::ldexp((Q)fx_from_double(x, em), em - 1082) != (Q)trunc) ++wrong;
    if (fx_from_double(i & 1 ? 0.0 : -0.0, em) != 0 || fx_from_double(4e-320, em) != 0) ++wrong;
    const int64_t k = (int64_t)(g() >> (1 + g() % 62)) * ((i & 1) ? 1 : -1);
    const double back = fx_to_double(k, -40), want = std::ldexp((double)k, -40);
    if (std::fabs((Q)back - std::ldexp((Q)k, -40)) > std::fabs((Q)want - std::ldexp((Q)k, -40))) ++wrong;
    int um;
    const double y = i == 0 ? 0.0 : x;
    const int64_t m = fx_mantissa(y, um);
    if (std::ldexp((Q)m, i == 0 ? 0 : um) != (Q)y) ++wrong;
  }
  printf("%g %ld %d\n", std::log2(rel), wrong, (int)bad);
  return 0;
}
