// The forward pass of the adjoint, in FP64: one RK stage's sweeps and node update (nonlinear weights, characteristic
// projection) in floating point, where the solver's own stages (hw_kernels2d.cu) use fixed point.
//
// The gradient with respect to the bottom is a small difference of large terms (the flux's and the source's parts
// balance at rest: its plane is 1e3 and more below the terms it sums), so its last digits follow every rounding of
// the states it is taken at: two forward passes that differ by one unit in the last place give bottom gradients
// that differ by 1e-10 to 3e-9 of their norm (measured on grids of 48 to 300 nodes a side). The recorded states therefore
// keep the arithmetic the gradients have always been taken at, operation for operation: part of the products are
// formed on the integer pipes (each bit-identical to DMUL), as is the node update's reciprocal. hw_gauge_loss,
// hw_adjoint_run and the block forms take these kernels; every other run of a solver takes the fixed-point ones.
#include "hw_fp64_int.h"
#include "hw_stencil2d.cuh"

namespace hw {
namespace {

// Products and reciprocals. Fp64: the plain product on the FP64 pipe (fused with a following add where the compiler
// does) and fast_rcp. Int<IRCP>: the correctly rounded product on the integer pipes (hw_fp64_int.h, bit-identical
// to DMUL, never fused) and, with IRCP, the integer-pipe reciprocal; it records whether an operand left its fast
// path, in which case the caller recomputes with Fp64. k(c, x) multiplies by a literal constant c.
struct Fp64 {
  static constexpr bool bad = false;
  __device__ __forceinline__ double operator()(double x, double y) { return x * y; }
  __device__ __forceinline__ double k(double c, double x) { return c * x; }
  __device__ __forceinline__ double rcp(double x) { return fast_rcp(x); }
};
template <bool IRCP>
struct Int {
  bool bad = false;
  __device__ __forceinline__ double operator()(double x, double y) {
    double r;
    bad |= !f64_mul_int(x, y, r);
    return r;
  }
  __device__ __forceinline__ double k(double c, double x) {
    double r;
    bad |= !f64_mul_int<true>(x, c, r);
    return r;
  }
  __device__ __forceinline__ double rcp(double x) {
    if constexpr (!IRCP) return fast_rcp(x);
    double r;
    bad |= !f64_rcp_int(x, r);
    return r;
  }
};

struct WeightsT {
  double n1, n2, n3, r;
};

template <class M>
__device__ __forceinline__ void inverse_squares(double t1, double t2, double t3, double& n1, double& n2, double& n3, M& mul) {
  const double s1 = mul(t1, t1), s2 = mul(t2, t2), s3 = mul(t3, t3);
  n1 = mul(s2, s3);
  n2 = mul(s1, s3);
  n3 = mul(s1, s2);
}

template <class M>
__device__ __forceinline__ double side_value(double f0, double f1, double f2, double p0, double p1, double p2, double eps, WeightsT& W, M& mul) {
  const double d1 = f0 - f1, d2 = f1 - f2;
  const double B1 = fma(2.0, d1, p0 + p1);
  const double A1 = B1 + (d1 + p1);
  const double B2 = fma(2.0, d2, p1 + p2);
  const double A2 = B2 + (d2 + p1);
  const double P = fma(0.5, p1, f1);
  const double e = d1 - d2;  // f0 - 2 f1 + f2
  const double g3 = fma(2.0, p1, f0 - f2);
  // t_l = beta_l + eps, with eps added once to the common term p1^2
  const double ppe = fma(p1, p1, eps);
  const double t1 = fma(mul.k((781.0 / 20.0), B1), B1, fma(mul.k((13.0 / 3.0), A1), A1, ppe));
  const double t2 = fma(mul.k((781.0 / 20.0), B2), B2, fma(mul.k((13.0 / 3.0), A2), A2, ppe));
  const double t3 = fma(mul.k((781.0 / 80.0), g3), g3, fma(mul.k((13.0 / 12.0), e), e, ppe));
  double n3;
  inverse_squares(t1, t2, t3, W.n1, W.n2, n3, mul);
  // gamma = (3, 3, 4)/10 -> proportional to (1, 1, 4/3)
  W.n3 = mul.k((4.0 / 3.0), n3);
  W.r = mul.rcp(W.n1 + W.n2 + W.n3);
  // sum(omega_l q_l) = P + (n1 A1 - n2 A2 + (n3'/2) e) / (6 (n1 + n2 + n3')), n3' = W.n3
  const double z = fma(mul.k(0.5, W.n3), e, fma(-W.n2, A2, mul(W.n1, A1)));
  return fma(mul.k((1.0 / 6.0), W.r), z, P);
}

template <class M>
__device__ __forceinline__ double weighted_value(const WeightsT& W, double c1, double c2, double c3, M& mul) {
  return mul(fma(W.n1, c1, fma(W.n2, c2, mul(W.n3, c3))), W.r);
}

template <class M>
__device__ __forceinline__ double limited_value(double m0, double m1, double m2, double nl, double nr, double eps, M& mul) {
  const double dl = m1 - m0, dr = m2 - m1;
  const double pl = fma(2.0, dl, -nl);
  const double pr = fma(2.0, dr, -nr);
  const double pc2 = dl + dr;  // 2 p'_3
  const double al = dl - nl, ar = dr - nr, ac = dr - dl;
  const double b1 = fma(mul.k((13.0 / 3.0), al), al, mul(pl, pl));
  const double b2 = fma(mul.k((13.0 / 3.0), ar), ar, mul(pr, pr));
  const double b3 = fma(mul.k((13.0 / 12.0), ac), ac, mul(mul.k(0.25, pc2), pc2));
  // d = (1, 1, 2)/4 -> proportional to (1, 1, 2); p'_3 = pc2 / 2 so its term is n3 pc2
  double n1, n2, n3;
  inverse_squares(b1 + eps, b2 + eps, b3 + eps, n1, n2, n3, mul);
  const double den = fma(2.0, n3, n1 + n2);
  const double num = fma(n1, pl, fma(n2, pr, mul(n3, pc2)));
  return mul(num, mul.rcp(den));
}

template <int DIR, class M>
__device__ __forceinline__ void record(const Node12& n, double g, double alpha, double rec[NREC], M& mul) {
  const double eta = n.v[0], m = n.v[1], w = n.v[2], b = n.v[9];
  const double h = eta - b;
  const double rh = fast_rcp(h);
  const double u = mul(m, rh), v = mul(w, rh);
  const double gh = mul(g, h), ge = mul(g, eta);
  const double pres = mul(ge, fma(0.5, eta, -b));  // g/2 (eta^2 - 2 eta b)
  const double uv = mul(u, v);
  // derivative data along the sweep (split) and across it (mixed)
  const int qs = DIR == 0 ? 3 : 6, qm = DIR == 0 ? 6 : 3;
  const double Hs = n.v[qs], Ms = n.v[qs + 1], Ws = n.v[qs + 2], Bs = n.v[DIR == 0 ? 10 : 11];
  const double Hm = n.v[qm], Mm = n.v[qm + 1], Wm = n.v[qm + 2], Bm = n.v[DIR == 0 ? 11 : 10];
  double F[3], Gs[3], Gm[3];
  const double mv = mul(m, v);
  if (DIR == 0) {
    const double uu = mul(u, u), a1 = gh - uu, a2 = uu - ge, u2 = u + u;
    F[0] = m; F[1] = fma(m, u, pres); F[2] = mv;
    Gs[0] = Ms;
    Gs[1] = fma(u2, Ms, fma(a1, Hs, mul(a2, Bs)));
    Gs[2] = fma(uv, Bs - Hs, fma(v, Ms, mul(u, Ws)));
    Gm[0] = Mm;
    Gm[1] = fma(u2, Mm, fma(a1, Hm, mul(a2, Bm)));
    Gm[2] = fma(uv, Bm - Hm, fma(v, Mm, mul(u, Wm)));
  } else {
    const double vv = mul(v, v), a1 = gh - vv, a2 = vv - ge, v2 = v + v;
    F[0] = w; F[1] = mv; F[2] = fma(w, v, pres);
    Gs[0] = Ws;
    Gs[1] = fma(uv, Bs - Hs, fma(v, Ms, mul(u, Ws)));
    Gs[2] = fma(v2, Ws, fma(a1, Hs, mul(a2, Bs)));
    Gm[0] = Wm;
    Gm[1] = fma(uv, Bm - Hm, fma(v, Mm, mul(u, Wm)));
    Gm[2] = fma(v2, Wm, fma(a1, Hm, mul(a2, Bm)));
  }
  const double U[3] = {eta, m, w}, D[3] = {Hs, Ms, Ws};
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    rec[R_FP + c] = fma(alpha, U[c], F[c]);
    rec[R_FM + c] = fma(-alpha, U[c], F[c]);
    rec[R_GP + c] = fma(alpha, D[c], Gs[c]);
    rec[R_GM + c] = fma(-alpha, D[c], Gs[c]);
    rec[R_MIX + c] = Gm[c];
  }
  rec[R_H] = h;
  rec[R_M] = m;
  rec[R_W] = w;
}

template <int DIR, class M>
__device__ __forceinline__ void interface_m(const double* r0, const double* r1, const double* r2,
                                                   const double* r3, int stride, const double qb[6], double g,
                                                   double eps_w, double out[12], M& mul) {
#define RV(r, f) (r)[(f) * stride]
  // interface state: h = (h_i + h_{i+1})/2, u = (m_i + m_{i+1})/(h_i + h_{i+1}), v likewise
  const double hs = RV(r1, R_H) + RV(r2, R_H);
  const double rhs = mul.rcp(hs);
  const double ub = mul(RV(r1, R_M) + RV(r2, R_M), rhs);
  const double vb = mul(RV(r1, R_W) + RV(r2, R_W), rhs);
  const double gh = mul(mul.k(0.5, g), hs);
  const double rs = fast_rsqrt(gh);
  const double ic2 = mul.k(0.5, rs);  // 1/(2c)
  // normal / tangential velocity of this sweep
  const double un = DIR == 0 ? ub : vb, ut = DIR == 0 ? vb : ub;
  // un +- c with c = gh / sqrt(gh): fmas (a product on the integer pipes would leave the adds)
  const double upc = fma(gh, rs, un), umc = fma(-gh, rs, un);
  // component indices: normal momentum and tangential momentum
  const int cn = DIR == 0 ? 1 : 2, ct = DIR == 0 ? 2 : 1;
  // scaled epsilon: fields 1, 3 carry s = 4c, field 2 carries s = 2 (both 2 without projection)
  const double eps2 = mul.k(4.0, eps_w);
  const double eps13 = mul(mul(mul.k(8.0, g), eps_w), hs);

  double G[3], GB1 = 0.0, GB3 = 0.0;  // per-field sums over both sides; source fields 1 and 3
  const double* rp[4] = {r0, r1, r2, r3};
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    // '+' uses nodes 0,1,2 of (F+, G+); '-' uses nodes 3,2,1 of (F-, G-) with the derivative negated.
    const int o0 = side == 0 ? 0 : 3, o1 = side == 0 ? 1 : 2, o2 = side == 0 ? 2 : 1;
    const int fo = side == 0 ? R_FP : R_FM, go = side == 0 ? R_GP : R_GM;
    const double sg = side == 0 ? 1.0 : -1.0;
    double f[3][3], p[3][3];  // [field][stencil point]
    const int os[3] = {o0, o1, o2};
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      const double* r = rp[os[t]];
      const double F0 = RV(r, fo), Fn = RV(r, fo + cn), Ft = RV(r, fo + ct);
      const double G0 = sg * RV(r, go), Gn = sg * RV(r, go + cn), Gt = sg * RV(r, go + ct);
      {
        // rows of L without 1/(2c): (un+c, -1, 0), (-ut, 0, 1), (-(un-c), 1, 0) on (rho, normal, tangential)
        f[0][t] = fma(upc, F0, -Fn);
        f[1][t] = fma(-ut, F0, Ft);
        f[2][t] = fma(-umc, F0, Fn);
        p[0][t] = fma(upc, G0, -Gn);
        p[1][t] = fma(-ut, G0, Gt);
        p[2][t] = fma(-umc, G0, Gn);
      }
    }
    const double* qbs = qb + 3 * side;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      WeightsT W;
      const double e = (k == 1) ? eps2 : eps13;
      const double v = side_value(f[k][0], f[k][1], f[k][2], p[k][0], p[k][1], p[k][2], e, W, mul);
      G[k] = side == 0 ? v : G[k] + v;
      // source data per field: (-b, 0, +b) (row entries of the normal-momentum column)
      if (k == 0) GB1 -= weighted_value(W, qbs[0], qbs[1], qbs[2], mul);
      if (k == 2) GB3 += weighted_value(W, qbs[0], qbs[1], qbs[2], mul);
    }
  }
  // back to physical components: 2 Fhat = double diag(1/s) G * 2
  double F2[3], B2[3];
  const double A = mul(G[0] + G[2], ic2);
  F2[0] = A;
  F2[cn] = fma(un, A, mul.k(0.5, G[2] - G[0]));
  F2[ct] = fma(ut, A, G[1]);
  const double Bs = mul(GB1 + GB3, ic2);
  B2[0] = Bs;
  B2[cn] = fma(un, Bs, mul.k(0.5, GB3 - GB1));
  B2[ct] = mul(ut, Bs);
  // derivative-equation flux (eq. Rec-phi, component-wise): 24 dS Ghat = 3 fpart + gpart
  // mixed term (eq. mixed): 12 dT Mhat = 7 (X_i + X_{i+1}) - (X_{i-1} + X_{i+2})
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double fpart =
        fma(7.0, RV(r2, R_FP + c) - RV(r1, R_FM + c),
            fma(8.0, RV(r2, R_FM + c) - RV(r1, R_FP + c), RV(r0, R_FP + c) - RV(r3, R_FM + c)));
    const double gpart = fma(-5.0, RV(r2, R_GP + c) + RV(r1, R_GM + c),
                             fma(-2.0, RV(r1, R_GP + c) + RV(r2, R_GM + c), RV(r0, R_GP + c) + RV(r3, R_GM + c)));
    out[c] = F2[c];
    out[3 + c] = B2[c];
    out[6 + c] = fma(3.0, fpart, gpart);
    out[9 + c] = fma(7.0, RV(r1, R_MIX + c) + RV(r2, R_MIX + c), -(RV(r0, R_MIX + c) + RV(r3, R_MIX + c)));
  }
#undef RV
}

// ---- the same interface shared out over lanes and warps (small grids), operation for operation ----
// Eigenvectors of the interface between the records r1 and r2.
template <int DIR>
struct Eigen {
  double un, ut, upc, umc, ic2, eps2, eps13;
  template <class M>
  __device__ __forceinline__ void form(const double* r1, const double* r2, int stride, double g, double eps_w, M& mul) {
    const double hs = r1[R_H * stride] + r2[R_H * stride];
    const double rhs = mul.rcp(hs);
    const double ub = mul(r1[R_M * stride] + r2[R_M * stride], rhs);
    const double vb = mul(r1[R_W * stride] + r2[R_W * stride], rhs);
    const double gh = mul(mul.k(0.5, g), hs);
    const double rs = fast_rsqrt(gh);
    ic2 = mul.k(0.5, rs);
    un = DIR == 0 ? ub : vb;
    ut = DIR == 0 ? vb : ub;
    upc = fma(gh, rs, un);
    umc = fma(-gh, rs, un);
    eps2 = mul.k(4.0, eps_w);
    eps13 = mul(mul(mul.k(8.0, g), eps_w), hs);
  }
};

// One upwind side: q, step = its first record's split data and the way to the next (side 1 from the far end, its
// derivatives negated by mask): the three fields' values and the source with the weights of fields 1 and 3.
template <int DIR, class M>
__device__ __forceinline__ void side_values(const Eigen<DIR>& E, const double* q, int step, int stride, uint32_t mask,
                                            const double qbs[3], double v[3], double& b1, double& b3, M& mul) {
  const int cn = DIR == 0 ? 1 : 2, ct = DIR == 0 ? 2 : 1;
  double f[3][3], p[3][3];
#pragma unroll
  for (int t = 0; t < 3; ++t) {
    const double* r = q + t * step;
    const double F0 = r[0], Fn = r[cn * stride], Ft = r[ct * stride];
    const double G0 = flip_sign(r[R_GP * stride], mask), Gn = flip_sign(r[(R_GP + cn) * stride], mask),
                 Gt = flip_sign(r[(R_GP + ct) * stride], mask);
    f[0][t] = fma(E.upc, F0, -Fn);
    f[1][t] = fma(-E.ut, F0, Ft);
    f[2][t] = fma(-E.umc, F0, Fn);
    p[0][t] = fma(E.upc, G0, -Gn);
    p[1][t] = fma(-E.ut, G0, Gt);
    p[2][t] = fma(-E.umc, G0, Gn);
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    WeightsT W;
    v[k] = side_value(f[k][0], f[k][1], f[k][2], p[k][0], p[k][1], p[k][2], k == 1 ? E.eps2 : E.eps13, W, mul);
    if (k == 0) b1 = weighted_value(W, qbs[0], qbs[1], qbs[2], mul);
    if (k == 2) b3 = weighted_value(W, qbs[0], qbs[1], qbs[2], mul);
  }
}

// Back to physical components from the sums over both sides: the first six interface values.
template <int DIR, class M>
__device__ __forceinline__ void back_values(const Eigen<DIR>& E, const double G[3], double GB1, double GB3, double out[6], M& mul) {
  const int cn = DIR == 0 ? 1 : 2, ct = DIR == 0 ? 2 : 1;
  const double A = mul(G[0] + G[2], E.ic2);
  out[0] = A;
  out[cn] = fma(E.un, A, mul.k(0.5, G[2] - G[0]));
  out[ct] = fma(E.ut, A, G[1]);
  const double Bs = mul(GB1 + GB3, E.ic2);
  out[3] = Bs;
  out[3 + cn] = fma(E.un, Bs, mul.k(0.5, GB3 - GB1));
  out[3 + ct] = mul(E.ut, Bs);
}

// The derivative flux and the mixed term: the other six.
__device__ __forceinline__ void linear_values(const double* r0, int sstep, int stride, double out[6]) {
  const double *r1 = r0 + sstep, *r2 = r1 + sstep, *r3 = r2 + sstep;
#define RV(r, f) (r)[(f) * stride]
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double fpart =
        fma(7.0, RV(r2, R_FP + c) - RV(r1, R_FM + c),
            fma(8.0, RV(r2, R_FM + c) - RV(r1, R_FP + c), RV(r0, R_FP + c) - RV(r3, R_FM + c)));
    const double gpart = fma(-5.0, RV(r2, R_GP + c) + RV(r1, R_GM + c),
                             fma(-2.0, RV(r1, R_GP + c) + RV(r2, R_GM + c), RV(r0, R_GP + c) + RV(r3, R_GM + c)));
    out[c] = fma(3.0, fpart, gpart);
    out[3 + c] = fma(7.0, RV(r1, R_MIX + c) + RV(r2, R_MIX + c), -(RV(r0, R_MIX + c) + RV(r3, R_MIX + c)));
  }
#undef RV
}

template <int DIR, class M>
__device__ __forceinline__ void limit_along(const double Um[3], const double U0[3], const double Up[3],
                                          const double Dm[3], const double Dp[3], double u, double v, double c,
                                          double ic2, double gh, double eps, double out[3], M& mul) {
  const int cn = DIR == 0 ? 1 : 2, ct = DIR == 0 ? 2 : 1;
  const double un = DIR == 0 ? u : v, ut = DIR == 0 ? v : u;
  const double upc = un + c, umc = un - c;
  auto proj = [&](const double* a, double o[3]) {
    o[0] = fma(upc, a[0], -a[cn]);
    o[1] = fma(-ut, a[0], a[ct]);
    o[2] = fma(-umc, a[0], a[cn]);
  };
  double m0[3], m1[3], m2[3], nl[3], nr[3];
  proj(Um, m0); proj(U0, m1); proj(Up, m2); proj(Dm, nl); proj(Dp, nr);
  const double e13 = mul(mul.k(4.0, eps), gh);
  double nu[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) nu[k] = limited_value(m0[k], m1[k], m2[k], nl[k], nr[k], k == 1 ? eps : e13, mul);
  const double A = mul(nu[0] + nu[2], ic2);
  out[0] = A;
  out[cn] = fma(un, A, mul.k(0.5, nu[2] - nu[0]));
  out[ct] = fma(ut, A, nu[1]);
}

// RHS (eq. swe-form-2d-dis) in scaled units: R_U, dx R_V, dy R_Q, of the node at o with the left x-interface ox and
// the lower y-interface oy.
template <class M>
__device__ __forceinline__ void right_hand_side(const Dev2D& d, const double cur[9], size_t o, size_t ox, size_t oy, double Rv[9],
                                                M& mul) {
  const double eta = cur[0], H1 = cur[3], H2 = cur[6];
  const double g = d.g;
  const double c_bx = d.c_bx, c_by = d.c_by, c_gx = d.c_gx, c_gy = d.c_gy, c_mx = d.c_mx,
          c_my = d.c_my;
  const double ge = mul(g, eta);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double dFx = __ldg(d.X[c] + ox + 1) - __ldg(d.X[c] + ox);
    const double dFy = __ldg(d.Y[c] + oy + d.nx) - __ldg(d.Y[c] + oy);
    const double dbx = __ldg(d.X[3 + c] + ox + 1) - __ldg(d.X[3 + c] + ox);
    const double dby = __ldg(d.Y[3 + c] + oy + d.nx) - __ldg(d.Y[3 + c] + oy);
    const double dGx = __ldg(d.X[6 + c] + ox + 1) - __ldg(d.X[6 + c] + ox);
    const double dGy = __ldg(d.Y[6 + c] + oy + d.nx) - __ldg(d.Y[6 + c] + oy);
    const double dMx = __ldg(d.X[9 + c] + ox + 1) - __ldg(d.X[9 + c] + ox);
    const double dMy = __ldg(d.Y[9 + c] + oy + d.nx) - __ldg(d.Y[9 + c] + oy);
    const double db = fma(c_bx, dbx, mul(c_by, dby));  // [b~]_x/dx + [b-]_y/dy
    Rv[c] = fma(-ge, db, fma(-c_bx, dFx, -mul(c_by, dFy)));
    double rv = fma(-c_gx, dGx, -mul(c_my, dMy));
    double rq = fma(-c_mx, dMx, -mul(c_gy, dGy));
    if (c > 0) {
      rv = fma(-ge, __ldg(d.sv[c - 1] + o), rv);
      rq = fma(-ge, __ldg(d.sq[c - 1] + o), rq);
    }
    Rv[3 + c] = fma(-mul(g, H1), db, rv);
    Rv[6 + c] = fma(-mul(g, H2), db, rq);
  }
}

// The node's velocities, wave speed c, 1/(2c) and g h.
template <class M>
__device__ __forceinline__ void node_speeds(const Dev2D& d, const double cur[9], size_t o, double& u, double& v, double& c,
                                            double& ic2, double& gh, M& mul) {
  const double b0 = __ldg(d.stat[0] + o);
  const double h = cur[0] - b0;
  gh = mul(d.g, h);
  const double rh = mul.rcp(h);
  u = mul(cur[1], rh);
  v = mul(cur[2], rh);
  const double rs = fast_rsqrt(gh);
  c = mul(gh, rs);
  ic2 = mul.k(0.5, rs);
}

template <class M>
__device__ __forceinline__ void node_update_m(const Dev2D& d, const StageArgs& sa, int i, int j, M& mul) {
  const size_t o = (size_t)j * d.nx + i;
  const size_t ox = (size_t)j * (d.nx + 1) + i;  // left x-interface; right is ox + 1
  const size_t oy = (size_t)j * d.nx + i;             // lower y-interface; upper is oy + nx
  double cur[9];
#pragma unroll
  for (int q = 0; q < 9; ++q) cur[q] = __ldg(d.S[q] + o);
  if (!(*sa.dt > 0.0)) {
    // a step of size 0 (e.g. clipped at the end time) leaves the state unchanged
#pragma unroll
    for (int q = 0; q < 9; ++q) sa.out[q][o] = cur[q];
    return;
  }
  double Rv[9];
  right_hand_side(d, cur, o, ox, oy, Rv, mul);
  // ---- limiter (Sec. 2.2, dimension by dimension) ----
  double mod[6];
  if (sa.limiter) {
    double u, v, c, ic2, gh;
    node_speeds(d, cur, o, u, v, c, ic2, gh, mul);
    Node12 nm, np;
    // x neighbours
    load_node(d, i - 1, j, nm);
    load_node(d, i + 1, j, np);
    limit_along<0>(nm.v, cur, np.v, nm.v + 3, np.v + 3, u, v, c, ic2, gh, d.eps_lim, mod, mul);
    load_node(d, i, j - 1, nm);
    load_node(d, i, j + 1, np);
    limit_along<1>(nm.v, cur, np.v, nm.v + 6, np.v + 6, u, v, c, ic2, gh, d.eps_lim, mod + 3, mul);
  } else {
#pragma unroll
    for (int q = 0; q < 6; ++q) mod[q] = cur[3 + q];
  }
  // ---- SSP-RK3 combination (eq. RK) ----
  const double dt = *sa.dt;
  if (sa.k == 1) {
    if (mul.bad) return;
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      const double cq = q < 3 ? cur[q] : mod[q - 3];
      if (sa.base) sa.base[q][o] = cq;
      sa.out[q][o] = fma(dt, Rv[q], cq);
    }
  } else {
    const double a = sa.k == 2 ? 0.75 : 1.0 / 3.0;
    const double b = sa.k == 2 ? 0.25 : 2.0 / 3.0;
    double res[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      const double cq = q < 3 ? cur[q] : mod[q - 3];
      res[q] = fma(a, __ldg(sa.base[q] + o), mul(b, fma(dt, Rv[q], cq)));
    }
    if (mul.bad) return;
#pragma unroll
    for (int q = 0; q < 9; ++q) sa.out[q][o] = res[q];
  }
}

constexpr int FT = 128;  // threads per tile: three blocks of 168 registers per SM

// One interface of a sweep: the reciprocals on the FP64 pipe, the products on the integer pipes; again on the FP64
// pipe if an operand left the fast path.
template <int DIR>
__device__ __forceinline__ void interface_point(const double* s, int step, int stride, const double qb[6], double g,
                                                double eps_w, double out[12]) {
  Int<false> mi;
  interface_m<DIR>(s, s + step, s + 2 * step, s + 3 * step, stride, qb, g, eps_w, out, mi);
  if (mi.bad) {
    Fp64 mf;
    interface_m<DIR>(s, s + step, s + 2 * step, s + 3 * step, stride, qb, g, eps_w, out, mf);
  }
}

// Both sweeps over the flattened extended lines of hw_stencil2d.cuh: blocks below nxt take x-tiles, the others
// y-tiles of pairs of columns.
__global__ void __launch_bounds__(FT, 3) k_sweeps_fp64(Dev2D d, const double* __restrict__ alpha, unsigned nxt) {
  __shared__ double sm[NREC * FT];
  const int t = threadIdx.x;
  Fp64 mf;
  double qb[6], out[12];
  if (blockIdx.x < nxt) {
    const unsigned W = d.nx + 4, total = (unsigned)d.ny * W, E = blockIdx.x * (FT - 3) + t;
    const unsigned j = E / W, e = E - j * W;
    if (E < total) {
      Node12 n;
      load_node(d, (int)e - 2, (int)j, n);
      double rec[NREC];
      record<0>(n, d.g, alpha[0], rec, mf);
#pragma unroll
      for (int f = 0; f < NREC; ++f) sm[f * FT + t] = rec[f];
    }
    __syncthreads();
    if (t >= FT - 3 || E >= total || e > (unsigned)d.nx) return;
    const size_t o = (size_t)j * (d.nx + 1) + e;
#pragma unroll
    for (int q = 0; q < 6; ++q) qb[q] = __ldg(d.qbx[q] + o);
    interface_point<0>(sm + t, 1, FT, qb, d.g, d.eps_w, out);
#pragma unroll
    for (int q = 0; q < 12; ++q) d.X[q][o] = out[q];
  } else {
    constexpr int yc = 2, rows = FT / yc, ifs = rows - 3;
    const unsigned H = d.ny + 4, total = (unsigned)((d.nx + yc - 1) / yc) * H;
    const int c = t % yc, r = t / yc;
    const unsigned E = (blockIdx.x - nxt) * ifs + r, g = E / H, e = E - g * H;
    const int i = (int)g * yc + c;
    if (E < total && i < d.nx) {
      Node12 n;
      load_node(d, i, (int)e - 2, n);
      double rec[NREC];
      record<1>(n, d.g, alpha[1], rec, mf);
#pragma unroll
      for (int f = 0; f < NREC; ++f) sm[f * FT + t] = rec[f];
    }
    __syncthreads();
    if (r >= ifs || E >= total || e > (unsigned)d.ny || i >= d.nx) return;
    const size_t o = (size_t)e * d.nx + i;
#pragma unroll
    for (int q = 0; q < 6; ++q) qb[q] = __ldg(d.qby[q] + o);
    interface_point<1>(sm + t, yc, FT, qb, d.g, d.eps_w, out);
#pragma unroll
    for (int q = 0; q < 12; ++q) d.Y[q][o] = out[q];
  }
}

// The same for small grids, where a tile's time is one warp's chain of dependent operations: SR - 3 x-interfaces per tile, each
// side a lane's (pairs of lanes exchange their sums), the derivative flux and the mixed term other warps': 60 -> 39 us a
// stage at 150 x 97. The sums keep their order, so the values are those of k_sweeps_fp64 bit for bit.
constexpr int SR = 64, ST = 3 * SR;  // records and threads per tile

template <int DIR>
__device__ __forceinline__ void sweep_split(const Dev2D& d, const double* sm, int rs, int u, bool valid, size_t o) {
  // u: the interface's first record; rs: records to the next one of its line
  double* const* P = DIR == 0 ? d.X : d.Y;
  if (threadIdx.x < 2 * SR) {
    const int side = threadIdx.x & 1;
    double v[3] = {}, b1 = 0.0, b3 = 0.0, qbs[3];
    Int<false> mi;
    const double* r0 = sm + u;
    Eigen<DIR> E{};
    if (valid) {
#pragma unroll
      for (int q = 0; q < 3; ++q) qbs[q] = __ldg((DIR == 0 ? d.qbx : d.qby)[3 * side + q] + o);
      E.form(r0 + rs, r0 + 2 * rs, SR, d.g, d.eps_w, mi);
      side_values<DIR>(E, side ? r0 + 3 * rs + R_FM * SR : r0, side ? -rs : rs, SR, side ? 0x80000000u : 0u, qbs, v, b1, b3, mi);
    }
    double w[3], c1, c3;
#pragma unroll
    for (int k = 0; k < 3; ++k) w[k] = __shfl_xor_sync(0xffffffffu, v[k], 1);
    c1 = __shfl_xor_sync(0xffffffffu, b1, 1);
    c3 = __shfl_xor_sync(0xffffffffu, b3, 1);
    bool bad = mi.bad;
    bad |= __shfl_xor_sync(0xffffffffu, (int)bad, 1) != 0;
    if (valid && side == 0) {
      double out[12];
      if (!bad) {
        const double G[3] = {v[0] + w[0], v[1] + w[1], v[2] + w[2]};
        const double GB1 = (0.0 - b1) - c1, GB3 = (0.0 + b3) + c3;
        back_values<DIR>(E, G, GB1, GB3, out, mi);
        bad = mi.bad;
      }
      if (bad) {
        double qb[6];
#pragma unroll
        for (int q = 0; q < 6; ++q) qb[q] = __ldg((DIR == 0 ? d.qbx : d.qby)[q] + o);
        Fp64 mf;
        interface_m<DIR>(r0, r0 + rs, r0 + 2 * rs, r0 + 3 * rs, SR, qb, d.g, d.eps_w, out, mf);
      }
#pragma unroll
      for (int q = 0; q < 6; ++q) P[q][o] = out[q];
    }
  } else if (valid) {
    double out[6];
    linear_values(sm + u, rs, SR, out);
#pragma unroll
    for (int q = 0; q < 6; ++q) P[6 + q][o] = out[q];
  }
}

__global__ void __launch_bounds__(ST, 2) k_sweeps_fp64_split(const __grid_constant__ Dev2D d, const double* __restrict__ alpha,
                                                             unsigned nxt) {
  __shared__ double sm[NREC * SR];
  const int t = threadIdx.x, u = t < 2 * SR ? t >> 1 : t - 2 * SR;  // the thread's interface
  Fp64 mf;
  if (blockIdx.x < nxt) {
    const unsigned W = d.nx + 4, total = (unsigned)d.ny * W, E0 = blockIdx.x * (SR - 3);
    if (t < SR && E0 + t < total) {
      const unsigned j = (E0 + t) / W;
      Node12 n;
      load_node(d, (int)(E0 + t - j * W) - 2, (int)j, n);
      double rec[NREC];
      record<0>(n, d.g, alpha[0], rec, mf);
#pragma unroll
      for (int f = 0; f < NREC; ++f) sm[f * SR + t] = rec[f];
    }
    __syncthreads();
    const unsigned E = E0 + u, j = E / W, e = E - j * W;
    sweep_split<0>(d, sm, 1, u, u < SR - 3 && E < total && e <= (unsigned)d.nx, (size_t)j * (d.nx + 1) + e);
  } else {
    constexpr int yc = 2, ifs = SR / yc - 3;
    const unsigned H = d.ny + 4, total = (unsigned)((d.nx + yc - 1) / yc) * H, E0 = (blockIdx.x - nxt) * ifs;
    if (t < SR) {
      const unsigned E = E0 + t / yc, g = E / H;
      const int i = (int)g * yc + t % yc;
      if (E < total && i < d.nx) {
        Node12 n;
        load_node(d, i, (int)(E - g * H) - 2, n);
        double rec[NREC];
        record<1>(n, d.g, alpha[1], rec, mf);
#pragma unroll
        for (int f = 0; f < NREC; ++f) sm[f * SR + t] = rec[f];
      }
    }
    __syncthreads();
    const unsigned E = E0 + u / yc, g = E / H, e = E - g * H;
    const int i = (int)g * yc + u % yc;
    sweep_split<1>(d, sm, yc, u, u / yc < ifs && E < total && e <= (unsigned)d.ny && i < d.nx, (size_t)e * d.nx + i);
  }
}

// The node update of small grids: 64 nodes a block, their right-hand sides, x-limiters and y-limiters two warps' each, the
// RK combination of three planes likewise: 46 -> 30 us a stage at 150 x 97, the values those of k_node_fp64.
__global__ void __launch_bounds__(192, 3) k_node_fp64_split(const __grid_constant__ Dev2D d, StageArgs sa) {
  __shared__ double s_mod[6 * 64], s_R[9 * 64];
  __shared__ int s_bad[64];
  const int t = threadIdx.x & 63, role = threadIdx.x >> 6;
  if (sa.nsteps && blockIdx.x == 0 && threadIdx.x == 0) {
    *sa.t = sa.snapped ? sa.clock[1] : *sa.t + sa.clock[0];
    if (sa.clock[0] > 0.0) ++*sa.nsteps;
  }
  const unsigned o = blockIdx.x * 64 + t;
  const int j = (int)(o / (unsigned)d.nx), i = (int)(o - (unsigned)j * d.nx);
  const bool in = j < d.ny;
  if (!(*sa.dt > 0.0)) {  // a step of size 0
    if (in)
#pragma unroll
      for (int q = 0; q < 3; ++q) sa.out[3 * role + q][o] = __ldg(d.S[3 * role + q] + o);
    return;
  }
  if (role == 0) s_bad[t] = 0;
  __syncthreads();
  Int<true> mi;
  if (in) {
    double cur[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) cur[q] = __ldg(d.S[q] + o);
    if (role == 0) {
      double Rv[9];
      right_hand_side(d, cur, o, (size_t)j * (d.nx + 1) + i, o, Rv, mi);
#pragma unroll
      for (int q = 0; q < 9; ++q) s_R[q * 64 + t] = Rv[q];
    } else {
      double mod[3];
      if (sa.limiter) {
        double u, v, c, ic2, gh;
        node_speeds(d, cur, o, u, v, c, ic2, gh, mi);
        Node12 nm, np;
        if (role == 1) {
          load_node(d, i - 1, j, nm);
          load_node(d, i + 1, j, np);
          limit_along<0>(nm.v, cur, np.v, nm.v + 3, np.v + 3, u, v, c, ic2, gh, d.eps_lim, mod, mi);
        } else {
          load_node(d, i, j - 1, nm);
          load_node(d, i, j + 1, np);
          limit_along<1>(nm.v, cur, np.v, nm.v + 6, np.v + 6, u, v, c, ic2, gh, d.eps_lim, mod, mi);
        }
      } else {
#pragma unroll
        for (int q = 0; q < 3; ++q) mod[q] = role == 1 ? cur[3 + q] : cur[6 + q];
      }
#pragma unroll
      for (int q = 0; q < 3; ++q) s_mod[(3 * (role - 1) + q) * 64 + t] = mod[q];
    }
    if (mi.bad) s_bad[t] = 1;
  }
  __syncthreads();
  double cq[3], res[3];
  if (in) {
    const double dt = *sa.dt, a = sa.k == 2 ? 0.75 : 1.0 / 3.0, b = sa.k == 2 ? 0.25 : 2.0 / 3.0;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const double R = s_R[(3 * role + q) * 64 + t];
      cq[q] = role == 0 ? __ldg(d.S[q] + o) : s_mod[(3 * (role - 1) + q) * 64 + t];
      res[q] = fma(dt, R, cq[q]);
      if (sa.k != 1) res[q] = fma(a, __ldg(sa.base[3 * role + q] + o), mi(b, res[q]));
    }
    if (mi.bad) s_bad[t] = 1;
  }
  __syncthreads();
  if (!in) return;
  if (s_bad[t]) {
    if (role == 0) {
      Fp64 mf;
      node_update_m(d, sa, i, j, mf);
    }
    return;
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    if (sa.k == 1 && sa.base) sa.base[3 * role + q][o] = cq[q];
    sa.out[3 * role + q][o] = res[q];
  }
}

template <int T>
__global__ void __launch_bounds__(T, T == 256 ? 3 : 8) k_node_fp64(Dev2D d, StageArgs sa) {
  const int i = blockIdx.x * 32 + threadIdx.x, j = blockIdx.y * (T / 32) + threadIdx.y;
  if (sa.nsteps && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0 && threadIdx.y == 0) {
    *sa.t = sa.snapped ? sa.clock[1] : *sa.t + sa.clock[0];
    if (sa.clock[0] > 0.0) ++*sa.nsteps;
  }
  if (i >= d.nx || j >= d.ny) return;
  Int<true> mi;
  node_update_m(d, sa, i, j, mi);
  if (mi.bad) {
    Fp64 mf;
    node_update_m(d, sa, i, j, mf);
  }
}

}  // namespace

// Nodes up to which the sweeps are split over lanes and warps, and the node update is: the split sweeps are the faster form as
// long as the tiles fill the GPU a few times at most (129 against 141 us a stage at 256^2, 39 against 60 at 150 x 97), the
// split node update while its blocks are resident at once (59 against 51 us at 256^2, 30 against 46 at 150 x 97).
constexpr size_t kSweepSplitMax = (size_t)152 * 16 * 32, kNodeSplitMax = (size_t)152 * 3 * 64;

void launch_stage_fp64(const Dev2D& d, const StageArgs& sa, const double* alpha, cudaStream_t st) {
  const size_t n = (size_t)d.nx * d.ny;
  const bool split = n <= kSweepSplitMax;
  const int IX = (split ? SR : FT) - 3, IY = (split ? SR : FT) / 2 - 3;
  const unsigned long long nxt = ((unsigned long long)d.ny * (d.nx + 4) + IX - 1) / IX;
  const unsigned long long nyt = ((unsigned long long)((d.nx + 1) / 2) * (d.ny + 4) + IY - 1) / IY;
  if (split) k_sweeps_fp64_split<<<(unsigned)(nxt + nyt), ST, 0, st>>>(d, alpha, (unsigned)nxt);
  else k_sweeps_fp64<<<(unsigned)(nxt + nyt), FT, 0, st>>>(d, alpha, (unsigned)nxt);
  if (n <= kNodeSplitMax) k_node_fp64_split<<<(unsigned)((n + 63) / 64), 192, 0, st>>>(d, sa);
  else if (n <= (size_t)152 * 16 * 32)
    k_node_fp64<64><<<dim3((d.nx + 31) / 32, (d.ny + 1) / 2), dim3(32, 2), 0, st>>>(d, sa);
  else
    k_node_fp64<256><<<dim3((d.nx + 31) / 32, (d.ny + 7) / 8), dim3(32, 8), 0, st>>>(d, sa);
}

}  // namespace hw
