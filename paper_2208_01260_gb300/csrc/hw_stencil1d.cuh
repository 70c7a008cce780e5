// Stencil building blocks of the 1D scheme (Zhao & Zhang, arXiv:2208.01260, Sec. 2) shared by its kernels:
// state (eta, m, dx H, dx M), static (b, dx b_x). Same conventions as the 2D kernels (see hw_device.cuh): split
// without 1/2, projection rows without 1/(2c), epsilon rescaled.
#pragma once
#include "hw_device.cuh"
#include "hw_internal.h"

namespace hw {

enum { Q_FP = 0, Q_FM = 2, Q_GP = 4, Q_GM = 6, Q_H = 8, Q_M = 9, NREC1 = 10 };

struct Node6 {
  double v[6];  // eta m H' M' b bxs
};

__device__ __forceinline__ void load_node1d(const Dev1D& d, int i, Node6& n) {
  bool f;
  const int ii = map_index(i, d.nx, d.bc, f);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    double x = __ldg(d.S[q] + ii);
    n.v[q] = f ? x * par_1d(q) : x;
  }
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    double x = __ldg(d.stat[q] + ii);
    n.v[4 + q] = f ? x * par_1d(4 + q) : x;
  }
}

// F and Phi of Sec. 2 (eq. swe-form-1d-e and the printed Phi), split with alpha (no 1/2).
__device__ __forceinline__ void node_record1d(const Node6& n, double g, double alpha, double rec[NREC1]) {
  const double eta = n.v[0], m = n.v[1], H = n.v[2], M = n.v[3], b = n.v[4], B = n.v[5];
  const double h = eta - b;
  const double u = m * fast_rcp(h);
  const double gh = g * h, ge = g * eta;
  const double pres = ge * fma(0.5, eta, -b);
  const double uu = u * u;
  const double F0 = m, F1 = fma(m, u, pres);
  const double G0 = M, G1 = fma(u + u, M, fma(gh - uu, H, (uu - ge) * B));
  rec[Q_FP] = fma(alpha, eta, F0);
  rec[Q_FP + 1] = fma(alpha, m, F1);
  rec[Q_FM] = fma(-alpha, eta, F0);
  rec[Q_FM + 1] = fma(-alpha, m, F1);
  rec[Q_GP] = fma(alpha, H, G0);
  rec[Q_GP + 1] = fma(alpha, M, G1);
  rec[Q_GM] = fma(-alpha, H, G0);
  rec[Q_GM + 1] = fma(-alpha, M, G1);
  rec[Q_H] = h;
  rec[Q_M] = m;
}

// Outputs (6): 2 Fhat (2), 2 bhat (2), 24 dx Phihat (2).
template <bool LINEAR, bool CHAR>
__device__ __forceinline__ void interface_values1d(const double* r0, const double* r1, const double* r2,
                                                   const double* r3, int stride, const double qb[6], double g,
                                                   double eps_w, double out[6]) {
#define RV(r, f) (r)[(f) * stride]
  const double hs = RV(r1, Q_H) + RV(r2, Q_H);
  const double ub = (RV(r1, Q_M) + RV(r2, Q_M)) * fast_rcp(hs);
  const double gh = (0.5 * g) * hs;
  const double rs = fast_rsqrt(gh);
  const double cb = gh * rs, ic2 = 0.5 * rs;
  const double upc = ub + cb, umc = ub - cb;
  const double eps = CHAR ? (8.0 * g * eps_w) * hs : 4.0 * eps_w;
  const double* rp[4] = {r0, r1, r2, r3};
  double G[2], GB1 = 0.0, GB2 = 0.0;
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    const int os[3] = {side == 0 ? 0 : 3, side == 0 ? 1 : 2, side == 0 ? 2 : 1};
    const int fo = side == 0 ? Q_FP : Q_FM, go = side == 0 ? Q_GP : Q_GM;
    const double sg = side == 0 ? 1.0 : -1.0;
    double f[2][3], p[2][3];
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      const double* r = rp[os[t]];
      const double F0 = RV(r, fo), F1 = RV(r, fo + 1);
      const double G0 = sg * RV(r, go), G1 = sg * RV(r, go + 1);
      if (CHAR) {
        // rows of L without 1/(2c): (u+c, -1), (-(u-c), 1)
        f[0][t] = fma(upc, F0, -F1);
        f[1][t] = fma(-umc, F0, F1);
        p[0][t] = fma(upc, G0, -G1);
        p[1][t] = fma(-umc, G0, G1);
      } else {
        f[0][t] = F0; f[1][t] = F1; p[0][t] = G0; p[1][t] = G1;
      }
    }
    const double* qbs = qb + 3 * side;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      Weights W;
      const double v = hweno_side<LINEAR>(f[k][0], f[k][1], f[k][2], p[k][0], p[k][1], p[k][2], eps, W);
      G[k] = side == 0 ? v : G[k] + v;
      if (CHAR) {
        if (k == 0) GB1 -= weighted(W, qbs[0], qbs[1], qbs[2]);
        else GB2 += weighted(W, qbs[0], qbs[1], qbs[2]);
      } else if (k == 1) {
        GB2 += weighted(W, qbs[0], qbs[1], qbs[2]);
      }
    }
  }
  if (CHAR) {
    const double A = (G[0] + G[1]) * ic2;
    out[0] = A;
    out[1] = fma(ub, A, 0.5 * (G[1] - G[0]));
    const double B = (GB1 + GB2) * ic2;
    out[2] = B;
    out[3] = fma(ub, B, 0.5 * (GB2 - GB1));
  } else {
    out[0] = G[0]; out[1] = G[1];
    out[2] = 0.0;  out[3] = GB2;
  }
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const double fpart =
        fma(7.0, RV(r2, Q_FP + c) - RV(r1, Q_FM + c),
            fma(8.0, RV(r2, Q_FM + c) - RV(r1, Q_FP + c), RV(r0, Q_FP + c) - RV(r3, Q_FM + c)));
    const double gpart = fma(-5.0, RV(r2, Q_GP + c) + RV(r1, Q_GM + c),
                             fma(-2.0, RV(r1, Q_GP + c) + RV(r2, Q_GM + c), RV(r0, Q_GP + c) + RV(r3, Q_GM + c)));
    out[4 + c] = fma(3.0, fpart, gpart);
  }
#undef RV
}

// alpha from its key; with dt_out, dt = CFL dx / alpha, the step that reaches t_end ending on it.
__device__ __forceinline__ void finish_alpha1d(unsigned long long key, double* alpha, double* dt_out, double cfl,
                                               double dx, const double* t_now, double t_end) {
  const double a = __longlong_as_double((long long)key);
  alpha[0] = a;
  alpha[1] = 0.0;
  if (dt_out) {
    double dt = cfl * dx / a;
    double t_next = t_now ? *t_now + dt : 0.0;
    if (t_now && t_end > 0.0) {
      // the step that reaches t_end (within a relative 1e-12) ends exactly on it
      const double rem = t_end - *t_now;
      if (dt >= rem - 1e-12 * t_end) {
        dt = rem > 0.0 ? rem : 0.0;
        t_next = rem > 0.0 ? t_end : *t_now;
      }
    }
    *dt_out = dt;
    if (t_now) dt_out[1] = t_next;
  }
}

}  // namespace hw
