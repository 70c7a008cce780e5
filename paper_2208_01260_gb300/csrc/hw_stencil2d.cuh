// Stencil building blocks of the 2D scheme shared by the single-grid kernels (hw_kernels2d.cu) and
// the batched kernels (hw_batch.cu): boundary-mapped node loads, per-node flux records, one interface
// of a sweep (Sec. 2.1 Steps 1-2 along x or y, eq. mixed), the limiter along one direction (Sec. 2.2)
// and the node update (eq. swe-form-2d-dis, limiter, eq. RK). See hw_device.cuh for the conventions.
#pragma once
#include "hw_device.cuh"
#include "hw_fixed.h"
#include "hw_internal.h"

namespace hw {

// ---------------------------------------------------------------------------------------------
// Loading a node with boundary mapping
// ---------------------------------------------------------------------------------------------
template <class R>
struct Node12T {
  R v[12];  // eta m w H1' M1' W1' H2' M2' W2' b bxs bys
};
using Node12 = Node12T<double>;

// Load of a plane that changes between launches. COH = false: through the read-only data path (valid
// while no block of the running kernel writes the plane). COH = true: an ordinary global load, for a
// kernel whose later phases read what its earlier phases wrote (a persistent kernel with grid
// barriers); the read-only path is not kept coherent with such writes.
template <bool COH, class T>
__device__ __forceinline__ T ldp(const T* p) {
  if constexpr (COH) return *p;
  else return __ldg(p);
}

// x with its sign flipped where mask is 0x80000000 (0: x itself), on the integer pipes.
__device__ __forceinline__ double flip_sign(double x, uint32_t mask) {
  uint32_t lo, hi;
  f64_words(x, lo, hi);
  return f64_from_words(lo, hi ^ mask);
}
__device__ __forceinline__ float flip_sign(float x, uint32_t mask) { return __uint_as_float(__float_as_uint(x) ^ mask); }

// base: offset of the grid's first node in the node planes (0 unless the planes pool several grids).
template <bool COH = false, class R>
__device__ __forceinline__ void load_node(const Dev2DT<R>& d, int i, int j, Node12T<R>& n, size_t base = 0) {
  bool fx, fy;
  const int ii = map_index(i, d.nx, d.bc_x, fx);
  const int jj = map_index(j, d.ny, d.bc_y, fy);
  const size_t o = base + (size_t)jj * d.nx + ii;
  const uint32_t mx = fx ? 0x80000000u : 0u, my = fy ? 0x80000000u : 0u;
#pragma unroll
  for (int q = 0; q < 12; ++q)
    n.v[q] = flip_sign(q < 9 ? ldp<COH>(d.S[q] + o) : __ldg(d.stat[q - 9] + o),
                       (par_x2d(q) < 0 ? mx : 0u) ^ (par_y2d(q) < 0 ? my : 0u));
}

// Per-node record a sweep keeps for its stencil (18 doubles).
enum { R_FP = 0, R_FM = 3, R_GP = 6, R_GM = 9, R_MIX = 12, R_H = 15, R_M = 16, R_W = 17, NREC = 18 };

// Pointwise fluxes of eq. (swe-form-2d-e) and their chain-rule derivatives of eq. (swe-form-2d-h). DIR = 0:
// x-sweep (F1, d_x F1 along the sweep, d_y F1 for the mixed term); DIR = 1: y-sweep (F2, d_y F2, d_x F2).
template <int DIR, class R>
__device__ __forceinline__ void node_fluxes(const Node12T<R>& n, R g, R F[3], R Gs[3], R Gm[3], R& h) {
  const R eta = n.v[0], m = n.v[1], w = n.v[2], b = n.v[9];
  h = eta - b;
  const R rh = fast_rcp(h);
  const R u = m * rh, v = w * rh;
  const R gh = g * h, ge = g * eta;
  const R pres = ge * fma(R(0.5), eta, -b);  // g/2 (eta^2 - 2 eta b)
  const R uv = u * v;
  // derivative data along the sweep (split) and across it (mixed)
  const int qs = DIR == 0 ? 3 : 6, qm = DIR == 0 ? 6 : 3;
  const R Hs = n.v[qs], Ms = n.v[qs + 1], Ws = n.v[qs + 2], Bs = n.v[DIR == 0 ? 10 : 11];
  const R Hm = n.v[qm], Mm = n.v[qm + 1], Wm = n.v[qm + 2], Bm = n.v[DIR == 0 ? 11 : 10];
  const R mv = m * v;
  if (DIR == 0) {
    const R uu = u * u, a1 = gh - uu, a2 = uu - ge, u2 = u + u;
    F[0] = m; F[1] = fma(m, u, pres); F[2] = mv;
    Gs[0] = Ms;
    Gs[1] = fma(u2, Ms, fma(a1, Hs, a2 * Bs));
    Gs[2] = fma(uv, Bs - Hs, fma(v, Ms, u * Ws));
    Gm[0] = Mm;
    Gm[1] = fma(u2, Mm, fma(a1, Hm, a2 * Bm));
    Gm[2] = fma(uv, Bm - Hm, fma(v, Mm, u * Wm));
  } else {
    const R vv = v * v, a1 = gh - vv, a2 = vv - ge, v2 = v + v;
    F[0] = w; F[1] = mv; F[2] = fma(w, v, pres);
    Gs[0] = Ws;
    Gs[1] = fma(uv, Bs - Hs, fma(v, Ms, u * Ws));
    Gs[2] = fma(v2, Ws, fma(a1, Hs, a2 * Bs));
    Gm[0] = Wm;
    Gm[1] = fma(uv, Bm - Hm, fma(v, Mm, u * Wm));
    Gm[2] = fma(v2, Wm, fma(a1, Hm, a2 * Bm));
  }
}

// The node's record: fluxes split with the global alpha (Sec. R(2.1) Step 1, without the factor 1/2).
template <int DIR, class R>
__device__ __forceinline__ void node_record(const Node12T<R>& n, R g, R alpha, R rec[NREC]) {
  R F[3], Gs[3], Gm[3];
  node_fluxes<DIR>(n, g, F, Gs, Gm, rec[R_H]);
  const int qs = DIR == 0 ? 3 : 6;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    rec[R_FP + c] = fma(alpha, n.v[c], F[c]);
    rec[R_FM + c] = fma(-alpha, n.v[c], F[c]);
    rec[R_GP + c] = fma(alpha, n.v[qs + c], Gs[c]);
    rec[R_GM + c] = fma(-alpha, n.v[qs + c], Gs[c]);
    rec[R_MIX + c] = Gm[c];
  }
  rec[R_M] = n.v[1];
  rec[R_W] = n.v[2];
}

// The record with its split fluxes and derivative fluxes (entries R_FP .. R_GM + 2) in fixed point for the
// nonlinear reconstruction (hw_fixed.h): per component, the four entries as 64-bit integers (below 2^60) of one
// unit, set by the exponents of F, G and alpha times U, D; the split itself is formed in fixed point (six products
// for the twelve fmas of node_record). R_GM holds -G-, the derivative the mirrored side takes. R_X holds the three
// units' biased exponents and, above them, whether an operand does not fit (infinite, NaN or subnormal data, or
// near the ends of the range).
enum { R_X = NREC, NRECX = NREC + 1 };
constexpr int kFxExpMin = 256, kFxExpMax = 1900;  // exponents whose products and squares stay far from the ends

template <int DIR>
__device__ __forceinline__ void node_record_fixed(const Node12& n, double g, double alpha, double rec[NRECX]) {
  double F[3], Gs[3], Gm[3];
  node_fluxes<DIR>(n, g, F, Gs, Gm, rec[R_H]);
  const int qs = DIR == 0 ? 3 : 6;
  int ua;
  const FxS al = fx_split(fx_mantissa(alpha, ua));
  const int ea = ua + 1084;  // alpha's biased exponent
  bool bad = (unsigned)(ea - 600) > 600u;
  int em[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double U = n.v[c], D = n.v[qs + c];
    const uint32_t wf = max(fx_absw(F[c]), fx_absw(Gs[c])), wu = max(fx_absw(U), fx_absw(D));
    em[c] = max((int)(wf >> 20) + 1, (int)(wu >> 20) + ea - 1020);
    const bool any = (fx_any(F[c]) | fx_any(Gs[c]) | fx_any(U) | fx_any(D)) != 0u;
    bad |= (max(wf, wu) >= (uint32_t)kFxExpMax << 20) | (em[c] > kFxExpMax) | ((em[c] < kFxExpMin) & any);
    em[c] = max(em[c], kFxExpMin);
    const int eu = em[c] - ea + 1020;  // alpha times a multiple of 2^(eu - 1082) is one of 2^(em - 1082)
    const int64_t f = fx_from_double(F[c], em[c]), q = fx_from_double(Gs[c], em[c]);
    const int64_t pu = fx_mulhi(fx_split(fx_from_double(U, eu)), al, 0), pd = fx_mulhi(fx_split(fx_from_double(D, eu)), al, 0);
    rec[R_FP + c] = __longlong_as_double(f + pu);
    rec[R_FM + c] = __longlong_as_double(f - pu);
    rec[R_GP + c] = __longlong_as_double(q + pd);
    rec[R_GM + c] = __longlong_as_double(pd - q);
    rec[R_MIX + c] = Gm[c];
  }
  rec[R_M] = n.v[1];
  rec[R_W] = n.v[2];
  rec[R_X] = f64_from_words((uint32_t)(em[0] | (em[1] << 16)), (uint32_t)em[2] | (bad ? 0x10000u : 0u));
}

// ---------------------------------------------------------------------------------------------
// One interface from the four stencil records (nodes i-1, i, i+1, i+2 along the sweep).
// Outputs (12): 2 Fhat, 2 bhat, 24 dS Ghat (derivative-equation flux), 12 dT Mhat (mixed term),
// where dS is the spacing along the sweep and dT the spacing across it. In double the first three carry the factors
// the node update would apply to their differences (interface_scales): there each costs the FP64 pipe an operation per
// difference, here most are part of the fixed-point form's conversions.
// qb[6] = source candidates q_1..q_3 of (b, dS b_s) for the '+' side then the mirrored '-' side.
// ---------------------------------------------------------------------------------------------
// Factors of the double interface values of sweep DIR: cf of 2 Fhat is 12 c_g = 1/(2dS), cb of 2 bhat is g/(2dS), cg of
// 24 dS Ghat is 1/(24dS).
template <int DIR>
__device__ __forceinline__ double scale_g(const Dev2D& d) { return DIR == 0 ? d.c_gx : d.c_gy; }
template <int DIR>
__device__ __forceinline__ double scale_b(const Dev2D& d) { return DIR == 0 ? d.c_bgx : d.c_bgy; }
template <int DIR>
__device__ __forceinline__ void interface_scales(const Dev2D& d, double out[12]) {
  const double cg = scale_g<DIR>(d), cf = 12.0 * cg, cb = scale_b<DIR>(d);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    out[c] *= cf;
    out[3 + c] *= cb;
    out[6 + c] *= cg;
  }
}

template <int DIR, bool LINEAR, bool CHAR, class R>
__device__ __forceinline__ void interface_values(const R* r0, const R* r1, const R* r2,
                                                   const R* r3, int stride, const R qb[6], R g,
                                                   R eps_w, R out[12]) {
#define RV(r, f) (r)[(f) * stride]
  // interface state: h = (h_i + h_{i+1})/2, u = (m_i + m_{i+1})/(h_i + h_{i+1}), v likewise
  const R hs = RV(r1, R_H) + RV(r2, R_H);
  const R rhs = fast_rcp(hs);
  const R ub = (RV(r1, R_M) + RV(r2, R_M)) * rhs;
  const R vb = (RV(r1, R_W) + RV(r2, R_W)) * rhs;
  const R gh = (R(0.5) * g) * hs;
  const R rs = fast_rsqrt(gh);
  const R ic2 = R(0.5) * rs;  // 1/(2c)
  // normal / tangential velocity of this sweep
  const R un = DIR == 0 ? ub : vb, ut = DIR == 0 ? vb : ub;
  // un +- c with c = gh / sqrt(gh)
  const R upc = fma(gh, rs, un), umc = fma(-gh, rs, un);
  // component indices: normal momentum and tangential momentum
  const int cn = DIR == 0 ? 1 : 2, ct = DIR == 0 ? 2 : 1;
  // scaled epsilon: fields 1, 3 carry s = 4c, field 2 carries s = 2 (both 2 without projection)
  const R eps2 = R(4.0) * eps_w;
  const R eps13 = CHAR ? (((R(8.0) * g) * eps_w) * hs) : eps2;

  R G[3], GB1 = R(0.0), GB3 = R(0.0);  // per-field sums over both sides; source fields 1 and 3
  const R* rp[4] = {r0, r1, r2, r3};
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    // '+' uses nodes 0,1,2 of (F+, G+); '-' uses nodes 3,2,1 of (F-, G-) with the derivative negated.
    const int o0 = side == 0 ? 0 : 3, o1 = side == 0 ? 1 : 2, o2 = side == 0 ? 2 : 1;
    const int fo = side == 0 ? R_FP : R_FM, go = side == 0 ? R_GP : R_GM;
    const R sg = side == 0 ? R(1.0) : -R(1.0);
    R f[3][3], p[3][3];  // [field][stencil point]
    const int os[3] = {o0, o1, o2};
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      const R* r = rp[os[t]];
      const R F0 = RV(r, fo), Fn = RV(r, fo + cn), Ft = RV(r, fo + ct);
      const R G0 = sg * RV(r, go), Gn = sg * RV(r, go + cn), Gt = sg * RV(r, go + ct);
      if (CHAR) {
        // rows of L without 1/(2c): (un+c, -1, 0), (-ut, 0, 1), (-(un-c), 1, 0) on (rho, normal, tangential)
        f[0][t] = fma(upc, F0, -Fn);
        f[1][t] = fma(-ut, F0, Ft);
        f[2][t] = fma(-umc, F0, Fn);
        p[0][t] = fma(upc, G0, -Gn);
        p[1][t] = fma(-ut, G0, Gt);
        p[2][t] = fma(-umc, G0, Gn);
      } else {
        f[0][t] = F0; f[1][t] = Fn; f[2][t] = Ft;
        p[0][t] = G0; p[1][t] = Gn; p[2][t] = Gt;
      }
    }
    const R* qbs = qb + 3 * side;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      WeightsT<R> W;
      const R e = (k == 1) ? eps2 : eps13;
      const R v = hweno_side<LINEAR>(f[k][0], f[k][1], f[k][2], p[k][0], p[k][1], p[k][2], e, W);
      G[k] = side == 0 ? v : G[k] + v;
      if (CHAR) {
        // source data per field: (-b, 0, +b) (row entries of the normal-momentum column)
        if (k == 0) GB1 -= weighted(W, qbs[0], qbs[1], qbs[2]);
        if (k == 2) GB3 += weighted(W, qbs[0], qbs[1], qbs[2]);
      } else {
        if (k == 1) GB1 += weighted(W, qbs[0], qbs[1], qbs[2]);  // the normal-momentum component itself
      }
    }
  }
  // back to physical components: 2 Fhat = R diag(1/s) G * 2
  R F2[3], B2[3];
  if (CHAR) {
    const R A = (G[0] + G[2]) * ic2;
    F2[0] = A;
    F2[cn] = fma(un, A, R(0.5) * (G[2] - G[0]));
    F2[ct] = fma(ut, A, G[1]);
    const R Bs = (GB1 + GB3) * ic2;
    B2[0] = Bs;
    B2[cn] = fma(un, Bs, R(0.5) * (GB3 - GB1));
    B2[ct] = ut * Bs;
  } else {
    F2[0] = G[0]; F2[cn] = G[1]; F2[ct] = G[2];
    B2[0] = R(0.0); B2[cn] = GB1; B2[ct] = R(0.0);
  }
  // derivative-equation flux (eq. Rec-phi, component-wise): 24 dS Ghat = 3 fpart + gpart
  // mixed term (eq. mixed): 12 dT Mhat = 7 (X_i + X_{i+1}) - (X_{i-1} + X_{i+2})
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const R fpart =
        fma(R(7.0), RV(r2, R_FP + c) - RV(r1, R_FM + c),
            fma(R(8.0), RV(r2, R_FM + c) - RV(r1, R_FP + c), RV(r0, R_FP + c) - RV(r3, R_FM + c)));
    const R gpart = fma(-R(5.0), RV(r2, R_GP + c) + RV(r1, R_GM + c),
                             fma(-R(2.0), RV(r1, R_GP + c) + RV(r2, R_GM + c), RV(r0, R_GP + c) + RV(r3, R_GM + c)));
    out[c] = F2[c];
    out[3 + c] = B2[c];
    out[6 + c] = fma(R(3.0), fpart, gpart);
    out[9 + c] = fma(R(7.0), RV(r1, R_MIX + c) + RV(r2, R_MIX + c), -(RV(r0, R_MIX + c) + RV(r3, R_MIX + c)));
  }
#undef RV
}

// The same interface with the reconstruction and the derivative flux in fixed point (hw_fixed.h), from four
// records of node_record_fixed. Returns false, with out unspecified, when an operand does not fit. PAIR: the lanes 2k
// and 2k + 1 share one interface, each forms the side of its lowest bit, and both return the result (the sums over the
// sides are of integers, so it is the same).
template <int DIR, bool CHAR, bool PAIR = false>
__device__ __forceinline__ bool interface_values_fixed(const double* r0, const double* r1, const double* r2,
                                                       const double* r3, int stride, const double qb[6],
                                                       const Dev2D& d, double out[12]) {
#define RV(r, f) (r)[(f) * stride]
  const int cn = DIR == 0 ? 1 : 2, ct = DIR == 0 ? 2 : 1;
  const double* rp[4] = {r0, r1, r2, r3};
  bool bad = false;
  // per component: the largest exponent over the four nodes; node s is shifted down by the difference
  int e0[4], en[4], et[4];
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    uint32_t lo, hi;
    f64_words(RV(rp[s], R_X), lo, hi);
    e0[s] = (int)(lo & 0xffffu);
    const int e1 = (int)(lo >> 16), e2 = (int)(hi & 0xffffu);
    en[s] = DIR == 0 ? e1 : e2;
    et[s] = DIR == 0 ? e2 : e1;
    bad |= (hi >> 16) != 0u;
  }
  if (bad) return false;
  const int m0 = max(max(e0[0], e0[1]), max(e0[2], e0[3])), mn = max(max(en[0], en[1]), max(en[2], en[3])),
            mt = max(max(et[0], et[1]), max(et[2], et[3]));
  // interface state (as interface_values)
  const double hs = RV(r1, R_H) + RV(r2, R_H);
  const double rhs = fast_rcp(hs);
  const double ub = (RV(r1, R_M) + RV(r2, R_M)) * rhs;
  const double vb = (RV(r1, R_W) + RV(r2, R_W)) * rhs;
  const double gh = d.half_g * hs;
  const double rs = fast_rsqrt(gh);
  const double un = DIR == 0 ? ub : vb, ut = DIR == 0 ? vb : ub;
  const double upc = fma(gh, rs, un), umc = fma(-gh, rs, un);
  const FxEps eps2 = fx_eps(d.fx_eps2, bad);
  const FxEps eps13 = CHAR ? fx_eps(d.fx_eps13 * hs, bad) : eps2;
  const FxScale kg = fx_scale(scale_g<DIR>(d), bad), kb = fx_scale(scale_b<DIR>(d), bad);
  // units of the fields' data (below 2^57): field k is its component (normal, tangential, normal) plus c_k F_0,
  // c = (-(un + c), -ut, -(un - c)); a coefficient's shift brings its products to the field's unit
  int U02 = 0, U1 = 0;
  FxS ck[3] = {};
  if (CHAR) {
    int up, um, uv;
    const int64_t xp = fx_mantissa(-upc, up), xm = fx_mantissa(-umc, um), xv = fx_mantissa(-ut, uv);
    const int u0 = m0 - 1082 + 64;
    U02 = max(max(max(up, um) + u0 + 2, mn - 1078), -900);
    U1 = max(max(uv + u0 + 2, mt - 1078), -900);
    bad |= max(U02, U1) > 900;
    ck[0] = fx_split(xp >> min(U02 - up - u0, 63));
    ck[1] = fx_split(xv >> min(U1 - uv - u0, 63));
    ck[2] = fx_split(xm >> min(U02 - um - u0, 63));
  }
  // shifts of the four nodes, one byte each
  auto shifts = [](int b, const int e[4]) {
    return (uint32_t)min(b - e[0], 63) | ((uint32_t)min(b - e[1], 63) << 8) | ((uint32_t)min(b - e[2], 63) << 16) |
           ((uint32_t)min(b - e[3], 63) << 24);
  };
  const uint32_t s0 = shifts(CHAR ? m0 : m0 + 4, e0), sn = shifts(CHAR ? U02 + 1082 : mn + 4, en),
                 st = shifts(CHAR ? U1 + 1082 : mt + 4, et);
  int64_t G[3] = {0, 0, 0}, BA = 0, BD = 0, Q[3] = {0, 0, 0};
  uint32_t bw = 0;
#pragma unroll
  for (int q = 0; q < 6; ++q) bw = max(bw, fx_absw(qb[q]));
  const int eb = max((int)(bw >> 20), kFxExpMin);  // source candidates: below 2^60, of one unit
  bad |= eb > kFxExpMax;
  // derivative of the quintic (eq. Rec-phi), exact: 3 (f_0 - 8 f_1 + 7 f_2) + p_0 - 2 p_1 - 5 p_2 for data below 2^56
  auto quintic = [](const int64_t f[3], const int64_t p[3]) {
    return 3 * ((f[0] - f[1]) - 7 * (f[1] - f[2])) + (p[0] - 2 * p[1] - 5 * p[2]);
  };
  const int own = PAIR ? (int)(threadIdx.x & 1) : 0;
#pragma unroll 1
  for (int side = PAIR ? own : 1; side >= own; --side) {
    // '+': nodes 0, 1, 2 of (F+, G+); '-': nodes 3, 2, 1 of (F-, -G-)
    const double* const q = side == 0 ? r0 : r3 + R_FM * stride;
    const int step = side == 0 ? (int)(r1 - r0) : -(int)(r1 - r0);
    const uint32_t rev = side == 0 ? 0x3210u : 0x0123u;
    const uint32_t z0 = __byte_perm(s0, 0, rev), zn = __byte_perm(sn, 0, rev), zt = __byte_perm(st, 0, rev);
    auto load = [&](int t, int f, uint32_t z) {
      return (int64_t)__double_as_longlong(q[t * step + f * stride]) >> ((z >> (8 * t)) & 0xffu);
    };
    FxS x[3], y[3];
    if (CHAR) {
      int64_t f[3], p[3];
#pragma unroll
      for (int t = 0; t < 3; ++t) {
        f[t] = load(t, 0, z0);
        p[t] = load(t, R_GP, z0);
        x[t] = fx_split(f[t]);
        y[t] = fx_split(p[t]);
        f[t] >>= 4;
        p[t] >>= 4;
      }
      Q[0] = quintic(f, p) - Q[0];  // the mirrored side's derivative counts negative
    }
    int64_t v1 = 0, v2 = 0;  // field 1's weights
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int c = CHAR ? (k == 1 ? ct : cn) : (k == 0 ? 0 : k == 1 ? cn : ct);
      const uint32_t z = CHAR ? (k == 1 ? zt : zn) : (k == 0 ? z0 : k == 1 ? zn : zt);
      int64_t f[3], p[3];
#pragma unroll
      for (int t = 0; t < 3; ++t) {
        f[t] = load(t, c, z);
        p[t] = load(t, R_GP + c, z);
      }
      if (CHAR) {
        if (k == 0) Q[1] = quintic(f, p) - Q[1];
        const FxS a = k == 0 ? ck[0] : k == 1 ? ck[1] : ck[2];
#pragma unroll
        for (int t = 0; t < 3; ++t) {
          f[t] = fx_mulhi(x[t], a, f[t]);
          p[t] = fx_mulhi(y[t], a, p[t]);
        }
      } else {
        Q[k] = quintic(f, p) - Q[k];
      }
      const FxEps ek = k == 1 ? eps2 : eps13;
      const int u = CHAR ? (k == 1 ? U1 : U02) : (k == 0 ? m0 : k == 1 ? mn : mt) - 1078;
      int64_t w1, w2;
      const int64_t v = fx_hweno_side(f[0], f[1], f[2], p[0], p[1], p[2], ek, u, w1, w2);
      if (k == 0) G[0] += v;
      if (k == 1) G[1] += v;
      if (k == 2) G[2] += v;
      // the source with the weights of fields 1 and 3 (of the normal component without projection)
      if (k == (CHAR ? 0 : 1)) { v1 = w1; v2 = w2; }
      if (k == 2) {
        const int64_t c3 = fx_from_double(qb[3 * side + 2], eb);
        const FxS d1 = fx_split(fx_from_double(qb[3 * side], eb) - c3), d2 = fx_split(fx_from_double(qb[3 * side + 1], eb) - c3);
        if (CHAR) {
          BA += fx_dot2<2>(d1, fx_split(w1 - v1), d2, fx_split(w2 - v2));
          BD += c3 + fx_dot2<2>(d1, fx_split(w1 + v1), d2, fx_split(w2 + v2));
        } else {
          BD += c3 + fx_dot2<3>(d1, fx_split(v1), d2, fx_split(v2));
        }
      }
    }
  }
  if constexpr (PAIR) {
    const unsigned pair = 3u << (threadIdx.x & 30);
    auto other = [&](int64_t x) { return (int64_t)__shfl_xor_sync(pair, (long long)x, 1); };
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      G[k] += other(G[k]);
      if (k < 2 || !CHAR) {
        const int64_t q = other(Q[k]);
        Q[k] = own == 0 ? Q[k] - q : q - Q[k];
      }
    }
    BA += other(BA);
    BD += other(BD);
  }
  // back to physical components: G carries a factor 6, BA and BD (the sums over fields 1 and 3 of -+ and of
  // the source values) a factor 1/2
  const int ub_ = eb - 1082;
  if (CHAR) {
    // 2 Fhat = (A, un A + (G2 + G0)/12, ut A + G1/6) with A = (G2 - G0) / (12 c), times 12 c_g
    const double A = fx_to_double(G[2] - G[0], U02) * (scale_g<DIR>(d) * rs);
    out[0] = A;
    out[cn] = fma(un, A, fx_to_double_scaled(G[2] + G[0], U02, kg));
    out[ct] = fma(ut, A, fx_to_double_scaled(G[1], U1 + 1, kg));
    const double Bs = fx_to_double(BA, ub_) * (scale_b<DIR>(d) * rs);
    out[3] = Bs;
    out[3 + cn] = fma(un, Bs, fx_to_double_scaled(BD, ub_, kb));
    out[3 + ct] = ut * Bs;
  } else {
    out[0] = fx_to_double_scaled(G[0], m0 - 1077, kg);
    out[cn] = fx_to_double_scaled(G[1], mn - 1077, kg);
    out[ct] = fx_to_double_scaled(G[2], mt - 1077, kg);
    out[3] = 0.0;
    out[3 + cn] = fx_to_double_scaled(BD, ub_, kb);
    out[3 + ct] = 0.0;
  }
  // derivative-equation flux and mixed term
  if (CHAR) {
    // the tangential component in its own unit (the field's may be coarser)
    auto load = [&](int s, int q) { return (int64_t)__double_as_longlong(RV(rp[s], q + ct)) >> min(mt + 4 - et[s], 63); };
    const int64_t f0[3] = {load(0, R_FP), load(1, R_FP), load(2, R_FP)}, p0[3] = {load(0, R_GP), load(1, R_GP), load(2, R_GP)};
    const int64_t f1[3] = {load(3, R_FM), load(2, R_FM), load(1, R_FM)}, p1[3] = {load(3, R_GM), load(2, R_GM), load(1, R_GM)};
    Q[2] = quintic(f0, p0) - quintic(f1, p1);
  }
  out[6] = fx_to_double_scaled(Q[0], m0 - 1078, kg);
  out[6 + cn] = fx_to_double_scaled(Q[1], CHAR ? U02 : mn - 1078, kg);
  out[6 + ct] = fx_to_double_scaled(Q[2], mt - 1078, kg);
#pragma unroll
  for (int c = 0; c < 3; ++c)
    out[9 + c] = fma(7.0, RV(r1, R_MIX + c) + RV(r2, R_MIX + c), -(RV(r0, R_MIX + c) + RV(r3, R_MIX + c)));
#undef RV
  return !bad;
}

// Where the two fallback calls below find their grid: a kernel parameter's address for one grid; the batched kernels,
// which form a Dev2D per thread, have the call form it again (BatchSource), because a local block whose address went
// into a call would be written to local memory, all 560 bytes of it, by every thread that never makes the call.
template <class R>
struct GridSource {
  const Dev2DT<R>* p;
  __device__ __forceinline__ const Dev2DT<R>& dev() const { return *p; }
};

// An interface whose data does not fit the fixed-point form, from its nodes again on the FP64 pipe: nodes
// (i - 2 .. i + 1, j) for DIR = 0, (i, j - 2 .. j + 1) for DIR = 1.
template <int DIR, bool CHAR, bool COH, class S>
__device__ __noinline__ void interface_fallback(const S src, double alpha, int i, int j, size_t on, const double qb[6],
                                                double out[12]) {
  const Dev2D& d = src.dev();
  double rec[4 * NREC];
#pragma unroll 1
  for (int s = 0; s < 4; ++s) {
    Node12 n;
    load_node<COH>(d, DIR == 0 ? i - 2 + s : i, DIR == 0 ? j : j - 2 + s, n, on);
    node_record<DIR>(n, d.g, alpha, rec + s * NREC);
  }
  interface_values<DIR, false, CHAR>(rec, rec + NREC, rec + 2 * NREC, rec + 3 * NREC, 1, qb, d.g, d.eps_w, out);
  interface_scales<DIR>(d, out);
}

// ---------------------------------------------------------------------------------------------
// alpha_x, alpha_y = max over nodes of |u| + c, |v| + c (exact max via ordered 64-bit keys) in two
// passes that keep the FP64 pipe out of most nodes: a coarse pass evaluates |u| + c in float (from the
// depth formed in double, converted by integer operations) and reduces the float maxima M; an exact pass
// re-evaluates every node in float and computes the double value only where the float one is within a
// relative 1e-5 of M (or cannot be trusted: values outside float's range, NaN, infinity). The float
// values are within about 1e-6 of the double ones, so the node attaining the double maximum is always
// re-evaluated and the result is the exact double maximum (a re-evaluated node contributes to both
// directions, which is harmless: no node's value exceeds a direction's maximum).
// ---------------------------------------------------------------------------------------------
// double -> float by truncation with integer operations (the FP64 pipe stays free): relative error
// below 2^-23 for values in float's normal range. Values below it become 0 (tiny is true); values
// above it, infinities and NaN set huge.
__device__ __forceinline__ float d2f_trunc(double x, bool& tiny, bool& huge) {
  const long long b = __double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ff);
  tiny = e <= 1023 - 127;
  huge = e >= 1023 + 128;
  const unsigned int sign = (unsigned int)((unsigned long long)b >> 32) & 0x80000000u;
  const unsigned int f = sign | ((unsigned int)(e - 1023 + 127) << 23) | (unsigned int)((b >> 29) & 0x7fffff);
  return tiny ? 0.0f : __uint_as_float(f);
}

// Float estimates of |u| + c and |v| + c at node o from the depth formed in double. exact: the node
// needs the double evaluation regardless (a depth or momentum outside float's range, NaN, infinity);
// neg: the depth is negative.
template <bool COH = false>
__device__ __forceinline__ void alpha_coarse(const Dev2D& d, size_t o, float& ax, float& ay, bool& exact,
                                             bool& neg) {
  const double hd = ldp<COH>(d.S[0] + o) - __ldg(d.stat[0] + o);
  bool t0, h0, t1, h1, t2, h2;
  const float h = d2f_trunc(hd, t0, h0);
  const float m = d2f_trunc(ldp<COH>(d.S[1] + o), t1, h1);
  const float w = d2f_trunc(ldp<COH>(d.S[2] + o), t2, h2);
  exact = t0 || h0 || h1 || h2;
  neg = h < 0.0f;
  const float rh = fast_rcp(h);
  const float gh = (float)d.g * h;
  const float c = gh * fast_rsqrt(gh);
  ax = fabsf(m) * rh + c;
  ay = fabsf(w) * rh + c;
}

// The exact pass over nodes o = begin, begin + step, ... < end, with the coarse maxima m32[0..1]: keys of
// the double maxima into kx, ky and status flags into bad.
// The double evaluation of the exact pass at node o: keys of |u| + c and |v| + c into kx, ky (maxima),
// status flags into bad.
template <bool COH = false>
__device__ __forceinline__ void alpha_exact_node(const Dev2D& d, size_t o, unsigned long long& kx,
                                                 unsigned long long& ky, int& bad) {
  const double hd = ldp<COH>(d.S[0] + o) - __ldg(d.stat[0] + o);
  if (!(hd > 0.0) || !(hd < 1e300)) {
    bad |= hd == hd ? HW_STATUS_DEPTH : HW_STATUS_NONFINITE;
    return;
  }
  const double rh = fast_rcp(hd);
  const double gh = d.g * hd;
  const double c = gh * fast_rsqrt(gh);
  const double ax = dabs(ldp<COH>(d.S[1] + o) * rh) + c, ay = dabs(ldp<COH>(d.S[2] + o) * rh) + c;
  if (!(ax < 1e300) || !(ay < 1e300)) {
    bad |= HW_STATUS_NONFINITE;
    return;
  }
  kx = max(kx, dkey(ax));
  ky = max(ky, dkey(ay));
}

// Whether the exact pass evaluates a node, from its coarse estimates and the thresholds tx, ty (the coarse
// maxima lowered by the estimates' error bound).
__device__ __forceinline__ bool alpha_needs_exact(float fx, float fy, bool exact, bool neg, float tx, float ty) {
  return exact || (!neg && !(fx < tx && fy < ty));
}

template <bool COH = false>
__device__ __forceinline__ void alpha_exact_range(const Dev2D& d, const unsigned int* m32, size_t begin, size_t end,
                                                  size_t step, unsigned long long& kx, unsigned long long& ky,
                                                  int& bad) {
  const float tx = __uint_as_float(m32[0]) * (1.0f - 1e-5f), ty = __uint_as_float(m32[1]) * (1.0f - 1e-5f);
  for (size_t o = begin; o < end; o += step) {
    float fx, fy;
    bool exact, neg;
    alpha_coarse<COH>(d, o, fx, fy, exact, neg);
    if (alpha_needs_exact(fx, fy, exact, neg, tx, ty)) alpha_exact_node<COH>(d, o, kx, ky, bad);
  }
}

// alpha keys of one block of 256 threads and 256 U nodes in one pass: float maxima first, then the double values of
// the block's nodes near those (the grid's maximum is one block's, so it is among them). Node u of a thread has number
// o0 + 256 u below n and lies at at(number). kx, ky: the block's maxima, in thread 0; status flags go to *status.
template <int U, class At>
__device__ __forceinline__ void alpha_block_keys(const Dev2D& d, size_t o0, size_t n, At at, unsigned long long& kx,
                                                 unsigned long long& ky, int* status) {
  __shared__ float s_m[2][8];
  __shared__ unsigned long long s_k[2][8];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float fx[U], fy[U], mx = 0.0f, my = 0.0f;
  bool exact[U], neg[U];
  int bad = 0;
#pragma unroll
  for (int u = 0; u < U; ++u) {
    exact[u] = false;
    neg[u] = true;  // past the end: skipped
    fx[u] = fy[u] = 0.0f;
    if (o0 + u * 256 < n) {
      alpha_coarse(d, at(o0 + u * 256), fx[u], fy[u], exact[u], neg[u]);
      if (neg[u] && !exact[u]) bad |= HW_STATUS_DEPTH;
    }
    if (!exact[u] && !neg[u]) {
      mx = fmaxf(mx, fx[u]);
      my = fmaxf(my, fy[u]);
    }
  }
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) {
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, s));
    my = fmaxf(my, __shfl_xor_sync(0xffffffffu, my, s));
  }
  if (lane == 0) { s_m[0][w] = mx; s_m[1][w] = my; }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    mx = fmaxf(mx, s_m[0][k]);
    my = fmaxf(my, s_m[1][k]);
  }
  const float tx = mx * (1.0f - 1e-5f), ty = my * (1.0f - 1e-5f);
  kx = ky = 0;
#pragma unroll
  for (int u = 0; u < U; ++u)
    if (o0 + u * 256 < n && alpha_needs_exact(fx[u], fy[u], exact[u], neg[u], tx, ty))
      alpha_exact_node(d, at(o0 + u * 256), kx, ky, bad);
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) {
    kx = max(kx, __shfl_xor_sync(0xffffffffu, kx, s));
    ky = max(ky, __shfl_xor_sync(0xffffffffu, ky, s));
  }
  if (bad) atomicOr(status, bad);
  if (lane == 0) { s_k[0][w] = kx; s_k[1][w] = ky; }
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int k = 1; k < 8; ++k) {
    kx = max(kx, s_k[0][k]);
    ky = max(ky, s_k[1][k]);
  }
}

// ---------------------------------------------------------------------------------------------
// Sweep tiles over flattened extended lines (shared by the single-grid and the batched kernels).
// x: extended node E = j (nx + 4) + e stands for node (e - 2, j), e = 0 .. nx + 3 (each row with two halo
// nodes on either side, rows one after the other); the x-interface k of row j (between nodes k - 1 and k,
// k = 0 .. nx) sits at E = j (nx + 4) + k and reads the records of E .. E + 3, all in its row.
// y: the same over groups of yc adjacent columns: extended row E = g (ny + 4) + e of group g stands for
// nodes (g yc + c, e - 2), c = 0 .. yc - 1.
// A tile of TILE_T threads forms the node records of TILE_T consecutive extended nodes (x; yc columns of
// TILE_T / yc extended rows in y), then, after one barrier, the interfaces whose four records lie in the
// tile: tiles run across line ends, so no grid size leaves a ragged tile. All TILE_T threads must call;
// sm holds NRECX * TILE_T values (NREC
// in single precision). on / oi: offsets of the grid in pooled node / interface planes (the
// batched form keeps the planes' base pointers in the kernel parameters and adds these, so that no
// per-grid pointer occupies a register). COH: state loads as in ldp.
// ---------------------------------------------------------------------------------------------
constexpr int TILE_T = 128;

template <bool LINEAR, bool CHAR, bool FIXED, bool COH = false, int T = TILE_T, class S, class R>
__device__ __forceinline__ void sweep_x_tile(const Dev2DT<R>& d, const S src, R ax, unsigned E0, R* sm, size_t on = 0,
                                             size_t oi = 0) {
  const unsigned W = d.nx + 4, total = (unsigned)d.ny * W;
  const int t = threadIdx.x;
  {
    const unsigned E = E0 + t;
    if (E < total) {
      const unsigned j = E / W, e = E - j * W;
      Node12T<R> n;
      load_node<COH>(d, (int)e - 2, (int)j, n, on);
      if constexpr (FIXED && !LINEAR) {
        R rec[NRECX];
        node_record_fixed<0>(n, d.g, ax, rec);
#pragma unroll
        for (int f = 0; f < NRECX; ++f) sm[f * T + t] = rec[f];
      } else {
        R rec[NREC];
        node_record<0>(n, R(d.g), ax, rec);
#pragma unroll
        for (int f = 0; f < NREC; ++f) sm[f * T + t] = rec[f];
      }
    }
  }
  __syncthreads();
  const unsigned E = E0 + t;
  if (t >= T - 3 || E >= total) return;
  const unsigned j = E / W, k = E - j * W;
  if (k > (unsigned)d.nx) return;
  const size_t o = oi + (size_t)j * (d.nx + 1) + k;
  R qb[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) qb[q] = __ldg(d.qbx[q] + o);
  R out[12];
  if constexpr (FIXED && !LINEAR) {
    if (!interface_values_fixed<0, CHAR>(sm + t, sm + t + 1, sm + t + 2, sm + t + 3, T, qb, d, out))
      interface_fallback<0, CHAR, COH>(src, ax, (int)k, (int)j, on, qb, out);
  } else {
      interface_values<0, LINEAR, CHAR>(sm + t, sm + t + 1, sm + t + 2, sm + t + 3, T, qb, R(d.g), R(d.eps_w), out);
      if constexpr (std::is_same<R, double>::value) interface_scales<0>(d, out);
  }
#pragma unroll
  for (int q = 0; q < 12; ++q) d.X[q][o] = out[q];
}

template <bool LINEAR, bool CHAR, bool FIXED, bool COH = false, class S, class R>
__device__ __forceinline__ void sweep_y_tile(const Dev2DT<R>& d, const S src, R ay, unsigned E0, int yc, R* sm, size_t on = 0,
                                             size_t oi = 0) {
  const int rows = TILE_T / yc, ifs = rows - 3;
  const unsigned H = d.ny + 4, total = (unsigned)((d.nx + yc - 1) / yc) * H;
  const int t = threadIdx.x, c = t % yc, r = t / yc;
  {
    const unsigned E = E0 + r;
    if (r < rows && E < total) {
      const unsigned g = E / H, e = E - g * H;
      const int i = (int)g * yc + c;
      if (i < d.nx) {
        Node12T<R> n;
        load_node<COH>(d, i, (int)e - 2, n, on);
        if constexpr (FIXED && !LINEAR) {
          R rec[NRECX];
          node_record_fixed<1>(n, d.g, ay, rec);
#pragma unroll
          for (int f = 0; f < NRECX; ++f) sm[f * TILE_T + t] = rec[f];
        } else {
          R rec[NREC];
          node_record<1>(n, R(d.g), ay, rec);
#pragma unroll
          for (int f = 0; f < NREC; ++f) sm[f * TILE_T + t] = rec[f];
        }
      }
    }
  }
  __syncthreads();
  const unsigned E = E0 + r;
  if (r >= ifs || E >= total) return;
  const unsigned g = E / H, k = E - g * H;
  const int i = (int)g * yc + c;
  if (k > (unsigned)d.ny || i >= d.nx) return;
  const size_t o = oi + (size_t)k * d.nx + i;
  R qb[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) qb[q] = __ldg(d.qby[q] + o);
  R out[12];
  const R* s0 = sm + t;
  if constexpr (FIXED && !LINEAR) {
    if (!interface_values_fixed<1, CHAR>(s0, s0 + yc, s0 + 2 * yc, s0 + 3 * yc, TILE_T, qb, d, out))
      interface_fallback<1, CHAR, COH>(src, ay, i, (int)k, on, qb, out);
  } else {
      interface_values<1, LINEAR, CHAR>(s0, s0 + yc, s0 + 2 * yc, s0 + 3 * yc, TILE_T, qb, R(d.g), R(d.eps_w), out);
      if constexpr (std::is_same<R, double>::value) interface_scales<1>(d, out);
  }
#pragma unroll
  for (int q = 0; q < 12; ++q) d.Y[q][o] = out[q];
}

// ---------------------------------------------------------------------------------------------
// Node kernel: RHS assembly, limiter, RK combination (or the bare RHS).
// ---------------------------------------------------------------------------------------------
// Limiter along one direction at one node (Sec. R(2.2)), scaled data. L-rows without 1/(2c):
// x: (u+c, -1, 0), (-v, 0, 1), (-(u-c), 1, 0); y: (v+c, 0, -1), (-u, 1, 0), (-(v-c), 0, 1).
template <int DIR, bool LINEAR, bool CHAR, class R>
__device__ __forceinline__ void limit_dir(const R Um[3], const R U0[3], const R Up[3],
                                          const R Dm[3], const R Dp[3], R u, R v, R c,
                                          R ic2, R gh, R eps, R out[3]) {
  const int cn = DIR == 0 ? 1 : 2, ct = DIR == 0 ? 2 : 1;
  const R un = DIR == 0 ? u : v, ut = DIR == 0 ? v : u;
  const R upc = un + c, umc = un - c;
  auto proj = [&](const R* a, R o[3]) {
    if (CHAR) {
      o[0] = fma(upc, a[0], -a[cn]);
      o[1] = fma(-ut, a[0], a[ct]);
      o[2] = fma(-umc, a[0], a[cn]);
    } else {
      o[0] = a[0]; o[1] = a[cn]; o[2] = a[ct];
    }
  };
  R m0[3], m1[3], m2[3], nl[3], nr[3];
  proj(Um, m0); proj(U0, m1); proj(Up, m2); proj(Dm, nl); proj(Dp, nr);
  const R e13 = CHAR ? ((R(4.0) * eps) * gh) : eps;
  R nu[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) nu[k] = limiter_field<LINEAR>(m0[k], m1[k], m2[k], nl[k], nr[k], k == 1 ? eps : e13);
  if (CHAR) {
    const R A = (nu[0] + nu[2]) * ic2;
    out[0] = A;
    out[cn] = fma(un, A, R(0.5) * (nu[2] - nu[0]));
    out[ct] = fma(ut, A, nu[1]);
  } else {
    out[0] = nu[0]; out[cn] = nu[1]; out[ct] = nu[2];
  }
}

// The limiter of both directions at node (i, j) on the FP64 pipe: scaled V and Q of the node into mod.
// b: the node's bottom; at(di, dj, n): its neighbours.
template <bool LINEAR, bool CHAR, class R, class At>
__device__ __forceinline__ void limit_node(const Dev2DT<R>& d, R b, const R cur[9], R mod[6], const At& at) {
  const R h = cur[0] - b;
  const R gh = R(d.g) * h;
  const R rh = fast_rcp(h);
  const R u = cur[1] * rh, v = cur[2] * rh;
  const R rs = fast_rsqrt(gh);
  const R c = gh * rs, ic2 = R(0.5) * rs;
  Node12T<R> nm, np;
  at(-1, 0, nm);
  at(1, 0, np);
  limit_dir<0, LINEAR, CHAR>(nm.v, cur, np.v, nm.v + 3, np.v + 3, u, v, c, ic2, gh, R(d.eps_lim), mod);
  at(0, -1, nm);
  at(0, 1, np);
  limit_dir<1, LINEAR, CHAR>(nm.v, cur, np.v, nm.v + 6, np.v + 6, u, v, c, ic2, gh, R(d.eps_lim), mod + 3);
}

// The same as a call, for the nodes whose data does not fit the fixed-point form.
template <bool CHAR, bool COH, class S>
__device__ __noinline__ void limit_node_fallback(const S src, int i, int j, size_t on, const double* cur, double* mod) {
  const Dev2D& d = src.dev();
  limit_node<false, CHAR>(d, __ldg(d.stat[0] + on + (size_t)j * d.nx + i), cur, mod,
                          [&](int di, int dj, Node12& n) { load_node<COH>(d, i + di, j + dj, n, on); });
}

// The same in fixed point (hw_fixed.h), direction by direction: the node and its two neighbours as integers of one unit
// per component (mass, normal, tangential), the differences and derivatives projected and limited field by field. One
// copy of the code for both directions, each with its own loads and units: with both directions' 27 values loaded
// first the node kernel spilled 380 bytes a thread at 80 registers, whose write-back was half of its DRAM writes (now about 90 bytes; a
// job of two steps at 2048^2 15.97 -> 15.55 ms).
// False (out unspecified) when an operand does not fit.
struct LimitNode {  // the node's velocities, g h, 1/sqrt(g h) and the weights' epsilons
  double u, v, gh, rs;
  FxEps eps2, eps13;
  bool bad;
  template <bool CHAR>
  __device__ __forceinline__ void form(const Dev2D& d, double b, const double cur[9]) {
    bad = false;
    const double h = cur[0] - b;
    gh = d.g * h;
    const double rh = fast_rcp(h);
    u = cur[1] * rh;
    v = cur[2] * rh;
    rs = fast_rsqrt(gh);
    eps2 = fx_eps(d.fx_eps2l, bad);
    eps13 = CHAR ? fx_eps(d.fx_eps13l * h, bad) : eps2;
  }
};

// out: mass, normal, tangential.
template <bool CHAR, bool COH>
__device__ __forceinline__ bool limit_dir_fixed(const Dev2D& d, int i, int j, size_t on, const double cur[9], const LimitNode& L,
                                                int dir, double out[3]) {
  const double u = L.u, v = L.v, gh = L.gh, rs = L.rs;
  const FxEps eps2 = L.eps2, eps13 = L.eps13;
  bool bad = L.bad;
  // planes of (mass, normal, tangential) and of their derivatives along the direction; across a wall the normal
  // component and the others' derivatives change sign
  const double* const pu[3] = {d.S[0], dir == 0 ? d.S[1] : d.S[2], dir == 0 ? d.S[2] : d.S[1]};
  const double* const pd[3] = {dir == 0 ? d.S[3] : d.S[6], dir == 0 ? d.S[4] : d.S[8], dir == 0 ? d.S[5] : d.S[7]};
  double U[3][3], D[2][3];
  U[0][0] = cur[0];
  U[0][1] = dir == 0 ? cur[1] : cur[2];
  U[0][2] = dir == 0 ? cur[2] : cur[1];
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    bool fx, fy;
    const int ii = map_index(dir == 0 ? i - 1 + 2 * s : i, d.nx, d.bc_x, fx);
    const int jj = map_index(dir == 0 ? j : j - 1 + 2 * s, d.ny, d.bc_y, fy);
    const size_t o = on + (size_t)jj * d.nx + ii;
    const uint32_t m = (dir == 0 ? fx : fy) ? 0x80000000u : 0u;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      U[s + 1][c] = flip_sign(ldp<COH>(pu[c] + o), c == 1 ? m : 0u);
      D[s][c] = flip_sign(ldp<COH>(pd[c] + o), c == 1 ? 0u : m);
    }
  }
  int em[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const uint32_t w = max(max(max(fx_absw(U[0][c]), fx_absw(U[1][c])), fx_absw(U[2][c])), max(fx_absw(D[0][c]), fx_absw(D[1][c])));
    const uint32_t any = fx_any(U[0][c]) | fx_any(U[1][c]) | fx_any(U[2][c]) | fx_any(D[0][c]) | fx_any(D[1][c]);
    em[c] = (int)(w >> 20);
    bad |= (em[c] > kFxExpMax) | ((em[c] < kFxExpMin) & (any != 0u));
    em[c] = max(em[c], kFxExpMin);
  }
  if (bad) return false;
  // differences to the two neighbours and their derivatives, below 2^61
  int64_t a[4][3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int64_t c0 = fx_from_double(U[0][c], em[c]);
    a[0][c] = c0 - fx_from_double(U[1][c], em[c]);
    a[1][c] = fx_from_double(U[2][c], em[c]) - c0;
    a[2][c] = fx_from_double(D[0][c], em[c]);
    a[3][c] = fx_from_double(D[1][c], em[c]);
  }
  if (CHAR) {
    // rows (-(un + c), 1, 0), (-ut, 0, 1), (-(un - c), 1, 0) on (mass, normal, tangential)
    const double un = dir == 0 ? u : v, ut = dir == 0 ? v : u;
    const double upc = fma(gh, rs, un), umc = fma(-gh, rs, un);
    int up, um, uv;
    const int64_t xp = fx_mantissa(-upc, up), xm = fx_mantissa(-umc, um), xv = fx_mantissa(-ut, uv);
    const int u0 = em[0] - 1082 + 64;
    const int U02 = max(max(max(up, um) + u0 + 2, em[1] - 1078), -900), U1 = max(max(uv + u0 + 2, em[2] - 1078), -900);
    if (max(U02, U1) > 900) return false;
    const FxS kp = fx_split(xp >> min(U02 - up - u0, 63)), km = fx_split(xm >> min(U02 - um - u0, 63)),
              kv = fx_split(xv >> min(U1 - uv - u0, 63));
    const int sn = min(U02 + 1082 - em[1], 63), st = min(U1 + 1082 - em[2], 63);
    int64_t nu[3];
    FxS x[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) x[s] = fx_split(a[s][0]);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const FxS kk = k == 0 ? kp : k == 1 ? kv : km;
      int64_t f[4];
#pragma unroll
      for (int s = 0; s < 4; ++s) f[s] = fx_mulhi(x[s], kk, k == 1 ? a[s][2] >> st : a[s][1] >> sn);
      nu[k] = fx_limiter_field(f[0], f[1], f[2], f[3], k == 1 ? eps2 : eps13, k == 1 ? U1 : U02);
    }
    const double A = fx_to_double(nu[2] - nu[0], U02 - 1) * (0.5 * rs);
    out[0] = A;
    out[1] = fma(un, A, fx_to_double(nu[2] + nu[0], U02 - 2));
    out[2] = fma(ut, A, fx_to_double(nu[1], U1 - 1));
  } else {
#pragma unroll
    for (int c = 0; c < 3; ++c)
      out[c] = fx_to_double(fx_limiter_field(a[0][c] >> 3, a[1][c] >> 3, a[2][c] >> 3, a[3][c] >> 3, eps2, em[c] - 1079),
                            em[c] - 1080);
  }
  return true;
}

template <bool CHAR, bool COH>
__device__ __forceinline__ bool limit_node_fixed(const Dev2D& d, int i, int j, size_t on, const double cur[9],
                                                 double mod[6]) {
  LimitNode L;
  L.form<CHAR>(d, __ldg(d.stat[0] + on + (size_t)j * d.nx + i), cur);
#pragma unroll 1
  for (int dir = 0; dir < 2; ++dir) {
    double out[3];
    if (!limit_dir_fixed<CHAR, COH>(d, i, j, on, cur, L, dir, out)) return false;
    if (dir == 0) {
      mod[0] = out[0]; mod[1] = out[1]; mod[2] = out[2];
    } else {
      mod[3] = out[0]; mod[4] = out[2]; mod[5] = out[1];
    }
  }
  return true;
}

// What the update of node (i, j) reads of the grid, from the planes: its state, bottom and neighbours, and the differences
// of interface value q over it along x and y. o, ox, oy: the node, its left x-interface and its lower y-interface.
template <bool COH, class R>
struct PlaneFaces {
  const Dev2DT<R>& d;
  const int i, j;
  const size_t on, o, ox, oy;
  __device__ __forceinline__ R state(int q) const { return ldp<COH>(d.S[q] + o); }
  __device__ __forceinline__ R bottom() const { return __ldg(d.stat[0] + o); }
  __device__ __forceinline__ void neighbour(int di, int dj, Node12T<R>& n) const { load_node<COH>(d, i + di, j + dj, n, on); }
  __device__ __forceinline__ R x(int q) const { return ldp<COH>(d.X[q] + ox + 1) - ldp<COH>(d.X[q] + ox); }
  __device__ __forceinline__ R y(int q) const { return ldp<COH>(d.Y[q] + oy + d.nx) - ldp<COH>(d.Y[q] + oy); }
};

// RHS (eq. swe-form-2d-dis) in scaled units: R_U, dx R_V, dy R_Q, of node o with state cur.
template <class R, class Faces>
__device__ __forceinline__ void right_hand_side(const Dev2DT<R>& d, size_t o, const R cur[9], const Faces& faces, R Rv[9]) {
  // In double: of the negative, whose 50 operations bound this part (64 with the factors applied here, 3 more per node in
  // the RK combination; node kernel at 2048^2 1.04 -> 0.94 ms, the sweeps within 2% of what they were).
  const R eta = cur[0], H1 = cur[3], H2 = cur[6];
  const R g = R(d.g);
  const R c_mx = R(d.c_mx), c_my = R(d.c_my);
  const R ge = g * eta;
  if constexpr (std::is_same<R, double>::value) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const R db = faces.x(3 + c) + faces.y(3 + c);  // g ([b~]_x/dx + [b-]_y/dy)
      Rv[c] = fma(eta, db, faces.x(c) + faces.y(c));
      R rv = fma(H1, db, fma(c_my, faces.y(9 + c), faces.x(6 + c)));
      R rq = fma(H2, db, fma(c_mx, faces.x(9 + c), faces.y(6 + c)));
      if (c > 0) {
        rv = fma(ge, __ldg(d.sv[c - 1] + o), rv);
        rq = fma(ge, __ldg(d.sq[c - 1] + o), rq);
      }
      Rv[3 + c] = rv;
      Rv[6 + c] = rq;
    }
  } else {
    const R c_bx = d.c_bx, c_by = d.c_by, c_gx = d.c_gx, c_gy = d.c_gy;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const R dFx = faces.x(c), dFy = faces.y(c), dbx = faces.x(3 + c), dby = faces.y(3 + c);
      const R dGx = faces.x(6 + c), dGy = faces.y(6 + c), dMx = faces.x(9 + c), dMy = faces.y(9 + c);
      const R db = fma(c_bx, dbx, c_by * dby);  // [b~]_x/dx + [b-]_y/dy
      Rv[c] = fma(-ge, db, fma(-c_bx, dFx, -(c_by * dFy)));
      R rv = fma(-c_gx, dGx, -(c_my * dMy));
      R rq = fma(-c_mx, dMx, -(c_gy * dGy));
      if (c > 0) {
        rv = fma(-ge, __ldg(d.sv[c - 1] + o), rv);
        rq = fma(-ge, __ldg(d.sq[c - 1] + o), rq);
      }
      Rv[3 + c] = fma(-(g * H1), db, rv);
      Rv[6 + c] = fma(-(g * H2), db, rq);
    }
  }
}

// RHS assembly, limiter and RK combination (or the bare RHS) at node (i, j) of one grid, read through faces. FIXED: the
// limiter in fixed point where the node's data fits it. on: offset of the grid in pooled node planes (0 for one grid). COH:
// loads of the state and base planes as in ldp.
template <int MODE, bool LINEAR, bool CHAR, bool FIXED, bool COH, class S, class R, class Faces>
__device__ __forceinline__ void node_update_faces(const Dev2DT<R>& d, const S src, const StageArgsT<R>& sa, int i, int j, size_t on,
                                                  const Faces& faces) {
  const size_t o = on + (size_t)j * d.nx + i;
  R cur[9];
#pragma unroll
  for (int q = 0; q < 9; ++q) cur[q] = faces.state(q);
  if (MODE == MODE_STAGE && !(*sa.dt > 0.0)) {
    // a step of size 0 (e.g. clipped at the end time) leaves the state unchanged
#pragma unroll
    for (int q = 0; q < 9; ++q) sa.out[q][o] = cur[q];
    return;
  }
  // ---- limiter (Sec. R(2.2), dimension by dimension) ----
  R mod[6];
  if (MODE == MODE_STAGE) {
    if (sa.limiter) {
      if constexpr (FIXED && !LINEAR && std::is_same<R, double>::value) {
        if (!limit_node_fixed<CHAR, COH>(d, i, j, on, cur, mod)) limit_node_fallback<CHAR, COH>(src, i, j, on, cur, mod);
      } else {
        limit_node<LINEAR, CHAR>(d, faces.bottom(), cur, mod, [&](int di, int dj, Node12T<R>& n) { faces.neighbour(di, dj, n); });
      }
    } else {
#pragma unroll
      for (int q = 0; q < 6; ++q) mod[q] = cur[3 + q];
    }
  }
  R Rv[9];
  right_hand_side<R>(d, o, cur, faces, Rv);
  if (MODE == MODE_RHS) {
    // physical units: R_V = (dx R_V)/dx, R_Q = (dy R_Q)/dy
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      const R s = q < 3 ? R(1.0) : R(q < 6 ? d.inv_dx : d.inv_dy);
      const R r = q < 3 ? Rv[q] : Rv[q] * s;
      sa.rhs_out[q][o] = std::is_same<R, double>::value ? flip_sign(r, 0x80000000u) : r;
    }
    return;
  }
  // ---- SSP-RK3 combination (eq. RK) ----
  const R dt = std::is_same<R, double>::value ? -R(*sa.dt) : R(*sa.dt);
  if (sa.k == 1) {
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      const R cq = q < 3 ? cur[q] : mod[q - 3];
      if (sa.base) sa.base[q][o] = cq;
      sa.out[q][o] = fma(dt, Rv[q], cq);
    }
    return;
  }
  if constexpr (std::is_same<R, double>::value) {
    // 3/4 base + (cq + dt R)/4, the quarter without the FP64 pipe. As (3 base + cq + dt R)/4, also two operations, the sum
    // 3 base + cq is rounded at the result's own last place where here only a quarter of a rounding comes in: errors of runs
    // against 64 bits were 5 to 8% larger with it.
    if (sa.k == 2) {
#pragma unroll
      for (int q = 0; q < 9; ++q) {
        const R cq = q < 3 ? cur[q] : mod[q - 3];
        sa.out[q][o] = fma(0.75, ldp<COH>(sa.base[q] + o), fx_quarter(fma(dt, Rv[q], cq)));
      }
      return;
    }
  }
  {
    const R a = sa.k == 2 ? R(0.75) : R(1.0) / R(3.0);
    const R b = sa.k == 2 ? R(0.25) : R(2.0) / R(3.0);
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      const R cq = q < 3 ? cur[q] : mod[q - 3];
      sa.out[q][o] = fma(a, ldp<COH>(sa.base[q] + o), b * fma(dt, Rv[q], cq));
    }
  }
}

// The same from the interface planes; oxo, oyo: the grid's offsets in pooled ones. COH: their loads too.
template <int MODE, bool LINEAR, bool CHAR, bool FIXED = false, bool COH = false, class S, class R>
__device__ __forceinline__ void node_update(const Dev2DT<R>& d, const S src, const StageArgsT<R>& sa, int i, int j, size_t on = 0,
                                            size_t oxo = 0, size_t oyo = 0) {
  const size_t o = (size_t)j * d.nx + i;
  const PlaneFaces<COH, R> faces{d, i, j, on, on + o, oxo + o + j, oyo + o};
  node_update_faces<MODE, LINEAR, CHAR, FIXED, COH>(d, src, sa, i, j, on, faces);
}

}  // namespace hw
