// One RK stage of the 1D scheme (Zhao & Zhang, arXiv:2208.01260, Sec. 2) in one launch, and whole runs of steps of
// a small grid in one launch.
//
// A 1D grid of the paper's sizes occupies a fraction of the GPU, so a stage lasts as long as one warp's chain of
// instructions plus the launches. On GB300 a warp issues an FP64 instruction every 64 cycles, whatever its
// parallelism, an integer one every 2 to 7 (measured), so the chain is kept short by
//   * the reconstruction and the limiter in fixed point (hw_fixed.h),
//   * lanes: four per interface (field x side of Sec. 2.1 Step 1), two per node in the limiter (its two fields),
//     four per node in the update (one per state plane),
//   * warps side by side: the limiter needs the stage's input only and runs beside the reconstruction,
//   * everything of a block's nodes kept in shared memory between the phases; alpha's reduction over the stage's
//     output closes the launch (the last block to finish forms alpha, the time and the next step), so a stage is
//     one launch instead of three.
// Blocks own N = 31 or 63 nodes and compute the two interfaces on their ends themselves. Grids of at most 504 nodes
// run whole steps in one launch of one thread-block cluster (k_run1d), larger ones a launch per stage (k_stage1d).
// Measured (a job of 20 steps at N = 200, of 10 at N = 12801): 1.14 -> 0.41 ms and 0.90 -> 0.51 ms against three
// launches per stage on the FP64 pipe; one launch per stage takes 0.66 ms at N = 200. k_stage1d at N = 12801 holds
// three blocks per SM (96 registers), all 413 at once: 17 us per stage against 21 with two.
#include "hw_fixed.h"
#include "hw_stencil1d.cuh"

namespace hw {

namespace {

// Fixed-point record: F+, F-, G+, -G- of both components as integers of one unit per component (below 2^60),
// depth and momentum as doubles, the units' biased exponents.
enum { Q_X = NREC1, NREC1X = NREC1 + 1 };
constexpr int kExpMin = 256, kExpMax = 1900;

template <int N>
struct Smem {
  double S[2][4][N + 4];  // state planes of nodes a - 2 .. a + n + 1 (a run's stages alternate)
  double T[2][N + 4];     // b, dx b_x
  double qb[6][N + 1];    // source candidates of interfaces a .. a + n
  double sv[N];
  double base[4][N];      // a run's step base
  double dt[3];           // step, time after it, time
  double rec[NREC1X][N + 4];
  double st[7][N + 1]; // interface states (I_* below)
  double X[6][N + 1];  // interface values a .. a + n
  double mod[2][N];
  unsigned long long key[12];
  int bad[12];
};

template <int N>
constexpr int kThreads = 4 * (N + 1) + 2 * (N + 1);

// Record of one node (node_record1d with the split in fixed point).
__device__ __forceinline__ void record_fixed(const double v[6], double g, double alpha, double* rec, int stride) {
  const double eta = v[0], m = v[1], H = v[2], M = v[3], b = v[4], B = v[5];
  const double h = eta - b;
  const double u = m * fast_rcp(h);
  const double ge = g * eta, uu = u * u;
  const double F[2] = {m, fma(m, u, ge * fma(0.5, eta, -b))};
  const double Gs[2] = {M, fma(u + u, M, fma(g * h - uu, H, (uu - ge) * B))};
  int ua;
  const FxS al = fx_split(fx_mantissa(alpha, ua));
  const int ea = ua + 1084;
  bool bad = (unsigned)(ea - 600) > 600u;
  int em[2];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const double U = v[c], D = v[2 + c];
    const uint32_t wf = max(fx_absw(F[c]), fx_absw(Gs[c])), wu = max(fx_absw(U), fx_absw(D));
    em[c] = max((int)(wf >> 20) + 1, (int)(wu >> 20) + ea - 1020);
    const bool any = (fx_any(F[c]) | fx_any(Gs[c]) | fx_any(U) | fx_any(D)) != 0u;
    bad |= (max(wf, wu) >= (uint32_t)kExpMax << 20) | (em[c] > kExpMax) | ((em[c] < kExpMin) & any);
    em[c] = max(em[c], kExpMin);
    const int eu = em[c] - ea + 1020;
    const int64_t f = fx_from_double(F[c], em[c]), q = fx_from_double(Gs[c], em[c]);
    const int64_t pu = fx_mulhi(fx_split(fx_from_double(U, eu)), al, 0), pd = fx_mulhi(fx_split(fx_from_double(D, eu)), al, 0);
    rec[(Q_FP + c) * stride] = __longlong_as_double(f + pu);
    rec[(Q_FM + c) * stride] = __longlong_as_double(f - pu);
    rec[(Q_GP + c) * stride] = __longlong_as_double(q + pd);
    rec[(Q_GM + c) * stride] = __longlong_as_double(pd - q);
  }
  rec[Q_H * stride] = h;
  rec[Q_M * stride] = m;
  rec[Q_X * stride] = f64_from_words((uint32_t)(em[0] | (em[1] << 16)), bad ? 1u : 0u);
}

__device__ __forceinline__ int64_t shfl64(int64_t x, int m) { return __shfl_xor_sync(0xffffffffu, (long long)x, m); }

// State of an interface (Sec. 2.1: averages of the two nodes), formed once per interface beside the records: u,
// 1 / sqrt(g h), the coefficients -(u + c) and -(u - c) of component 0 as mantissas with their units, and epsilon.
enum { I_U = 0, I_RS = 1, I_CP = 2, I_CM = 3, I_UNITS = 4, I_EPS = 5, I_EPSU = 6 };
template <bool CHAR>
__device__ __forceinline__ void interface_state(const Dev1D& d, const double* S, const double* b, int stride, double* st,
                                                int xstride) {
  const double hs = (S[1] - b[1]) + (S[2] - b[2]);
  const double ub = (S[stride + 1] + S[stride + 2]) * fast_rcp(hs);
  const double gh = d.half_g * hs;
  const double rs = fast_rsqrt(gh);
  bool bad = false;
  const FxEps eps = fx_eps(CHAR ? d.fx_eps13 * hs : d.fx_eps2, bad);
  int up, um;
  const int64_t xp = fx_mantissa(-fma(gh, rs, ub), up), xm = fx_mantissa(-fma(-gh, rs, ub), um);
  st[I_U * xstride] = ub;
  st[I_RS * xstride] = rs;
  st[I_CP * xstride] = __longlong_as_double(xp);
  st[I_CM * xstride] = __longlong_as_double(xm);
  st[I_UNITS * xstride] = f64_from_words((uint32_t)up, (uint32_t)um);
  st[I_EPS * xstride] = __longlong_as_double((int64_t)eps.m);
  st[I_EPSU * xstride] = f64_from_words((uint32_t)eps.u, bad ? 1u : 0u);
}

// All six values of interface k from its nodes on the FP64 pipe (data that does not fit).
template <bool CHAR>
__device__ __noinline__ void interface_fp64(const Dev1D& d, double alpha, const double* S, const double* T, int stride,
                                            const double* qb_, int qstride, double out[6]) {
  double rec[4 * NREC1], qb[6];
#pragma unroll 1
  for (int s = 0; s < 4; ++s) {
    Node6 n;
    for (int q = 0; q < 6; ++q) n.v[q] = q < 4 ? S[q * stride + s] : T[(q - 4) * stride + s];
    node_record1d(n, d.g, alpha, rec + s * NREC1);
  }
  for (int q = 0; q < 6; ++q) qb[q] = qb_[q * qstride];
  interface_values1d<false, CHAR>(rec, rec + NREC1, rec + 2 * NREC1, rec + 3 * NREC1, 1, qb, d.g, d.eps_w, out);
}

// Interface k by four lanes of a warp: lane r takes field r >> 1 (without projection: component r >> 1) on side
// r & 1; the sides and fields meet by shuffles. r0: the first of its four records in shared memory; S: the first
// of its four nodes (T: static planes); ist: its state; qb: its source candidates. Lane r writes X components {0, 1},
// {2, 3}, {4}, {5} for r = 0 .. 3 unless live is false.
template <bool CHAR>
__device__ __forceinline__ void interface_lanes(const Dev1D& d, double alpha, const double* r0, const double* S, const double* T,
                                                int stride, const double* ist, const double* qb, int r, bool live,
                                                double* X, int xstride) {
  const int fld = r >> 1, side = r & 1;
  // per component: the four nodes' exponents, the unit, each node's shift
  bool bad = false;
  int e[2][4], m[2];
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    uint32_t lo, hi;
    f64_words(r0[Q_X * stride + s], lo, hi);
    e[0][s] = (int)(lo & 0xffffu);
    e[1][s] = (int)(lo >> 16);
    bad |= hi != 0u;
  }
#pragma unroll
  for (int c = 0; c < 2; ++c) m[c] = max(max(e[c][0], e[c][1]), max(e[c][2], e[c][3]));
  const double ub = ist[I_U * xstride], rs = ist[I_RS * xstride];
  FxEps eps;
  {
    uint32_t lo, hi;
    f64_words(ist[I_EPSU * xstride], lo, hi);
    eps.m = (uint64_t)__double_as_longlong(ist[I_EPS * xstride]);
    eps.u = (int)lo;
    bad |= hi != 0u;
  }
  // this side's source candidates, below 2^60 (one unit for both sides)
  double qv[6];
  uint32_t bw = 0;
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    qv[q] = qb[q * xstride];
    bw = max(bw, fx_absw(qv[q]));
  }
  const int eb = max((int)(bw >> 20), kExpMin);
  bad |= eb > kExpMax;
  const int64_t c3 = fx_from_double(side ? qv[5] : qv[2], eb);
  const FxS d1 = fx_split(fx_from_double(side ? qv[3] : qv[0], eb) - c3), d2 = fx_split(fx_from_double(side ? qv[4] : qv[1], eb) - c3);
  // the fields' unit and this field's coefficient -(u +- c) of component 0
  int U = 0;
  FxS ck = {0, 0};
  if (CHAR) {
    uint32_t lo, hi;
    f64_words(ist[I_UNITS * xstride], lo, hi);
    const int up = (int)lo, um = (int)hi;
    const int64_t xp = __double_as_longlong(ist[I_CP * xstride]), xm = __double_as_longlong(ist[I_CM * xstride]);
    const int u0 = m[0] - 1082 + 64;
    U = max(max(max(up, um) + u0 + 2, m[1] - 1078), -900);
    bad |= U > 900;
    const int64_t x = fld == 0 ? xp : xm;
    ck = fx_split(x >> min(U - (fld == 0 ? up : um) - u0, 63));
  }
  // '+': nodes 0, 1, 2 of (F+, G+); '-': nodes 3, 2, 1 of (F-, -G-)
  const double* const q = side == 0 ? r0 : r0 + Q_FM * stride + 3;
  const int step = side == 0 ? 1 : -1;
  auto load = [&](int t, int f, int c, int b) {
    const int es = side == 0 ? e[c][t] : e[c][3 - t];
    return (int64_t)__double_as_longlong(q[t * step + f * stride]) >> min(b - es, 63);
  };
  int64_t f0[3], p0[3], f1[3], p1[3];
#pragma unroll
  for (int t = 0; t < 3; ++t) {
    f0[t] = load(t, 0, 0, CHAR ? m[0] : m[0] + 4);
    p0[t] = load(t, Q_GP, 0, CHAR ? m[0] : m[0] + 4);
    f1[t] = load(t, 1, 1, CHAR ? U + 1082 : m[1] + 4);
    p1[t] = load(t, Q_GP + 1, 1, CHAR ? U + 1082 : m[1] + 4);
  }
  int64_t f[3], p[3], qf[3], qp[3];  // this lane's field, and the component whose derivative flux it forms
#pragma unroll
  for (int t = 0; t < 3; ++t) {
    qf[t] = fld == 0 ? (CHAR ? f0[t] >> 4 : f0[t]) : f1[t];
    qp[t] = fld == 0 ? (CHAR ? p0[t] >> 4 : p0[t]) : p1[t];
    f[t] = CHAR ? fx_mulhi(fx_split(f0[t]), ck, f1[t]) : qf[t];
    p[t] = CHAR ? fx_mulhi(fx_split(p0[t]), ck, p1[t]) : qp[t];
  }
  const int64_t quint = 3 * ((qf[0] - qf[1]) - 7 * (qf[1] - qf[2])) + (qp[0] - 2 * qp[1] - 5 * qp[2]);
  const int uf = CHAR ? U : m[fld] - 1078;
  int64_t w1, w2;
  const int64_t v = fx_hweno_side(f[0], f[1], f[2], p[0], p[1], p[2], eps, uf, w1, w2);
  const int64_t b = c3 + fx_dot2<3>(d1, fx_split(w1), d2, fx_split(w2));
  // sum over the sides, exchange with the other field
  const int64_t Gk = v + shfl64(v, 1), Bk = b + shfl64(b, 1), qo = shfl64(quint, 1);
  const int64_t Gx = shfl64(Gk, 2), Bx = shfl64(Bk, 2), qs = side == 0 ? quint - qo : qo - quint, qx = shfl64(qs, 2);
  const int ub_ = eb - 1082, uq0 = m[0] - 1078, uq1 = CHAR ? U : m[1] - 1078;
  double o0, o1 = 0.0;
  if (CHAR) {
    // lane 0: (G_2 - G_1, G_2 + G_1) / 6; lane 1: the same of the source; lanes 2, 3: derivative fluxes
    const int64_t A0 = fld == 0 ? Gk : Gx, A1 = fld == 0 ? Gx : Gk, B0 = fld == 0 ? Bk : Bx, B1 = fld == 0 ? Bx : Bk;
    const int64_t P = r == 0 ? A1 - A0 : r == 1 ? B1 - B0 : r == 2 ? qx : qs;
    const int64_t M = r == 0 ? A1 + A0 : B1 + B0;
    const int u = r == 0 ? U : r == 1 ? ub_ : r == 2 ? uq0 : uq1;
    const double sc = r == 0 ? 1.0 / 12.0 : 0.5;
    const double z = fx_to_double(P, u);
    o0 = r < 2 ? z * (sc * rs) : z;
    o1 = fma(ub, o0, sc * fx_to_double(M, r == 0 ? U : ub_));
  } else {
    const int64_t P = r == 0 ? Gk : r == 1 ? 0 : r == 2 ? qx : qs;
    const int64_t M = r == 0 ? Gx : Bx;
    const double z = fx_to_double(P, r == 0 ? m[0] - 1078 : r == 2 ? uq0 : uq1);
    o0 = r == 0 ? (1.0 / 6.0) * z : z;
    const double y = fx_to_double(M, r == 0 ? m[1] - 1078 : ub_);
    o1 = r == 0 ? (1.0 / 6.0) * y : y;
  }
  if (!live) return;
  if (bad) {
    if (r == 0) {
      double out[6];
      interface_fp64<CHAR>(d, alpha, S, T, stride, qb, xstride, out);
      for (int c = 0; c < 6; ++c) X[c * xstride] = out[c];
    }
    return;
  }
  if (r < 2) {
    X[2 * r * xstride] = o0;
    X[(2 * r + 1) * xstride] = o1;
  } else {
    X[(2 + r) * xstride] = o0;
  }
}

// Limited derivatives of a node on the FP64 pipe (data that does not fit). S: the node before it; b: its depth plane.
template <bool CHAR>
__device__ __noinline__ void limit_fp64(const Dev1D& d, const double* S, const double* b, int stride, double mod[2]) {
  const double *E = S, *M = S + stride, *H = S + 2 * stride, *D = S + 3 * stride;
  if (!CHAR) {
    mod[0] = limiter_field<false>(E[0], E[1], E[2], H[0], H[2], d.eps_lim);
    mod[1] = limiter_field<false>(M[0], M[1], M[2], D[0], D[2], d.eps_lim);
    return;
  }
  const double h = E[1] - b[1], gh = d.g * h;
  const double u = M[1] * fast_rcp(h);
  const double rs = fast_rsqrt(gh);
  const double c = gh * rs, ic2 = 0.5 * rs, upc = u + c, umc = u - c, e = (4.0 * d.eps_lim) * gh;
  const double a = limiter_field<false>(fma(upc, E[0], -M[0]), fma(upc, E[1], -M[1]), fma(upc, E[2], -M[2]),
                                        fma(upc, H[0], -D[0]), fma(upc, H[2], -D[2]), e);
  const double f = limiter_field<false>(fma(-umc, E[0], M[0]), fma(-umc, E[1], M[1]), fma(-umc, E[2], M[2]),
                                        fma(-umc, H[0], D[0]), fma(-umc, H[2], D[2]), e);
  const double A = (a + f) * ic2;
  mod[0] = A;
  mod[1] = fma(u, A, 0.5 * (f - a));
}

// The limiter of a node by two lanes, one per field (component): lane r returns limited component r. S, b: the
// node before it in shared memory. Every lane of the warp must call.
template <bool CHAR>
__device__ __forceinline__ double limit_lanes(const Dev1D& d, const double* S, const double* b, int stride, int r) {
  const double *E = S, *M = S + stride, *H = S + 2 * stride, *D = S + 3 * stride;
  const double v[2][5] = {{E[0], E[1], E[2], H[0], H[2]}, {M[0], M[1], M[2], D[0], D[2]}};
  bool bad = false;
  int em[2];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    uint32_t w = 0, any = 0;
#pragma unroll
    for (int s = 0; s < 5; ++s) {
      w = max(w, fx_absw(v[c][s]));
      any |= fx_any(v[c][s]);
    }
    em[c] = (int)(w >> 20);
    bad |= (em[c] > kExpMax) | ((em[c] < kExpMin) & (any != 0u));
    em[c] = max(em[c], kExpMin);
  }
  const double h = E[1] - b[1], gh = d.g * h;
  const FxEps eps = fx_eps(CHAR ? d.fx_eps13l * h : d.fx_eps2l, bad);
  int64_t a[2][4];  // differences to the neighbours and their derivatives, below 2^61
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const int64_t m = fx_from_double(v[c][1], em[c]);
    a[c][0] = m - fx_from_double(v[c][0], em[c]);
    a[c][1] = fx_from_double(v[c][2], em[c]) - m;
    a[c][2] = fx_from_double(v[c][3], em[c]);
    a[c][3] = fx_from_double(v[c][4], em[c]);
  }
  double o;
  if (CHAR) {
    const double u = M[1] * fast_rcp(h);
    const double rs = fast_rsqrt(gh);
    int up, um;
    const int64_t xp = fx_mantissa(-fma(gh, rs, u), up), xm = fx_mantissa(-fma(-gh, rs, u), um);
    const int u0 = em[0] - 1082 + 64;
    const int U = max(max(max(up, um) + u0 + 2, em[1] - 1078), -900);
    bad |= U > 900;
    const FxS k = fx_split((r == 0 ? xp : xm) >> min(U - (r == 0 ? up : um) - u0, 63));
    const int sn = min(U + 1082 - em[1], 63);
    int64_t f[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) f[s] = fx_mulhi(fx_split(a[0][s]), k, a[1][s] >> sn);
    const int64_t nu = fx_limiter_field(f[0], f[1], f[2], f[3], eps, U);
    const int64_t nx = shfl64(nu, 1), n0 = r == 0 ? nu : nx, n1 = r == 0 ? nx : nu;
    const double A = fx_to_double(n1 - n0, U - 1) * (0.5 * rs);
    o = r == 0 ? A : fma(u, A, fx_to_double(n1 + n0, U - 2));
  } else {
    const int64_t x0 = r == 0 ? a[0][0] : a[1][0], x1 = r == 0 ? a[0][1] : a[1][1], x2 = r == 0 ? a[0][2] : a[1][2],
                  x3 = r == 0 ? a[0][3] : a[1][3];
    const int e = r == 0 ? em[0] : em[1];
    o = fx_to_double(fx_limiter_field(x0 >> 3, x1 >> 3, x2 >> 3, x3 >> 3, eps, e - 1079), e - 1080);
  }
  if (bad) {
    double mod[2];
    limit_fp64<CHAR>(d, S, b, stride, mod);
    o = r == 0 ? mod[0] : mod[1];
  }
  return o;
}

// alpha of a node from eta, m and b as an ordered key (0 and a status flag if the depth or the speed is not a
// positive finite number).
__device__ __forceinline__ unsigned long long alpha_key(double g, double eta, double m, double b, int& bad) {
  const double h = eta - b;
  if (!(h > 0.0) || !(h < 1e300)) {
    bad |= h == h ? HW_STATUS_DEPTH : HW_STATUS_NONFINITE;
    return 0;
  }
  const double gh = g * h;
  const double s = dabs(m * fast_rcp(h)) + gh * fast_rsqrt(gh);
  if (!(s < 1e300)) {
    bad |= HW_STATUS_NONFINITE;
    return 0;
  }
  return dkey(s);
}

// Static planes and source terms of nodes [a, a + n) into shared memory.
template <int N>
__device__ __forceinline__ void load_static(const Dev1D& d, int a, int n, Smem<N>& sm) {
  for (int l = threadIdx.x; l < 2 * (n + 4); l += kThreads<N>) {
    const int q = l >= n + 4, i = l - q * (n + 4);
    bool fl;
    const int ii = map_index(a - 2 + i, d.nx, d.bc, fl);
    const double x = __ldg((q ? d.stat[1] : d.stat[0]) + ii);
    sm.T[q][i] = fl && q ? -x : x;
  }
  for (int l = threadIdx.x; l < n + 1; l += kThreads<N>) {
#pragma unroll
    for (int q = 0; q < 6; ++q) sm.qb[q][l] = __ldg(d.qb[q] + a + l);
    if (l < n) sm.sv[l] = __ldg(d.sv + a + l);
  }
}

// State planes of nodes a - 2 .. a + n + 1 (boundary-mapped) into buffer p.
template <int N>
__device__ __forceinline__ void load_state(const Dev1D& d, int a, int n, int p, Smem<N>& sm) {
  for (int l = threadIdx.x; l < 4 * (n + 4); l += kThreads<N>) {
    const int q = l / (n + 4), i = l - q * (n + 4);
    bool fl;
    const int ii = map_index(a - 2 + i, d.nx, d.bc, fl);
    const double x = (q == 0 ? d.S[0] : q == 1 ? d.S[1] : q == 2 ? d.S[2] : d.S[3])[ii];
    sm.S[p][q][i] = fl && (q == 1 || q == 2) ? -x : x;  // par_1d
  }
}

// One stage k of nodes [a, a + n) from buffer p (all of a - 2 .. a + n + 1, the static planes and sm.dt loaded).
// put(q, j, value) takes component q of the stage's output (or of the right-hand side, MODE_RHS) at node a + j;
// base(q, j, value, store) stores or returns the step's base. All threads call.
template <int MODE, bool CHAR, int N, class Put, class Base>
__device__ __forceinline__ void stage_block(const Dev1D& d, int k, int limiter, double alpha, int n, int p, Smem<N>& sm,
                                            Put&& put, Base&& base) {
  constexpr int W = N + 4, TI = 4 * (N + 1);
  const int t = threadIdx.x;
  double(*const S)[W] = sm.S[p];
  if (t < TI) {
    if (t < n + 4) {
      const double v[6] = {S[0][t], S[1][t], S[2][t], S[3][t], sm.T[0][t], sm.T[1][t]};
      record_fixed(v, d.g, alpha, &sm.rec[0][t], W);
    } else if (t >= TI / 2 && t - TI / 2 <= n) {  // other warps than the records'
      const int j = t - TI / 2;
      interface_state<CHAR>(d, &S[0][j], &sm.T[0][j], W, &sm.st[0][j], N + 1);
    }
    asm volatile("bar.sync 1, %0;" ::"n"(TI) : "memory");  // the reconstruction's warps only
    const int j = t >> 2;
    const bool live = j <= n;
    const int jj = live ? j : 0;  // past the last interface: the first again, not written
    interface_lanes<CHAR>(d, alpha, &sm.rec[0][jj], &S[0][jj], &sm.T[0][jj], W, &sm.st[0][jj], &sm.qb[0][jj], t & 3, live,
                          &sm.X[0][jj], N + 1);
  } else if (MODE == MODE_STAGE && limiter) {
    const int l = t - TI, j = l >> 1;
    const int jj = min(j, n - 1);
    const double o = limit_lanes<CHAR>(d, &S[0][jj + 1], &sm.T[0][jj + 1], W, l & 1);
    if (j < n) sm.mod[l & 1][j] = o;
  }
  __syncthreads();
  // node update: lane q of node j forms state plane q (eq. swe-form-1d-semi, eq. RK)
  if (t < 4 * n) {
    const int j = t >> 2, q = t & 3, c = q & 1;
    const double cur = S[q][j + 2], ge = d.g * S[0][j + 2];
    const double db = d.c_b * (sm.X[2 + c][j + 1] - sm.X[2 + c][j]);
    const int xp = q < 2 ? c : 4 + c;
    const double dd = sm.X[xp][j + 1] - sm.X[xp][j];
    double R = fma(q < 2 ? -ge : -d.g * S[2][j + 2], db, -(q < 2 ? d.c_b : d.c_g) * dd);
    if (q == 3) R = fma(-ge, sm.sv[j], R);
    if (MODE == MODE_RHS) {
      put(q, j, q < 2 ? R : R * d.inv_dx);
    } else {
      const double dt = sm.dt[0];
      double res = cur;
      if (dt > 0.0) {  // a step of size 0 leaves the state unchanged
        const double cq = q < 2 || !limiter ? cur : sm.mod[c][j];
        res = fma(dt, R, cq);
        if (k == 1) {
          base(q, j, cq, true);
        } else {
          const double wa = k == 2 ? 0.75 : 1.0 / 3.0, wb = k == 2 ? 0.25 : 2.0 / 3.0;
          res = fma(wa, base(q, j, 0.0, false), wb * res);
        }
      }
      put(q, j, res);
    }
  }
}

// The block's maximum key and status flags, in thread 0 (all threads call).
template <int N>
__device__ __forceinline__ void block_key(Smem<N>& sm, unsigned long long& key, int& bad) {
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) {
    key = max(key, __shfl_xor_sync(0xffffffffu, key, s));
    bad |= __shfl_xor_sync(0xffffffffu, bad, s);
  }
  if ((threadIdx.x & 31) == 0) {
    sm.key[threadIdx.x >> 5] = key;
    sm.bad[threadIdx.x >> 5] = bad;
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int w = 1; w < kThreads<N> / 32; ++w) {
      key = max(key, sm.key[w]);
      bad |= sm.bad[w];
    }
}

// One stage per launch. slot[0], slot[1]: key and arrival count of the output's alpha (both zero between launches);
// slot[2]: the status flags of the output, which count once a stage uses it; slot[3] collects them. With next, the
// last block forms the next stage's alpha and, after stage 3, the time and the next step's size.
struct Step1D {
  unsigned long long* slot;
  int* status;
  double* alpha;
  double* dt;  // dt[0] step, dt[1] time after it, dt[2] time
  unsigned long long* nsteps;
  double cfl, t_end;
  int next;
};

template <int MODE, bool CHAR, int N>
__global__ void __launch_bounds__(kThreads<N>, 3) k_stage1d(Dev1D d, StageArgs1D sa, Step1D st) {
  __shared__ Smem<N> sm;
  const int a = blockIdx.x * N, n = min(N, d.nx - a);
  load_static(d, a, n, sm);
  load_state(d, a, n, 0, sm);
  const double alpha = st.alpha[0];
  if (MODE == MODE_STAGE && threadIdx.x == 0) {
    sm.dt[0] = *sa.dt;
    // flags of this stage's input, found by the launch that wrote it
    if (blockIdx.x == 0 && st.slot[2]) atomicOr(st.status, (int)st.slot[2]);
  }
  __syncthreads();
  auto put = [&](int q, int j, double x) {
    if (MODE == MODE_RHS) {
      (q == 0 ? sa.rhs_out[0] : q == 1 ? sa.rhs_out[1] : q == 2 ? sa.rhs_out[2] : sa.rhs_out[3])[a + j] = x;
    } else {
      (q == 0 ? sa.out[0] : q == 1 ? sa.out[1] : q == 2 ? sa.out[2] : sa.out[3])[a + j] = x;
      if (q < 2) sm.S[1][q][j + 2] = x;
    }
  };
  auto base = [&](int q, int j, double x, bool store) {
    double* const p = (q == 0 ? sa.base[0] : q == 1 ? sa.base[1] : q == 2 ? sa.base[2] : sa.base[3]) + a + j;
    if (!store) return *p;
    *p = x;
    return x;
  };
  stage_block<MODE, CHAR, N>(d, sa.k, sa.limiter, alpha, n, 0, sm, put, base);
  if (MODE == MODE_RHS || !st.next) return;
  __syncthreads();
  int bad = 0;
  unsigned long long key = 0;
  if (threadIdx.x < n) key = alpha_key(d.g, sm.S[1][0][threadIdx.x + 2], sm.S[1][1][threadIdx.x + 2], sm.T[0][threadIdx.x + 2], bad);
  block_key(sm, key, bad);
  if (threadIdx.x != 0) return;
  // one thread per block: the block's maximum and flags, a fence, then the arrival count, so the last block to
  // arrive finds every block's; every block has read alpha, dt and slot[2] by then
  atomicMax(st.slot, key);
  if (bad) atomicOr(reinterpret_cast<unsigned int*>(st.slot + 3), (unsigned)bad);
  __threadfence();
  if (atomicAdd(st.slot + 1, 1ull) != (unsigned long long)gridDim.x - 1) return;
  __threadfence();
  if (sa.k == 3) {
    st.dt[2] = st.dt[1];
    if (sm.dt[0] > 0.0) ++*st.nsteps;
  }
  finish_alpha1d(atomicMax(st.slot, 0ull), st.alpha, sa.k == 3 ? st.dt : nullptr, st.cfl, d.dx, st.dt + 2, st.t_end);
  st.slot[2] = atomicExch(st.slot + 3, 0ull);
  st.slot[0] = 0;
  st.slot[1] = 0;
}

// Whole steps of a small grid in one launch: the grid's blocks form one thread-block cluster, which holds the state
// in shared memory from stage to stage. After a stage every block has its own nodes' new values; the cluster's
// barrier then publishes them and the blocks' alpha maxima, and each block fetches its four ghost nodes from the
// blocks that own them. Buffers alternate with the stages: a block overwrites what others read in one stage
// only after the barrier that ends the next.
constexpr int kCluster = 8;

__device__ __forceinline__ uint32_t smem_of_rank(const void* p, uint32_t rank) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ double ld_cluster(uint32_t a) {
  double x;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(x) : "r"(a) : "memory");
  return x;
}
__device__ __forceinline__ void st_cluster(uint32_t a, unsigned long long x) {
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(a), "l"(x) : "memory");
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

struct Run1D {
  double* base[4];
  Time1D tm;
  double t_end;
  int nsteps, limiter;
};

template <bool CHAR, int N>
__global__ void __launch_bounds__(kThreads<N>) k_run1d(Dev1D d, Run1D r) {
  __shared__ Smem<N> sm;
  __shared__ unsigned long long peer[2][2][kCluster];  // [parity][key, flags][block]
  const int t = threadIdx.x, rank = blockIdx.x, C = gridDim.x;  // one cluster
  const int a = rank * N, n = min(N, d.nx - a);
  load_static(d, a, n, sm);
  load_state(d, a, n, 0, sm);
  double alpha = r.tm.alpha[0];
  if (t < 3) sm.dt[t] = r.tm.dt[t];
  unsigned long long steps = 0;
  // flags of the state that the next stage reads, from the launch before (slot[2], as k_stage1d's) and to the next one
  int p = 0, pending = (int)r.tm.slot[2], used = 0;
  cluster_barrier();  // every block runs; shared memory and slot[2] read
  for (int step = 0; step < r.nsteps; ++step) {
    if (r.t_end > 0.0 && sm.dt[2] >= r.t_end) break;  // the same in every block
    for (int k = 1; k <= 3; ++k) {
      used |= pending;
      auto put = [&](int q, int j, double x) { sm.S[p ^ 1][q][j + 2] = x; };
      auto base = [&](int q, int j, double x, bool store) {
        if (store) sm.base[q][j] = x;
        return sm.base[q][j];
      };
      stage_block<MODE_STAGE, CHAR, N>(d, k, r.limiter, alpha, n, p, sm, put, base);
      __syncthreads();
      int bad = 0;
      unsigned long long key = 0;
      if (t < n) key = alpha_key(d.g, sm.S[p ^ 1][0][t + 2], sm.S[p ^ 1][1][t + 2], sm.T[0][t + 2], bad);
      block_key(sm, key, bad);
      if (t == 0) {
        for (int b = 0; b < C; ++b) {
          st_cluster(smem_of_rank(&peer[p][0][rank], b), key);
          st_cluster(smem_of_rank(&peer[p][1][rank], b), (unsigned long long)bad);
        }
      }
      cluster_barrier();
      unsigned long long m = 0;
      pending = 0;
      for (int b = 0; b < C; ++b) {
        m = max(m, peer[p][0][b]);
        pending |= (int)peer[p][1][b];
      }
      alpha = __longlong_as_double((long long)m);
      if (t < 16) {  // ghost nodes
        const int q = t >> 2, g = t & 3, i = g < 2 ? g : n + g;
        bool fl;
        const int ii = map_index(a - 2 + i, d.nx, d.bc, fl);
        const double x = ld_cluster(smem_of_rank(&sm.S[p ^ 1][q][ii % N + 2], ii / N));
        sm.S[p ^ 1][q][i] = fl && (q == 1 || q == 2) ? -x : x;
      } else if (k == 3 && t == 32) {  // the time, and the next step
        if (sm.dt[0] > 0.0) ++steps;
        double al[2], dt[2];
        const double now = sm.dt[1];
        finish_alpha1d(m, al, dt, r.tm.cfl, d.dx, &now, r.t_end);
        sm.dt[0] = dt[0];
        sm.dt[1] = dt[1];
        sm.dt[2] = now;
      }
      p ^= 1;
      __syncthreads();
    }
  }
  for (int l = t; l < 4 * n; l += kThreads<N>) {
    const int q = l / n, j = l - q * n;
    (q == 0 ? d.S[0] : q == 1 ? d.S[1] : q == 2 ? d.S[2] : d.S[3])[a + j] = sm.S[p][q][j + 2];
    (q == 0 ? r.base[0] : q == 1 ? r.base[1] : q == 2 ? r.base[2] : r.base[3])[a + j] = sm.base[q][j];
  }
  if (rank == 0) {
    if (t < 3) r.tm.dt[t] = sm.dt[t];
    if (t == 0) {
      r.tm.alpha[0] = alpha;
      r.tm.slot[2] = (unsigned long long)pending;
      if (used) atomicOr(r.tm.status, used);
    }
    if (t == 32) *r.tm.nsteps += steps;
  }
  cluster_barrier();  // no block leaves while another may read its shared memory
}

}  // namespace

template <int MODE, bool CHAR>
static void launch(const Dev1D& d, const StageArgs1D& sa, const Step1D& st, cudaStream_t stream) {
  constexpr int N = 31;
  k_stage1d<MODE, CHAR, N><<<(d.nx + N - 1) / N, kThreads<N>, 0, stream>>>(d, sa, st);
}

template <bool CHAR, int N>
static cudaError_t launch_run(const Dev1D& d, const Run1D& r, cudaStream_t stream) {
  cudaLaunchConfig_t cfg{};
  const unsigned blocks = (unsigned)((d.nx + N - 1) / N);
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(kThreads<N>);
  cfg.stream = stream;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = blocks;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_run1d<CHAR, N>, d, r);
}

bool run1d_fits(const Dev1D& d) { return d.nx <= kCluster * 63; }

int launch_run1d(const Dev1D& d, double* const base[4], const Time1D& tm, int nsteps, int limiter, double t_end, bool chr,
                 cudaStream_t stream) {
  Run1D r{};
  for (int q = 0; q < 4; ++q) r.base[q] = base[q];
  r.tm = tm;
  r.t_end = t_end;
  r.nsteps = nsteps;
  r.limiter = limiter;
  if (d.nx <= kCluster * 31) return (int)(chr ? launch_run<true, 31>(d, r, stream) : launch_run<false, 31>(d, r, stream));
  return (int)(chr ? launch_run<true, 63>(d, r, stream) : launch_run<false, 63>(d, r, stream));
}

void launch_rhs1d(const Dev1D& d, const StageArgs1D& sa, const double* alpha, bool chr, cudaStream_t stream) {
  Step1D st{};
  st.alpha = const_cast<double*>(alpha);  // read only
  if (chr) launch<MODE_RHS, true>(d, sa, st, stream);
  else launch<MODE_RHS, false>(d, sa, st, stream);
}

void launch_stage1d(const Dev1D& d, const StageArgs1D& sa, const Time1D& tm, bool next, double t_end, bool chr,
                    cudaStream_t stream) {
  Step1D st{tm.slot, tm.status, tm.alpha, tm.dt, tm.nsteps, tm.cfl, t_end, next ? 1 : 0};
  if (chr) launch<MODE_STAGE, true>(d, sa, st, stream);
  else launch<MODE_STAGE, false>(d, sa, st, stream);
}

}  // namespace hw
