// Internal structures shared by the kernels and the C-ABI layer (not part of the public header).
#pragma once
#include <algorithm>
#include <cstddef>
#include <cuda_runtime.h>

#include "../../include/hwswe.h"

namespace hw {

enum { MODE_STAGE = 0, MODE_RHS = 1 };
enum { HW_STATUS_DEPTH = 1, HW_STATUS_NONFINITE = 2, HW_STATUS_TIMEOUT = 4, HW_STATUS_BOUNDS = 8 };

// Everything a 2D kernel needs, passed by value. R is the working precision (double for the scheme,
// float for the single-precision variant) of the planes and of the grid constants.
template <class R>
struct Dev2DT {
  int nx, ny, bc_x, bc_y;
  R dx, dy, inv_dx, inv_dy, g, eps_w, eps_lim;
  // assembly constants: 1/(2dx), 1/(2dy), 1/(24dx), 1/(24dy), 1/(12dx), 1/(12dy)
  R c_bx, c_by, c_gx, c_gy, c_mx, c_my;
  R half_g;            // g / 2
  R c_bgx, c_bgy;      // g / (2dx), g / (2dy) (double grids; set_spacing_products)
  R fx_eps13, fx_eps2;    // the weights' epsilon of the fixed-point sweeps: (160/781) g eps_w, (80/781) eps_w
  R fx_eps13l, fx_eps2l;  // and of the limiter: (12/13) g eps_lim, (3/13) eps_lim
  R* S[9];      // current state (eta, m, w, dx V, dy Q)
  R* stat[3];   // b, dx b_x, dy b_y
  R* bxy[2];    // b_x, b_y (physical, for conversions and static terms)
  R* X[12];     // x-interface values, pitch nx+1
  R* Y[12];     // y-interface values, pitch nx, ny+1 rows
  R* qbx[6];    // source candidates at x-interfaces ('+' q1..q3, '-' q1..q3)
  R* qby[6];
  R* sv[2];     // static derivative-source terms of the V equations (m, w components)
  R* sq[2];     // ... of the Q equations
};
using Dev2D = Dev2DT<double>;

// g and the weights' epsilons with the constants derived from them.
template <class D>
inline void set_physics(D& d, double g, double eps_w, double eps_lim) {
  using R = decltype(d.g);
  d.g = (R)g;
  d.eps_w = (R)eps_w;
  d.eps_lim = (R)eps_lim;
  d.half_g = (R)(0.5 * g);
  d.fx_eps13 = (R)((160.0 / 781.0) * eps_w * g);
  d.fx_eps2 = (R)((80.0 / 781.0) * eps_w);
  d.fx_eps13l = (R)((12.0 / 13.0) * eps_lim * g);
  d.fx_eps2l = (R)((3.0 / 13.0) * eps_lim);
}

// g c_b, rounded once from c_g = c_b / 12: the interface values carry c_g (fluxes) and this (bottom), whose quotient
// decides how well the two balance at rest.
template <class D>
inline void set_spacing_products(D& d, double g) {
  d.c_bgx = (double)(12.0L * (long double)g * (long double)d.c_gx);
  d.c_bgy = (double)(12.0L * (long double)g * (long double)d.c_gy);
}

template <class R>
struct StageArgsT {
  int k;             // RK stage 1..3
  int limiter;
  const R* dt;       // device scalar
  R* out[9];
  R* base[9];
  R* rhs_out[9];
  // with nsteps (stage 3): the step's end, *t = clock[1] (snapped) or *t + clock[0], counted if clock[0] > 0
  unsigned long long* nsteps;
  double* t;
  const double* clock;
  int snapped;
};
using StageArgs = StageArgsT<double>;

struct Ptr9 {
  double* p[9];
};

struct Ptr12 {
  void* p[12];  // planes of either precision
};

struct PhysIn {
  const double* p[12];  // h, hu, hv, b, h_x, hu_x, hv_x, h_y, hu_y, hv_y, b_x, b_y
};

// 1D
struct Dev1D {
  int nx, bc;
  double dx, inv_dx, g, eps_w, eps_lim;
  double c_b, c_g;   // 1/(2dx), 1/(24dx)
  double half_g, fx_eps13, fx_eps2, fx_eps13l, fx_eps2l;  // as in Dev2DT
  double* S[4];      // eta, m, dx H, dx M
  double* stat[2];   // b, dx b_x
  double* bx;        // b_x
  double* X[9];      // interface values: 2Fhat (2), 2bhat (2), 24dx Ghat (2), + 3 spare
  double* qb[6];
  double* sv;        // dx [B^]_x / dx (m component)
};

struct StageArgs1D {
  int k, limiter;
  const double* dt;
  double* out[4];
  double* base[4];
  double* rhs_out[4];
};

struct PhysIn1D {
  const double* p[6];  // h, hu, b, h_x, hu_x, b_x
};

// launchers (hw_kernels2d.cu)
int set_kernel_attributes2d();
// amax (double grids): kAlpha2dScratch device slots: the alpha_x and alpha_y keys, then scratch of the
// reduction (its float maxima, then one slot per tile); the first three are cleared here. The float
// variant's reduction uses the first three.
constexpr int kAlpha2dTiles = 152 * 8;
constexpr int kAlpha2dSlots = 3 + kAlpha2dTiles;      // then the slots of launch_alpha_finish2d (zero between launches)
constexpr int kAlpha2dScratch = kAlpha2dSlots + 4;
void launch_alpha2d(const Dev2D& d, unsigned long long* amax, int* status, cudaStream_t st);
// The reduction with its finish (the last block to end forms alpha; with_dt also the CFL step dt[0], clipped to end
// at t_end > 0, and the time after it dt[1], from the time *t_now): amax as above, zero before the first launch.
// fsc (single precision): receives alpha_x, alpha_y and dt rounded to float.
struct AlphaOut {
  double* alpha;
  double* dt;
  int with_dt;
  double cfl, inv_dx, inv_dy;
  const double* t_now;
  double t_end;
  float* fsc;
};
// Nodes up to which the double reduction is one launch. The two forms are within 0.5% of a step of each other from 131,072
// nodes on (10 steps, one launch / two: 3.41 / 3.43 ms at 131,044 nodes, 5.84 / 5.84 at 2^18, 6.08 / 6.06 at 266,240, 20.13 /
// 20.10 at 2^20); two keep the FP64 pipe out of the tiles that cannot hold the maximum.
constexpr size_t kAlphaOneMax = (size_t)1 << 18;
void launch_alpha_finish2d(const Dev2D& d, unsigned long long* amax, int* status, const AlphaOut& out, cudaStream_t st);
void launch_alpha_finish2d(const Dev2DT<float>& d, unsigned long long* amax, int* status, const AlphaOut& out,
                           cudaStream_t st);
// One block of a decomposed grid on this device: both state plane sets over its extended (nx + 4) x (ny + 4) nodes,
// its faces as in hw_part_info, and where its alpha, step and time live.
struct PartBlock {
  double* S[2][9];
  double* b;
  int nx, ny;
  int mode[4], nbr[4];
  double *alpha, *dt;
  const double* t;
  int* status;
};
// The start of a stage of all blocks (parts: np of them on the device, host: the same on the host), reading plane set
// cur: ring exchange, alpha, with_dt also the step as AlphaOut. slots: 4, zero before the first launch. d: any block's
// (spacings and g are common).
void launch_parts_begin(const PartBlock* parts, const PartBlock* host, int np, int cur, const Dev2D& d, unsigned oddx,
                        unsigned oddy, unsigned long long* slots, bool with_dt, double cfl, double t_end,
                        cudaStream_t st);
// both sweeps (one launch while the grid is small)
void launch_sweeps2d(const Dev2D& d, const double* alpha, bool linear, bool chr, cudaStream_t st);
void launch_finish_alpha2d(const Dev2D& d, const unsigned long long* amax, double* alpha, double* dt_out,
                           double cfl, const double* t_now, double t_end, cudaStream_t st);
void launch_sweep_x2d(const Dev2D& d, const double* alpha, bool linear, bool chr, cudaStream_t st);
void launch_sweep_y2d(const Dev2D& d, const double* alpha, bool linear, bool chr, cudaStream_t st);
void launch_node2d(const Dev2D& d, const StageArgs& sa, int mode, bool linear, bool chr, cudaStream_t st);
void launch_init2d(const Dev2D& d, const PhysIn& in, int* status, cudaStream_t st);
// the b-only source terms alone (launch_init2d runs them after the conversion)
void launch_static2d(const Dev2D& d, cudaStream_t st);
void launch_convert2d(const Dev2D& d, const Ptr9& src, const Ptr9& dst, int layout, int dir, cudaStream_t st);
// single-precision variant of the stage kernels, and plane casts between precisions
void launch_sweep_x2d(const Dev2DT<float>& d, const float* alpha, bool linear, bool chr, cudaStream_t st);
void launch_sweep_y2d(const Dev2DT<float>& d, const float* alpha, bool linear, bool chr, cudaStream_t st);
void launch_node2d(const Dev2DT<float>& d, const StageArgsT<float>& sa, int mode, bool linear, bool chr,
                   cudaStream_t st);
// a stage of the single-precision variant in one launch, nonlinear weights (hw_stage32.cu)
void launch_stage2d_f32(const Dev2DT<float>& d, const StageArgsT<float>& sa, const float* alpha, bool chr, cudaStream_t st);
void launch_cast_planes(int nplanes, size_t n, const Ptr12& src, const Ptr12& dst, int to_float, cudaStream_t st);

// One RK stage of the adjoint's forward pass (hw_forward64.cu): sweeps and node update in FP64.
void launch_stage_fp64(const Dev2D& d, const StageArgs& sa, const double* alpha, cudaStream_t st);
void solver_fp64_stages(hw_solver* s, bool on);  // this solver's stages (2D double, nonlinear, projected) take it

// record an error message for hw_last_error (hw_api.cu); returns code
int set_last_error(int code, const char* msg);

// launchers (hw_kernels1d.cu)
void launch_alpha1d(const Dev1D& d, unsigned long long* amax, int* status, cudaStream_t st);
void launch_finish_alpha1d(const Dev1D& d, const unsigned long long* amax, double* alpha, double* dt_out,
                           double cfl, const double* t_now, double t_end, cudaStream_t st);
// linear weights only (hw_step1d.cu has the scheme's own)
void launch_sweep1d(const Dev1D& d, const double* alpha, bool chr, cudaStream_t st);
void launch_node1d(const Dev1D& d, const StageArgs1D& sa, int mode, bool chr, cudaStream_t st);
// The scheme's 1D right-hand side, and one RK stage (hw_step1d.cu), each one launch with alpha on the device. With
// next the stage also forms the next stage's alpha and, after stage 3, the time and the next step's size.
struct Time1D {
  unsigned long long* slot;  // 4, zero before the first launch
  int* status;
  double* alpha;
  double* dt;  // step, time after it, time
  unsigned long long* nsteps;
  double cfl;
};
void launch_rhs1d(const Dev1D& d, const StageArgs1D& sa, const double* alpha, bool chr, cudaStream_t st);
// Up to nsteps whole steps of a small grid (run1d_fits) in one launch, from d.S back into d.S, with alpha and the
// first step's size on the device; ends early at t_end > 0. Returns the launch's cudaError_t.
bool run1d_fits(const Dev1D& d);
int launch_run1d(const Dev1D& d, double* const base[4], const Time1D& tm, int nsteps, int limiter, double t_end, bool chr,
                 cudaStream_t st);
void launch_stage1d(const Dev1D& d, const StageArgs1D& sa, const Time1D& tm, bool next, double t_end, bool chr,
                    cudaStream_t st);
void launch_init1d(const Dev1D& d, const PhysIn1D& in, int* status, cudaStream_t st);
void launch_convert1d(const Dev1D& d, const Ptr9& src, const Ptr9& dst, int layout, int dir, cudaStream_t st);



// Solver internals used by the adjoint (hw_adjoint.cu); defined in hw_api.cu.
struct SolverView {
  cudaStream_t stream;
  Dev2D* d2;            // null for 1D solvers
  double** state;       // current state planes (9)
  double* base[9];
  double* alpha;
  double* dt;
  const hw_params* params;
  size_t n;
};
int solver_view(hw_solver* s, SolverView* v);
// Sub-domain solvers (hw_dd.cu): the planes a halo exchange moves (set 0: the 9 state planes of the current
// state; set 1: those and the static planes b, dx b_x, dy b_y, b_x, b_y), the extended grid's Dev2D, and
// the stream the solver launches on (swapped for graph capture; returns the previous one).
int part_planes(hw_solver* s, int set, double** planes, int* nplanes);
const Dev2D* part_dev(hw_solver* s);
void part_block(hw_solver* s, PartBlock* b);
// stage k of an initialised block whose ring, alpha and step are in place (launch_parts_begin)
void part_stage(hw_solver* s, int k);
cudaStream_t solver_swap_stream(hw_solver* s, cudaStream_t st);
int solver_cur(hw_solver* s);                  // which of the two state buffers holds the state
cudaStream_t solver_stream(hw_solver* s);
const hw_part_info* part_info(hw_solver* s);   // null unless a block solver
// still water (h = 1, everything else 0) on the 2-node ring of 12 extended input planes (hw_dd.cu)
void launch_fill_ring(double* const* planes12, int nxe, int nye, cudaStream_t st);
// The blocks of a single-GPU block decomposition (hw_dd.cu), and its halo exchange on any set of
// nplanes planes per block (planes[p][q], extended grids; oddx / oddy: bit q set for planes that change
// sign across x- / y-walls), and the transpose of that exchange (for adjoints: the ring's values are
// added to the nodes they were copied from and the ring is cleared). Stream-ordered on st.
int dd_blocks(hw_dd* d, int* np, hw_solver* const** parts, const hw_part_info** info, cudaStream_t* st,
              const hw_grid** grid);
int dd_exchange_planes(hw_dd* d, double* const* const* planes, int nplanes, unsigned oddx, unsigned oddy,
                       cudaStream_t st);
int dd_exchange_adjoint(hw_dd* d, double* const* const* planes, int nplanes, unsigned oddx, unsigned oddy,
                        cudaStream_t st);
// every block's stream waits for st (fork); st waits for every block's stream (join)
int dd_fork_blocks(hw_dd* d, cudaStream_t st);
int dd_join_blocks(hw_dd* d, cudaStream_t st);
void adjoint_release(hw_solver* s);  // frees a solver's adjoint working buffers; hw_destroy calls it
// Frees what solvers that are in no call keep for their next adjoint call; whether there was any.
bool release_idle_memory();
// cudaMalloc, once more after release_idle_memory while memory is short.
cudaError_t device_alloc(void** p, size_t bytes);

}  // namespace hw
