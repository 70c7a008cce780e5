// 2D kernels of the well-balanced fifth-order FD HWENO scheme (Zhao & Zhang, arXiv:2208.01260,
// Sec. 3) for sm_103a. One RK stage is four launches on the solver's stream (three on grids whose sweeps share one, two
// in single precision, hw_stage32.cu; the adjoint's forward pass has its own, hw_forward64.cu):
//   k_alpha2d_* global Lax-Friedrichs constants alpha_x = max(|u|+c), alpha_y = max(|v|+c)
//   k_sweep_x   x-interfaces: Sec. 2.1 Steps 1-2 along x for (F1, Phi1, tilde-b, tilde-B1) and the
//               mixed term Psi1 of eq. (mixed)
//   k_sweep_y   y-interfaces: Steps 1-2 along y for (F2, Psi2, bar-b, bar-B2) and the mixed Phi2
//   k_node2d    eq. (swe-form-2d-dis) (source signs read as '-'), the HWENO limiter of Sec. 2.2
//               applied dimension by dimension, and the SSP-RK3 combination of eq. (RK)
// Interface values go through global memory: the FP64 pipe, not memory, bounds this scheme on
// GB300, so each interface is computed exactly once. Every kernel is instantiated for double and for
// the single-precision variant (float planes and constants).
#include "hw_stencil2d.cuh"

namespace hw {

// ---------------------------------------------------------------------------------------------
// Sweeps: one tile of TILE_T threads per block over the flattened extended lines (hw_stencil2d.cuh),
// TILE_T - 3 x-interfaces, or YS_C (TILE_T / YS_C - 3) y-interfaces, per block.
// ---------------------------------------------------------------------------------------------
constexpr int YS_C = 2;  // columns per y-tile group of the double y-sweep (measured: 2 beats 1 and 4)

// The double kernels run the nonlinear reconstruction and the limiter in fixed point (hw_fixed.h): on the FP64
// pipe alone these kernels took 2.80 (x), 2.85 (y) and 2.03 ms (node) per stage at 2048^2, its operations at the
// pipe's rate; now 0.80, 0.85 and 0.91 ms. What bounds the sweeps is the sum of what is left on the FP64 pipe (69
// operations per x-interface, 58% busy) and integer work (4110 instructions per warp, 54% of the issue slots, the integer
// pipe 60% busy); the node kernel the FP64 pipe (100 operations, 73-79% busy) with the latency of its loads.
template <class R>
constexpr bool kFixed = std::is_same<R, double>::value;
template <class R>
constexpr int kTileRec = std::is_same<R, double>::value ? NRECX : NREC;
// Threads per x-tile and blocks per SM the kernels are compiled for. The register file holds 3, 4, 5 or 6 warps per
// SM partition at 168, 128, 96 or 80 registers: measured at 2048^2, x-sweep 0.79 / 0.77 ms at 4 / 5 (tiles of 192
// threads 0.79, of 96 0.84), y-sweep 0.83 / 0.85, node kernel 1.16 / 1.15 / 1.04 ms at 4 / 5 / 6.
template <class R>
constexpr int kXT = std::is_same<R, double>::value ? TILE_T : 192;
constexpr int kXsBlocks = 5, kYsBlocks = 4;
constexpr int kNodeT = 256;
template <class R>
constexpr int kNodeBlocks = std::is_same<R, double>::value ? 3 : 5;

template <bool LINEAR, bool CHAR, class R>
__global__ void __launch_bounds__(kXT<R>, kXsBlocks) k_sweep_x(const __grid_constant__ Dev2DT<R> d, const R* __restrict__ alpha) {
  __shared__ R sm[kTileRec<R> * kXT<R>];
  sweep_x_tile<LINEAR, CHAR, kFixed<R>, false, kXT<R>>(d, GridSource<R>{&d}, alpha[0], blockIdx.x * (kXT<R> - 3), sm);
}

template <bool LINEAR, bool CHAR>
__global__ void __launch_bounds__(TILE_T, kYsBlocks) k_sweep_y(const __grid_constant__ Dev2D d, const double* __restrict__ alpha) {
  __shared__ double sm[NRECX * TILE_T];
  sweep_y_tile<LINEAR, CHAR, true>(d, GridSource<double>{&d}, alpha[1], blockIdx.x * (TILE_T / YS_C - 3), YS_C, sm);
}

// Both sweeps in one launch, for grids whose tiles fill the GPU a few times at most: a sweep of few tiles lasts as
// long as one tile's chain, and each sweep's last wave runs partly empty.
template <bool CHAR>
__global__ void __launch_bounds__(TILE_T, kYsBlocks) k_sweep_xy(const __grid_constant__ Dev2D d, const double* __restrict__ alpha, int nxt) {
  __shared__ double sm[NRECX * TILE_T];
  if ((int)blockIdx.x < nxt) sweep_x_tile<false, CHAR, true>(d, GridSource<double>{&d}, alpha[0], blockIdx.x * (TILE_T - 3), sm);
  else sweep_y_tile<false, CHAR, true>(d, GridSource<double>{&d}, alpha[1], (blockIdx.x - nxt) * (TILE_T / YS_C - 3), YS_C, sm);
}

// Small grids, where a stage is as long as one warp's chain: both sweeps with two lanes per interface, and the node update
// split over three pairs of warps, below; the values are those of the other forms bit for bit. 10 steps at 64x66 0.95 ->
// 0.75 ms, at 100x90 0.97 -> 0.84, at 128^2 1.06 -> 0.97, at 170^2 1.36 -> 1.30.
constexpr int SP_R = TILE_T / 2;  // records per tile

template <int DIR, bool CHAR>
__device__ __forceinline__ void sweep_pair(const Dev2D& d, const double* s, int step, size_t o, int i, int j, double alpha) {
  double* const* const P = DIR == 0 ? d.X : d.Y;
  double qb[6], out[12];
#pragma unroll
  for (int q = 0; q < 6; ++q) qb[q] = __ldg((DIR == 0 ? d.qbx : d.qby)[q] + o);
  if (!interface_values_fixed<DIR, CHAR, true>(s, s + step, s + 2 * step, s + 3 * step, SP_R, qb, d, out))
    interface_fallback<DIR, CHAR, false>(GridSource<double>{&d}, alpha, i, j, 0, qb, out);
  const int own = threadIdx.x & 1;
#pragma unroll
  for (int q = 0; q < 6; ++q) P[6 * own + q][o] = own ? out[6 + q] : out[q];
}

template <bool CHAR>
__global__ void __launch_bounds__(TILE_T, 4) k_sweep_xy_pair(const __grid_constant__ Dev2D d, const double* __restrict__ alpha, int nxt) {
  __shared__ double sm[NRECX * SP_R];
  const int t = threadIdx.x, u = t >> 1;
  if ((int)blockIdx.x < nxt) {
    const unsigned W = d.nx + 4, total = (unsigned)d.ny * W, E0 = blockIdx.x * (SP_R - 3);
    if (t < SP_R && E0 + t < total) {
      const unsigned j = (E0 + t) / W;
      Node12 n;
      load_node(d, (int)(E0 + t - j * W) - 2, (int)j, n);
      double rec[NRECX];
      node_record_fixed<0>(n, d.g, alpha[0], rec);
#pragma unroll
      for (int f = 0; f < NRECX; ++f) sm[f * SP_R + t] = rec[f];
    }
    __syncthreads();
    const unsigned E = E0 + u, j = E / W, k = E - j * W;
    if (u >= SP_R - 3 || E >= total || k > (unsigned)d.nx) return;
    sweep_pair<0, CHAR>(d, sm + u, 1, (size_t)j * (d.nx + 1) + k, (int)k, (int)j, alpha[0]);
  } else {
    constexpr int ifs = SP_R / YS_C - 3;
    const unsigned H = d.ny + 4, total = (unsigned)((d.nx + YS_C - 1) / YS_C) * H, E0 = (blockIdx.x - nxt) * ifs;
    if (t < SP_R) {
      const unsigned E = E0 + t / YS_C, g = E / H;
      const int i = (int)g * YS_C + t % YS_C;
      if (E < total && i < d.nx) {
        Node12 n;
        load_node(d, i, (int)(E - g * H) - 2, n);
        double rec[NRECX];
        node_record_fixed<1>(n, d.g, alpha[1], rec);
#pragma unroll
        for (int f = 0; f < NRECX; ++f) sm[f * SP_R + t] = rec[f];
      }
    }
    __syncthreads();
    const unsigned E = E0 + u / YS_C, g = E / H, k = E - g * H;
    const int i = (int)g * YS_C + u % YS_C;
    if (u / YS_C >= ifs || E >= total || k > (unsigned)d.ny || i >= d.nx) return;
    sweep_pair<1, CHAR>(d, sm + u, YS_C, (size_t)k * d.nx + i, i, (int)k, alpha[1]);
  }
}

// A stage's node update of small grids: of 64 nodes a block, the right-hand side, the limiter along x and the limiter along
// y are two warps' each, then the RK combination of three planes is. The values are node_update's.
template <bool CHAR>
__global__ void __launch_bounds__(192, 3) k_node2d_split(const __grid_constant__ Dev2D d, const __grid_constant__ StageArgs sa) {
  __shared__ double s_R[9 * 64];
  __shared__ int s_bad[64];
  const int t = threadIdx.x & 63, role = threadIdx.x >> 6;
  if (sa.nsteps && blockIdx.x == 0 && threadIdx.x == 0) {
    *sa.t = sa.snapped ? sa.clock[1] : *sa.t + sa.clock[0];
    if (sa.clock[0] > 0.0) ++*sa.nsteps;
  }
  const unsigned o = blockIdx.x * 64 + t;
  const int j = (int)(o / (unsigned)d.nx), i = (int)(o - (unsigned)j * d.nx);
  const bool in = j < d.ny;
  if (!(*sa.dt > 0.0)) {  // a step of size 0 leaves the state unchanged
    if (in)
#pragma unroll
      for (int q = 0; q < 3; ++q) sa.out[3 * role + q][o] = __ldg(d.S[3 * role + q] + o);
    return;
  }
  if (role == 0) s_bad[t] = 0;
  __syncthreads();
  double cur[9], mod[3];
  if (in) {
#pragma unroll
    for (int q = 0; q < 9; ++q) cur[q] = __ldg(d.S[q] + o);
    if (role == 0) {
      const PlaneFaces<false, double> faces{d, i, j, 0, o, (size_t)o + j, o};
      double Rv[9];
      right_hand_side<double>(d, o, cur, faces, Rv);
#pragma unroll
      for (int q = 0; q < 9; ++q) s_R[q * 64 + t] = Rv[q];
    } else if (sa.limiter) {
      LimitNode L;
      L.form<CHAR>(d, __ldg(d.stat[0] + o), cur);
      double out[3];
      if (!limit_dir_fixed<CHAR, false>(d, i, j, 0, cur, L, role - 1, out)) s_bad[t] = 1;
      mod[0] = out[0];
      mod[1] = role == 1 ? out[1] : out[2];
      mod[2] = role == 1 ? out[2] : out[1];
    } else {
#pragma unroll
      for (int q = 0; q < 3; ++q) mod[q] = role == 1 ? cur[3 + q] : cur[6 + q];
    }
  }
  __syncthreads();
  if (!in) return;
  if (role != 0 && s_bad[t]) {
    double both[6];
    limit_node_fallback<CHAR, false>(GridSource<double>{&d}, i, j, 0, cur, both);
#pragma unroll
    for (int q = 0; q < 3; ++q) mod[q] = role == 1 ? both[q] : both[3 + q];
  }
  const double dt = -*sa.dt;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const double R = s_R[(3 * role + q) * 64 + t];
    const double cq = role == 0 ? cur[q] : mod[q];
    double* const out = sa.out[3 * role + q] + o;
    if (sa.k == 1) {
      if (sa.base) sa.base[3 * role + q][o] = cq;
      *out = fma(dt, R, cq);
    } else if (sa.k == 2) {
      *out = fma(0.75, __ldg(sa.base[3 * role + q] + o), fx_quarter(fma(dt, R, cq)));
    } else {
      *out = fma(1.0 / 3.0, __ldg(sa.base[3 * role + q] + o), (2.0 / 3.0) * fma(dt, R, cq));
    }
  }
}

// Single-precision y-sweep: bound by memory rather than arithmetic, it keeps the column march, whose
// loads are 32 consecutive nodes of a row: each thread owns one column and marches down `seg`
// interfaces with the last four node records in a private shared-memory ring (no block barrier and
// only 3 extra records per segment). Measured at 2048^2: 0.139 ms against 0.164 ms for the best tile.
constexpr int YS_W = 32;

template <bool LINEAR, bool CHAR>
__global__ void __launch_bounds__(YS_W, 32) k_sweep_y_col(Dev2DT<float> d, const float* __restrict__ alpha, int seg) {
  __shared__ float ring[4 * NREC * YS_W];
  const int i = blockIdx.x * YS_W + threadIdx.x;
  if (i >= d.nx) return;
  const int k0 = blockIdx.y * seg;
  const float ay = alpha[1];
  const int rend = min(k0 + seg, d.ny + 1);
  for (int r = k0 - 2; r <= rend; ++r) {
    Node12T<float> n;
    load_node(d, i, r, n);
    float rec[NREC];
    node_record<1>(n, d.g, ay, rec);
    float* slot = ring + (size_t)(r & 3) * NREC * YS_W + threadIdx.x;
#pragma unroll
    for (int f = 0; f < NREC; ++f) slot[f * YS_W] = rec[f];
    const int k = r - 1;
    if (k >= k0 && k < k0 + seg && k <= d.ny) {
      const float* s0 = ring + (size_t)((k - 2) & 3) * NREC * YS_W + threadIdx.x;
      const float* s1 = ring + (size_t)((k - 1) & 3) * NREC * YS_W + threadIdx.x;
      const float* s2 = ring + (size_t)((k) & 3) * NREC * YS_W + threadIdx.x;
      const float* s3 = ring + (size_t)((k + 1) & 3) * NREC * YS_W + threadIdx.x;
      const size_t o = (size_t)k * d.nx + i;
      float qb[6];
#pragma unroll
      for (int q = 0; q < 6; ++q) qb[q] = __ldg(d.qby[q] + o);
      float out[12];
      interface_values<1, LINEAR, CHAR>(s0, s1, s2, s3, YS_W, qb, d.g, d.eps_w, out);
#pragma unroll
      for (int q = 0; q < 12; ++q) d.Y[q][o] = out[q];
    }
  }
}

// T threads per block: 256, or 64 for grids that do not fill the GPU with those (their warps then spread over more
// SMs, and need not spill).
template <int MODE, bool LINEAR, bool CHAR, class R, int T = kNodeT>
__global__ void __launch_bounds__(T, T == kNodeT ? kNodeBlocks<R> : 8) k_node2d(const __grid_constant__ Dev2DT<R> d, StageArgsT<R> sa) {
  const int i = blockIdx.x * 32 + threadIdx.x;
  const int j = blockIdx.y * (T / 32) + threadIdx.y;
  if (MODE == MODE_STAGE && sa.nsteps && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0 && threadIdx.y == 0) {
    *sa.t = sa.snapped ? sa.clock[1] : *sa.t + sa.clock[0];
    if (sa.clock[0] > 0.0) ++*sa.nsteps;
  }
  if (i >= d.nx || j >= d.ny) return;
  node_update<MODE, LINEAR, CHAR, kFixed<R>>(d, GridSource<R>{&d}, sa, i, j);
}

// ---------------------------------------------------------------------------------------------
// alpha_x, alpha_y = max over nodes of |u| + c, |v| + c, plus a status flag for non-finite or
// non-positive depth: in double the two passes of hw_stencil2d.cuh (coarse float maxima, then the exact
// double maximum near them), in single precision one pass.
// ---------------------------------------------------------------------------------------------
// Each block reduces one contiguous tile of nodes; each thread keeps kAlphaU nodes' loads in flight. The
// coarse pass records every tile's float maxima (bit 31 set when a node of the tile needs the exact
// evaluation regardless), so the exact pass skips the tiles that cannot hold a maximum: it evaluates the
// same nodes, by the same rule, as a pass over all nodes would.
constexpr int kAlphaU = 4;
constexpr unsigned kTileExact = 0x80000000u;

__device__ __forceinline__ void alpha_tile(size_t n, size_t& begin, size_t& end) {
  const size_t per = (n + gridDim.x - 1) / gridDim.x;
  begin = min(n, (size_t)blockIdx.x * per);
  end = min(n, begin + per);
}

__global__ void __launch_bounds__(256) k_alpha2d_coarse(Dev2D d, unsigned int* m32, uint2* tiles, int* status) {
  __shared__ float s_m[2][8];
  __shared__ int s_ex[8];
  size_t begin, end;
  alpha_tile((size_t)d.nx * d.ny, begin, end);
  float mx = 0.0f, my = 0.0f;
  int bad = 0, ex = 0;
  for (size_t o0 = begin + threadIdx.x; o0 < end; o0 += kAlphaU * blockDim.x) {
    float ax[kAlphaU], ay[kAlphaU];
    bool exact[kAlphaU], neg[kAlphaU];
#pragma unroll
    for (int u = 0; u < kAlphaU; ++u) {
      exact[u] = false;
      neg[u] = true;  // past the end: skipped
      if (o0 + u * blockDim.x < end) alpha_coarse(d, o0 + u * blockDim.x, ax[u], ay[u], exact[u], neg[u]);
    }
#pragma unroll
    for (int u = 0; u < kAlphaU; ++u) {
      if (o0 + u * blockDim.x >= end) continue;
      if (exact[u]) { ex = 1; continue; }  // the exact pass evaluates (and, if need be, flags) this node
      if (neg[u]) { bad |= HW_STATUS_DEPTH; continue; }
      mx = fmaxf(mx, ax[u]);
      my = fmaxf(my, ay[u]);
    }
  }
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) {
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, s));
    my = fmaxf(my, __shfl_xor_sync(0xffffffffu, my, s));
  }
  ex = __any_sync(0xffffffffu, ex);
  const int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) { s_m[0][w] = mx; s_m[1][w] = my; s_ex[w] = ex; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < (int)(blockDim.x >> 5); ++k) {
      mx = fmaxf(mx, s_m[0][k]);
      my = fmaxf(my, s_m[1][k]);
      ex |= s_ex[k];
    }
    // non-negative floats order as their bit patterns
    atomicMax(m32, __float_as_uint(mx));
    atomicMax(m32 + 1, __float_as_uint(my));
    const unsigned f = ex ? kTileExact : 0u;
    tiles[blockIdx.x] = make_uint2(__float_as_uint(mx) | f, __float_as_uint(my) | f);
  }
  if (bad) atomicOr(status, bad);
}

// alpha keys -> doubles; dt = cfl / (alpha_x/dx + alpha_y/dy), optionally clipped to t_end - t.
__device__ __forceinline__ void finish_alpha(unsigned long long kx, unsigned long long ky, const AlphaOut& f) {
  const double ax = __longlong_as_double((long long)kx), ay = __longlong_as_double((long long)ky);
  f.alpha[0] = ax;
  f.alpha[1] = ay;
  if (f.with_dt) {
    double dt = f.cfl / fma(ax, f.inv_dx, ay * f.inv_dy);
    double t_next = f.t_now ? *f.t_now + dt : 0.0;
    if (f.t_now && f.t_end > 0.0) {
      // the step that reaches t_end (within a relative 1e-12) ends exactly on it
      const double rem = f.t_end - *f.t_now;
      if (dt >= rem - 1e-12 * f.t_end) {
        dt = rem > 0.0 ? rem : 0.0;
        t_next = rem > 0.0 ? f.t_end : *f.t_now;
      }
    }
    f.dt[0] = dt;
    if (f.t_now) f.dt[1] = t_next;
  }
  if (f.fsc) {
    f.fsc[0] = (float)ax;
    f.fsc[1] = (float)ay;
    f.fsc[2] = (float)f.dt[0];
  }
}

// The end of a block of a reduction into slots[0..1] (keys; slots[2] scratch, slots[3] the blocks done): called by
// one thread once the block's maxima are in; the last block finishes and clears the slots. No block waits.
__device__ __forceinline__ void alpha_block_done(unsigned long long* slots, const AlphaOut& f) {
  __threadfence();
  if (atomicAdd(slots + 3, 1ull) != (unsigned long long)gridDim.x - 1) return;
  __threadfence();
  finish_alpha(atomicMax(slots, 0ull), atomicMax(slots + 1, 0ull), f);
  slots[0] = slots[1] = slots[2] = slots[3] = 0;
}

// The nodes alpha_exact_range would evaluate, in the tiles whose coarse maxima reach the thresholds. keys: the
// maxima; FINISH: keys are the slots of alpha_block_done, and m32 one of them.
template <bool FINISH>
__global__ void __launch_bounds__(256) k_alpha2d_exact(Dev2D d, const unsigned int* m32, const uint2* tiles,
                                                       unsigned long long* keys, int* status, AlphaOut f) {
  const float tx = __uint_as_float(m32[0]) * (1.0f - 1e-5f), ty = __uint_as_float(m32[1]) * (1.0f - 1e-5f);
  const uint2 tile = tiles[blockIdx.x];
  if (((tile.x | tile.y) & kTileExact) || !(__uint_as_float(tile.x) < tx && __uint_as_float(tile.y) < ty)) {
    size_t begin, end;
    alpha_tile((size_t)d.nx * d.ny, begin, end);
    unsigned long long kx = 0, ky = 0;
    int bad = 0;
    for (size_t o0 = begin + threadIdx.x; o0 < end; o0 += kAlphaU * blockDim.x) {
      float fx[kAlphaU], fy[kAlphaU];
      bool exact[kAlphaU], neg[kAlphaU], in[kAlphaU];
#pragma unroll
      for (int u = 0; u < kAlphaU; ++u) {
        in[u] = o0 + u * blockDim.x < end;
        if (in[u]) alpha_coarse(d, o0 + u * blockDim.x, fx[u], fy[u], exact[u], neg[u]);
      }
#pragma unroll
      for (int u = 0; u < kAlphaU; ++u)
        if (in[u] && alpha_needs_exact(fx[u], fy[u], exact[u], neg[u], tx, ty))
          alpha_exact_node(d, o0 + u * blockDim.x, kx, ky, bad);
    }
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
      kx = max(kx, __shfl_xor_sync(0xffffffffu, kx, s));
      ky = max(ky, __shfl_xor_sync(0xffffffffu, ky, s));
    }
    if ((threadIdx.x & 31) == 0) {
      if (kx) atomicMax(keys, kx);
      if (ky) atomicMax(keys + 1, ky);
      if (FINISH) __threadfence();
    }
    if (bad) atomicOr(status, bad);
  }
  if (!FINISH) return;
  // also in a skipped tile: the last block to arrive clears m32, which every warp of every block must have read by then
  __syncthreads();
  if (threadIdx.x == 0) alpha_block_done(keys, f);
}

// The whole reduction in one launch, for small grids (kAlphaOneMax): each block takes 256 U nodes.
// Measured: 3.8 + 4.5 + 2.5 us and a memset in three launches at 64x66 become one of 4.3 us.
template <int U>
__global__ void __launch_bounds__(256) k_alpha2d_one(Dev2D d, unsigned long long* slots, int* status, AlphaOut f) {
  unsigned long long kx, ky;
  alpha_block_keys<U>(d, (size_t)blockIdx.x * (256 * U) + threadIdx.x, (size_t)d.nx * d.ny, [](size_t o) { return o; },
                      kx, ky, status);
  if (threadIdx.x != 0) return;
  if (kx) atomicMax(slots, kx);
  if (ky) atomicMax(slots + 1, ky);
  alpha_block_done(slots, f);
}

// The start of a stage of all blocks of a decomposed grid: alpha over the blocks' own nodes (alpha_blocks thread
// blocks of 1024 nodes per block of the grid) and the exchange of their rings (the other thread blocks). A ring node
// takes its value through at most one y face and one x face straight from the node it is a copy of; only own nodes
// are read and only ring nodes written, so the two parts need no order. Bound by latency: 600x512 in 2x2 blocks moves
// 0.6 MB of rings and reads 10 MB for alpha.
__global__ void __launch_bounds__(256) k_parts_begin(const PartBlock* __restrict__ parts, int np, int cur, double g,
                                                     unsigned oddx, unsigned oddy, int alpha_blocks,
                                                     unsigned long long* slots, AlphaOut f) {
  const int chunk = (int)(blockIdx.x / (unsigned)np);
  const PartBlock& P = parts[blockIdx.x - (unsigned)chunk * np];
  if (chunk < alpha_blocks) {
    Dev2D d;
    d.g = g;
    for (int q = 0; q < 3; ++q) d.S[q] = P.S[cur][q];
    d.stat[0] = P.b;
    const unsigned nx = (unsigned)P.nx;
    unsigned long long kx, ky;
    alpha_block_keys<4>(d, (size_t)chunk * 1024 + threadIdx.x, (size_t)P.nx * P.ny,
                        [nx](size_t o) {
                          const unsigned j = (unsigned)o / nx, i = (unsigned)o - j * nx;
                          return (size_t)(j + 2) * (nx + 4) + i + 2;
                        },
                        kx, ky, P.status);
    if (threadIdx.x == 0) {
      if (kx) atomicMax(slots, kx);
      if (ky) atomicMax(slots + 1, ky);
    }
  } else {
    const int r = (chunk - alpha_blocks) * 256 + threadIdx.x, W = P.nx + 4;
    if (r < 4 * (W + P.ny)) {
      // the ring: rows 0, 1, ny + 2, ny + 3 in full width, then columns 0, 1, nx + 2, nx + 3 of the other rows
      int i, j;
      if (r < 4 * W) {
        const int row = r / W;
        i = r - row * W;
        j = row < 2 ? row : P.ny + row;
      } else {
        const int q = r - 4 * W, c = q & 3;
        j = 2 + (q >> 2);
        i = c < 2 ? c : P.nx + c;
      }
      // the node's source across a face of block b, in b's direction of length n: coordinate k (0, 1 or n + 2, n + 3)
      auto cross = [&](const PartBlock*& b, int lo, int n, int n_of_nbr, int& k) {
        const bool low = k < 2;
        const int face = low ? lo : lo + 1, c = low ? k : k - (n + 2), mode = b->mode[face];
        if (mode == HW_HALO_NEIGHBOR) {
          k = low ? n_of_nbr + c : 2 + c;
          b = parts + b->nbr[face];
          return false;
        }
        const int sc = mode == HW_HALO_MIRROR ? 1 - c : low ? 0 : 1;
        k = (low ? 2 : n) + sc;
        return mode == HW_HALO_MIRROR;
      };
      const PartBlock* s = &P;
      int si = i, sj = j;
      bool fx = false, fy = false;
      if (sj < 2 || sj >= s->ny + 2) fy = cross(s, HW_FACE_S, s->ny, parts[s->nbr[sj < 2 ? HW_FACE_S : HW_FACE_N]].ny, sj);
      if (si < 2 || si >= s->nx + 2) fx = cross(s, HW_FACE_W, s->nx, parts[s->nbr[si < 2 ? HW_FACE_W : HW_FACE_E]].nx, si);
      const size_t from = (size_t)sj * (s->nx + 4) + si, to = (size_t)j * W + i;
      double v[9];
#pragma unroll
      for (int q = 0; q < 9; ++q) v[q] = s->S[cur][q][from];
#pragma unroll
      for (int q = 0; q < 9; ++q) {
        if (fx && ((oddx >> q) & 1u)) v[q] = -v[q];
        if (fy && ((oddy >> q) & 1u)) v[q] = -v[q];
        P.S[cur][q][to] = v[q];
      }
    }
  }
  // the last thread block to end forms every block's alpha (and dt)
  __shared__ int s_last;
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(slots + 3, 1ull) == (unsigned long long)gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const unsigned long long ax = atomicMax(slots, 0ull), ay = atomicMax(slots + 1, 0ull);
  for (int p = threadIdx.x; p < np; p += 256) {
    f.alpha = parts[p].alpha;
    f.dt = parts[p].dt;
    f.t_now = f.with_dt ? parts[p].t : nullptr;
    finish_alpha(ax, ay, f);
  }
  __syncthreads();
  if (threadIdx.x == 0) slots[0] = slots[1] = slots[2] = slots[3] = 0;
}

// Single precision: the maximum in float, widened to a double key once per block. Each thread keeps the
// loads of kAlphaU nodes in flight (the pass is bound by memory latency otherwise).
__global__ void __launch_bounds__(256) k_alpha2d_f32(Dev2DT<float> d, unsigned long long* slots, int* status, AlphaOut f) {
  __shared__ float s_m[2][8];
  int bad = 0;
  const size_t n = (size_t)d.nx * d.ny, step = (size_t)gridDim.x * blockDim.x;
  float mx = 0.0f, my = 0.0f;
  for (size_t o0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x; o0 < n; o0 += kAlphaU * step) {
    float hn[kAlphaU], mn[kAlphaU], wn[kAlphaU];
#pragma unroll
    for (int q = 0; q < kAlphaU; ++q) {
      const size_t o = o0 + q * step;
      hn[q] = 1.0f;
      mn[q] = wn[q] = 0.0f;
      if (o < n) {
        hn[q] = __ldg(d.S[0] + o) - __ldg(d.stat[0] + o);
        mn[q] = __ldg(d.S[1] + o);
        wn[q] = __ldg(d.S[2] + o);
      }
    }
#pragma unroll
    for (int q = 0; q < kAlphaU; ++q) {
      if (o0 + q * step >= n) continue;
      const float h = hn[q];
      if (!(h > 0.0f) || !(h < 3e38f)) { bad |= h == h ? HW_STATUS_DEPTH : HW_STATUS_NONFINITE; continue; }
      const float rh = fast_rcp(h);
      const float gh = d.g * h;
      const float c = gh * fast_rsqrt(gh);
      const float u = mn[q] * rh, v = wn[q] * rh;
      const float ax = fabsf(u) + c, ay = fabsf(v) + c;
      if (!(ax < 3e38f) || !(ay < 3e38f)) { bad |= HW_STATUS_NONFINITE; continue; }
      mx = fmaxf(mx, ax);
      my = fmaxf(my, ay);
    }
  }
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) {
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, s));
    my = fmaxf(my, __shfl_xor_sync(0xffffffffu, my, s));
  }
  if (bad) atomicOr(status, bad);
  if ((threadIdx.x & 31) == 0) { s_m[0][threadIdx.x >> 5] = mx; s_m[1][threadIdx.x >> 5] = my; }
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int k = 1; k < 8; ++k) {
    mx = fmaxf(mx, s_m[0][k]);
    my = fmaxf(my, s_m[1][k]);
  }
  atomicMax(slots, dkey((double)mx));
  atomicMax(slots + 1, dkey((double)my));
  alpha_block_done(slots, f);
}

// alpha and dt from keys that a launch of its own found (blocks of a decomposition).
__global__ void k_finish_alpha2d(const unsigned long long* amax, AlphaOut f) { finish_alpha(amax[0], amax[1], f); }

// ---------------------------------------------------------------------------------------------
// Initialisation and conversion kernels
// ---------------------------------------------------------------------------------------------
// physical (h, hu, hv, b, h_x, hu_x, hv_x, h_y, hu_y, hv_y, b_x, b_y) -> equilibrium state with
// scaled derivatives (eta = h + b, H = h_x + b_x; Sec. 3) and static (b, dx b_x, dy b_y).
__global__ void k_init2d(Dev2D d, PhysIn in, int* status) {
  const size_t n = (size_t)d.nx * d.ny;
  for (size_t o = (size_t)blockIdx.x * blockDim.x + threadIdx.x; o < n; o += (size_t)gridDim.x * blockDim.x) {
    const double h = in.p[0][o], b = in.p[3][o], bx = in.p[10][o], by = in.p[11][o];
    if (!(h > 0.0) || !(h < 1e300)) atomicOr(status, h == h ? HW_STATUS_DEPTH : HW_STATUS_NONFINITE);
    d.S[0][o] = h + b;
    d.S[1][o] = in.p[1][o];
    d.S[2][o] = in.p[2][o];
    d.S[3][o] = d.dx * (in.p[4][o] + bx);
    d.S[4][o] = d.dx * in.p[5][o];
    d.S[5][o] = d.dx * in.p[6][o];
    d.S[6][o] = d.dy * (in.p[7][o] + by);
    d.S[7][o] = d.dy * in.p[8][o];
    d.S[8][o] = d.dy * in.p[9][o];
    d.stat[0][o] = b;
    d.stat[1][o] = d.dx * bx;
    d.stat[2][o] = d.dy * by;
    d.bxy[0][o] = bx;
    d.bxy[1][o] = by;
  }
}

// state <-> user planes. layout 0: physical (h, hu, hv, h_x, hu_x, hv_x, h_y, hu_y, hv_y);
// layout 1: equilibrium (eta, m, w, eta_x, m_x, w_x, eta_y, m_y, w_y). dir 0: export, 1: import.
__global__ void k_convert2d(Dev2D d, Ptr9 src9, Ptr9 dst9, int layout, int dir) {
  double* const* S = d.S;
  const size_t n = (size_t)d.nx * d.ny;
  for (size_t o = (size_t)blockIdx.x * blockDim.x + threadIdx.x; o < n; o += (size_t)gridDim.x * blockDim.x) {
    const double b = d.stat[0][o], bx = d.bxy[0][o], by = d.bxy[1][o];
    if (dir == 0) {
      double x[9];
      for (int q = 0; q < 9; ++q) x[q] = S[q][o];
      dst9.p[0][o] = layout == 0 ? x[0] - b : x[0];
      dst9.p[1][o] = x[1];
      dst9.p[2][o] = x[2];
      dst9.p[3][o] = layout == 0 ? x[3] * d.inv_dx - bx : x[3] * d.inv_dx;
      dst9.p[4][o] = x[4] * d.inv_dx;
      dst9.p[5][o] = x[5] * d.inv_dx;
      dst9.p[6][o] = layout == 0 ? x[6] * d.inv_dy - by : x[6] * d.inv_dy;
      dst9.p[7][o] = x[7] * d.inv_dy;
      dst9.p[8][o] = x[8] * d.inv_dy;
    } else {
      double x[9];
      for (int q = 0; q < 9; ++q) x[q] = src9.p[q][o];
      S[0][o] = layout == 0 ? x[0] + b : x[0];
      S[1][o] = x[1];
      S[2][o] = x[2];
      S[3][o] = d.dx * (layout == 0 ? x[3] + bx : x[3]);
      S[4][o] = d.dx * x[4];
      S[5][o] = d.dx * x[5];
      S[6][o] = d.dy * (layout == 0 ? x[6] + by : x[6]);
      S[7][o] = d.dy * x[7];
      S[8][o] = d.dy * x[8];
    }
  }
}

// Static parts of the source terms that depend on b only (Sec. 2.1 Step 2 and eq. mixed):
//   qbx/qby: Hermite candidates q_1..q_3 of (b, dS b_s) per interface and side (the nonlinear
//            weights are applied per stage),
//   sv, sq : dx [tilde-B1^]_x/dx + dx [bar-B1^]_y/dy and dy [tilde-B2^]_x/dx + dy [bar-B2^]_y/dy
//            (normal-momentum and tangential-momentum components; the first component is zero).
__device__ __forceinline__ double bval(const Dev2D& d, int q, int i, int j) {
  // q: 0 b, 1 b_x, 2 b_y (physical); parities: b even; b_x odd across x-walls; b_y odd across y-walls
  bool fx, fy;
  const int ii = map_index(i, d.nx, d.bc_x, fx);
  const int jj = map_index(j, d.ny, d.bc_y, fy);
  const size_t o = (size_t)jj * d.nx + ii;
  double x = q == 0 ? d.stat[0][o] : d.bxy[q - 1][o];
  if (fx && q == 1) x = -x;
  if (fy && q == 2) x = -x;
  return x;
}

__device__ __forceinline__ void cands(double f0, double f1, double f2, double p0, double p1, double p2, double q[3]) {
  q[0] = 0.5 * (f0 + f1) + (p0 + 5.0 * p1) / 6.0;
  q[1] = 0.5 * (f1 + f2) + (p1 - p2) / 6.0;
  q[2] = (f0 + 10.0 * f1 + f2) / 12.0 + 0.5 * p1;
}

// Derivative of the quintic at the interface, both sides summed, on (b/2, b_s/2) (eq. Rec-phi).
__device__ __forceinline__ double qprime_sum(double b0, double b1, double b2, double b3, double s0, double s1,
                                             double s2, double s3, double del) {
  const double qp = (b0 - 8.0 * b1 + 7.0 * b2) / (4.0 * del) + (s0 - 2.0 * s1 - 5.0 * s2) / 12.0;
  const double qm = (-7.0 * b1 + 8.0 * b2 - b3) / (4.0 * del) + (-5.0 * s1 - 2.0 * s2 + s3) / 12.0;
  return 0.5 * (qp + qm);
}

__device__ __forceinline__ double mixed4(double a, double b, double c, double e) {
  return (-a + 7.0 * b + 7.0 * c - e) / 12.0;
}

__global__ void k_static2d(Dev2D d) {
  const int i = blockIdx.x * 32 + threadIdx.x;
  const int j = blockIdx.y * 8 + threadIdx.y;
  // x-interfaces k = i (0..nx) of row j; y-interfaces k = j (0..ny) of column i
  if (j < d.ny && i <= d.nx) {
    double b[4], s[4];
    for (int t = 0; t < 4; ++t) {
      b[t] = bval(d, 0, i - 2 + t, j);
      s[t] = d.dx * bval(d, 1, i - 2 + t, j);
    }
    double qp[3], qm[3];
    cands(b[0], b[1], b[2], s[0], s[1], s[2], qp);
    cands(b[3], b[2], b[1], -s[3], -s[2], -s[1], qm);
    const size_t o = (size_t)j * (d.nx + 1) + i;
    for (int q = 0; q < 3; ++q) { d.qbx[q][o] = qp[q]; d.qbx[3 + q][o] = qm[q]; }
  }
  if (i < d.nx && j <= d.ny) {
    double b[4], s[4];
    for (int t = 0; t < 4; ++t) {
      b[t] = bval(d, 0, i, j - 2 + t);
      s[t] = d.dy * bval(d, 2, i, j - 2 + t);
    }
    double qp[3], qm[3];
    cands(b[0], b[1], b[2], s[0], s[1], s[2], qp);
    cands(b[3], b[2], b[1], -s[3], -s[2], -s[1], qm);
    const size_t o = (size_t)j * d.nx + i;
    for (int q = 0; q < 3; ++q) { d.qby[q][o] = qp[q]; d.qby[3 + q][o] = qm[q]; }
  }
  if (i < d.nx && j < d.ny) {
    // x-interfaces i-1/2 (left, stencil i-2..i+1) and i+1/2 (right, i-1..i+2)
    auto B1x = [&](int k) {  // tilde-B1 hat (normal-momentum component) at x-interface k-1/2
      return qprime_sum(bval(d, 0, k - 2, j), bval(d, 0, k - 1, j), bval(d, 0, k, j), bval(d, 0, k + 1, j),
                        bval(d, 1, k - 2, j), bval(d, 1, k - 1, j), bval(d, 1, k, j), bval(d, 1, k + 1, j), d.dx);
    };
    auto B2x = [&](int k) {  // tilde-B2 hat = mixed(b_y) at x-interface k-1/2
      return mixed4(bval(d, 2, k - 2, j), bval(d, 2, k - 1, j), bval(d, 2, k, j), bval(d, 2, k + 1, j));
    };
    auto B1y = [&](int k) {  // bar-B1 hat = mixed(b_x) at y-interface k-1/2
      return mixed4(bval(d, 1, i, k - 2), bval(d, 1, i, k - 1), bval(d, 1, i, k), bval(d, 1, i, k + 1));
    };
    auto B2y = [&](int k) {  // bar-B2 hat (tangential = y-momentum component) at y-interface k-1/2
      return qprime_sum(bval(d, 0, i, k - 2), bval(d, 0, i, k - 1), bval(d, 0, i, k), bval(d, 0, i, k + 1),
                        bval(d, 2, i, k - 2), bval(d, 2, i, k - 1), bval(d, 2, i, k), bval(d, 2, i, k + 1), d.dy);
    };
    const size_t o = (size_t)j * d.nx + i;
    // dx * (tilde-B1 hat)_x / dx = difference; dx * (bar-B1 hat)_y / dy
    d.sv[0][o] = B1x(i + 1) - B1x(i);
    d.sv[1][o] = d.dx * (B1y(j + 1) - B1y(j)) * d.inv_dy;
    // dy * (tilde-B2 hat)_x / dx; dy * (bar-B2 hat)_y / dy = difference
    d.sq[0][o] = d.dy * (B2x(i + 1) - B2x(i)) * d.inv_dx;
    d.sq[1][o] = B2y(j + 1) - B2y(j);
  }
}

// ---------------------------------------------------------------------------------------------
// Host launchers
// ---------------------------------------------------------------------------------------------
template <bool L, bool C, class R>
static void launch_sx(const Dev2DT<R>& d, const R* alpha, cudaStream_t st) {
  const unsigned long long total = (unsigned long long)d.ny * (d.nx + 4);
  constexpr int T = kXT<R>;
  k_sweep_x<L, C, R><<<(unsigned)((total + T - 4) / (T - 3)), T, 0, st>>>(d, alpha);
}

// Segment length of the float column march: one balanced wave of resident blocks when the grid allows
// it (the blocks of a column segment all do the same work), at least 8 interfaces per segment.
static int sweep_y_segment(int nx, int ny, int blocks_per_sm) {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 1;
  }
  const int cols = (nx + YS_W - 1) / YS_W;
  const long resident = (long)sms * std::max(blocks_per_sm, 1);
  long segs = std::max(1L, resident / cols);
  int seg = (int)((ny + 1 + segs - 1) / segs);
  return std::max(seg, std::min(8, ny + 1));
}

template <bool L, bool C, class R>
static void launch_sy(const Dev2DT<R>& d, const R* alpha, cudaStream_t st) {
  if constexpr (std::is_same<R, float>::value) {
    static int bps = -1;
    if (bps < 0 && cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, k_sweep_y_col<L, C>, YS_W, 0) != cudaSuccess)
      bps = 1;
    const int seg = sweep_y_segment(d.nx, d.ny, bps);
    dim3 gy((d.nx + YS_W - 1) / YS_W, (d.ny + 1 + seg - 1) / seg);
    k_sweep_y_col<L, C><<<gy, YS_W, 0, st>>>(d, alpha, seg);
  } else {
    constexpr int IFS = TILE_T / YS_C - 3;
    const unsigned long long total = (unsigned long long)((d.nx + YS_C - 1) / YS_C) * (d.ny + 4);
    k_sweep_y<L, C><<<(unsigned)((total + IFS - 1) / IFS), TILE_T, 0, st>>>(d, alpha);
  }
}

// Nodes up to which the node update runs in blocks of 64 threads: what those hold at once (16 warps per SM).
constexpr size_t kNodeSmallMax = (size_t)152 * 16 * 32;
// ... and up to which it is split over warps, and interfaces have two lanes: one wave of the split node update's blocks.
constexpr size_t kNodeSplitMax = (size_t)152 * 3 * 64, kPairMax = (size_t)152 * 3 * 64;

template <int MODE, bool L, bool C, class R>
static void launch_node(const Dev2DT<R>& d, const StageArgsT<R>& sa, cudaStream_t st) {
  if constexpr (std::is_same<R, double>::value && !L) {
    if (MODE == MODE_STAGE && (size_t)d.nx * d.ny <= kNodeSplitMax) {
      k_node2d_split<C><<<(unsigned)(((size_t)d.nx * d.ny + 63) / 64), 192, 0, st>>>(d, sa);
      return;
    }
    if ((size_t)d.nx * d.ny <= kNodeSmallMax) {
      k_node2d<MODE, L, C, R, 64><<<dim3((d.nx + 31) / 32, (d.ny + 1) / 2), dim3(32, 2), 0, st>>>(d, sa);
      return;
    }
  }
  constexpr int rows = kNodeT / 32;
  dim3 g((d.nx + 31) / 32, (d.ny + rows - 1) / rows);
  k_node2d<MODE, L, C, R><<<g, dim3(32, rows), 0, st>>>(d, sa);
}

int set_kernel_attributes2d() { return 0; }

static int alpha_blocks(const Dev2D& d) {
  return (int)std::min<size_t>(((size_t)d.nx * d.ny + 255) / 256, (size_t)kAlpha2dTiles);
}
void launch_alpha2d(const Dev2D& d, unsigned long long* amax, int* status, cudaStream_t st) {
  cudaMemsetAsync(amax, 0, 3 * sizeof(unsigned long long), st);
  unsigned int* m32 = reinterpret_cast<unsigned int*>(amax + 2);
  uint2* tiles = reinterpret_cast<uint2*>(amax + 3);
  const int blocks = alpha_blocks(d);
  k_alpha2d_coarse<<<blocks, 256, 0, st>>>(d, m32, tiles, status);
  k_alpha2d_exact<false><<<blocks, 256, 0, st>>>(d, m32, tiles, amax, status, AlphaOut{});
}
void launch_alpha_finish2d(const Dev2D& d, unsigned long long* amax, int* status, const AlphaOut& out, cudaStream_t st) {
  unsigned long long* slots = amax + kAlpha2dSlots;
  const size_t n = (size_t)d.nx * d.ny;
  // one node a thread while one block an SM takes the grid; beyond, four a thread, which is the slower form up to 2^18 nodes (10
  // steps at 65,536 nodes 1.90 ms with one, 2.00 with four; at 131,044 3.35 and 3.39; at 2^18 5.74 and 5.80)
  if (n <= (size_t)152 * 256) {
    k_alpha2d_one<1><<<(unsigned)((n + 255) / 256), 256, 0, st>>>(d, slots, status, out);
  } else if (n <= kAlphaOneMax) {
    k_alpha2d_one<4><<<(unsigned)((n + 1023) / 1024), 256, 0, st>>>(d, slots, status, out);
  } else {
    unsigned int* m32 = reinterpret_cast<unsigned int*>(slots + 2);
    uint2* tiles = reinterpret_cast<uint2*>(amax + 3);
    const int blocks = alpha_blocks(d);
    k_alpha2d_coarse<<<blocks, 256, 0, st>>>(d, m32, tiles, status);
    k_alpha2d_exact<true><<<blocks, 256, 0, st>>>(d, m32, tiles, slots, status, out);
  }
}
void launch_alpha_finish2d(const Dev2DT<float>& d, unsigned long long* amax, int* status, const AlphaOut& out,
                           cudaStream_t st) {
  const size_t n = (size_t)d.nx * d.ny;
  const int blocks = (int)std::min<size_t>((n + 255) / 256, (size_t)152 * 8);
  k_alpha2d_f32<<<blocks, 256, 0, st>>>(d, amax + kAlpha2dSlots, status, out);
}

void launch_parts_begin(const PartBlock* parts, const PartBlock* host, int np, int cur, const Dev2D& d, unsigned oddx,
                        unsigned oddy, unsigned long long* slots, bool with_dt, double cfl, double t_end,
                        cudaStream_t st) {
  size_t na = 0, nr = 0;
  for (int p = 0; p < np; ++p) {
    na = std::max(na, ((size_t)host[p].nx * host[p].ny + 1023) / 1024);
    nr = std::max(nr, ((size_t)4 * (host[p].nx + 4 + host[p].ny) + 255) / 256);
  }
  k_parts_begin<<<(unsigned)((na + nr) * np), 256, 0, st>>>(
      parts, np, cur, d.g, oddx, oddy, (int)na, slots,
      AlphaOut{nullptr, nullptr, with_dt, cfl, d.inv_dx, d.inv_dy, nullptr, t_end, nullptr});
}

void launch_finish_alpha2d(const Dev2D& d, const unsigned long long* amax, double* alpha, double* dt_out,
                           double cfl, const double* t_now, double t_end, cudaStream_t st) {
  k_finish_alpha2d<<<1, 1, 0, st>>>(amax, AlphaOut{alpha, dt_out, dt_out != nullptr, cfl, d.inv_dx, d.inv_dy, t_now, t_end, nullptr});
}

template <class R>
static void sweep_x_impl(const Dev2DT<R>& d, const R* alpha, bool linear, bool chr, cudaStream_t st) {
  if (linear) { if (chr) launch_sx<true, true>(d, alpha, st); else launch_sx<true, false>(d, alpha, st); }
  else        { if (chr) launch_sx<false, true>(d, alpha, st); else launch_sx<false, false>(d, alpha, st); }
}
template <class R>
static void sweep_y_impl(const Dev2DT<R>& d, const R* alpha, bool linear, bool chr, cudaStream_t st) {
  if (linear) { if (chr) launch_sy<true, true>(d, alpha, st); else launch_sy<true, false>(d, alpha, st); }
  else        { if (chr) launch_sy<false, true>(d, alpha, st); else launch_sy<false, false>(d, alpha, st); }
}
template <class R>
static void node_impl(const Dev2DT<R>& d, const StageArgsT<R>& sa, int mode, bool linear, bool chr, cudaStream_t st) {
  if (mode == MODE_RHS) {
    if (linear) { if (chr) launch_node<MODE_RHS, true, true>(d, sa, st); else launch_node<MODE_RHS, true, false>(d, sa, st); }
    else        { if (chr) launch_node<MODE_RHS, false, true>(d, sa, st); else launch_node<MODE_RHS, false, false>(d, sa, st); }
  } else {
    if (linear) { if (chr) launch_node<MODE_STAGE, true, true>(d, sa, st); else launch_node<MODE_STAGE, true, false>(d, sa, st); }
    else        { if (chr) launch_node<MODE_STAGE, false, true>(d, sa, st); else launch_node<MODE_STAGE, false, false>(d, sa, st); }
  }
}

void launch_sweep_x2d(const Dev2D& d, const double* alpha, bool linear, bool chr, cudaStream_t st) {
  sweep_x_impl(d, alpha, linear, chr, st);
}
void launch_sweep_y2d(const Dev2D& d, const double* alpha, bool linear, bool chr, cudaStream_t st) {
  sweep_y_impl(d, alpha, linear, chr, st);
}
// Tiles of both sweeps up to which they share a launch: one launch has one partly empty last wave instead of two. Four steps
// in one / two launches: 1.39 / 1.49 ms at 131,044 nodes, 2.61 / 2.67 at 291,600, 2.81 / 2.87 at 313,600 (this line lies
// between), 8.05 / 8.08 at 2^20, 30.7 / 30.6 at 2^22.
constexpr unsigned long long kSweepsOneMax = 152 * 4 * 8;

void launch_sweeps2d(const Dev2D& d, const double* alpha, bool linear, bool chr, cudaStream_t st) {
  const bool pair = !linear && (size_t)d.nx * d.ny <= kPairMax;
  const int IX = (pair ? SP_R : TILE_T) - 3, IY = (pair ? SP_R : TILE_T) / YS_C - 3;
  const unsigned long long nxt = ((unsigned long long)d.ny * (d.nx + 4) + IX - 1) / IX;
  const unsigned long long nyt = ((unsigned long long)((d.nx + YS_C - 1) / YS_C) * (d.ny + 4) + IY - 1) / IY;
  if (pair) {
    if (chr) k_sweep_xy_pair<true><<<(unsigned)(nxt + nyt), TILE_T, 0, st>>>(d, alpha, (int)nxt);
    else k_sweep_xy_pair<false><<<(unsigned)(nxt + nyt), TILE_T, 0, st>>>(d, alpha, (int)nxt);
    return;
  }
  if (!linear && nxt + nyt <= kSweepsOneMax) {
    if (chr) k_sweep_xy<true><<<(unsigned)(nxt + nyt), TILE_T, 0, st>>>(d, alpha, (int)nxt);
    else k_sweep_xy<false><<<(unsigned)(nxt + nyt), TILE_T, 0, st>>>(d, alpha, (int)nxt);
    return;
  }
  launch_sweep_x2d(d, alpha, linear, chr, st);
  launch_sweep_y2d(d, alpha, linear, chr, st);
}
void launch_node2d(const Dev2D& d, const StageArgs& sa, int mode, bool linear, bool chr, cudaStream_t st) {
  node_impl(d, sa, mode, linear, chr, st);
}
void launch_sweep_x2d(const Dev2DT<float>& d, const float* alpha, bool linear, bool chr, cudaStream_t st) {
  sweep_x_impl(d, alpha, linear, chr, st);
}
void launch_sweep_y2d(const Dev2DT<float>& d, const float* alpha, bool linear, bool chr, cudaStream_t st) {
  sweep_y_impl(d, alpha, linear, chr, st);
}
void launch_node2d(const Dev2DT<float>& d, const StageArgsT<float>& sa, int mode, bool linear, bool chr,
                   cudaStream_t st) {
  node_impl(d, sa, mode, linear, chr, st);
}

// Plane conversion between precisions (the single-precision variant keeps double copies for the
// initialisation and the exchange with the caller).
__global__ void k_cast_planes(int nplanes, size_t n, Ptr12 src, Ptr12 dst, int to_float) {
  for (size_t o = (size_t)blockIdx.x * blockDim.x + threadIdx.x; o < n; o += (size_t)gridDim.x * blockDim.x)
    for (int q = 0; q < nplanes; ++q) {
      if (to_float) ((float*)dst.p[q])[o] = (float)((const double*)src.p[q])[o];
      else ((double*)dst.p[q])[o] = (double)((const float*)src.p[q])[o];
    }
}

void launch_cast_planes(int nplanes, size_t n, const Ptr12& src, const Ptr12& dst, int to_float, cudaStream_t st) {
  int blocks = (int)std::min<size_t>((n + 255) / 256, (size_t)152 * 16);
  k_cast_planes<<<blocks, 256, 0, st>>>(nplanes, n, src, dst, to_float);
}

void launch_init2d(const Dev2D& d, const PhysIn& in, int* status, cudaStream_t st) {
  const size_t n = (size_t)d.nx * d.ny;
  int blocks = (int)std::min<size_t>((n + 255) / 256, (size_t)152 * 16);
  k_init2d<<<blocks, 256, 0, st>>>(d, in, status);
  dim3 g((d.nx + 1 + 31) / 32, (d.ny + 1 + 7) / 8);
  k_static2d<<<g, dim3(32, 8), 0, st>>>(d);
}

void launch_static2d(const Dev2D& d, cudaStream_t st) {
  dim3 g((d.nx + 1 + 31) / 32, (d.ny + 1 + 7) / 8);
  k_static2d<<<g, dim3(32, 8), 0, st>>>(d);
}

void launch_convert2d(const Dev2D& d, const Ptr9& src, const Ptr9& dst, int layout, int dir, cudaStream_t st) {
  const size_t n = (size_t)d.nx * d.ny;
  int blocks = (int)std::min<size_t>((n + 255) / 256, (size_t)152 * 16);
  k_convert2d<<<blocks, 256, 0, st>>>(d, src, dst, layout, dir);
}

}  // namespace hw
