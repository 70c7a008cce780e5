// One RK stage of the single-precision variant in one launch: both sweeps and the node update of a tile of nodes, with
// the interface values in shared memory.
//
// As three launches (hw_kernels2d.cu) a stage wrote 24 interface planes and read them back, 192 of its 440 bytes per
// node, and each kernel lay between the memory and the issue limit. A tile of 16 x 16 nodes forms (16 + 4) x 16 records
// along each direction (1.25 per node) and 17 x 16 interfaces (1.06 per node). What bounds it is instruction issue (59% of
// the slots, 2290 instructions per node) with the latency of its loads, at 30 warps per SM. Measured at 2048^2: 0.411 ms a stage,
// a job of four steps 6.14 -> 5.78 ms; with 4 blocks per SM (48 registers) 6.01 ms, with the tile's nodes held in shared
// memory (68 KB a block) 6.13 ms.
#include "hw_stencil2d.cuh"

namespace hw {
namespace {

constexpr int FX = 16, FY = 16;           // tile
constexpr int F_T = FX * (FY + 4);        // threads: one per record (the same number along x and y)
constexpr int F_NX = (FX + 1) * FY, F_NY = FX * (FY + 1);
static_assert(FX == FY, "one record per thread in both directions");
constexpr int kF32Blocks = 3;

// What the update of a node reads: its state and neighbours from the planes, the interface values from the tile (xs, ys at
// its left x-interface and its lower y-interface).
struct TileFaces {
  const PlaneFaces<false, float> planes;
  const float *xs, *ys;
  __device__ __forceinline__ float state(int q) const { return planes.state(q); }
  __device__ __forceinline__ float bottom() const { return planes.bottom(); }
  __device__ __forceinline__ void neighbour(int di, int dj, Node12T<float>& n) const { planes.neighbour(di, dj, n); }
  __device__ __forceinline__ float x(int q) const { return xs[q * F_NX + 1] - xs[q * F_NX]; }
  __device__ __forceinline__ float y(int q) const { return ys[q * F_NY + FX] - ys[q * F_NY]; }
};

template <bool CHAR>
__global__ void __launch_bounds__(F_T, kF32Blocks) k_stage2d_f32(const __grid_constant__ Dev2DT<float> d,
                                                                 const __grid_constant__ StageArgsT<float> sa,
                                                                 const float* __restrict__ alpha) {
  __shared__ float rec[NREC * F_T], xs[12 * F_NX], ys[12 * F_NY];
  const int t = threadIdx.x, i0 = blockIdx.x * FX, j0 = blockIdx.y * FY;
  if (sa.nsteps && blockIdx.x == 0 && blockIdx.y == 0 && t == 0) {
    *sa.t = sa.snapped ? sa.clock[1] : *sa.t + sa.clock[0];
    if (sa.clock[0] > 0.0) ++*sa.nsteps;
  }
  {  // x-records of nodes i0 - 2 .. i0 + FX + 1
    const int r = t / (FX + 4), e = t - r * (FX + 4), i = i0 - 2 + e, j = j0 + r;
    if (i < d.nx + 2 && j < d.ny) {
      Node12T<float> n;
      load_node(d, i, j, n);
      float v[NREC];
      node_record<0>(n, d.g, alpha[0], v);
#pragma unroll
      for (int f = 0; f < NREC; ++f) rec[f * F_T + t] = v[f];
    }
  }
  __syncthreads();
  if (t < F_NX) {
    const int r = t / (FX + 1), k = t - r * (FX + 1), i = i0 + k, j = j0 + r;
    if (i <= d.nx && j < d.ny) {
      const size_t o = (size_t)j * (d.nx + 1) + i;
      float qb[6], out[12];
#pragma unroll
      for (int q = 0; q < 6; ++q) qb[q] = __ldg(d.qbx[q] + o);
      const float* s = rec + r * (FX + 4) + k;
      interface_values<0, false, CHAR>(s, s + 1, s + 2, s + 3, F_T, qb, d.g, d.eps_w, out);
#pragma unroll
      for (int q = 0; q < 12; ++q) xs[q * F_NX + t] = out[q];
    }
  }
  __syncthreads();
  const int c = t % FX, r = t / FX, i = i0 + c;
  {  // y-records of rows j0 - 2 .. j0 + FY + 1
    const int j = j0 - 2 + r;
    if (i < d.nx && j < d.ny + 2) {
      Node12T<float> n;
      load_node(d, i, j, n);
      float v[NREC];
      node_record<1>(n, d.g, alpha[1], v);
#pragma unroll
      for (int f = 0; f < NREC; ++f) rec[f * F_T + t] = v[f];
    }
  }
  __syncthreads();
  const int j = j0 + r;
  if (t < F_NY && i < d.nx && j <= d.ny) {
    const size_t o = (size_t)j * d.nx + i;
    float qb[6], out[12];
#pragma unroll
    for (int q = 0; q < 6; ++q) qb[q] = __ldg(d.qby[q] + o);
    const float* s = rec + t;
    interface_values<1, false, CHAR>(s, s + FX, s + 2 * FX, s + 3 * FX, F_T, qb, d.g, d.eps_w, out);
#pragma unroll
    for (int q = 0; q < 12; ++q) ys[q * F_NY + t] = out[q];
  }
  __syncthreads();
  if (t < FX * FY && i < d.nx && j < d.ny) {
    const TileFaces faces{{d, i, j, 0, (size_t)j * d.nx + i, 0, 0}, xs + r * (FX + 1) + c, ys + t};
    node_update_faces<MODE_STAGE, false, CHAR, false, false>(d, GridSource<float>{&d}, sa, i, j, 0, faces);
  }
}

}  // namespace

void launch_stage2d_f32(const Dev2DT<float>& d, const StageArgsT<float>& sa, const float* alpha, bool chr, cudaStream_t st) {
  const dim3 g((d.nx + FX - 1) / FX, (d.ny + FY - 1) / FY);
  if (chr) k_stage2d_f32<true><<<g, F_T, 0, st>>>(d, sa, alpha);
  else k_stage2d_f32<false><<<g, F_T, 0, st>>>(d, sa, alpha);
}

}  // namespace hw
