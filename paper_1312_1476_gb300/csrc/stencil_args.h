// stencil_args.h -- kernel arguments of the fused stencil step (Algorithm 1
// with the matrix-free lattice apply of Q, Section 2), shared by the
// stencil kernels.
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"

namespace gmrf {

template <typename T>
struct StencilArgs {
  const T* Win;  // apply mode: v
  T* Wout;       // apply mode: y = scale Q v
  T scale;
  T* W0;         // step mode: q ping-pong, W[j & 1] read, W[(j+1) & 1] written
  T* W1;
  T* V;  // basis ring base
  const float* kappa2;
  T kappa2_const;
  int nx, ny, nz;
  size_t n;
  int nzc;  // z chunks (3-D register kernel)
  StepParams P;
  VecState* st;
  double* alpha;
  double* beta;
  float* alpha_f;
  float* beta2_f;
  Dots<T>* partials;
  unsigned* counters;
};

struct Grid;

// ---- 2-D tiles and the arithmetic of a cell, shared by the one-step kernel
// (lanczos_stencil.cu) and the resident one (stencil2d_resident.cu), whose results are
// the same bits.
// Rows of a 2-D tile, two of them a thread's: half the additions of a sum over
// the block, and half its barriers, per cell.  FP64 tiles are 8 rows, so that a
// small grid spreads over more SMs (their FP64 lanes bound it), FP32 tiles 16.
// 64 x 64 periodic, about 26 steps, one vector and 256, 16 rows and one a thread
// (512 threads) before: FP64 636 -> 588 us and 3119 -> 2732, FP32 514 -> 508 and
// 1872 -> 1549.
constexpr int kTileX = 32, kTileCells = 2;
template <typename T>
__host__ __device__ constexpr int tile2d_y() { return sizeof(T) == 8 ? 8 : 16; }
template <typename T>
__host__ __device__ constexpr int tile2d_threads() { return kTileX * tile2d_y<T>() / kTileCells; }

// Explicit roundings: what the compiler may contract differs with the code around.
__device__ __forceinline__ float next_v(float q, float vp, float coef, float inv_b, bool later) {
  return __fmul_rn(later ? __fmaf_rn(-coef, vp, q) : q, inv_b);
}
__device__ __forceinline__ double next_v(double q, double vp, double coef, double inv_b, bool later) {
  return __dmul_rn(later ? __fma_rn(-coef, vp, q) : q, inv_b);
}
__device__ __forceinline__ float edge(float c, float x) { return __fsub_rn(c, x); }
__device__ __forceinline__ double edge(double c, double x) { return __dsub_rn(c, x); }
// kappa^2 c + the differences along the edges (0 for one that leaves a Neumann grid)
__device__ __forceinline__ float b_cell(float k, float c, float l, float r, float u, float d) {
  return __fadd_rn(__fadd_rn(__fmaf_rn(k, c, l), r), __fadd_rn(u, d));
}
__device__ __forceinline__ double b_cell(double k, double c, double l, double r, double u, double d) {
  return __dadd_rn(__dadd_rn(__fma_rn(k, c, l), r), __dadd_rn(u, d));
}
__device__ __forceinline__ float less(float q, float b, float v) { return __fmaf_rn(-b, v, q); }
__device__ __forceinline__ double less(double q, double b, double v) { return __fma_rn(-b, v, q); }

// stencil3d_tma.cu (eligibility and item counts are declared in internal.h)
// 16-byte alignment of the vector and coefficient pointers the kernel maps.
bool stencil3d_tma_pointers_ok(const void* win, const void* wout, const float* kappa2);
// step = true: fused Lanczos step on a.W0/W1/V; false: a.Wout = Q a.Win.
cudaError_t launch_stencil3d_tma(const Grid& g, const StencilArgs<float>& a, int nvec, bool step, cudaStream_t s);

// stencil3d_flat.cu: 3-D grids up to 512 wide, any precision and pointer alignment.
bool stencil3d_flat_eligible(const Grid& g);
int stencil3d_flat_blocks_per_vector(const Grid& g);
template <typename T>
cudaError_t launch_stencil3d_flat(const Grid& g, const StencilArgs<T>& a, int nvec, bool step, cudaStream_t s);

// stencil2d_strip.cu: the 2-D step streamed down strips of 128 (FP32) / 64
// (FP64) columns, for grids of at least half a strip and 65536 cells.
bool stencil2d_strip_eligible(const Grid& g, bool fp64);
int stencil2d_strip_blocks_per_vector(const Grid& g, bool fp64);
template <typename T>
cudaError_t launch_stencil2d_strip(const Grid& g, const StencilArgs<T>& a, int nvec, bool step, cudaStream_t s);

// stencil2d_resident.cu: up to nsteps steps on a 2-D grid that a thread-block cluster holds.
template <typename T>
cudaError_t launch_stencil2d_resident(const Grid& g, const StencilArgs<T>& a, int nvec, int nsteps, cudaStream_t s);

}  // namespace gmrf
