// precond_line.h -- entry points of the preconditioner kernels that transform
// along x and solve along y (precond_line.cuh), one translation unit per
// precision and preconditioner kind.
#pragma once

#include <cuda_runtime.h>

#include <vector>

#include "precond.h"

namespace gmrf {
namespace line {

template <typename R>
struct C2;
template <>
struct C2<float> { typedef float2 T; };
template <>
struct C2<double> { typedef double2 T; };

// Column coefficients of the recurrence along y, one record per real of a
// packed spectrum row (see precond_line.cuh): rho the root below 1 of
// rho + 1/rho = 2 + kappa_bar^2 + lambda_x.
template <typename R>
struct ColCoef {
  R delta;   // 1 - rho
  R dchunk;  // 1 - rho^(rows of a chunk)
  R pseg;    // rho^(rows of a scan lane)
  R pn;      // rho^ny
  R close;   // 1 / (1 - rho^(2 ny)) (reflecting ends) or 1 / (1 - rho^ny) (periodic)
  R gain;    // (2 / nx) / (1/rho - rho): Green's function at 0 times the transform's normalisation
  R pad0, pad1;
};

template <typename R>
struct Args {
  typedef typename C2<R>::T C;
  int nx, ny, bc;
  int form;             // FORM_CTC / FORM_DIAG (precond.h)
  R roff;               // R = K - roff
  const C* tw;          // FFT twiddles, pass after pass (fft_twiddles)
  const R* pair;        // {tw_k, d_k} of the pairs k = 0 .. nx/4 - 1 (mirror), {tw_k} (circulant)
  const ColCoef<R>* col;  // [nx]
  R* T;                 // spectrum, packed rows [ny][nx] per vector
  size_t tstride;
  R* G;                 // g = C v (squared operator)
  R* Wg;                // w when the y-boundary terms need a separate pass
  const R* in;
  R* out;
  R scale;              // of out (L_INV)
  bool in_elem, out_elem;  // in / out not aligned for vectors (L_FWD, L_INV)
  const float* kappa2;
  R kappa2_const;
  size_t n;
  R* W0;
  R* W1;
  R* V;
  StepParams P;
  VecState* st;
  double* alpha;
  double* beta;
  float* alpha_f;
  float* beta2_f;
  Dots<R>* partials;
  unsigned* counters;
};

// Host tables of a grid: FFT twiddles, pair factors and column coefficients.
struct HostTables {
  std::vector<double> tw;    // complex pairs
  std::vector<double> pair;
  std::vector<double> col;   // records of 8
};
void host_tables(int kind, int nx, int ny, double kbar2, HostTables& t);

template <typename R>
cudaError_t step_circ(const Args<R>& a, int nvec, cudaStream_t s);
template <typename R>
cudaError_t apply_circ(const Args<R>& a, int nvec, cudaStream_t s);
template <typename R>
cudaError_t operator_circ(const Args<R>& a, int nvec, cudaStream_t s);
template <typename R>
cudaError_t step_mirror(const Args<R>& a, int nvec, cudaStream_t s);
template <typename R>
cudaError_t apply_mirror(const Args<R>& a, int nvec, cudaStream_t s);
template <typename R>
cudaError_t operator_mirror(const Args<R>& a, int nvec, cudaStream_t s);

}  // namespace line

// Squared operators (power 2: M^{-1/2} = B_bar^{-1}) with nx a power of two in
// [64, 4096] and ny one in [8, 4096].
bool line_eligible(int power, int nx, int ny);
int line_blocks_per_vector(int nx, int ny);

}  // namespace gmrf
