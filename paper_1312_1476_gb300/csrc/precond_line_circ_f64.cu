// precond_line_circ_f64.cu -- instantiation of the line kernels: circulant (torus) preconditioner, FP64.
#include "precond_line.cuh"

namespace gmrf {
namespace line {

template <>
cudaError_t step_circ<double>(const Args<double>& a, int nvec, cudaStream_t s) {
  return step_k<double, GMRF_PREC_CIRCULANT>(a, nvec, s);
}
template <>
cudaError_t apply_circ<double>(const Args<double>& a, int nvec, cudaStream_t s) {
  return apply_k<double, GMRF_PREC_CIRCULANT>(a, nvec, s);
}
template <>
cudaError_t operator_circ<double>(const Args<double>& a, int nvec, cudaStream_t s) {
  return operator_k<double, GMRF_PREC_CIRCULANT>(a, nvec, s);
}

}  // namespace line
}  // namespace gmrf
