// precond_line_circ_f32.cu -- instantiation of the line kernels: circulant (torus) preconditioner, FP32.
#include "precond_line.cuh"

namespace gmrf {
namespace line {

template <>
cudaError_t step_circ<float>(const Args<float>& a, int nvec, cudaStream_t s) {
  return step_k<float, GMRF_PREC_CIRCULANT>(a, nvec, s);
}
template <>
cudaError_t apply_circ<float>(const Args<float>& a, int nvec, cudaStream_t s) {
  return apply_k<float, GMRF_PREC_CIRCULANT>(a, nvec, s);
}
template <>
cudaError_t operator_circ<float>(const Args<float>& a, int nvec, cudaStream_t s) {
  return operator_k<float, GMRF_PREC_CIRCULANT>(a, nvec, s);
}

}  // namespace line
}  // namespace gmrf
