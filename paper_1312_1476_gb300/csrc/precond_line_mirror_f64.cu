// precond_line_mirror_f64.cu -- instantiation of the line kernels: mirror-extended (DCT-II) preconditioner, FP64.
#include "precond_line.cuh"

namespace gmrf {
namespace line {

template <>
cudaError_t step_mirror<double>(const Args<double>& a, int nvec, cudaStream_t s) {
  return step_k<double, GMRF_PREC_MIRROR>(a, nvec, s);
}
template <>
cudaError_t apply_mirror<double>(const Args<double>& a, int nvec, cudaStream_t s) {
  return apply_k<double, GMRF_PREC_MIRROR>(a, nvec, s);
}
template <>
cudaError_t operator_mirror<double>(const Args<double>& a, int nvec, cudaStream_t s) {
  return operator_k<double, GMRF_PREC_MIRROR>(a, nvec, s);
}

}  // namespace line
}  // namespace gmrf
