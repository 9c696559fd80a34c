// precond_line_mirror_f32.cu -- instantiation of the line kernels: mirror-extended (DCT-II) preconditioner, FP32.
#include "precond_line.cuh"

namespace gmrf {
namespace line {

template <>
cudaError_t step_mirror<float>(const Args<float>& a, int nvec, cudaStream_t s) {
  return step_k<float, GMRF_PREC_MIRROR>(a, nvec, s);
}
template <>
cudaError_t apply_mirror<float>(const Args<float>& a, int nvec, cudaStream_t s) {
  return apply_k<float, GMRF_PREC_MIRROR>(a, nvec, s);
}
template <>
cudaError_t operator_mirror<float>(const Args<float>& a, int nvec, cudaStream_t s) {
  return operator_k<float, GMRF_PREC_MIRROR>(a, nvec, s);
}

}  // namespace line
}  // namespace gmrf
