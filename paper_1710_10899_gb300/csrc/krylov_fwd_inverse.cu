// Krylov forward: the inverse, refined from double-float or in FP64.
#include "krylov_fwd.cuh"

namespace submat {
namespace kry {

cudaError_t launch_inverse_df(const Args& a, const Class& c, int grid, cudaStream_t s) {
  return dispatch<true, df>(a, c, grid, s);
}
cudaError_t set_attr_inverse_df() { return attrs<true, df>(); }
cudaError_t launch_inverse_fp64(const Args& a, const Class& c, int grid, cudaStream_t s) {
  return dispatch<true, double>(a, c, grid, s);
}
cudaError_t set_attr_inverse_fp64() { return attrs<true, double>(); }

}  // namespace kry
}  // namespace submat
