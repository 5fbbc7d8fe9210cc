// Krylov forward: roots (and A itself) in FP64.
#include "krylov_fwd.cuh"

namespace submat {
namespace kry {

cudaError_t launch_roots_fp64(const Args& a, const Class& c, int grid, cudaStream_t s) {
  return dispatch<false, double>(a, c, grid, s);
}
cudaError_t set_attr_roots_fp64() { return attrs<false, double>(); }

}  // namespace kry
}  // namespace submat
