// Krylov forward: roots (and A itself) in double-float, wide rows again in FP64.
#include "krylov_fwd.cuh"

namespace submat {
namespace kry {

cudaError_t launch_roots_df(const Args& a, const Class& c, int grid, cudaStream_t s) {
  return dispatch<false, df>(a, c, grid, s);
}
cudaError_t set_attr_roots_df() { return attrs<false, df>(); }

}  // namespace kry
}  // namespace submat
