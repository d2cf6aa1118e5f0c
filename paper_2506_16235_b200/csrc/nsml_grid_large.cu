// The grid select's instances for large buckets: a source file of their own, compiled beside nsml_api.cu.
#include "nsml_grid.cuh"

namespace nsml {

template <int DTYPE>
GridKernel<DTYPE> large_grid_kernel(bool feedback, bool masked) {
  return feedback ? (masked ? k_select_grid<DTYPE, true, true, true> : k_select_grid<DTYPE, true, false, true>)
                  : (masked ? k_select_grid<DTYPE, false, true, true> : k_select_grid<DTYPE, false, false, true>);
}
template GridKernel<NSML_F32> large_grid_kernel<NSML_F32>(bool, bool);
template GridKernel<NSML_BF16> large_grid_kernel<NSML_BF16>(bool, bool);

}  // namespace nsml
