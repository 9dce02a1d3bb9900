// Instances of the resident kernel for the second-order sweep.
#include "pc_resident.cuh"

namespace pcx {

cudaError_t launch_resident2(const pc_plan *p, const Sweep &s, const double *x0, cudaStream_t st, size_t *scratch) {
  return res_choose<2, 1, 4, 8, 16>(p, s, x0, st, scratch);
}

}  // namespace pcx
