// Instances of the resident kernel for the first-order sweep.
#include "pc_resident.cuh"

namespace pcx {

cudaError_t launch_resident1(const pc_plan *p, const Sweep &s, const double *x0, cudaStream_t st, size_t *scratch) {
  return res_choose<1, 1, 2, 4, 8>(p, s, x0, st, scratch);
}

}  // namespace pcx
