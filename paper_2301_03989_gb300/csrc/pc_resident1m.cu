// Instances of the resident kernel: first-order sweep, mixed precision.
#include "pc_resident.cuh"

namespace pcx {

cudaError_t launch_resident1m(const pc_plan *p, const Sweep &s, const double *x0, cudaStream_t st, size_t *scratch) {
  return res_choose<1, true, ResKernel<1, 256, 1>, ResKernel<1, 256, 2>, ResKernel<1, 128, 4>,
                    ResKernel<2, 128, 4>, ResKernel<4, 256, 2>, ResKernel<8, 512, 1, true>, ResKernel<2, 256, 2>>(p, s, x0, st, scratch);
}

}  // namespace pcx
