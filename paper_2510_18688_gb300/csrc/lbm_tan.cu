// lbm_tan.cu -- the initial state with forward-mode tangent arithmetic (FP64
// value and derivative, sm_103a); the step is the node step's.
#include "lbm_launch.h"

namespace lbmk {

cudaError_t launch_init_tan(const InitArgs<Dual>& a, cudaStream_t s) {
  lbm_init_kernel<Dual, Dual><<<grid_dims(a.g), block_dims(), 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace lbmk
