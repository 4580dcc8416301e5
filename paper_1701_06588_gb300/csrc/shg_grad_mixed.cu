// Mixed-precision gradients: radial orders as the FP64 form, angular part in double-float on the FP32 pipes (min(la, lb)
// = 3; the other classes run in FP64, launch_2c_grad, beside this launch).
#include "shg_grad2c.cuh"

namespace shg {

cudaError_t launch_2c_grad_mixed(const ArgsGrad &a, cudaStream_t s, int threads) { return launch_grad<true>(a, s, threads); }

}  // namespace shg
