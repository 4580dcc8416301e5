// Mixed-precision two-center passes of any set of operators.
#define SHG_XF_CALLS
#include "shg_mixed2c.cuh"

namespace shg {

cudaError_t launch_2c_mixed_all(const ArgsMixFused &a, cudaStream_t s, int threads, int ctas_per_sm, int variant)
{
    switch (variant) {
    case 0: return launch_mix<kSumAll, 4>(a, s, threads, ctas_per_sm);
    case 1: return launch_mix<kSumAll, 6>(a, s, threads, ctas_per_sm);
    default: return launch_mix<kSumAll, 5>(a, s, threads, ctas_per_sm);
    }
}

}  // namespace shg
