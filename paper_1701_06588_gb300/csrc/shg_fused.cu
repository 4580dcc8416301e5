// FP64 two-center passes of 1/r and erfc (the pair of a range-separated step) and the choice of an instantiation.
#include "shg_pair2c.cuh"

namespace shg {

cudaError_t launch_2c_fused(const ArgsFused &a, cudaStream_t s, int threads, int ctas_per_sm, int variant)
{
    const unsigned w = a.r.want;
    if (w & ~(unsigned)(kSumCo | kSumX)) {
        if (w == kSumOv || w == kSumEr || w == kSumGa || w == kSumGc) return launch_2c_one(a, s, threads, ctas_per_sm);
        return launch_2c_all(a, s, threads, ctas_per_sm, variant);
    }
    if (w == kSumCo) return launch_2c_one(a, s, threads, ctas_per_sm);
    switch (variant) {
    case 0: return launch_pass<kSumCo | kSumX, 4>(a, s, threads, ctas_per_sm);
    case 1: return launch_pass<kSumCo | kSumX, 8>(a, s, threads, ctas_per_sm);
    default: return launch_pass<kSumCo | kSumX, 6>(a, s, threads, ctas_per_sm);
    }
}

}  // namespace shg
