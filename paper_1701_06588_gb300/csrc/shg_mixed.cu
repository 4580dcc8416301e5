// Mixed-precision two-center passes of one operator and of 1/r and erfc, and the choice of an instantiation.
#include "shg_mixed2c.cuh"

namespace shg {

cudaError_t launch_2c_mixed(const ArgsMixFused &a, cudaStream_t s, int threads, int ctas_per_sm, int variant)
{
    const unsigned w = a.f.r.want;
    switch (w) {
    case kSumOv: return launch_mix<kSumOv, 4>(a, s, threads, ctas_per_sm);
    case kSumEr: return launch_mix<kSumEr, 4>(a, s, threads, ctas_per_sm);
    case kSumGa: return launch_mix<kSumGa, 4>(a, s, threads, ctas_per_sm);
    case kSumGc: return launch_mix<kSumGc, 4>(a, s, threads, ctas_per_sm);
    default: break;
    }
    if (!(w & ~(unsigned)(kSumCo | kSumX))) {
        switch (variant) {
        case 0: return launch_mix<kSumCo | kSumX, 4>(a, s, threads, ctas_per_sm);
        case 1: return launch_mix<kSumCo | kSumX, 8>(a, s, threads, ctas_per_sm);
        default: return launch_mix<kSumCo | kSumX, 6>(a, s, threads, ctas_per_sm);
        }
    }
    return launch_2c_mixed_all(a, s, threads, ctas_per_sm, variant);
}

}  // namespace shg
