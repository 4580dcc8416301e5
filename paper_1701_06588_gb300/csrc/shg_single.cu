// FP64 two-center passes of one operator (erfc: shg_fused.cu).
#include "shg_pair2c.cuh"

namespace shg {

cudaError_t launch_2c_one(const ArgsFused &a, cudaStream_t s, int threads, int ctas_per_sm)
{
    switch (a.r.want) {
    case kSumOv: return launch_pass<kSumOv, 4>(a, s, threads, ctas_per_sm);
    case kSumCo: return launch_pass<kSumCo, 4>(a, s, threads, ctas_per_sm);
    case kSumEr: return launch_pass<kSumEr, 4>(a, s, threads, ctas_per_sm);
    case kSumGa: return launch_pass<kSumGa, 4>(a, s, threads, ctas_per_sm);
    case kSumGc: return launch_pass<kSumGc, 4>(a, s, threads, ctas_per_sm);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace shg
