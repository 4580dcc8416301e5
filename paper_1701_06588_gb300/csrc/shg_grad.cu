// Gradients of the two-center SHG integrals with respect to the centers (Sec. II C of arXiv:1701.06588, Eq. dev_ab), as a
// vector-Jacobian product with upstream weights W:
//   g = sum_{ma,mb} W[ma][mb] d(a|O|b)[ma][mb] / dR_a,     d/dR_b = -d/dR_a (translation invariance).
// Radial orders up to la+lb+1 as in the integral pass (shg_xradial.cuh; nothing is kept from a forward evaluation), the
// angular part in shg_grad_angular.cuh.  Tiles and groups as the integral pass; the lanes of a group share the primitive
// pairs and the projection of W, and add up their gradients.
#include "shg_grad2c.cuh"
#include "shg_tilemap.cuh"

namespace shg {

cudaError_t launch_2c_grad(const ArgsGrad &a, cudaStream_t s, int threads) { return launch_grad<false>(a, s, threads); }

namespace {
using namespace dev;

template <int J>
__device__ void pair_grad_ra2n(const Args2c &g, int p)
{
    const ShellRec sa = g.shells[g.pair_a[p]];
    const ShellRec sb = g.shells[g.pair_b[p]];
    const int la = sa.l, lb = sb.l;
    const Vec4 A = g.centers[sa.center];
    const Vec4 B = g.centers[sb.center];
    const double v[3] = {A.x - B.x, A.y - B.y, A.z - B.z};
    const double R2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
    double Q[J + 1];
#pragma unroll
    for (int j = 0; j <= J; ++j) Q[j] = 0.0;
    const int Kb = sb.nprim, npp = sa.nprim * Kb;
    for (int q = 0; q < npp; ++q) {
        const int ia = q / Kb, ib = q - ia * Kb;
        radial_acc_ra2n<J + 1>(g.prims[sa.prim_off + ia], g.prims[sb.prim_off + ib], R2, la + lb + 1, la, g, Q);
    }
    double G[3];
    vjp_d<J>(g.cg, g.k, la, lb, v, R2, Q, 0.0, 0.0, g.w + g.w_off[p], 0, 1, G);
    for (int d = 0; d < 3; ++d) {
        g.grad_a[3 * (int64_t)p + d] = G[d];
        if (g.grad_b) g.grad_b[3 * (int64_t)p + d] = -G[d];
    }
}

__global__ void __launch_bounds__(128) k_2c_grad_ra2n(const Args2c g)
{
    const int lane = threadIdx.x & 31;
    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(g.counter, 1);
        t = __shfl_sync(0xffffffffu, t, 0) + g.tile_begin;
        if (t >= g.tile_end) break;
        int cls;
        const int q = map_pair(g.map, t, lane, cls);
        if (q >= 0) {
            const int la = cls / (kLmax2c + 1), lb = cls % (kLmax2c + 1), p = g.perm[q];
            switch ((la < lb ? la : lb) + 1) {
            case 1: pair_grad_ra2n<1>(g, p); break;
            case 2: pair_grad_ra2n<2>(g, p); break;
            case 3: pair_grad_ra2n<3>(g, p); break;
            case 4: pair_grad_ra2n<4>(g, p); break;
            case 5: pair_grad_ra2n<5>(g, p); break;
            case 6: pair_grad_ra2n<6>(g, p); break;
            default: pair_grad_ra2n<7>(g, p); break;
            }
        }
        __syncwarp();
    }
}

}  // namespace

cudaError_t launch_2c_grad_ra2n(const Args2c &a, cudaStream_t s)
{
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_2c_grad_ra2n, 128, 0) != cudaSuccess || per < 1) per = 1;
    k_2c_grad_ra2n<<<(sms > 0 ? sms : 1) * per, 128, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace shg
