// Mixed-precision two-center passes: the radial sums of the FP64 pass (their extended-float terms cost less than
// double-float ones and carry more digits), the angular part in double-float on the FP32 pipes (a double-float
// multiply-add is 18 FP32 instructions of about one cycle, an FP64 one holds its unit for 64).  Only the classes for which
// that is sooner done (kMixedDfMinL, kMixedFp64MinL); the others run in FP64 (launch_2c_fused) beside this launch.
#pragma once

#include "shg_cg_mix.cuh"
#include "shg_pair2c.cuh"

namespace shg {
namespace {

template <unsigned MASK, int J>
__device__ __forceinline__ void tile_2c_mix(const ArgsMixFused &a, const Tile &t, int lane)
{
    // as tile_2c
    const ArgsFused &g = a.f;
    const int group = t.group, gl = lane & (group - 1), slot = lane / group;
    const bool own = slot < t.count;
    const int p = g.perm[t.start + (own ? slot : t.count - 1)];
    const int ia = g.pair_a[p], ib = g.pair_b[p];
    const ShellRec sa = g.shells[ia];
    const ShellRec sb = g.shells[ib];
    const int la = sa.l, lb = sb.l, kmax = la + lb;
    const Vec4 A = g.centers[sa.center];
    const Vec4 B = g.centers[sb.center];
    const double vx = A.x - B.x, vy = A.y - B.y, vz = A.z - B.z;
    const double R2 = vx * vx + vy * vy + vz * vz;
    const long long off = g.out_off[p];
    const bool off_screen = screened<MASK>(g, ia, ib, R2, (2 * la + 1) * (2 * lb + 1), off, own && gl == 0);
    xrad::Sums<J> s;
    xrad::radial<MASK, J>(g.r, sa, sb, R2, kmax, g.k, off_screen || (group == 1 && !own) ? kNoPrims : gl, group, s);
    const double far = (MASK & kSumCo) ? xrad::far_order(s.far, R2, kmax, g.k) : 0.0;
    const bool store = own && !off_screen;

    const int er = R2 > 0.0 ? cgm::exponent(R2) >> 1 : 0;
    const dfm::df x = cgm::split(cgm::scale_exp(vx, -er)), y = cgm::split(cgm::scale_exp(vy, -er)),
                  z = cgm::split(cgm::scale_exp(vz, -er)), r2 = cgm::split(cgm::scale_exp(R2, -2 * er));
    if (!store) return;
    constexpr int kN = (cgm::kMixMaxL + 1) * kMixedFp64MinL;
    dfm::df P[kN], PF[kN], C[cgm::kMixMaxL + 1], S[cgm::kMixMaxL + 1];
    cgm::harmonics(x, y, z, r2, kmax, J, a.kappa, P, C, S);
#pragma unroll 1
    for (int op = 0; op < 6; ++op) {
        double *out = g.out[op];
        if (!out) continue;
        double O[J];
        orders_of<MASK, J>(s, g.r.want, op, O);
        const double top = op == OP_COULOMB || op == OP_ERFC ? far : 0.0;
        cgm::block_from_orders<J>(g.cg, la, lb, R2, er, O, top, P, C, S, PF, gl, group, out + off);
    }
}

template <unsigned MASK>
__device__ __forceinline__ void run_tile_mix(const ArgsMixFused &a, const Tile &t, int lane)
{
    const int la = t.cls / (kLmax2c + 1), lb = t.cls % (kLmax2c + 1);
    static_assert(kMixedDfMinL == 2 && kMixedFp64MinL == 4, "cases below");
    switch ((la < lb ? la : lb) + 1) {
    case 3: tile_2c_mix<MASK, 3>(a, t, lane); break;
    case 4: tile_2c_mix<MASK, 4>(a, t, lane); break;
    default: break;
    }
}

template <unsigned MASK, int MinB>
__global__ void __launch_bounds__(128, MinB) k_2c_mixed_fused(const ArgsMixFused a)
{
    const int lane = threadIdx.x & 31;
    const ArgsFused &g = a.f;
    cudaTriggerProgrammaticLaunchCompletion();
    if (!g.counter) {
        const int t = g.tile_begin + launch_warp(blockIdx.x, blockDim.x, threadIdx.x);
        if (t < g.tile_end) run_tile_mix<MASK>(a, g.tiles[t], lane);
        if (g.beside) cudaGridDependencySynchronize();
        return;
    }
    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(g.counter, 1);
        t = __shfl_sync(0xffffffffu, t, 0) + g.tile_begin;
        if (t >= g.tile_end) break;
        run_tile_mix<MASK>(a, g.tiles[t], lane);
        __syncwarp();
    }
    if (g.beside) cudaGridDependencySynchronize();
}

template <unsigned MASK, int MinB>
cudaError_t launch_mix(const ArgsMixFused &a, cudaStream_t s, int threads, int ctas_per_sm)
{
    const int grid = pass_grid(a.f, (const void *)k_2c_mixed_fused<MASK, MinB>, threads, ctas_per_sm);
    return launch_on(k_2c_mixed_fused<MASK, MinB>, a, a.f.beside, grid, threads, s);
}

}  // namespace
}  // namespace shg
