// Kernel of the two-center vector-Jacobian product of one operator (shg_grad.cu, shg_grad_mixed.cu).
#pragma once

#include "shg_grad_angular.cuh"
#include "shg_pair2c.cuh"

namespace shg {
namespace {

// Gradient of one pair from Q[j] = O^{(la+lb+1-j)} (top, top1: harmonic contributions to the orders la+lb, la+lb+1),
// over the element sets of lane gl of `group`
template <int J>
__device__ __forceinline__ void vjp_d(const CGTab &t, const Consts &k, int la, int lb, const double (&v)[3], double R2,
                                      const double (&Q)[J + 1], double top, double top1, const double *__restrict__ w,
                                      int gl, int group, double (&G)[3])
{
    using N = gradang::NumD;
    const int c = la * (kLmax2c + 1) + lb;
    const double *fc = t.fc + 28 * c;
    double F[J], D[J];
    gradang::laplace_orders_d<J>(fc, R2, Q, F, D);
    F[0] = fma(__ldg(fc), top, F[0]);
    D[0] = fma(__ldg(fc), top1, D[0]);
    double Ac[cg::kNP2], As[cg::kNP2], P[cg::kNP2], R[cg::kNP2];
    gradang::project<N>(t.g + __ldg(t.gbase + c), la, lb, J, gl, group, [&](int i) { return w[i]; }, Ac, As);
    gradang::contract<N, J>(v[0], v[1], v[2], R2, la + lb, gradang::KapD{k}, F, D, Ac, As, P, R, G);
}

// the same in double-float
template <int J>
__device__ __forceinline__ void vjp_f(const CGTab &t, const KappaMix &k, int la, int lb, const double (&v)[3], double R2,
                                      const double (&Q)[J + 1], double top, double top1, const double *__restrict__ w,
                                      int gl, int group, double (&G)[3])
{
    using N = gradang::NumF;
    const int c = la * (kLmax2c + 1) + lb, kmax = la + lb, ne = (2 * la + 1) * (2 * lb + 1);
    const double *fc = t.fc + 28 * c;
    double F[J], D[J];
    gradang::laplace_orders_d<J>(fc, R2, Q, F, D);
    F[0] = fma(__ldg(fc), top, F[0]);
    D[0] = fma(__ldg(fc), top1, D[0]);
    // the separation in units of 2^er, F_p 2^{er L} and F_p' 2^{er (L + 2)} scaled by 2^-e, W by 2^-ew
    const int er = R2 > 0.0 ? cgm::exponent(R2) >> 1 : 0;
    int e = -4000, ew = -4000;
#pragma unroll
    for (int p = 0; p < J; ++p) {
        const int x = er * (kmax - 2 * p);
        if (F[p] != 0.0) e = max(e, cgm::exponent(F[p]) + x);
        if (D[p] != 0.0) e = max(e, cgm::exponent(D[p]) + x + 2 * er);
    }
    for (int i = 0; i < ne; ++i) {
        const double x = w[i];
        if (x != 0.0) ew = max(ew, cgm::exponent(x));
    }
    dfm::df Ff[J], Df[J];
#pragma unroll
    for (int p = 0; p < J; ++p) {
        const int x = er * (kmax - 2 * p) - e;
        Ff[p] = cgm::split(cgm::scale_exp(F[p], x));
        Df[p] = cgm::split(cgm::scale_exp(D[p], x + 2 * er));
    }
    constexpr int kN = (cgm::kMixMaxL + 1) * kMixedFp64MinL;
    dfm::df Ac[kN], As[kN], P[kN], R[kN], g[3];
    gradang::project<N>(t.gm + __ldg(t.gbase + c), la, lb, J, gl, group,
                        [&](int i) { return cgm::split(cgm::scale_exp(w[i], -ew)); }, Ac, As);
    gradang::contract<N, J>(cgm::split(cgm::scale_exp(v[0], -er)), cgm::split(cgm::scale_exp(v[1], -er)),
                            cgm::split(cgm::scale_exp(v[2], -er)), cgm::split(cgm::scale_exp(R2, -2 * er)), kmax,
                            gradang::KapF{k}, Ff, Df, Ac, As, P, R, g);
    for (int d = 0; d < 3; ++d) G[d] = cgm::scale_exp(cgm::scale_exp((double)g[d].hi + (double)g[d].lo, e - er), ew);
}

template <unsigned MASK, bool MIXED, int J>
__device__ __forceinline__ void tile_grad(const ArgsGrad &a, const Tile &t, int lane)
{
    // as tile_2c
    const ArgsFused &g = a.f;
    const int group = t.group, gl = lane & (group - 1), slot = lane / group;
    const bool own = slot < t.count;
    const int p = g.perm[t.start + (own ? slot : t.count - 1)];
    const ShellRec sa = g.shells[g.pair_a[p]];
    const ShellRec sb = g.shells[g.pair_b[p]];
    const int la = sa.l, lb = sb.l, kmax = la + lb;
    const Vec4 A = g.centers[sa.center];
    const Vec4 B = g.centers[sb.center];
    const double v[3] = {A.x - B.x, A.y - B.y, A.z - B.z};
    const double R2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
    xrad::Sums<J + 1> s;
    xrad::radial<MASK, J + 1>(g.r, sa, sb, R2, kmax + 1, g.k, own ? gl : kNoPrims, group, s);
    const int op = MASK == kSumOv ? OP_OVERLAP : MASK == kSumCo ? OP_COULOMB : MASK == kSumEr ? OP_ERF
                   : MASK == kSumGa ? OP_GAUSS : MASK == kSumGc ? OP_GCOUL : OP_ERFC;
    double Q[J + 1], top = 0.0, top1 = 0.0, G[3];
    orders_of<MASK, J + 1>(s, g.r.want, op, Q);
    if (MASK & kSumCo) {
        top = xrad::far_order(s.far, R2, kmax, g.k);
        top1 = xrad::far_order(s.far, R2, kmax + 1, g.k);
    }
    const double *w = a.w + g.out_off[p];
    if (MIXED) vjp_f<J>(g.cg, a.kappa, la, lb, v, R2, Q, top, top1, w, gl, group, G);
    else vjp_d<J>(g.cg, g.k, la, lb, v, R2, Q, top, top1, w, gl, group, G);
    xrad::group_sum<3>(G, group);
    if (own && gl == 0) {
        for (int d = 0; d < 3; ++d) {
            a.grad_a[3 * (int64_t)p + d] = G[d];
            if (a.grad_b) a.grad_b[3 * (int64_t)p + d] = -G[d];
        }
    }
}

template <unsigned MASK, bool MIXED>
__device__ __forceinline__ void run_tile_grad(const ArgsGrad &a, const Tile &t, int lane)
{
    const int la = t.cls / (kLmax2c + 1), lb = t.cls % (kLmax2c + 1);
    const int J = (la < lb ? la : lb) + 1;
    static_assert(kMixedDfMinLGrad == 3 && kMixedFp64MinL == 4, "one class of J in double-float");
    if (MIXED) {
        if (J == 4) tile_grad<MASK, MIXED, 4>(a, t, lane);
    } else {
        switch (J) {
        case 1: tile_grad<MASK, false, 1>(a, t, lane); break;
        case 2: tile_grad<MASK, false, 2>(a, t, lane); break;
        case 3: tile_grad<MASK, false, 3>(a, t, lane); break;
        case 4: tile_grad<MASK, false, 4>(a, t, lane); break;
        case 5: tile_grad<MASK, false, 5>(a, t, lane); break;
        case 6: tile_grad<MASK, false, 6>(a, t, lane); break;
        default: tile_grad<MASK, false, 7>(a, t, lane); break;
        }
    }
}

template <unsigned MASK, bool MIXED>
__global__ void __launch_bounds__(128, 4) k_2c_grad(const ArgsGrad a)
{
    const int lane = threadIdx.x & 31;
    const ArgsFused &g = a.f;
    if (MIXED) cudaTriggerProgrammaticLaunchCompletion();
    if (!g.counter) {
        const int t = tile_at(g, launch_warp(blockIdx.x, blockDim.x, threadIdx.x));
        if (t >= 0) run_tile_grad<MASK, MIXED>(a, g.tiles[t], lane);
        if (!MIXED && g.beside) cudaGridDependencySynchronize();
        return;
    }
    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(g.counter, 1);
        t = tile_at(g, __shfl_sync(0xffffffffu, t, 0));
        if (t < 0) break;
        run_tile_grad<MASK, MIXED>(a, g.tiles[t], lane);
        __syncwarp();
    }
    if (!MIXED && g.beside) cudaGridDependencySynchronize();
}

template <unsigned MASK, bool MIXED>
cudaError_t launch_grad_mask(const ArgsGrad &a, cudaStream_t s, int threads)
{
    const int grid = pass_grid(a.f, (const void *)k_2c_grad<MASK, MIXED>, threads, 0);
    return launch_on(k_2c_grad<MASK, MIXED>, a, a.f.beside, grid, threads, s);
}

template <bool MIXED>
cudaError_t launch_grad(const ArgsGrad &a, cudaStream_t s, int threads)
{
    switch (a.f.r.want) {
    case kSumOv: return launch_grad_mask<kSumOv, MIXED>(a, s, threads);
    case kSumCo: return launch_grad_mask<kSumCo, MIXED>(a, s, threads);
    case kSumEr: return launch_grad_mask<kSumEr, MIXED>(a, s, threads);
    case kSumGa: return launch_grad_mask<kSumGa, MIXED>(a, s, threads);
    case kSumGc: return launch_grad_mask<kSumGc, MIXED>(a, s, threads);
    case kSumCo | kSumX: return launch_grad_mask<kSumCo | kSumX, MIXED>(a, s, threads);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace
}  // namespace shg
