// Kernel of the FP64 two-center pass over one or several of overlap, 1/r, erfc, erf and the Gaussian operator:
// everything that depends on the geometry only (the harmonics) and the primitive-pair setup is shared by the operators,
// erfc(wr)/r is formed as 1/r - erf(wr)/r (Table S1), and erf and erfc with one omega share the attenuated sum.
//
// Work mapping: a warp per class-pure tile of pairs with similar Ka Kb, 1, 2, 4 or 8 lanes per pair (Tile), which share
// the primitive pairs and the elements; each lane forms the harmonics.  MASK: the sums the instantiation holds
// accumulators for (RadialIn::want selects among them per launch).
#pragma once

#include "shg_cg.cuh"
#include "shg_tilemap.cuh"
#include "shg_xradial.cuh"

namespace shg {
namespace {
using namespace dev;

constexpr int kNoPrims = 1 << 20;       // first primitive pair of a lane that sums none

// orders of operator op from the sums
template <unsigned MASK, int J>
__device__ __forceinline__ void orders_of(const xrad::Sums<J> &s, unsigned want, int op, double (&O)[J])
{
#pragma unroll
    for (int j = 0; j < J; ++j) {
        double v = 0.0;
        if ((MASK & kSumOv) && op == OP_OVERLAP) v = s.ov[j];
        if ((MASK & kSumGa) && op == OP_GAUSS) v = s.ga[j];
        if (MASK & kSumGc) v = s.gc[j];
        if ((MASK & kSumEr) && op == OP_ERF) v = s.er[j];
        if ((MASK & kSumCo) && op == OP_COULOMB) v = s.co[j];
        if ((MASK & kSumX) && op == OP_ERFC) v = s.co[j] - ((want & kSumX) || !(MASK & kSumEr) ? s.x[j] : s.er[j]);
        O[j] = v;
    }
}

template <unsigned MASK>
__device__ __forceinline__ bool screened(const ArgsFused &g, int ia, int ib, double R2, int n, long long off,
                                         bool write)
{
    if (!(MASK == kSumOv || MASK == kSumGa) || !(g.screen_thresh > 0.0)) return false;
    const int op = MASK == kSumOv ? OP_OVERLAP : OP_GAUSS;
    if (screen_bound(g.screen[ia], g.screen[ib], R2, op, g.screen_omega) >= g.screen_thresh) return false;
    double *o = g.out[op] + off;
    for (int i = 0; write && i < n; ++i) o[i] = 0.0;
    return true;
}

template <unsigned MASK, int J>
__device__ __forceinline__ void tile_2c(const ArgsFused &g, const Tile &t, int lane)
{
    // lanes without a pair of their own (the end of a chunk) repeat the last one and store nothing
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

    if (!store) return;
    double P[cg::kNP2], PF[cg::kNP2], C[2 * kLmax2c + 1], S[2 * kLmax2c + 1];
    cg::harmonics(vx, vy, vz, R2, kmax, J, g.k, P, C, S);
#pragma unroll 1
    for (int op = 0; op < 6; ++op) {
        double *out = g.out[op];
        if (!out) continue;
        double O[J];
        orders_of<MASK, J>(s, g.r.want, op, O);
        const double top = op == OP_COULOMB || op == OP_ERFC ? far : 0.0;
        cg::block_from_orders<J>(g.cg, la, lb, R2, O, top, P, C, S, PF, gl, group, out + off);
    }
}

template <unsigned MASK>
__device__ __forceinline__ void run_tile(const ArgsFused &g, const Tile &t, int lane)
{
    const int la = t.cls / (kLmax2c + 1), lb = t.cls % (kLmax2c + 1);
    switch ((la < lb ? la : lb) + 1) {
    case 1: tile_2c<MASK, 1>(g, t, lane); break;
    case 2: tile_2c<MASK, 2>(g, t, lane); break;
    case 3: tile_2c<MASK, 3>(g, t, lane); break;
    case 4: tile_2c<MASK, 4>(g, t, lane); break;
    case 5: tile_2c<MASK, 5>(g, t, lane); break;
    case 6: tile_2c<MASK, 6>(g, t, lane); break;
    default: tile_2c<MASK, 7>(g, t, lane); break;
    }
}

// i-th tile of a launch, or -1 past the last
__device__ __forceinline__ int tile_at(const ArgsFused &g, int i)
{
    int t = g.tile_begin + i;
    if (t >= g.skip_at) t += g.skip_n;
    return t < g.tile_end ? t : -1;
}

// With a tile counter every warp takes tiles from it until none are left; without one (static launch) warp w of block b
// takes tile tile_begin + b * warps_per_block + w once.  MinB: CTAs of 128 threads that must fit on an SM (a register
// cap).
template <unsigned MASK, int MinB>
__global__ void __launch_bounds__(128, MinB) k_2c_fp64_fused(const ArgsFused g)
{
    const int lane = threadIdx.x & 31;
    cudaTriggerProgrammaticLaunchCompletion();
    if (!g.counter) {
        const int t = tile_at(g, launch_warp(blockIdx.x, blockDim.x, threadIdx.x));
        if (t >= 0) run_tile<MASK>(g, g.tiles[t], lane);
        if (g.beside) cudaGridDependencySynchronize();
        return;
    }
    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(g.counter, 1);
        t = tile_at(g, __shfl_sync(0xffffffffu, t, 0));
        if (t < 0) break;
        run_tile<MASK>(g, g.tiles[t], lane);
        __syncwarp();
    }
    if (g.beside) cudaGridDependencySynchronize();
}

// CTAs of a pass: a static launch takes a warp per tile, a persistent one at most that and no more than fit (or
// ctas_per_sm)
inline int pass_grid(const ArgsFused &a, const void *kernel, int threads, int ctas_per_sm)
{
    const int all = (a.tile_end - a.tile_begin - a.skip_n + threads / 32 - 1) / (threads / 32);
    if (!a.counter) return all;
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, 0) != cudaSuccess || per < 1) per = 1;
    if (ctas_per_sm > 0 && ctas_per_sm < per) per = ctas_per_sm;
    per *= sms > 0 ? sms : 1;
    return per < all ? per : all;
}

// Launch of a pass.  One that runs beside the launch before it starts when the CTAs of that launch are all resident or
// done (they announce it at their start) and waits for its end before it ends itself, so that later work of the stream is
// ordered after both; nothing of the one is read by the other.
template <typename A>
cudaError_t launch_on(void (*kernel)(const A), const A &a, bool beside, int grid, int threads, cudaStream_t s)
{
    if (grid <= 0) return cudaSuccess;
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(grid);
    c.blockDim = dim3(threads);
    c.stream = s;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &at;
    c.numAttrs = beside ? 1 : 0;
    return cudaLaunchKernelEx(&c, kernel, a);
}

template <unsigned MASK, int MinB>
cudaError_t launch_pass(const ArgsFused &a, cudaStream_t s, int threads, int ctas_per_sm)
{
    const int grid = pass_grid(a, (const void *)k_2c_fp64_fused<MASK, MinB>, threads, ctas_per_sm);
    return launch_on(k_2c_fp64_fused<MASK, MinB>, a, a.beside, grid, threads, s);
}

}  // namespace
}  // namespace shg
