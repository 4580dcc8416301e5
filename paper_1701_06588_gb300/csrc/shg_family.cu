// Family basis sets (all shells of an element share one exponent set, as in
// the MOLOPT bases the paper measures): the radial terms G^{(k)} of Table S1
// depend on the primitive pair and the separation only, so for a group of
// shell pairs whose a-shells share one family on one center (and likewise
// for b) they are computed once per primitive pair, for every order the
// group needs, and each shell pair contracts them with its own weights,
//   O^{(k)}_{ab} = sum_{i,j} w_a[i] w_b[j] G^{(k)}[i][j],
//   w = N c (2 alpha)^{-l}                               (Eq. O_rab2_deriv),
// instead of recomputing the radial terms per shell pair.  One warp per
// group: G in shared memory, lanes over primitive pairs, then over (shell
// pair, order) items.  The angular part follows in the class-tiled kernel
// (OP_PRE).
#include "shg_xradial.cuh"

namespace shg {
namespace {
using namespace dev;
using namespace xfp;

constexpr int kFamWarps = 4;

// X_n = P q^n F_n(T), n = kmin..kmax, into G[n - kmin] (added, with the sign of (-1)^n times `sign`): the top order from the
// Boys head, the others by X_n = (-2R^2 X_{n+1} + P q^n exp(-T)) / (2n+1) (2T/q = -2R^2)
__device__ __forceinline__ void boys_orders(const ArgsFam &g, xf pre, xf q, xf T, double R2, int kmin, int kmax,
                                            uint32_t sign, double *G)
{
    xf F, e;
    xrad::boys_any(T, kmax, g.t, g.k.dfact[kmax], kmax > kmin, F, e);
    xf t = pre;
    if (kmin) t = mul(t, xfp::powi(q, kmin));
    double E[kFamOrd];
    for (int n = kmin; n < kmax; ++n) {
        E[n - kmin] = to_double(mul(t, e), xrad::order_sign(sign, n));
        t = mul(t, q);
    }
    double x = to_double(mul(t, F), xrad::order_sign(sign, kmax));
    G[kmax - kmin] += x;
    const double m2R2 = -2.0 * R2;
    for (int n = kmax - 1; n >= kmin; --n) {
        x = fma(m2R2, x, E[n - kmin]) * g.k.inv_int[2 * n + 1];
        G[n - kmin] += x;
    }
}

// Unit-weight radial terms G[k - kmin] = (0_a|O|0_b)^{(k)}, k = kmin..kmax, of one primitive pair, in extended floats up
// to the recursion (as shg_xradial.cuh; the FP64 form took 0.27 of the 0.53 ms of a 300-atom pass)
template <int OP>
__device__ __forceinline__ void radial_all(xf a, xf b, double R2, int kmin, int kmax, const ArgsFam &g, double *G)
{
    const xf rc = xfp::rsqrt(add(a, b)), ic = mul(rc, rc), ab = mulr(a, b);
    const xf rho = muln(ab, ic);
    const xf T = mul(rho, from_double(R2));
    if (OP == OP_OVERLAP || OP == OP_GAUSS) {
        xf t = mul(ic, rc), f = rho;
        double c = kPi32;
        if (OP == OP_OVERLAP) {
            t = mul(t, xrad::exp_neg(T, g.t.exp));
        } else {
            const xf w = {g.omega.w_m, g.omega.w_e};
            const xf rd = xfp::rsqrt(add(rho, w)), id = mul(rd, rd), wd = mul(w, id);
            f = mul(rho, wd);
            t = mul(mul(t, mul(id, rd)), xrad::exp_neg(mul(T, wd), g.t.exp));
            c = kPi3;
        }
        if (kmin) t = mul(t, xfp::powi(f, kmin));
        for (int k = kmin; k <= kmax; ++k) {
            G[k - kmin] = c * to_double(t, xrad::order_sign(0, k));
            t = mul(t, f);
        }
        return;
    }
    if (OP == OP_GCOUL) {
        // (pi/c)^{3/2} (2 pi/d) exp(-w T/d) (-rho)^k sum_i C(k,i) (w/d)^{k-i} (rho/d)^i F_i(T rho/d)
        const xf w = {g.omega.w_m, g.omega.w_e};
        const xf rd = xfp::rsqrt(add(rho, w)), id = mul(rd, rd), sw = mul(w, id), sr = mul(rho, id);
        xf T2 = mul(T, sr), F[kBoysOrders], e;
        xrad::boys_any(T2, kmax, g.t, g.k.dfact[kmax], true, F[kmax], e);
        T2.e += 1;
        for (int n = kmax; n > 0; --n) F[n - 1] = mul(add(mul(T2, F[n]), e), from_double(g.k.inv_int[2 * n - 1]));
        xf pre = mul(mul(mul(ic, rc), id), xrad::exp_neg(mul(T, sw), g.t.exp));
        for (int k = 0; k <= kmax; ++k) {
            if (k >= kmin) G[k - kmin] = kTwoPi52 * to_double(mul(pre, F[0]), xrad::order_sign(0, k));
            for (int i = 0; i < kmax - k; ++i) F[i] = add(mul(sw, F[i]), mul(sr, F[i + 1]));
            pre = mul(pre, rho);
        }
        return;
    }
    // 2 pi^{5/2} / (alpha beta sqrt(c)): 1 / (alpha beta) = 1 / (c rho)
    const xf rr = xfp::rsqrt(rho);
    const xf pre = mul(mul(mul(rr, rr), mul(ic, rc)), from_double(kTwoPi52));
    for (int k = kmin; k <= kmax; ++k) G[k - kmin] = 0.0;
    if (OP == OP_COULOMB || OP == OP_ERFC) boys_orders(g, pre, rho, T, R2, kmin, kmax, 0, G);
    if (OP == OP_ERF || OP == OP_ERFC) {
        const xf w = {g.omega.w_m, g.omega.w_e}, w2 = {g.omega.w2_m, g.omega.w2_e};
        const xf u = mul(w, xfp::rsqrt(add(rho, w2))), s = mul(u, u);
        boys_orders(g, mul(pre, u), mul(rho, s), mul(s, T), R2, kmin, kmax, OP == OP_ERFC ? 0x80000000u : 0u, G);
    }
}

template <int OP>
__global__ void __launch_bounds__(32 * kFamWarps) k_family_radial(const ArgsFam g)
{
    __shared__ double Gs[kFamWarps][kFamOrd * kFamPP];
    __shared__ int Js[kFamWarps][33];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    double *gs = Gs[w];
    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(g.counter, 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= g.n_groups) break;
        const FamGroup gr = g.groups[t];
        const Vec4 A = g.centers[gr.ca], B = g.centers[gr.cb];
        const double vx = A.x - B.x, vy = A.y - B.y, vz = A.z - B.z;
        const double R2 = vx * vx + vy * vy + vz * vz;
        const int npp = gr.fa_k * gr.fb_k;
        for (int ij = lane; ij < npp; ij += 32) {
            const int i = ij / gr.fb_k, j = ij - i * gr.fb_k;
            const XPrim pa = g.xprims[gr.fa_prim + i], pb = g.xprims[gr.fb_prim + j];
            double G[kFamOrd];
            radial_all<OP>(xf{pa.am, pa.ae}, xf{pb.am, pb.ae}, R2, gr.kmin, gr.kmax, g, G);
            for (int k = gr.kmin; k <= gr.kmax; ++k) gs[(k - gr.kmin) * kFamPP + ij] = G[k - gr.kmin];
        }
        __syncwarp();
        // contraction: lanes over (shell pair, order) items, 32 shell pairs at a
        // time; item it belongs to the pair r with js[r] <= it < js[r + 1]
        int *js = Js[w];
        for (int q0 = 0; q0 < gr.count; q0 += 32) {
            int Jq = 0;
            if (q0 + lane < gr.count) {
                const int p = gr.start + q0 + lane;
                const int la = g.shells[g.pair_a[p]].l, lb = g.shells[g.pair_b[p]].l;
                Jq = (la < lb ? la : lb) + 1;
            }
            int inc = Jq;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += v;
            }
            js[lane + 1] = inc;
            if (lane == 0) js[0] = 0;
            const int total = __shfl_sync(0xffffffffu, inc, 31);
            __syncwarp();
            for (int it = lane; it < total; it += 32) {
                int r = 0;
#pragma unroll
                for (int step = 16; step >= 1; step >>= 1)
                    if (js[r + step] <= it) r += step;
                const int tj = it - js[r];
                const int p = gr.start + q0 + r;      // the subset is stored in group order
                const ShellRec sa = g.shells[g.pair_a[p]], sb = g.shells[g.pair_b[p]];
                const int kmax = sa.l + sb.l;
                const double *gk = gs + (kmax - tj - gr.kmin) * kFamPP;
                double s = 0.0;
                for (int i = 0; i < gr.fa_k; ++i) {
                    double si = 0.0;
                    for (int j = 0; j < gr.fb_k; ++j) si = fma(g.prims[sb.prim_off + j].w2c, gk[i * gr.fb_k + j], si);
                    s = fma(g.prims[sa.prim_off + i].w2c, si, s);
                }
                g.o_pre[(int64_t)p * kJmax + tj] = s;
            }
            __syncwarp();
        }
    }
}

__global__ void k_gather_i64(const int64_t *__restrict__ src, const int32_t *__restrict__ idx, int64_t n,
                             int64_t *__restrict__ dst)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = src[idx[i]];
}

template <int OP>
cudaError_t launch_fam(const ArgsFam &a, cudaStream_t s)
{
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_family_radial<OP>, 32 * kFamWarps, 0) != cudaSuccess ||
        per < 1)
        per = 1;
    k_family_radial<OP><<<sms * per, 32 * kFamWarps, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_family_radial(const ArgsFam &a, int op, cudaStream_t s)
{
    if (a.n_groups <= 0) return cudaSuccess;
    switch (op) {
    case OP_OVERLAP: return launch_fam<OP_OVERLAP>(a, s);
    case OP_COULOMB: return launch_fam<OP_COULOMB>(a, s);
    case OP_ERFC: return launch_fam<OP_ERFC>(a, s);
    case OP_ERF: return launch_fam<OP_ERF>(a, s);
    case OP_GAUSS: return launch_fam<OP_GAUSS>(a, s);
    case OP_GCOUL: return launch_fam<OP_GCOUL>(a, s);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_gather_i64(const int64_t *src, const int32_t *idx, int64_t n, int64_t *dst, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    const int64_t blocks = (n + 255) / 256;
    k_gather_i64<<<(int)(blocks < 4096 ? blocks : 4096), 256, 0, s>>>(src, idx, n, dst);
    return cudaGetLastError();
}

}  // namespace shg
