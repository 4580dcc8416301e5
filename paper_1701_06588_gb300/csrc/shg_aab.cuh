// Three-index overlaps (a b a~), a and a~ on center A, b on center B, by the SHG scheme of Sec. II D (arXiv:1701.06588):
// shared parts of the integral and the gradient kernel.
//
// The product of the two functions on A is expanded in solid harmonics, S_{la,ma} S_{lt,mt} = sum_{L,M} c r^{2p} S_{L,M},
// L = la+lt, la+lt-2, .., |la-lt|, p = (la+lt-L)/2 (Eq. product_SHG_STGO); each L is a two-center block of a shell
// (L, alpha' = alpha + alpha~) times r_a^{2p} with b, whose radial orders P_L^{(k)} (Eq. Pa_aba) contract
// binom(p,j) (L)_j alpha'^{-j} (0_a'|r_a^{2(p-j)}|0_b)^{(k)} over the primitive triples and whose angular part is the
// expansion of shg_cg.cuh once more, for the class (L, lb).
//
// Work mapping: eight lanes per triple (four triples per warp, one warp per CTA), everything between the phases in
// shared memory: the lanes share the primitive triples, then the columns of the harmonics, the (|M|, |mb|) sets of
// the blocks and the (|ma|, |mt|) sets of the result.  With one thread per triple, 15 KB of arrays per thread went
// through L1 and L2 to DRAM (22 times the output), and a triple of 300 primitive combinations ran alone at the end.
#pragma once

#include "shg_cg.cuh"
#include "shg_xradial.cuh"

namespace shg {
namespace aab {
using namespace xfp;

constexpr int kLanes = 8;                          // lanes per triple
constexpr int kSlots = 32 / kLanes;

// Sizes of one (la, lt, lb) class
struct Shape {
    int la, lt, lb, Lmin, Lmax, nL, kmax;          // kmax = Lmax + lb
    __host__ __device__ constexpr Shape(int cls)
        : la(cls / 49), lt(cls / 7 % 7), lb(cls % 7), Lmin(la > lt ? la - lt : lt - la), Lmax(la + lt),
          nL((Lmax - Lmin) / 2 + 1), kmax(Lmax + lb)
    {
    }
    __host__ __device__ constexpr int L(int i) const { return Lmin + 2 * i; }
    __host__ __device__ constexpr int J(int i) const { return (L(i) < lb ? L(i) : lb) + 1; }
    // first (L, q) entry, first (L, M', q) entry (M' = 0..L+lb) and first (L, M) entry of L(i)
    __host__ __device__ constexpr int qbase(int i) const
    {
        int n = 0;
        for (int j = 0; j < i; ++j) n += J(j);
        return n;
    }
    __host__ __device__ constexpr int pbase(int i) const
    {
        int n = 0;
        for (int j = 0; j < i; ++j) n += (L(j) + lb + 1) * J(j);
        return n;
    }
    __host__ __device__ constexpr int mbase(int i) const
    {
        int n = 0;
        for (int j = 0; j < i; ++j) n += 2 * L(j) + 1;
        return n;
    }
};

// pi^{3/2} over the constants (2 pi^{5/2})^{1/2} of the three weights
constexpr double kWeight = dev::kPi32 / (dev::kTwoPi52 * 5.914967172795613);

// First primitive combination of a lane that sums none
constexpr int kNone = 1 << 30;

// Radial orders of one triple, summed over the primitive combinations first, first + 8, ..: P_L^{(L + lb + X - j)} of L(i),
// j = 0 .. min(L, lb) + X (X = 1 for gradients), at part[v * 8] with v counting (i, j).  Per combination
//   P_L^{(k)} += W (2 alpha')^{-L} (-rho)^k sum_o binom(k,o) r_o,
//   r_o = (-tau)^o sum_{m=o}^{p} K_{L,m} alpha'^{m-p} c^{-m} Lag_{m-o}^{(1/2+o)}(-u),    tau = beta/alpha', u = beta^2 R^2/c,
// K_{L,m} = binom(p,m) (L)_{p-m} m!, since d^o/du^o of the polynomial of (0|r_a^{2m}|0) (Eq. I_jab) is 2^m m! times that
// Laguerre polynomial; all terms of r_o are positive, and the polynomials of one combination follow from row o = 0 by one
// addition each.  About half the FP64 operations of summing (0|r_a^{2m}|0)^{(k)} order by order; the prefactors are
// extended floats on the integer pipes.  NP = number of L (min(la, la~) + 1): the polynomials stay in registers, the sums
// over the combinations in shared memory (an FP64 instruction holds its unit for 64 cycles, so the access beside it is
// free).  900,000 triples: 11.2 ms whole call; sums in registers (168 of them, warps waiting for instructions in 41% of
// their cycles) 13.4 ms, runtime loops over local arrays 12.3 ms.
template <int NP>
__device__ __forceinline__ void radial(const Args3c &g, const Shape &sh, int X, const ShellRec &sa, const ShellRec &st,
                                       const ShellRec &sb, double R2, int first, double *part)
{
    constexpr int nL = NP;
    const int Lmin = sh.Lmin, lb = sh.lb;
    const int nq = sh.qbase(nL) + X * nL;
    for (int v = 0; v < nq; ++v) part[v * kLanes] = 0.0;
    const int Kb = sb.nprim, Kt = st.nprim, n = sa.nprim * Kt * Kb;
    const float rKb = 1.0f / (float)Kb, rKt = 1.0f / (float)Kt;
    const xf R2x = from_double(R2);
    const int k0 = Lmin > lb ? Lmin : lb;                       // lowest order of Lmin
    for (int q = first; q < n; q += kLanes) {
        const int at = (int)(((float)q + 0.5f) * rKb), ib = q - at * Kb;     // exact: q < 2^15, K <= 32
        const int ia = (int)(((float)at + 0.5f) * rKt), it = at - ia * Kt;
        const XPrim A = g.orb_prims[sa.prim_off + ia], T = g.orb_prims[st.prim_off + it], B = g.aux_prims[sb.prim_off + ib];
        const xf al = {A.am, A.ae}, at_ = {T.am, T.ae}, be = {B.am, B.ae};
        const xf ap = add(al, at_);
        const xf rap = xfp::rsqrt(ap), iap = mul(rap, rap);
        const xf rc = xfp::rsqrt(add(ap, be)), ic = mul(rc, rc);
        const xf bic = mul(be, ic);
        const xf rho = mul(ap, bic);
        // N c = cw alpha (2 alpha)^l and N c / (2 beta)^lb = cw beta up to the constant of cw (kWeight)
        const uint32_t sw = hi32(A.wm) ^ hi32(T.wm) ^ hi32(B.wm);
        constexpr uint64_t mask = ~(1ull << 63);
        xf w = muln(mulr(xf{A.wm & mask, A.we}, xf{T.wm & mask, T.we}), xf{B.wm & mask, B.we});
        w = mul(w, muln(mulr(al, at_), be));
        if (sa.l) w = mul(w, xfp::powi(xf{al.m, al.e + 1}, sa.l));
        if (st.l) w = mul(w, xfp::powi(xf{at_.m, at_.e + 1}, st.l));
        w = mul(mul(w, mul(ic, rc)), xrad::exp_neg(mul(rho, R2x), g.exptab));
        if (Lmin) w = mul(w, xfp::powi(xf{iap.m, iap.e - 1}, Lmin));
        if (k0) w = mul(w, xfp::powi(rho, k0));
        double e = to_double(w, sw ^ ((uint32_t)k0 << 31));     // W (2 alpha')^{-Lmin} (-rho)^{k0}
        const double mrho = -to_double(rho, 0);
        double pa[nL], pc[nL], tp[nL], lam[nL][nL];
        pa[0] = pc[0] = tp[0] = 1.0;
        lam[0][0] = 1.0;
        double s2 = 0.0;
        if (nL > 1) {
            const double ia1 = to_double(iap, 0), c1 = to_double(ic, 0), mtau = -to_double(mul(be, iap), 0);
            const double u = to_double(mul(mul(be, bic), R2x), 0);
            s2 = 0.25 * ia1 * ia1;                              // (2 alpha')^{-2}
            pa[nL > 1 ? 1 : 0] = ia1;
            pc[nL > 1 ? 1 : 0] = c1;
            tp[nL > 1 ? 1 : 0] = mtau;
            lam[0][nL > 1 ? 1 : 0] = u + 1.5;
            lam[nL > 1 ? 1 : 0][0] = 1.0;
#pragma unroll
            for (int m = 2; m < nL; ++m) {
                pa[m] = pa[m - 1] * ia1;
                pc[m] = pc[m - 1] * c1;
                tp[m] = tp[m - 1] * mtau;
                double s = g.k3.lag[m][m];
#pragma unroll
                for (int j = m - 1; j >= 0; --j) s = fma(s, u, g.k3.lag[m][j]);
                lam[0][m] = s;
                // Lag_n^{(a+1)} = Lag_n^{(a)} + Lag_{n-1}^{(a+1)}
#pragma unroll
                for (int o = 1; o < m; ++o) lam[o][m - o] = lam[o - 1][m - o] + lam[o][m - o - 1];
                lam[m][0] = 1.0;
            }
        }
        double *acc = part;
#pragma unroll
        for (int i = 0; i < nL; ++i) {
            const int L = Lmin + 2 * i, p = nL - 1 - i, kl = L > lb ? L : lb, J = (L < lb ? L : lb) + 1 + X;
            double bm[nL], r[nL];
            const double *K = g.k3.K[L][p];
#pragma unroll
            for (int m = 0; m <= p; ++m) bm[m] = K[m] * (pa[p - m] * pc[m]);
            r[0] = bm[0];
#pragma unroll
            for (int m = 1; m <= p; ++m) r[0] = fma(bm[m], lam[0][m], r[0]);
#pragma unroll
            for (int o = 1; o <= p; ++o) {
                double s = bm[o];
#pragma unroll
                for (int m = o + 1; m <= p; ++m) s = fma(bm[m], lam[o][m - o], s);
                r[o] = s * tp[o];
            }
            double f = e;
#pragma unroll 1
            for (int j = J - 1; j >= 0; --j) {
                const double *bn = g.k3.binom[kl + J - 1 - j];
                double s = r[0];
#pragma unroll
                for (int o = 1; o <= p; ++o) s = fma(bn[o], r[o], s);
                acc[j * kLanes] = fma(f, s, acc[j * kLanes]);
                if (j) f *= mrho;
            }
            acc += J * kLanes;
            if (i + 1 < nL) {
                // next L: (2 alpha')^{-2} and the step of its lowest order
                const int d = (L + 2 > lb ? L + 2 : lb) - kl;
                e *= s2;
                if (d) e *= mrho;
                if (d == 2) e *= mrho;
            }
        }
    }
}

// the lanes' sums added up: sum[v] over part[v * 8 ..]
__device__ __forceinline__ void reduce(int nq, int gl, const double *part, double *sum)
{
    __syncwarp();
    for (int v = gl; v < nq; v += kLanes) {
        double s = 0.0;
        for (int l = 0; l < kLanes; ++l) s += part[v * kLanes + l];
        sum[v] = s * kWeight;
    }
    __syncwarp();
}

// C_M, S_M for M = 0..kmax by the lanes of a slot
__device__ __forceinline__ void circular(double x, double y, int kmax, int gl, double *C, double *S)
{
    double c = 1.0, s = 0.0;
    for (int m = 0; m <= kmax; ++m) {
        if ((m & (kLanes - 1)) == gl) {
            C[m] = c;
            S[m] = s;
        }
        const double t = x * c - y * s;
        s = x * s + y * c;
        c = t;
    }
}

// Dynamic shared memory that every kernel may take without raising its own limit.  That limit belongs to the function, not
// to a launch: a call that set it for its own list could lower it between another thread's setting and launch.  The largest
// class takes 20,160 bytes (integrals) and 43,456 bytes (gradients).
constexpr size_t kSharedLimit = 48 << 10;

// bytes of a warp's slots, the largest over the valid classes (la + la~ <= kLmaxAabA)
template <class Doubles>
constexpr size_t largest_slots(Doubles doubles)
{
    int most = 0;
    for (int cls = 0; cls < kNClass3; ++cls) {
        const Shape s(cls);
        if (s.Lmax <= kLmaxAabA && doubles(s) > most) most = doubles(s);
    }
    return kSlots * sizeof(double) * (size_t)most;
}

// Persistent launch of one-warp CTAs with the shared memory of four slots each
template <class Launch>
cudaError_t launch_slots(const void *kernel, const Args3c &a, Launch launch)
{
    const size_t bytes = (size_t)kSlots * a.slot_doubles * sizeof(double);
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, 32, bytes);
    if (e != cudaSuccess) return e;
    launch((sms > 0 ? sms : 1) * (per > 0 ? per : 1), bytes);
    return cudaGetLastError();
}

}  // namespace aab
}  // namespace shg
