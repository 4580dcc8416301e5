// Contracted radial orders of one shell pair (Table S1, Eq. O_rab2_deriv) in extended-float arithmetic (shg_xf.cuh).
//
// One near 1/r-type primitive pair took about 25 FP64 instructions (an inverse square root, the Boys head, the
// products of weights), each of which holds the FP64 unit of a sub-partition for 64 cycles; as integer operations the
// same work is about 250 issue cycles, and only the sums over the primitive pairs stay on the FP64 unit (one addition
// per order), which runs beside the integer pipes.  Every product carries 59 bits and more, so the primitive terms are
// rounded to FP64 once, where the FP64 form accumulated ten to twenty roundings.
//
// 1/r-type operators use the contracted downward recursion: per primitive pair only the top order and the exp(-T')
// terms E_j are summed, X_n = (-2 R^2 X_{n+1} + P q^n exp(-T')) / (2n+1) is applied once to the sums (the two terms
// of a step have one sign for every primitive pair).
#pragma once

#include "shg_device.cuh"
#include "shg_xf.cuh"

#ifdef SHG_XF_CALLS
#define SHG_XF_DEV static __device__ __noinline__
#else
#define SHG_XF_DEV __device__ __forceinline__
#endif

namespace shg {
namespace xrad {
using namespace xfp;

// exp(-T) for T < 1024 (2^-1477 and below: a value the conversion to FP64 flushes to 0).  n = ceil(T log2 e) or one more,
// r = n ln2 - T in [0, 0.6932), exp(r) from a table at r_j = j/512 and the series of the rest.
SHG_XF_DEV xf exp_neg(xf T, const uint64_t *__restrict__ tab)
{
    if (T.e > -53) return xf{1ull << 62, -100000};
    const int s = -53 - T.e;                                                 // >= 0
    const uint32_t t21 = s < 32 ? hi32(T.m) >> s : 0u;                       // T 2^21
    const uint32_t n = (uint32_t)(((uint64_t)(t21 + 1u) * 3098164010u) >> 52) + 1u;     // log2(e) 2^31, rounded up
    const int sl = T.e + 62;                                                 // T 2^62 mod 2^64
    const uint64_t v = sl >= 0 ? T.m << sl : shr(T.m, -sl);
    const uint64_t r = (uint64_t)n * 3196577161300663915ull - v;             // ln2 2^62
    const uint64_t E = __ldg(tab + (r >> 53));                               // exp(r_j) 2^62
    const uint64_t z = expm1_small((r & 0x1fffffffffffffull) << 2);
    const uint64_t m = E + (mulhi(E, z) << 1);
    const int c = (int)(hi32(m) >> 31);                                      // exp(r) may reach 2
    return xf{m >> c, c - 62 - (int)n};
}

// T in units 2^-56; false for T >= kFarT (out of the table)
__device__ __forceinline__ bool boys_fixed(xf T, uint64_t &Tf)
{
    if (T.e > -56) return false;
    Tf = shr(T.m, -56 - T.e);
    return hi32(Tf) < ((uint32_t)kFarT << 24);
}

// F_n(T) from the table of order n (BoysEnt): Taylor series about the upper end of T's cell of width 1/512, all terms
// positive
SHG_XF_DEV xf boys_series(const BoysEnt *__restrict__ tab, uint64_t Tf)
{
    const uint32_t i = hi32(Tf) >> 15;
    const uint64_t Y = ~(Tf << 8) & 0x7fffffffffffffull;                     // (T_{i+1} - T) 2^64, less 1
    const uint32_t y = (uint32_t)(Y >> 23);                                  // 2^41
    uint64_t c0, c1, c2, c35;
    asm("ld.global.nc.v4.u64 {%0, %1, %2, %3}, [%4];" : "=l"(c0), "=l"(c1), "=l"(c2), "=l"(c35) : "l"(tab + i));
    const uint32_t c45 = hi32(c35);
    const uint32_t p4 = (c45 & 0xffffffu) + (uint32_t)(((uint64_t)y * (c45 >> 24)) >> 27);
    const uint32_t p3 = lo32(c35) + (uint32_t)(((uint64_t)y * p4) >> 36);
    const uint64_t p2 = c2 + (((uint64_t)y * p3) >> 11);
    const uint64_t p1 = c1 + mulhi(Y, p2);
    uint64_t m = c0 + mulhi(Y, p1);
    int e = -62 - (int)(lo32(c2) & 255u);
    if (!(hi32(m) >> 30)) {
        m += m;
        e -= 1;
    }
    return xf{m, e};
}

// F_n(T) and, with need_e, exp(-T) for any T; n runtime, dfn = (2n-1)!!
__device__ __forceinline__ void boys_any(xf T, int n, const XTab &t, double dfn, bool need_e, xf &F, xf &e)
{
    uint64_t Tf;
    if (boys_fixed(T, Tf)) {
        F = boys_series(t.boys + (size_t)n * kBoysCells, Tf);
        if (need_e) e = exp_neg(T, t.exp);
    } else {
        // (2n-1)!! (2T)^-n sqrt(pi / (4T)); exp(-T) < 1e-31 is dropped
        const xf rT = xfp::rsqrt(T);
        F = mul(mul(from_double(dfn), rT), from_double(dev::kSqrtPiHalf));
        if (n) {
            xf h = mul(rT, rT);
            h.e -= 1;
            F = mul(F, xfp::powi(h, n));
        }
        e = xf{1ull << 62, -100000};
    }
}

// Sums of one shell pair: order kmax - j at [j].  far: sum of the far-field weights of the 1/r sum (T >= kFarT)
template <int J>
struct Sums {
    double ov[J], co[J], er[J], x[J], ga[J], gc[J], far;
};

template <int J>
__device__ __forceinline__ void zero(double (&v)[J])
{
#pragma unroll
    for (int j = 0; j < J; ++j) v[j] = 0.0;
}

// sign word of order k: the weights' sign times (-1)^k (bit 31)
__device__ __forceinline__ uint32_t order_sign(uint32_t sw, int k) { return sw ^ ((uint32_t)k << 31); }

// attenuated part: X_k = pre u s^k (-rho)^k F_k(s T), s = omega^2 / (omega^2 + rho), u = sqrt(s); pre_k = pre rho^kmin
template <int J>
__device__ __forceinline__ void att_term(const XOmega &om, const xf &rho, const xf &T, const xf &prek, int kmax,
                                         uint32_t sw, const RadialIn &g, const Consts &k, double (&O)[J], double (&E)[J])
{
    const int kmin = kmax - J + 1;
    const xf w = {om.w_m, om.w_e}, w2 = {om.w2_m, om.w2_e};
    const xf rd = xfp::rsqrt(add(rho, w2));
    const xf u = mul(w, rd);
    const xf s = mul(u, u);
    xf t = mul(prek, u);
    if (kmin) t = mul(t, xfp::powi(s, kmin));
    xf F, e;
    boys_any(mul(s, T), kmax, g.t, k.dfact[kmax], J > 1, F, e);
    if (J > 1) {
        const xf q = mul(rho, s);
        xf te = mul(t, e);
#pragma unroll
        for (int j = J - 1; j >= 1; --j) {
            E[j] += to_double(te, order_sign(sw, kmax - j));
            if (j > 1) te = mul(te, q);
            t = mul(t, q);
        }
    }
    O[0] += to_double(mul(t, F), order_sign(sw, kmax));
}

// exp(-w r^2)/r: (pi/c)^{3/2} (2 pi/d) exp(-w T/d) (-rho)^k sum_i C(k,i) (w/d)^{k-i} (rho/d)^i F_i(T rho/d), d = rho + w:
// the binomial weights of a convex combination, applied as v_i <- (w/d) v_i + (rho/d) v_{i+1} k times.
template <int J>
__device__ __forceinline__ void gcoul_term(const RadialIn &g, const xf &ab, const xf &ic, const xf &rc, const xf &rho,
                                           const xf &T, const xf &ww, int kmax, uint32_t sw, const Consts &k,
                                           double (&O)[J])
{
    const int kmin = kmax - J + 1;
    const xf w = {g.gauss.w_m, g.gauss.w_e};
    const xf rd = xfp::rsqrt(add(rho, w));
    const xf id = mul(rd, rd);
    const xf sw_ = mul(w, id), sr = mul(rho, id);
    xf T2 = mul(T, sr);
    xf F[kBoysOrders], e;
    boys_any(T2, kmax, g.t, k.dfact[kmax], true, F[kmax], e);
    T2.e += 1;
    for (int n = kmax; n > 0; --n) F[n - 1] = mul(add(mul(T2, F[n]), e), from_double(k.inv_int[2 * n - 1]));
    xf pre = mul(mul(muln(ww, rc), muln(ab, ic)), mul(id, exp_neg(mul(T, sw_), g.t.exp)));
    if (kmin) pre = mul(pre, xfp::powi(rho, kmin));
    for (int m = 1; m <= kmin; ++m)
        for (int i = 0; i <= kmax - m; ++i) F[i] = add(mul(sw_, F[i]), mul(sr, F[i + 1]));
#pragma unroll
    for (int t = 0; t < J; ++t) {
        O[J - 1 - t] += to_double(mul(pre, F[0]), order_sign(sw, kmin + t));
        if (t + 1 < J) {
            for (int i = 0; i < J - 1 - t; ++i) F[i] = add(mul(sw_, F[i]), mul(sr, F[i + 1]));
            pre = mul(pre, rho);
        }
    }
}

template <int J>
__device__ __forceinline__ void finish(double m2R2, int kmax, const Consts &k, double (&O)[J], const double (&E)[J])
{
#pragma unroll
    for (int j = 1; j < J; ++j) O[j] = fma(m2R2, O[j - 1], E[j]) * k.inv_int[2 * (kmax - j) + 1];
}

// sum over the group of `group` consecutive lanes (a power of two), in every lane; all lanes of the warp call it
template <int J>
__device__ __forceinline__ void group_sum(double (&v)[J], int group)
{
    for (int o = 1; o < group; o <<= 1)
#pragma unroll
        for (int j = 0; j < J; ++j) v[j] += __shfl_xor_sync(0xffffffffu, v[j], o);
}

// Orders kmax - J + 1 .. kmax of every wanted sum.  MASK: the sums this instantiation holds accumulators for.  Lane gl of
// a group of `group` lanes takes the primitive pairs gl, gl + group, ..; every lane of the group returns the sums.  The
// whole warp calls this with one group size.
template <unsigned MASK, int J>
__device__ __forceinline__ void radial(const RadialIn &g, const ShellRec &sa, const ShellRec &sb, double R2, int kmax,
                                       const Consts &k, int gl, int group, Sums<J> &o)
{
    const int kmin = kmax - J + 1;
    const unsigned want = g.want & MASK;
    const bool f_co = want & kSumCo, f_er = want & kSumEr, f_x = want & kSumX, f_ov = want & kSumOv, f_ga = want & kSumGa;
    double Eco[J], Eer[J], Ex[J];
    zero(o.ov), zero(o.co), zero(o.er), zero(o.x), zero(o.ga), zero(o.gc);
    zero(Eco), zero(Eer), zero(Ex);
    o.far = 0.0;
    // R^2 = 0: any small value, T stays below 2^-1000
    const xf R2x = from_double(R2);
    const int Kb = sb.nprim, npp = sa.nprim * Kb;
    const XPrim *pa = g.prims + sa.prim_off, *pb = g.prims + sb.prim_off;
    const float rKb = 1.0f / (float)Kb;
    int last = -1;
    xf a, wa;
    uint32_t swa;
    double fwa;
    for (int q = gl; q < npp; q += group) {
        const int ia = (int)(((float)q + 0.5f) * rKb), ib = q - ia * Kb;    // exact: q < 1024, Kb <= 32
        if (ia != last) {
            last = ia;
            const XPrim A = pa[ia];
            a = xf{A.am, A.ae};
            wa = xf{A.wm & ~(1ull << 63), A.we};
            swa = hi32(A.wm);
            fwa = A.fw;
        }
        const XPrim B = pb[ib];
        const xf b = {B.am, B.ae};
        const xf rc = xfp::rsqrt(add(a, b));
        const xf ab = mulr(a, b);
        const xf ic = mul(rc, rc);
        const xf rho = muln(ab, ic);
        const xf T = mul(rho, R2x);
        const uint32_t sw = swa ^ hi32(B.wm);
        const xf ww = mulr(wa, xf{B.wm & ~(1ull << 63), B.we});              // 2 pi^{5/2} w / (alpha beta)
        xf eT;
        bool have_e = false;
        if ((MASK & (kSumCo | kSumEr | kSumX)) && (f_co || f_er || f_x)) {
            xf pre = muln(ww, rc);
            uint64_t Tf;
            const bool near = boys_fixed(T, Tf);
            if (kmin && (f_er || f_x || near)) pre = mul(pre, xfp::powi(rho, kmin));
            if ((MASK & kSumCo) && f_co) {
                if (near) {
                    xf t = pre;
                    if (J > 1) {
                        eT = exp_neg(T, g.t.exp);
                        have_e = true;
                        xf te = mul(t, eT);
#pragma unroll
                        for (int j = J - 1; j >= 1; --j) {
                            Eco[j] += to_double(te, order_sign(sw, kmax - j));
                            if (j > 1) te = mul(te, rho);
                            t = mul(t, rho);
                        }
                    }
                    const xf F = boys_series(g.t.boys + (size_t)kmax * kBoysCells, Tf);
                    o.co[0] += to_double(mul(t, F), order_sign(sw, kmax));
                } else {
                    o.far = fma(fwa, B.fw, o.far);
                }
            }
            if ((MASK & kSumEr) && f_er) att_term<J>(g.erf, rho, T, pre, kmax, sw, g, k, o.er, Eer);
            if ((MASK & kSumX) && f_x) att_term<J>(g.erfc, rho, T, pre, kmax, sw, g, k, o.x, Ex);
        }
        if (MASK & kSumGc) gcoul_term<J>(g, ab, ic, rc, rho, T, ww, kmax, sw, k, o.gc);
        if ((MASK & (kSumOv | kSumGa)) && (f_ov || f_ga)) {
            // w c^{-3/2}; the powers of pi are applied to the sums
            const xf w3 = mul(muln(ww, rc), muln(ab, ic));
            if ((MASK & kSumOv) && f_ov) {
                // (pi/c)^{3/2} exp(-T) (-rho)^k
                xf t = mul(w3, have_e ? eT : exp_neg(T, g.t.exp));
                if (kmin) t = mul(t, xfp::powi(rho, kmin));
#pragma unroll
                for (int j = J - 1; j >= 0; --j) {
                    o.ov[j] += to_double(t, order_sign(sw, kmax - j));
                    if (j) t = mul(t, rho);
                }
            }
            if ((MASK & kSumGa) && f_ga) {
                // (pi^2/(c (rho+w)))^{3/2} exp(-w T/(rho+w)) (-w rho/(rho+w))^k
                const xf w = {g.gauss.w_m, g.gauss.w_e};
                const xf rd = xfp::rsqrt(add(rho, w));
                const xf id = mul(rd, rd);
                const xf wd = mul(w, id);
                const xf f = mul(rho, wd);
                xf t = mul(mul(w3, mul(id, rd)), exp_neg(mul(T, wd), g.t.exp));
                if (kmin) t = mul(t, xfp::powi(f, kmin));
#pragma unroll
                for (int j = J - 1; j >= 0; --j) {
                    o.ga[j] += to_double(t, order_sign(sw, kmax - j));
                    if (j) t = mul(t, f);
                }
            }
        }
    }
    if (group > 1) {
        if (MASK & kSumOv) group_sum(o.ov, group);
        if (MASK & kSumGa) group_sum(o.ga, group);
        if (MASK & kSumGc) group_sum(o.gc, group);
        if (MASK & kSumCo) {
            group_sum(o.co, group);
            group_sum(Eco, group);
            for (int s = 1; s < group; s <<= 1) o.far += __shfl_xor_sync(0xffffffffu, o.far, s);
        }
        if (MASK & kSumEr) {
            group_sum(o.er, group);
            group_sum(Eer, group);
        }
        if (MASK & kSumX) {
            group_sum(o.x, group);
            group_sum(Ex, group);
        }
    }
    // ww carries 2 pi^{5/2}
    constexpr double c_ov = dev::kPi32 / dev::kTwoPi52, c_ga = dev::kPi3 / dev::kTwoPi52;
#pragma unroll
    for (int j = 0; j < J; ++j) {
        o.ov[j] *= c_ov;
        o.ga[j] *= c_ga;
    }
    const double m2R2 = -2.0 * R2;
    if (MASK & kSumCo) finish<J>(m2R2, kmax, k, o.co, Eco);
    if (MASK & kSumEr) finish<J>(m2R2, kmax, k, o.er, Eer);
    if (MASK & kSumX) finish<J>(m2R2, kmax, k, o.x, Ex);
}

// Far-field order n = kmax of the 1/r sum: pi^3 (-1)^n (2n-1)!! (2R^2)^{-n} / R times the far weights (R > 0).  The far
// field of 1/r is harmonic, so only the top order enters a block (F_p with p >= 1 vanishes for it).
__device__ __forceinline__ double far_order(double far, double R2, int n, const Consts &k)
{
    if (far == 0.0) return 0.0;
    const double ir = ::rsqrt(R2);
    return far * dev::kPi3 * ir * k.dfact[n] * dev::powi(-0.5 * ir * ir, n);
}

}  // namespace xrad
}  // namespace shg
