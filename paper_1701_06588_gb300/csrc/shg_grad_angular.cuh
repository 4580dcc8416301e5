// Angular part of the two-center vector-Jacobian product (Sec. II E, Eq. dev_ab), from the expanded product of the solid
// harmonics (shg_cg.cuh): with the upstream weights W projected onto the expansion,
//   A_{L,M} = sum_{ma,mb} c W[ma][mb]        (J multiply-adds per element and |M|, cosine and sine parts),
// the scalar sum W (a|O|b) is sum_{L,M} A_{L,M} S_{L,M}(R) F_p(R^2), and its gradient
//   sum A_{L,M} (F_p grad S_{L,M} + 2 R F_p' S_{L,M}).
// With S_{L,M} = p_{L,M}(z, q) {C_M, S_M}(x, y), q = R^2:
//   dp/dq (z fixed) = -(L-M)(L-M-1) / (2 (2L-1)) p_{L-1,M+1},   dp/dz (x, y fixed) = (L-M)(L+M) / (2L-1) p_{L-1,M},
//   d(C_M + i S_M) = M (C_{M-1} + i S_{M-1}) (dx + i dy).
// The cost per element is J + 1 multiply-adds; the translation-matrix form took 2 J^2 and six rows of dW per function.
//
// The arithmetic is a parameter: FP64 (NumD) or double-float on the FP32 pipes (NumF, for the mixed-precision passes,
// operands scaled as in shg_cg_mix.cuh).
#pragma once

#include "shg_cg_mix.cuh"

namespace shg {
namespace gradang {

struct NumD {
    using T = double;
    using C = double;
    static __device__ __forceinline__ T zero() { return 0.0; }
    static __device__ __forceinline__ T one() { return 1.0; }
    static __device__ __forceinline__ T mul(T a, T b) { return a * b; }
    static __device__ __forceinline__ T add(T a, T b) { return a + b; }
    static __device__ __forceinline__ T sub(T a, T b) { return a - b; }
    static __device__ __forceinline__ T fma(T a, T b, T c) { return ::fma(a, b, c); }
    static __device__ __forceinline__ T fnma(T a, T b, T c) { return ::fma(-a, b, c); }
    static __device__ __forceinline__ T smul(float n, T a) { return (double)n * a; }       // exact small n
    static __device__ __forceinline__ T ld(const C *p) { return __ldg(p); }
};

struct NumF {
    using T = dfm::df;
    using C = float2;
    static __device__ __forceinline__ T zero() { return dfm::df_f(0.0f); }
    static __device__ __forceinline__ T one() { return dfm::df_f(1.0f); }
    static __device__ __forceinline__ T mul(T a, T b) { return dfm::mul(a, b); }
    static __device__ __forceinline__ T add(T a, T b) { return dfm::add(a, b); }
    static __device__ __forceinline__ T sub(T a, T b) { return dfm::sub(a, b); }
    static __device__ __forceinline__ T fma(T a, T b, T c) { return dfm::add(dfm::mul(a, b), c); }
    static __device__ __forceinline__ T fnma(T a, T b, T c) { return dfm::sub(c, dfm::mul(a, b)); }
    static __device__ __forceinline__ T smul(float n, T a) { return dfm::mul_f(a, n); }
    static __device__ __forceinline__ T ld(const C *p) { return cgm::ldf(__ldg(p)); }
};

// kappa of (l, M) and 1/n in the arithmetic
struct KapD {
    const Consts &k;
    __device__ __forceinline__ double operator()(int l, int M) const { return k.kappa[l][M]; }
    __device__ __forceinline__ double inv(int n) const { return k.inv_int[n]; }
};
struct KapF {
    const KappaMix &k;
    __device__ __forceinline__ dfm::df operator()(int l, int M) const { return cgm::ldf(k.v[l][M]); }
    __device__ __forceinline__ dfm::df inv(int n) const { return cgm::ldf(k.inv[n]); }
};

// F_p and F_p' = dF_p / dq from Q[j] = O^{(la+lb+1-j)}, j = 0..J; fc: coefficients of the class
template <int J>
__device__ __forceinline__ void laplace_orders_d(const double *__restrict__ fc, double q, const double (&Q)[J + 1],
                                                 double (&F)[J], double (&D)[J])
{
#pragma unroll
    for (int p = 0; p < J; ++p) {
        double f = 0.0, d = 0.0, e = 0.0;                      // Horner in q: value, derivative of the powers, next orders
#pragma unroll
        for (int j = 0; j <= p; ++j) {
            const double c = __ldg(fc + p * (p + 1) / 2 + j);
            d = fma(d, q, f);
            f = fma(f, q, c * Q[j + 1]);
            e = fma(e, q, c * Q[j]);
        }
        F[p] = f;
        D[p] = d + e;
    }
}

// A_{L,M}: cosine part at Ac[M * J + p], sine part at As, over the element sets gl, gl + group, .. of the pair;
// weight(i): W of element i of the block
template <class N, class Weight>
__device__ __forceinline__ void project(const typename N::C *__restrict__ g, int la, int lb, int J, int gl, int group,
                                        const Weight &weight, typename N::T *Ac, typename N::T *As)
{
    using T = typename N::T;
    const int nb = 2 * lb + 1, kmax = la + lb, c0 = la * nb + lb;
    for (int i = 0; i < (kmax + 1) * J; ++i) Ac[i] = As[i] = N::zero();
    for (int i = gl; i < (la + 1) * (lb + 1); i += group) {
        const int a = i / (lb + 1), b = i - a * (lb + 1);
        const typename N::C *gi = g + i * 2 * J;
        const int m1 = a > b ? a - b : b - a, m2 = a + b;
        const int n1 = min(J, (kmax - m1) / 2 + 1);
        const T cc = weight(c0 + a * nb + b);
        T u = cc, v = N::zero();
        if (a && b) {
            const T ss = weight(c0 - a * nb - b), sc = weight(c0 - a * nb + b), cs = weight(c0 + a * nb - b);
            const int n2 = min(J, (kmax - m2) / 2 + 1);
            const T u2 = N::sub(cc, ss), v2 = N::add(sc, cs);
            for (int p = 0; p < n2; ++p) {
                const T w = N::ld(gi + J + p);
                Ac[m2 * J + p] = N::fma(w, u2, Ac[m2 * J + p]);
                As[m2 * J + p] = N::fma(w, v2, As[m2 * J + p]);
            }
            u = N::add(cc, ss);
            v = a > b ? N::sub(sc, cs) : N::sub(cs, sc);
        } else if (m1) {
            v = weight(a ? c0 - a * nb : c0 - b);
        }
        for (int p = 0; p < n1; ++p) {
            const T w = N::ld(gi + p);
            Ac[m1 * J + p] = N::fma(w, u, Ac[m1 * J + p]);
            if (m1) As[m1 * J + p] = N::fma(w, v, As[m1 * J + p]);
        }
    }
}

// gradient of sum_{L,M} A_{L,M} S_{L,M} F_p: G = (dx, dy, dz).  P, R: work arrays of (kmax + 1) J entries
template <class N, int J, class Kap>
__device__ __forceinline__ void contract(typename N::T x, typename N::T y, typename N::T z, typename N::T q, int kmax,
                                         const Kap &kap, const typename N::T (&F)[J], const typename N::T (&D)[J],
                                         const typename N::T *Ac, const typename N::T *As, typename N::T *P,
                                         typename N::T *R, typename N::T (&G)[3])
{
    using T = typename N::T;
    // p_{L,M} at P[M J + p] and p_{L-1,M} at R[M J + p], L = kmax - 2p
    for (int M = 0; M <= kmax; ++M) {
        T p0 = N::zero(), p1 = N::one();
        for (int l = M;; ++l) {
            const int d = kmax - l, p = d >> 1;
            if (p < J) {
                if (d & 1) R[M * J + p] = p1;
                else P[M * J + p] = p1;
            }
            if (l == kmax) break;
            T n = N::mul(z, p1);
            if (l > M) n = N::fnma(N::mul(kap(l, M), q), p0, n);
            p0 = p1;
            p1 = n;
        }
    }
    const T z2 = N::smul(2.0f, z);
    T U = N::zero(), Z = N::zero(), X = N::zero(), Y = N::zero();
    T c = N::one(), s = N::zero(), c1 = N::zero(), s1 = N::zero();         // C_M, S_M and C_{M-1}, S_{M-1}
    for (int M = 0; M <= kmax; ++M) {
        T ac = N::zero(), as = N::zero(), bc = N::zero(), bs = N::zero(), dc = N::zero(), ds = N::zero();
#pragma unroll
        for (int p = 0; p < J; ++p) {
            const int L = kmax - 2 * p;
            if (L < M) continue;
            const T pl = P[M * J + p], wa = Ac[M * J + p], ws = As[M * J + p];
            const T f = N::mul(F[p], pl), dp = N::mul(D[p], pl);
            T b = dp, d = N::mul(z2, dp);
            if (L > M) {
                // F_p over 2L - 1, times the integer factors
                const T h = N::mul(F[p], kap.inv(2 * L - 1));
                d = N::fma(N::smul((float)((L - M) * (L + M)), h), R[M * J + p], d);
                if (L > M + 1) b = N::fnma(N::smul(0.5f * (float)((L - M) * (L - M - 1)), h), R[(M + 1) * J + p], b);
            }
            ac = N::fma(f, wa, ac);
            as = N::fma(f, ws, as);
            bc = N::fma(b, wa, bc);
            bs = N::fma(b, ws, bs);
            dc = N::fma(d, wa, dc);
            ds = N::fma(d, ws, ds);
        }
        U = N::fma(c, bc, N::fma(s, bs, U));
        Z = N::fma(c, dc, N::fma(s, ds, Z));
        if (M) {
            const T n = N::smul((float)M, ac), m = N::smul((float)M, as);
            X = N::fma(c1, n, N::fma(s1, m, X));
            Y = N::fma(c1, m, N::fnma(s1, n, Y));
        }
        c1 = c;
        s1 = s;
        c = N::fnma(y, s1, N::mul(x, c1));
        s = N::fma(y, c1, N::mul(x, s1));
    }
    G[0] = N::fma(N::smul(2.0f, x), U, X);
    G[1] = N::fma(N::smul(2.0f, y), U, Y);
    G[2] = Z;
}

}  // namespace gradang
}  // namespace shg
