// The expanded angular part (shg_cg.cuh) in double-float arithmetic on the FP32 pipes, for the mixed-precision passes.
// Range: the separation is scaled by a power of two to 1 <= |R| < 2 (each F_p takes the factor back), the F_p by a
// power of two to at most 2, so everything stays near 1 in FP32 whatever the exponents; the scale returns with the
// conversion of an element to FP64.
#pragma once

#include "shg_cg.cuh"
#include "shg_df.cuh"

namespace shg {
namespace cgm {
using namespace dfm;

constexpr int kMixMaxL = kLmax2c + kMixedFp64MinL - 1;      // largest la + lb of a mixed-precision class (J <= kMixedFp64MinL)

__device__ __forceinline__ df ldf(float2 v) { return df{v.x, v.y}; }

__device__ __forceinline__ df split(double v)
{
    const float hi = __double2float_rn(v);
    return df{hi, __double2float_rn(v - (double)hi)};
}

__device__ __forceinline__ int exponent(double v) { return (int)((__double2hiint(v) >> 20) & 0x7ff) - 1023; }

// v 2^e for normal v and a result in the normal range; 0 below it and for v = 0, infinity
// above; infinities and NaN unchanged
__device__ __forceinline__ double scale_exp(double v, int e)
{
    const int hi = __double2hiint(v), f = (hi >> 20) & 0x7ff, x = f + e;
    if (f == 0x7ff) return v;
    if (x <= 0 || !f) return 0.0;
    if (x >= 2047) return __hiloint2double((hi & (int)0x80000000u) | 0x7ff00000, 0);
    return __hiloint2double((hi & (int)0x800fffffu) | (x << 20), __double2loint(v));
}

// P[M * J + p], C[M], S[M] as cg::harmonics
__device__ __forceinline__ void harmonics(df x, df y, df z, df r2, int kmax, int J, const KappaMix &k, df *P, df *C, df *S)
{
    C[0] = df_f(1.0f);
    S[0] = df_f(0.0f);
    for (int m = 0; m < kmax; ++m) {
        const df c = C[m], s = S[m];
        C[m + 1] = sub(mul(x, c), mul(y, s));
        S[m + 1] = add(mul(x, s), mul(y, c));
    }
    for (int M = 0; M <= kmax; ++M) {
        df p0 = df_f(0.0f), p1 = df_f(1.0f);
        for (int l = M;; ++l) {
            const int d = kmax - l;
            if (!(d & 1) && (d >> 1) < J) P[M * J + (d >> 1)] = p1;
            if (l == kmax) break;
            df n = mul(z, p1);
            if (l > M) n = sub(n, mul(mul(ldf(k.v[l][M]), r2), p0));
            p0 = p1;
            p1 = n;
        }
    }
}

// sum_p g[p] v[p], p < n: compensated dot product (Dot2 of Ogita, Rump and Oishi)
__device__ __forceinline__ df dot(const float2 *__restrict__ g, const df *v, int n)
{
    float sh = 0.0f, sl = 0.0f;
    for (int p = 0; p < n; ++p) {
        const float2 c = __ldg(g + p);
        const df b = v[p];
        const float pr = c.x * b.hi;
        float ep = fmaf(c.x, b.hi, -pr);
        ep = fmaf(c.x, b.lo, ep);
        ep = fmaf(c.y, b.hi, ep);
        const df t = two_sum(sh, pr);
        sh = t.hi;
        sl += t.lo + ep;
    }
    return fast_two_sum(sh, sl);
}

__device__ __forceinline__ double out_of(df v, int e)
{
    return scale_exp(dev::flt_to_dbl(v.hi) + dev::flt_to_dbl(v.lo), e);
}

// the elements (+-a, +-b), scaled by 2^e at the store (arguments as cg::element)
__device__ __forceinline__ void element(const float2 *__restrict__ g, int a, int b, int kmax, int J, int nb, const df *PF,
                                        const df *C, const df *S, int e, double *__restrict__ o)
{
    const int m1 = a > b ? a - b : b - a, m2 = a + b;
    const df X1 = dot(g, PF + m1 * J, min(J, (kmax - m1) / 2 + 1));
    const df c1 = mul(C[m1], X1), s1 = mul(a < b ? neg(S[m1]) : S[m1], X1);
    if (a && b) {
        const df X2 = dot(g + J, PF + m2 * J, min(J, (kmax - m2) / 2 + 1));
        const df c2 = mul(C[m2], X2), s2 = mul(S[m2], X2);
        o[a * nb + b] = out_of(add(c1, c2), e);
        o[-a * nb - b] = out_of(sub(c1, c2), e);
        o[-a * nb + b] = out_of(add(s2, s1), e);
        o[a * nb - b] = out_of(sub(s2, s1), e);
    } else {
        o[a * nb + b] = out_of(c1, e);
        if (a) o[-a * nb] = out_of(s1, e);
        if (b) o[-b] = out_of(neg(s1), e);
    }
}

// Block of one operator from its FP64 radial orders; P, C, S in units of 2^er (harmonics of the scaled separation)
template <int J>
__device__ __forceinline__ void block_from_orders(const CGTab &t, int la, int lb, double r2, int er, const double (&O)[J],
                                                  double top, const df *P, const df *C, const df *S, df *PF, int gl, int group,
                                                  double *__restrict__ out)
{
    double F[J];
    const int c = la * (kLmax2c + 1) + lb, kmax = la + lb;
    const double *fc = t.fc + 28 * c;
    cg::laplace_orders<J>(fc, r2, O, F);
    F[0] = fma(__ldg(fc), top, F[0]);
    int e = -4000;
#pragma unroll
    for (int p = 0; p < J; ++p)
        if (F[p] != 0.0) e = max(e, exponent(F[p]) + er * (kmax - 2 * p));
    df Fs[J];
#pragma unroll
    for (int p = 0; p < J; ++p) Fs[p] = split(scale_exp(F[p], er * (kmax - 2 * p) - e));
    for (int M = 0; M <= kmax; ++M) {
#pragma unroll
        for (int p = 0; p < J; ++p)
            if (M + 2 * p <= kmax) PF[M * J + p] = mul(P[M * J + p], Fs[p]);
    }
    const float2 *g = t.gm + __ldg(t.gbase + c);
    const int nb = 2 * lb + 1;
    for (int i = gl; i < (la + 1) * (lb + 1); i += group) {
        const int a = i / (lb + 1), b = i - a * (lb + 1);
        element(g + i * 2 * J, a, b, kmax, J, nb, PF, C, S, e, out + la * nb + lb);
    }
}

}  // namespace cgm
}  // namespace shg
