// Angular part of a two-center block from its contracted radial orders (Eq. final_r12int_ab), with the product of
// the two solid harmonics expanded first.  The block is
//   (a|O|b) = (-1)^lb S_{la,ma}(grad) S_{lb,mb}(grad) G(R^2),   S_{la,ma} S_{lb,mb} = sum_{L,M} c r^{la+lb-L} S_{L,M},
// L = la+lb, la+lb-2, .., |la-lb| (J = min(la, lb) + 1 values, p = (la+lb-L)/2), |M| = ||ma| +- |mb||, and
//   S_{L,M}(grad) (grad^2)^p G = S_{L,M}(R) F_p,   F_p = 2^{la+lb} sum_i binom(p,i) (L+3/2+i)_{p-i} R^{2i} G^{(L+p+i)}.
// So F_p needs the J orders O^{(k)}, k = max(la,lb) .. la+lb, once per pair and operator, and an element is a sum
// over the J values of L for two |M|.  With S_{L,+-M} = nu p_{L,M}(z, R^2) {C_M, S_M}(x, y), C_M + i S_M = (x + i y)^M,
// the four sign combinations of (|ma|, |mb|) share two sums
//   X1 = sum_p g1_p p_{L,||ma|-|mb||} F_p,   X2 = sum_p g2_p p_{L,|ma|+|mb|} F_p :
//   cc = C1 X1 + C2 X2,  ss = C1 X1 - C2 X2,  (sine, cosine) = S2 X2 + s S1 X1,  (cosine, sine) = S2 X2 - s S1 X1,
// s = sign(|ma| - |mb|): J/2 + 2 operations per element, where the translation-matrix form (W_a W_b^T, Sec. II E)
// takes J^2 + J after building two sets of J^2-long rows.  Near the z axis an element keeps its relative accuracy
// (its terms carry the powers |M| of x + i y that the element has); the sum over p cancels less than the sum over j of
// the translation-matrix form (rms error of (6,6) Coulomb blocks against long double 3.4e-16 of the block maximum
// against 8.8e-16, (3,3) 1.4e-16 against 1.9e-16).
//
// The loops run over runtime l: one copy serves every class, and index arithmetic and loads hide behind the FP64
// instructions (64 cycles each per sub-partition).
#pragma once

#include "shg_device.cuh"

namespace shg {
namespace cg {

constexpr int kMaxL = kLmaxAabA + kLmax2c;                  // largest L of a table class

// largest number of (M, p) entries of a two-center pair: (2 l_max + 1) J
constexpr int kNP2 = (2 * kLmax2c + 1) * kJmax;

// p_{L,M}(z, r2) for L = kmax - 2p at P[M * J + p] (monic in z: p_{l+1} = z p_l - (l^2 - M^2)/(4 l^2 - 1) r2 p_{l-1}), and
// C_M, S_M, 0 <= M <= kmax
__device__ __forceinline__ void harmonics(double x, double y, double z, double r2, int kmax, int J, const Consts &k,
                                          double *P, double *C, double *S)
{
    C[0] = 1.0;
    S[0] = 0.0;
    for (int m = 0; m < kmax; ++m) {
        const double c = C[m], s = S[m];
        C[m + 1] = x * c - y * s;
        S[m + 1] = x * s + y * c;
    }
    for (int M = 0; M <= kmax; ++M) {
        double p0 = 0.0, p1 = 1.0;
        for (int l = M;; ++l) {
            const int d = kmax - l;
            if (!(d & 1) && (d >> 1) < J) P[M * J + (d >> 1)] = p1;
            if (l == kmax) break;
            const double n = z * p1 - (k.kappa[l][M] * r2) * p0;
            p0 = p1;
            p1 = n;
        }
    }
}

// F[p] of one operator from O[j] = O^{(kmax-j)}; fc: coefficients of the class, p (p+1)/2 + j
template <int J>
__device__ __forceinline__ void laplace_orders(const double *__restrict__ fc, double r2, const double (&O)[J],
                                               double (&F)[J])
{
#pragma unroll
    for (int p = 0; p < J; ++p) {
        double s = __ldg(fc + p * (p + 1) / 2) * O[0];
#pragma unroll
        for (int j = 1; j <= p; ++j) s = fma(s, r2, __ldg(fc + p * (p + 1) / 2 + j) * O[j]);
        F[p] = s;
    }
}

// the elements (+-a, +-b) of the block of one operator; PF[M * J + p] = p_{L,M} F_p, g: coefficients of (a, b), o: the
// block's element (0, 0)
__device__ __forceinline__ void element(const double *__restrict__ g, int a, int b, int kmax, int J, int nb,
                                        const double *PF, const double *C, const double *S, double *__restrict__ o)
{
    const int m1 = a > b ? a - b : b - a, m2 = a + b;
    // L >= M: p <= (kmax - M) / 2
    const int n1 = min(J, (kmax - m1) / 2 + 1);
    double X1 = __ldg(g) * PF[m1 * J];
    for (int p = 1; p < n1; ++p) X1 = fma(__ldg(g + p), PF[m1 * J + p], X1);
    if (a && b) {
        const int n2 = min(J, (kmax - m2) / 2 + 1);
        double X2 = __ldg(g + J) * PF[m2 * J];
        for (int p = 1; p < n2; ++p) X2 = fma(__ldg(g + J + p), PF[m2 * J + p], X2);
        const double c1 = C[m1] * X1, s2 = S[m2] * X2;
        const double s1 = a > b ? S[m1] : -S[m1];
        o[a * nb + b] = fma(C[m2], X2, c1);
        o[-a * nb - b] = fma(-C[m2], X2, c1);
        o[-a * nb + b] = fma(s1, X1, s2);
        o[a * nb - b] = fma(-s1, X1, s2);
    } else {
        o[a * nb + b] = C[m1] * X1;
        if (a) o[-a * nb] = S[m1] * X1;
        if (b) o[-b] = S[m1] * X1;
    }
}

// Block of one operator from its radial orders: lane gl of the `group` lanes of the pair stores every group-th set of
// elements.  top: a contribution to the order la + lb that
// belongs to a harmonic part of G (its F_p, p >= 1, vanish).
template <int J>
__device__ __forceinline__ void block_from_orders(const CGTab &t, int la, int lb, double r2, const double (&O)[J],
                                                  double top, const double *P, const double *C, const double *S,
                                                  double *PF, int gl, int group, double *__restrict__ out)
{
    double F[J];
    const double *fc = t.fc + 28 * (la * (kLmax2c + 1) + lb);
    laplace_orders<J>(fc, r2, O, F);
    F[0] = fma(__ldg(fc), top, F[0]);
    const int kmax = la + lb;
    for (int M = 0; M <= kmax; ++M) {
#pragma unroll
        for (int p = 0; p < J; ++p)
            if (M + 2 * p <= kmax) PF[M * J + p] = P[M * J + p] * F[p];
    }
    const double *g = t.g + __ldg(t.gbase + la * (kLmax2c + 1) + lb);
    const int nb = 2 * lb + 1;
    for (int i = gl; i < (la + 1) * (lb + 1); i += group) {
        const int a = i / (lb + 1), b = i - a * (lb + 1);
        element(g + i * 2 * J, a, b, kmax, J, nb, PF, C, S, out + la * nb + lb);
    }
}

}  // namespace cg
}  // namespace shg
