// Gradient kernel of the three-index overlaps: vector-Jacobian product of the (a b a~) blocks with respect to the common
// center R_a of a and a~ (d/dR_b = -d/dR_a).  The upstream block W[ma][mt][mb] is projected through the product expansion
// onto every (L, M, mb), that through the expansion of the class (L, lb) onto the solid harmonics of R_a - R_b, and the
// two-center contraction (shg_grad_angular.cuh) runs over all L.  See shg_aab.cuh for the radial part and the mapping.
#include "shg_aab.cuh"

namespace shg {
namespace {
using namespace dev;
using namespace aab;

// Orders (one more per L than the integrals), F and F', C and S, the coefficients A (cosine and sine), then the partial
// sums or the weight combinations of two columns and their projections
__host__ __device__ constexpr int slot_doubles(const Shape &s)
{
    const int nq = s.qbase(s.nL), n1 = nq + s.nL, work = kLanes * n1;
    const int ang = 2 * s.pbase(s.nL) + 8 * (s.la + 1) * (s.lt + 1) + 2 * s.mbase(s.nL);
    return n1 + 2 * nq + 2 * (s.kmax + 1) + (work > ang ? work : ang);
}
static_assert(largest_slots([](const Shape &s) constexpr { return slot_doubles(s); }) <= kSharedLimit, "see kSharedLimit");

__device__ __forceinline__ void tile_aab_grad(const Args3c &g, const Tile &t, int lane, double *smem)
{
    const Shape sh(t.cls);
    const int gl = lane & (kLanes - 1), slot = lane / kLanes;
    const bool own = slot < t.count;
    const int p = g.perm[t.start + (own ? slot : t.count - 1)];
    const ShellRec sa = g.orb_shells[g.t_a[p]], st = g.orb_shells[g.t_t[p]], sb = g.aux_shells[g.t_b[p]];
    const Vec4 A = g.orb_centers[sa.center], B = g.aux_centers[sb.center];
    const double x = A.x - B.x, y = A.y - B.y, z = A.z - B.z;
    const double R2 = x * x + y * y + z * z;

    const int la = sh.la, lt = sh.lt, lb = sh.lb, nL = sh.nL, nt = 2 * lt + 1, nb = 2 * lb + 1, kmax = sh.kmax;
    const int nq = sh.qbase(nL), np = sh.pbase(nL), nat = (la + 1) * (lt + 1);
    // (L, |M|) sets and (L, M') coefficients
    const int nset = (sh.mbase(nL) + nL) / 2, ncoef = nset + nL * lb;
    double *sum = smem + slot * g.slot_doubles, *F = sum + nq + nL, *D = F + nq, *C = D + nq, *S = C + kmax + 1;
    double *Ac = S + kmax + 1, *As = Ac + np, *Wc = As + np, *Uk = Wc + 8 * nat;
    const int first = own ? gl : kNone;
    switch (nL) {
    case 1: radial<1>(g, sh, 1, sa, st, sb, R2, first, Ac + gl); break;
    case 2: radial<2>(g, sh, 1, sa, st, sb, R2, first, Ac + gl); break;
    case 3: radial<3>(g, sh, 1, sa, st, sb, R2, first, Ac + gl); break;
    case 4: radial<4>(g, sh, 1, sa, st, sb, R2, first, Ac + gl); break;
    case 5: radial<5>(g, sh, 1, sa, st, sb, R2, first, Ac + gl); break;
    default: radial<6>(g, sh, 1, sa, st, sb, R2, first, Ac + gl); break;
    }
    reduce(nq + nL, gl, Ac, sum);

    // F_q and F_q' of every (L, q); O[j] = P^{(L+lb+1-j)}
    for (int v = gl; v < nq; v += kLanes) {
        int i = 0, q = v;
        while (q >= sh.J(i)) q -= sh.J(i++);
        const double *fc = g.cg.fc + 28 * (sh.L(i) * (kLmax2c + 1) + lb) + q * (q + 1) / 2;
        const double *O = sum + v - q + i;
        double f = 0.0, d = 0.0, e = 0.0;
        for (int j = 0; j <= q; ++j) {
            const double c = __ldg(fc + j);
            d = fma(d, R2, f);
            f = fma(f, R2, c * O[j + 1]);
            e = fma(e, R2, c * O[j]);
        }
        F[v] = f;
        D[v] = d + e;
    }
    circular(x, y, kmax, gl, C, S);
    for (int i = gl; i < 2 * np; i += kLanes) Ac[i] = 0.0;      // Ac and As
    __syncwarp();

    const double *w = g.w + g.w_off[p] + (la * nt + lt) * nb + lb;
    const double *h0 = g.cg.h + __ldg(g.cg.gbase + la * (kLmax2c + 1) + lt);
    for (int b = 0; b <= lb; ++b) {
        const int ncol = b ? 2 : 1;
        // weight combinations of the sets (+-ma, +-mt): u1, v1 (|M| = ||ma| - |mt||), u2, v2 (|M| = |ma| + |mt|)
        for (int v = gl; v < nat; v += kLanes) {
            const int a = v / (lt + 1), c = v - a * (lt + 1);
            for (int col = 0; col < ncol; ++col) {
                const double *wb = w + (col ? -b : b);
                double *o = Wc + 8 * v + 4 * col;
                const double cc = wb[(a * nt + c) * nb];
                if (a && c) {
                    const double ss = wb[(-a * nt - c) * nb], sc = wb[(-a * nt + c) * nb], cs = wb[(a * nt - c) * nb];
                    o[0] = cc + ss;
                    o[1] = a > c ? sc - cs : cs - sc;
                    o[2] = cc - ss;
                    o[3] = sc + cs;
                } else {
                    o[0] = cc;
                    o[1] = a ? wb[-a * nt * nb] : c ? wb[-c * nb] : 0.0;
                }
            }
        }
        __syncwarp();
        // U_{L,+-m} of both columns: the sets with ||ma| - |mt|| = m and |ma| + |mt| = m
        for (int v = gl, i = 0, m = gl, mb = 0; v < nset; v += kLanes, m += kLanes) {
            while (m > sh.L(i)) {
                m -= sh.L(i) + 1;
                mb += 2 * sh.L(i) + 1;
                ++i;
            }
            const double *hp = h0 + nL - 1 - i;
            double uc[2] = {0.0, 0.0}, us[2] = {0.0, 0.0};
            for (int a = 0; a <= la; ++a) {
                for (int k = 0; k < 2; ++k) {
                    const int c = k ? a + m : a - m;
                    if (c < 0 || c > lt || (k && !m)) continue;
                    const double hw = __ldg(hp + (a * (lt + 1) + c) * 2 * nL);
                    const double *o = Wc + 8 * (a * (lt + 1) + c);
                    uc[0] = fma(hw, o[0], uc[0]);
                    if (m) us[0] = fma(hw, o[1], us[0]);
                    if (b) {
                        uc[1] = fma(hw, o[4], uc[1]);
                        if (m) us[1] = fma(hw, o[5], us[1]);
                    }
                }
                const int c = m - a;
                if (a && c > 0 && c <= lt) {
                    const double hw = __ldg(hp + (a * (lt + 1) + c) * 2 * nL + nL);
                    const double *o = Wc + 8 * (a * (lt + 1) + c);
                    uc[0] = fma(hw, o[2], uc[0]);
                    us[0] = fma(hw, o[3], us[0]);
                    if (b) {
                        uc[1] = fma(hw, o[6], uc[1]);
                        us[1] = fma(hw, o[7], us[1]);
                    }
                }
            }
            double *o = Uk + 2 * (mb + sh.L(i));
            for (int col = 0; col < ncol; ++col) {
                o[2 * m + col] = uc[col];
                if (m) o[-2 * m + col] = us[col];
            }
        }
        __syncwarp();
        // A_{L,M'}: the sets (+-m, +-b) with |m - b| = M' and m + b = M'
        for (int v = gl, i = 0, M = gl, pb = 0, mb = 0; v < ncoef; v += kLanes, M += kLanes) {
            while (M > sh.L(i) + lb) {
                const int L = sh.L(i);
                M -= L + lb + 1;
                pb += (L + lb + 1) * sh.J(i);
                mb += 2 * L + 1;
                ++i;
            }
            const int L = sh.L(i), J = sh.J(i), n = min(J, (L + lb - M) / 2 + 1);
            const double *g0 = g.cg.g + __ldg(g.cg.gbase + L * (kLmax2c + 1) + lb) + 2 * J * b;
            const double *U = Uk + 2 * (mb + L);
            double *ac = Ac + pb + M * J, *as = As + pb + M * J;
            for (int k = 0; k < 3; ++k) {
                // m - b = M, b - m = M, m + b = M
                const int m = k == 0 ? M + b : k == 1 ? b - M : M - b;
                if (m < 0 || m > L || (k == 1 && !M) || (k == 2 && (!m || !b))) continue;
                const double *gm = g0 + 2 * J * (lb + 1) * m + (k == 2 ? J : 0);
                double u, w_;
                if (m && b) {
                    const double cc = U[2 * m], ss = U[-2 * m + 1], sc = U[-2 * m], cs = U[2 * m + 1];
                    u = k == 2 ? cc - ss : cc + ss;
                    w_ = k == 2 ? sc + cs : k == 0 ? sc - cs : cs - sc;
                } else {
                    u = U[2 * m];
                    w_ = m ? U[-2 * m] : b ? U[1] : 0.0;
                }
                for (int q = 0; q < n; ++q) {
                    const double c = __ldg(gm + q);
                    ac[q] = fma(c, u, ac[q]);
                    if (M) as[q] = fma(c, w_, as[q]);
                }
            }
        }
        __syncwarp();
    }

    // contraction: one column M' per lane and turn, with the columns M' and M'+1 of the harmonics
    double U = 0.0, Z = 0.0, X = 0.0, Y = 0.0;
    for (int M = gl; M <= kmax; M += kLanes) {
        double p0 = 0.0, p1 = 1.0, r0 = 0.0, r1 = 0.0;          // p_{l-1,M}, p_{l,M}; p_{l-1,M+1}, p_{l,M+1}
        double ac = 0.0, as = 0.0, bc = 0.0, bs = 0.0, dc = 0.0, ds = 0.0;
        for (int l = M;; ++l) {
            if (!((kmax - l) & 1)) {
                const double inv = l ? g.k.inv_int[2 * l - 1] : 0.0;
                const double fz = (double)((l - M) * (l + M)) * inv * p0;
                const double fq = -0.5 * (double)((l - M) * (l - M - 1)) * inv * r0;
                for (int i = 0, qb = 0, pb = 0; i < nL; ++i) {
                    const int L = sh.L(i), J = sh.J(i), q = (L + lb - l) >> 1;
                    if (q >= 0 && q < J) {
                        const double f = F[qb + q], d = D[qb + q] * p1;
                        const double wa = Ac[pb + M * J + q], ws = As[pb + M * J + q];
                        const double fp = f * p1, b = fma(f, fq, d), e = fma(2.0 * z, d, f * fz);
                        ac = fma(fp, wa, ac);
                        as = fma(fp, ws, as);
                        bc = fma(b, wa, bc);
                        bs = fma(b, ws, bs);
                        dc = fma(e, wa, dc);
                        ds = fma(e, ws, ds);
                    }
                    qb += J;
                    pb += (L + lb + 1) * J;
                }
            }
            if (l == kmax) break;
            const double n = z * p1 - (g.k.kappa[l][M] * R2) * p0;
            p0 = p1;
            p1 = n;
            // column M+1 starts with p_{M+1,M+1} = 1
            const double m = l > M ? z * r1 - (l > M + 1 ? g.k.kappa[l][M + 1] * R2 * r0 : 0.0) : 1.0;
            r0 = r1;
            r1 = m;
        }
        U = fma(C[M], bc, fma(S[M], bs, U));
        Z = fma(C[M], dc, fma(S[M], ds, Z));
        if (M) {
            const double c1 = C[M - 1], s1 = S[M - 1], n = (double)M * ac, m = (double)M * as;
            X = fma(c1, n, fma(s1, m, X));
            Y = fma(c1, m, fma(-s1, n, Y));
        }
    }
    double G[3] = {fma(2.0 * x, U, X), fma(2.0 * y, U, Y), Z};
    xrad::group_sum<3>(G, kLanes);
    if (own && gl == 0) {
        for (int d = 0; d < 3; ++d) {
            g.grad_a[3 * (int64_t)p + d] = G[d];
            if (g.grad_b) g.grad_b[3 * (int64_t)p + d] = -G[d];
        }
    }
    __syncwarp();
}

__global__ void __launch_bounds__(32, 16) k_3c_grad_fp64(const Args3c g)
{
    extern __shared__ double smem[];
    const int lane = threadIdx.x;
    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(g.counter, 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= g.tile_end) break;
        tile_aab_grad(g, g.tiles[t], lane, smem);
        __syncwarp();
    }
}

}  // namespace

int slot_doubles_3c_grad(int cls) { return slot_doubles(Shape(cls)); }

cudaError_t launch_3c_grad(const Args3c &a, cudaStream_t s)
{
    return launch_slots((const void *)k_3c_grad_fp64, a,
                        [&](int grid, size_t bytes) { k_3c_grad_fp64<<<grid, 32, bytes, s>>>(a); });
}

}  // namespace shg
