// Integral kernel of the three-index overlaps (a b a~); see shg_aab.cuh.
#include "shg_aab.cuh"

namespace shg {
namespace {
using namespace dev;
using namespace aab;

// Shared memory of a slot in doubles: orders, F_q, C and S, then the partial sums or (L, M', q) products and two columns
// of the blocks
__host__ __device__ constexpr int slot_doubles(const Shape &s)
{
    const int nq = s.qbase(s.nL), work = kLanes * nq, ang = s.pbase(s.nL) + 2 * s.mbase(s.nL);
    return 2 * nq + 2 * (s.kmax + 1) + (work > ang ? work : ang);
}
static_assert(largest_slots([](const Shape &s) constexpr { return slot_doubles(s); }) <= kSharedLimit, "see kSharedLimit");

// Screening of one triple: |phi_a phi_a~| <= 2 sabs_a sabs_a~ lfac_a lfac_a~
// exp(-(amin_a + amin_a~) r^2 / 2) (the single-shell bound of the two-center
// screen, multiplied), so the two-center overlap bound of the combined record
// and b bounds every element of the block.
__device__ __forceinline__ bool screened(const Args3c &g, int p, double R2)
{
    if (!(g.screen_thresh > 0.0)) return false;
    const ScreenRec ra = g.orb_screen[g.t_a[p]], rt = g.orb_screen[g.t_t[p]], rb = g.aux_screen[g.t_b[p]];
    const ScreenRec at{ra.amin + rt.amin, ra.sabs * rt.sabs, 1.4142135623730950488 * ra.lfac * rt.lfac, 0.0};
    return screen_bound(at, rb, R2, OP_OVERLAP, 0.0) < g.screen_thresh;
}

__device__ __forceinline__ void tile_aab(const Args3c &g, const Tile &t, int lane, double *smem)
{
    const Shape sh(t.cls);
    const int gl = lane & (kLanes - 1), slot = lane / kLanes;
    // slots without a triple of their own repeat the last one and store nothing
    const bool own = slot < t.count;
    const int p = g.perm[t.start + (own ? slot : t.count - 1)];
    const ShellRec sa = g.orb_shells[g.t_a[p]], st = g.orb_shells[g.t_t[p]], sb = g.aux_shells[g.t_b[p]];
    const Vec4 A = g.orb_centers[sa.center], B = g.aux_centers[sb.center];
    const double vx = A.x - B.x, vy = A.y - B.y, vz = A.z - B.z;
    const double R2 = vx * vx + vy * vy + vz * vz;
    const bool zero = screened(g, p, R2);
    const int first = own && !zero ? gl : kNone;

    const int nq = sh.qbase(sh.nL), np = sh.pbase(sh.nL);
    double *sum = smem + slot * g.slot_doubles, *F = sum + nq, *C = F + nq, *S = C + sh.kmax + 1, *PF = S + sh.kmax + 1;
    double *Bk = PF + np;                                       // [mbase + M + L][cosine, sine column]
    switch (sh.nL) {
    case 1: radial<1>(g, sh, 0, sa, st, sb, R2, first, PF + gl); break;
    case 2: radial<2>(g, sh, 0, sa, st, sb, R2, first, PF + gl); break;
    case 3: radial<3>(g, sh, 0, sa, st, sb, R2, first, PF + gl); break;
    case 4: radial<4>(g, sh, 0, sa, st, sb, R2, first, PF + gl); break;
    case 5: radial<5>(g, sh, 0, sa, st, sb, R2, first, PF + gl); break;
    default: radial<6>(g, sh, 0, sa, st, sb, R2, first, PF + gl); break;
    }
    reduce(nq, gl, PF, sum);

    // F_q of every (L, q)
    for (int v = gl; v < nq; v += kLanes) {
        int i = 0, q = v;
        while (q >= sh.J(i)) q -= sh.J(i++);
        const double *fc = g.cg.fc + 28 * (sh.L(i) * (kLmax2c + 1) + sh.lb) + q * (q + 1) / 2;
        const double *O = sum + v - q;
        double s = 0.0;
        for (int j = 0; j <= q; ++j) s = fma(s, R2, __ldg(fc + j) * O[j]);
        F[v] = s;
    }
    circular(vx, vy, sh.kmax, gl, C, S);
    __syncwarp();
    // p_{L',M'} F_q: one column M' per lane and turn
    for (int M = gl; M <= sh.kmax; M += kLanes) {
        double p0 = 0.0, p1 = 1.0;
        for (int l = M;; ++l) {
            if (!((sh.kmax - l) & 1)) {
                for (int i = 0, qb = 0, pb = 0; i < sh.nL; ++i) {
                    const int L = sh.L(i), J = sh.J(i), q = (L + sh.lb - l) >> 1;
                    if (q >= 0 && q < J) PF[pb + M * J + q] = p1 * F[qb + q];
                    qb += J;
                    pb += (L + sh.lb + 1) * J;
                }
            }
            if (l == sh.kmax) break;
            const double n = vz * p1 - (g.k.kappa[l][M] * R2) * p0;
            p0 = p1;
            p1 = n;
        }
    }
    __syncwarp();

    const int la = sh.la, lt = sh.lt, lb = sh.lb, nt = 2 * lt + 1, nb = 2 * lb + 1;
    double *out = g.out + g.out_off[p];
    const double *h0 = g.cg.h + __ldg(g.cg.gbase + la * (kLmax2c + 1) + lt);
    const int Jat = sh.nL, nat = (la + 1) * (lt + 1), nset = (sh.mbase(sh.nL) + sh.nL) / 2;      // (L, |M|) sets
    for (int b = 0; b <= lb; ++b) {
        // columns +b and -b of every block (L, lb): sets (+-m, +-b)
        for (int v = gl, i = 0, m = gl, pb = 0, mb = 0; v < nset; v += kLanes, m += kLanes) {
            while (m > sh.L(i)) {
                const int L = sh.L(i);
                m -= L + 1;
                pb += (L + lb + 1) * sh.J(i);
                mb += 2 * L + 1;
                ++i;
            }
            const int L = sh.L(i), J = sh.J(i), km = L + lb;
            const double *gm = g.cg.g + __ldg(g.cg.gbase + L * (kLmax2c + 1) + lb) + 2 * J * (b + (lb + 1) * m);
            const int m1 = m > b ? m - b : b - m, m2 = m + b;
            const int n1 = min(J, (km - m1) / 2 + 1);
            const double *f1 = PF + pb + m1 * J;
            double X1 = __ldg(gm) * f1[0];
            for (int q = 1; q < n1; ++q) X1 = fma(__ldg(gm + q), f1[q], X1);
            double *o = Bk + 2 * (mb + L);
            if (m && b) {
                const int n2 = min(J, (km - m2) / 2 + 1);
                const double *f2 = PF + pb + m2 * J;
                double X2 = __ldg(gm + J) * f2[0];
                for (int q = 1; q < n2; ++q) X2 = fma(__ldg(gm + J + q), f2[q], X2);
                const double c1 = C[m1] * X1, s2 = S[m2] * X2, s1 = m > b ? S[m1] : -S[m1];
                o[2 * m] = fma(C[m2], X2, c1);
                o[-2 * m + 1] = fma(-C[m2], X2, c1);
                o[-2 * m] = fma(s1, X1, s2);
                o[2 * m + 1] = fma(-s1, X1, s2);
            } else {
                o[2 * m] = C[m1] * X1;
                if (m) o[-2 * m] = S[m1] * X1;
                if (b) o[1] = S[m1] * X1;
            }
        }
        __syncwarp();
        // sums over (L, M) for the sets (+-ma, +-mt)
        for (int v = gl; own && v < nat; v += kLanes) {
            const int a = v / (lt + 1), c = v - a * (lt + 1);
            const double *h = h0 + v * 2 * Jat;
            const int m1 = a > c ? a - c : c - a, m2 = a + c;
            for (int col = 0; col <= (b ? 1 : 0); ++col) {
                double y1c = 0.0, y1s = 0.0, y2c = 0.0, y2s = 0.0;
                // table index p = (la + lt - L) / 2 = nL - 1 - i
                for (int i = sh.nL - 1, mb = sh.mbase(sh.nL), p_ = 0; i >= 0; --i, ++p_) {
                    const int L = sh.L(i);
                    mb -= 2 * L + 1;
                    if (L < m1) break;
                    const double *o = Bk + 2 * (mb + L) + col;
                    const double w1 = __ldg(h + p_);
                    y1c = fma(w1, o[2 * m1], y1c);
                    if (m1) y1s = fma(w1, o[-2 * m1], y1s);
                    if (a && c && m2 <= L) {
                        const double w2 = __ldg(h + Jat + p_);
                        y2c = fma(w2, o[2 * m2], y2c);
                        y2s = fma(w2, o[-2 * m2], y2s);
                    }
                }
                if (zero) y1c = y1s = y2c = y2s = 0.0;
                double *o = out + (la * nt + lt) * nb + lb + (col ? -b : b);
                if (a && c) {
                    const double s1 = a > c ? y1s : -y1s;
                    o[(a * nt + c) * nb] = y1c + y2c;
                    o[(-a * nt - c) * nb] = y1c - y2c;
                    o[(-a * nt + c) * nb] = y2s + s1;
                    o[(a * nt - c) * nb] = y2s - s1;
                } else {
                    o[(a * nt + c) * nb] = y1c;
                    if (a) o[-a * nt * nb] = y1s;
                    if (c) o[-c * nb] = y1s;
                }
            }
        }
        __syncwarp();
    }
}

__global__ void __launch_bounds__(32, 16) k_3c_fp64(const Args3c g)
{
    extern __shared__ double smem[];
    const int lane = threadIdx.x;
    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(g.counter, 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= g.tile_end) break;
        tile_aab(g, g.tiles[t], lane, smem);
        __syncwarp();
    }
}

}  // namespace

int slot_doubles_3c(int cls) { return slot_doubles(Shape(cls)); }

cudaError_t launch_3c(const Args3c &a, cudaStream_t s)
{
    return launch_slots((const void *)k_3c_fp64, a, [&](int grid, size_t bytes) { k_3c_fp64<<<grid, 32, bytes, s>>>(a); });
}

}  // namespace shg
