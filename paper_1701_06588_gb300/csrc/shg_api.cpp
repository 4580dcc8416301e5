// Host side of the SHG integral library: C ABI, input validation, shell
// normalisation, device tables, planning and kernel dispatch.
#include "../../include/shg.h"
#include "shg_internal.h"
#include "shg_xf.cuh"

#include <algorithm>
#include <string>
#include <unordered_map>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include <nvtx3/nvToolsExt.h>

namespace shg {

// NVTX range around one phase of a call (plan, exec, copies), visible to
// profilers that trace NVTX (ncu --nvtx, nsys); no cost without a tool.
struct Phase {
    explicit Phase(const char *name) { nvtxRangePushA(name); }
    ~Phase() { nvtxRangePop(); }
    Phase(const Phase &) = delete;
    Phase &operator=(const Phase &) = delete;
};

static thread_local std::string g_err;

int fail(int code, const char *fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_err = buf;
    return code;
}

void clear_error() { g_err.clear(); }

#define SHG_CUDA(call)                                                                                    \
    do {                                                                                                  \
        cudaError_t e_ = (call);                                                                          \
        if (e_ != cudaSuccess) return fail(SHG_ECUDA, "%s: %s (%s:%d)", #call, cudaGetErrorString(e_),   \
                                           __FILE__, __LINE__);                                          \
    } while (0)

// ------------------------------------------------------------------------- //
// Constant tables                                                           //
// ------------------------------------------------------------------------- //
static long double lfact(int n)
{
    long double f = 1;
    for (int i = 2; i <= n; ++i) f *= i;
    return f;
}

// Double-double arithmetic for the host precomputation (shell normalisation
// and per-primitive weights): as accurate as 80-bit long double and much
// faster than the software binary128 long double of aarch64 hosts.
struct dd {
    double hi, lo;
};
static inline dd dd_two_sum(double a, double b)
{
    const double s = a + b, bb = s - a;
    return dd{s, (a - (s - bb)) + (b - bb)};
}
static inline dd dd_norm(double h, double l) { const double s = h + l; return dd{s, l - (s - h)}; }
static inline dd dd_add(dd a, dd b)
{
    dd s = dd_two_sum(a.hi, b.hi), t = dd_two_sum(a.lo, b.lo);
    s.lo += t.hi;
    s = dd_norm(s.hi, s.lo);
    s.lo += t.lo;
    return dd_norm(s.hi, s.lo);
}
static inline dd dd_mul(dd a, dd b)
{
    const double p = a.hi * b.hi;
    double e = std::fma(a.hi, b.hi, -p);
    e += a.hi * b.lo + a.lo * b.hi;
    return dd_norm(p, e);
}
static inline dd dd_div(dd a, dd b)
{
    const double q1 = a.hi / b.hi;
    const dd r = dd_add(a, dd_mul(b, dd{-q1, 0.0}));
    const double q2 = r.hi / b.hi;
    const dd r2 = dd_add(r, dd_mul(b, dd{-q2, 0.0}));
    const double q3 = r2.hi / b.hi;
    return dd_add(dd_norm(q1, q2), dd{q3, 0.0});
}
static inline dd dd_sqrt(dd a)
{
    if (!(a.hi > 0)) return dd{0.0, 0.0};
    const double x = std::sqrt(a.hi);
    const dd x2 = dd_mul(dd{x, 0.0}, dd{x, 0.0});
    const dd d = dd_add(a, dd{-x2.hi, -x2.lo});
    return dd_norm(x, d.hi / (2 * x));
}
static inline dd dd_from(long double v)
{
    const double h = (double)v;
    return dd{h, (double)(v - (long double)h)};
}

void fill_consts(Consts &k)
{
    std::memset(&k, 0, sizeof k);
    // A_{l,mu} = (-1)^mu sqrt((2 - delta_{mu,0}) (l+mu)! (l-mu)!)      Eq. (A)
    for (int l = 0; l <= kLmaxR; ++l)
        for (int mu = 0; mu <= l; ++mu) {
            long double v = std::sqrt((long double)(mu == 0 ? 1 : 2) * lfact(l + mu) * lfact(l - mu));
            k.A[l][mu] = (double)((mu & 1) ? -v : v);
        }
    // (2j-1)!! B_{j,kappa},  B_{j,kappa} = 1 / ((2 - delta_{kappa,0}) (j+kappa)! (j-kappa)!)   Eq. (B)
    for (int j = 0; j < kJmax; ++j) {
        long double df = 1;
        for (int i = 2 * j - 1; i > 1; i -= 2) df *= i;
        for (int kp = 0; kp <= j; ++kp) {
            const long double v = df / ((kp == 0 ? 1 : 2) * lfact(j + kp) * lfact(j - kp));
            k.jB[j][kp] = (double)v;
            k.jB_lo[j][kp] = (double)(v - (long double)k.jB[j][kp]);
        }
    }
    for (int i = 0; i < 32; ++i) k.pow2[i] = std::ldexp(1.0, i);
    for (int i = 0; i < 64; ++i) k.dint[i] = (double)i;
    for (int i = 1; i < 192; ++i) k.inv_int[i] = (double)(1.0L / (long double)i);
    k.inv_int_lo[0] = 0.0;
    for (int i = 1; i < 64; ++i) k.inv_int_lo[i] = (double)(1.0L / (long double)i - (long double)k.inv_int[i]);
    for (int l = 1; l < 16; ++l)
        for (int m = 0; m <= l; ++m) k.kappa[l][m] = (double)((long double)(l * l - m * m) / (4 * l * l - 1));
    long double df = 1;
    for (int n = 0; n < 32; ++n) {
        k.dfact[n] = (double)df;                 // (2n-1)!!
        df *= (2 * n + 1);
    }
    // (a|r_a^{2n}|b): C(n, j) and the coefficients 2^{d-m} (2m+1)!! C(m,d) / (2d+1)!!
    // of Eqs. sra2ms and I_jab
    auto odd_fact = [](int n) { long double f = 1; for (int i = n; i > 1; i -= 2) f *= i; return f; };
    for (int n = 0; n <= kRa2nMax; ++n)
        for (int j = 0; j <= n; ++j) {
            k.binom[n][j] = (double)(lfact(n) / (lfact(j) * lfact(n - j)));
            k.ra2n_k[n][j] = (double)(std::ldexp(1.0L, j - n) * odd_fact(2 * n + 1) * (lfact(n) / (lfact(j) * lfact(n - j))) /
                                      odd_fact(2 * j + 1));
        }
}

// Extended floats from host values: FP64 (also denormal) and double-double, > 0
static xfp::xf xf_of(dd v)
{
    int x;
    const double f = std::frexp(v.hi, &x);                       // [1/2, 1)
    int64_t m = (int64_t)std::ldexp(f, 63) + (int64_t)std::llrint(std::ldexp(v.lo, 63 - x));
    if (m < 0) m = INT64_MAX;                                    // hi rounded up to a power of two
    int e = x - 63;
    if (m < (1ll << 62)) {                                       // hi a power of two, lo < 0
        m *= 2;
        --e;
    }
    return xfp::xf{(uint64_t)m, e};
}

static XOmega x_omega(double w)
{
    if (!(w > 0)) return XOmega{1ull << 62, 1ull << 62, -62, -62};
    const xfp::xf a = xf_of(dd{w, 0.0}), b = xfp::mul(a, a);
    return XOmega{a.m, b.m, a.e, b.e};
}

// Table of BoysEnt (layout there): at the coarse points T_i = i/32 the power series of F_48 and the downward recursion
// in long double; at the 16 nodes k/512 around each, F_20 by its Taylor series (|d| <= 1/64, ten terms) and downward.
static void make_boys_cells(std::vector<BoysEnt> &tab)
{
    const int ntop = 48, nf = 20;
    tab.assign((size_t)kBoysCells * kBoysOrders, BoysEnt{});
#pragma omp parallel for schedule(dynamic, 16)
    for (int i = 0; i <= kBoysCells / 16; ++i) {
        const long double T = (long double)i / 32;
        const long double e = std::exp(-T);
        long double term = 1.0L / (2 * ntop + 1), sum = term;
        for (int k = 1; k < 20000; ++k) {
            term *= 2 * T / (long double)(2 * ntop + 2 * k + 1);
            sum += term;
            if (term < sum * 1e-24L) break;
        }
        long double F[ntop + 1];
        F[ntop] = e * sum;
        for (int n = ntop; n > 0; --n) F[n - 1] = (2 * T * F[n] + e) / (long double)(2 * n - 1);
        for (int k = 16 * i - 8; k < 16 * i + 8; ++k) {
            if (k < 1 || k > kBoysCells) continue;
            const long double d = T - (long double)k / 512, Tk = (long double)k / 512;
            long double G[nf + 1], pw = 1;
            G[nf] = 0;
            for (int t = 0; t <= 10; ++t) {
                G[nf] += F[nf + t] * pw;
                pw *= d / (t + 1);
            }
            const long double ek = std::exp(-Tk);
            for (int n = nf; n > 0; --n) G[n - 1] = (2 * Tk * G[n] + ek) / (long double)(2 * n - 1);
            for (int n = 0; n < kBoysOrders; ++n) {
                int x;
                const long double f = std::frexp(G[n], &x);
                const int s = f < 1 - 1.0L / 256 ? 63 - x : 62 - x;
                auto fix = [&](int t, long double fac, int unit) {
                    return (uint64_t)std::rint(std::ldexp(G[n + t] / fac, s - unit));
                };
                BoysEnt &b = tab[(size_t)n * kBoysCells + (k - 1)];
                b.c0 = fix(0, 1, 0);
                b.c1 = fix(1, 1, 0);
                b.c2 = ((fix(2, 2, 0) + 128) & ~255ull) | (uint64_t)(s - 62);
                b.c3 = (uint32_t)fix(3, 6, 30);
                b.c45 = (uint32_t)fix(4, 24, 35) | (uint32_t)(fix(5, 120, 49) << 24);
            }
        }
    }
}

static float2 split2(long double v)
{
    const float hi = (float)v;
    return make_float2(hi, (float)(v - (long double)hi));
}

// same for a double: v - hi is exact in double (hi holds v's leading 24 bits)
static inline float2 split2d(double v)
{
    const float hi = (float)v;
    return make_float2(hi, (float)(v - (double)hi));
}

void fill_consts3(Consts3 &k)
{
    std::memset(&k, 0, sizeof k);
    for (int n = 0; n < 18; ++n)
        for (int i = 0; i <= n; ++i) k.binom[n][i] = (double)(lfact(n) / (lfact(i) * lfact(n - i)));
    // L_m^{(1/2)}(-u) = sum_j binom(m + 1/2, m - j) u^j / j!
    for (int m = 0; m < 6; ++m)
        for (int j = 0; j <= m; ++j) {
            long double v = 1;
            for (int i = 0; i < m - j; ++i) v *= (m + 0.5L - i) / (i + 1);
            k.lag[m][j] = (double)(v / lfact(j));
        }
    for (int L = 0; L < 11; ++L)
        for (int p = 0; p < 6; ++p)
            for (int m = 0; m <= p; ++m) {
                long double r = 1;
                for (int i = 0; i < p - m; ++i) r *= (L + i);
                k.K[L][p][m] = (double)((lfact(p) / (lfact(m) * lfact(p - m))) * r * lfact(m));
            }
}

// Gauss-Legendre nodes and weights on [-1, 1] (Newton on P_n).
static void gauss_legendre(int n, std::vector<long double> &x, std::vector<long double> &w)
{
    const long double pi = 3.14159265358979323846264338327950288L;
    x.assign(n, 0);
    w.assign(n, 0);
    for (int i = 0; i < n; ++i) {
        long double t = std::cos(pi * (i + 0.75L) / (n + 0.5L)), dp = 0;
        for (int it = 0; it < 100; ++it) {
            long double p0 = 1, p1 = t;
            for (int k = 2; k <= n; ++k) {
                const long double p2 = ((2 * k - 1) * t * p1 - (k - 1) * p0) / k;
                p0 = p1;
                p1 = p2;
            }
            dp = n * (t * p1 - p0) / (t * t - 1);
            const long double dt = p1 / dp;
            t -= dt;
            if (std::fabs(dt) < 1e-19L) break;
        }
        x[i] = t;
        w[i] = 2 / ((1 - t * t) * dp * dp);
    }
}

// Coefficients of the expanded angular part (layout at CGTab).  With S_{l,+-m} = nu_{l,m} p_{l,m}(z, r^2) {C_m, S_m},
// nu_{l,m} = sqrt((2 - delta_{m0}) (l-m)!/(l+m)!) (2l-1)!!/(l-m)!, the product of the two theta functions is
// expanded in those of (L, M) by Gauss-Legendre quadrature exact for the degrees (<= 2 (kLmaxAabA + kLmax2c)).
static void make_cg(std::vector<double> &g, std::vector<double> &h, std::vector<int> &gbase, std::vector<double> &fc)
{
    const int lmax = kLmaxAabA + kLmax2c, nq = 24;
    std::vector<long double> x, w;
    gauss_legendre(nq, x, w);
    // theta functions nu p sin^m at the nodes, and nu
    std::vector<long double> th((size_t)(lmax + 1) * (lmax + 1) * nq, 0), nu((size_t)(lmax + 1) * (lmax + 1), 0);
    for (int l = 0; l <= lmax; ++l)
        for (int m = 0; m <= l; ++m) {
            long double odd = 1;
            for (int i = 2 * l - 1; i > 1; i -= 2) odd *= i;
            nu[l * (lmax + 1) + m] = std::sqrt((m ? 2 : 1) * lfact(l - m) / lfact(l + m)) * odd / lfact(l - m);
        }
    for (int q = 0; q < nq; ++q)
        for (int m = 0; m <= lmax; ++m) {
            long double p0 = 0, p1 = 1, sm = 1;
            const long double s = std::sqrt(1 - x[q] * x[q]);
            for (int i = 0; i < m; ++i) sm *= s;
            for (int l = m; l <= lmax; ++l) {
                th[((size_t)l * (lmax + 1) + m) * nq + q] = nu[l * (lmax + 1) + m] * p1 * sm;
                const long double n = x[q] * p1 - (long double)(l * l - m * m) / (4 * l * l - 1) * p0;
                p0 = p1;
                p1 = n;
            }
        }
    auto theta = [&](int l, int m) { return &th[((size_t)l * (lmax + 1) + m) * nq]; };
    gbase.assign(kNClassCG, 0);
    fc.assign((size_t)kNClassCG * 28, 0.0);
    g.clear();
    for (int la = 0; la <= kLmaxAabA; ++la)
        for (int lb = 0; lb <= kLmax2c; ++lb) {
            const int J = std::min(la, lb) + 1, c = la * (kLmax2c + 1) + lb;
            gbase[c] = (int)g.size();
            for (int a = 0; a <= la; ++a)
                for (int b = 0; b <= lb; ++b)
                    for (int s = 0; s < 2; ++s)
                        for (int p = 0; p < J; ++p) {
                            const int L = la + lb - 2 * p, M = s ? a + b : std::abs(a - b);
                            long double v = 0, vh = 0;
                            if (M <= L && !(s && (!a || !b))) {
                                const long double *ta = theta(la, a), *tb = theta(lb, b), *tL = theta(L, M);
                                for (int q = 0; q < nq; ++q) v += w[q] * ta[q] * tb[q] * tL[q];
                                vh = v * (2 * L + 1) / (M ? 4.0L : 2.0L) * (a && b ? 0.5L : 1.0L);
                                v = vh * nu[L * (lmax + 1) + M];
                            }
                            g.push_back((double)v);
                            if (la <= kLmax2c) h.push_back((double)vh);
                        }
            for (int p = 0; p < J; ++p)
                for (int j = 0; j <= p; ++j) {
                    const int L = la + lb - 2 * p, i = p - j;
                    long double v = lfact(p) / (lfact(i) * lfact(p - i)) * std::ldexp((lb & 1) ? -1.0L : 1.0L, la + lb);
                    for (int q = i; q < p; ++q) v *= L + 1.5L + q;
                    fc[(size_t)c * 28 + p * (p + 1) / 2 + j] = (double)v;
                }
        }
}

// ------------------------------------------------------------------------- //
// Per-device tables                                                          //
// ------------------------------------------------------------------------- //
constexpr int kNBins = kNClass * kKbins2c;

constexpr int kNBins3 = kNClass3 * kKbins3c;

struct DevState {
    DeviceTables t{};
    int *bin_rank[2] = {nullptr, nullptr};   // [2 * kNBins]: rank of bin, then bin of rank
    int *bin_rank3 = nullptr;                // [2 * kNBins3], three-index bins by cost
    cudaMemPool_t pool = nullptr;            // plans (plan_alloc)
    int users = 0;                           // live bases and plans of the device
    bool ready = false;
};

// Estimated cost of a triple of kk primitive combinations, for the order of the tiles: operations of the form that sums order
// by order with translation matrices.  The present kernels take fewer per element (the expanded harmonics) and per
// combination, so it overrates large l.
static double class_cost3(int la, int lt, int lb, int kk)
{
    const int Lmin = std::abs(la - lt), Lmax = la + lt, nL = (Lmax - Lmin) / 2 + 1;
    double rad = 30.0, ang = 0;
    for (int L = Lmin; L <= Lmax; L += 2) {
        const int J = std::min(L, lb) + 1;
        rad += 4.0 * J * ((Lmax - L) / 2 + 1);
        ang += (2.0 * L + 1) * (2 * lb + 1) * (J * J + 2) + (2.0 * L + 1) * J * J;
    }
    return kk * rad + ang + (2.0 * la + 1) * (2 * lt + 1) * (2 * lb + 1) * nL * 2;
}

static int g_chunk_class3[kNClass3];        // class of every chunk of the three-index rank order
static uint8_t g_chunk_class[2][kNClass];   // class of every chunk of a schedule's rank order (the same on all devices)

static std::mutex g_mu;
static DevState g_dev[64];

// the same of a pair
static double class_cost(int la, int lb, int kk)
{
    const int J = std::min(la, lb) + 1;
    const double radial = kk * (40.0 + 4.0 * J);
    const double na = 2 * la + 1, nb = 2 * lb + 1;
    const double angular = na * nb * (J * J + 2) + (2 * na + nb) * J * J + 10.0 * (std::max(la, lb) + 1) * (std::max(la, lb) + 1);
    return radial + angular;
}

static void make_ranks(int schedule, std::vector<int> &rank, std::vector<int> &inv)
{
    rank.assign(kNBins, 0);
    inv.assign(kNBins, 0);
    std::vector<int> order(kNBins);
    for (int b = 0; b < kNBins; ++b) order[b] = b;
    if (schedule == SHG_SCHED_PER_CLASS) {
        // class-major, Ka*Kb descending inside a class
        std::sort(order.begin(), order.end(), [](int x, int y) {
            const int cx = x / kKbins2c, cy = y / kKbins2c;
            if (cx != cy) return cx < cy;
            return (x % kKbins2c) > (y % kKbins2c);
        });
    } else {
        // class-major; classes grouped by J = min(la, lb) + 1 (descending), then by
        // decreasing estimated cost of their heaviest pairs; Ka*Kb descending
        // inside a class.  Longest tiles come first (J-major is close to cost
        // order), and the warps resident on one SM mostly run one J
        // instantiation at a time (instruction-cache locality)
        std::vector<double> ccost(kNClass);
        std::vector<int> cJ(kNClass);
        for (int cls = 0; cls < kNClass; ++cls) {
            const int la = cls / (kLmax2c + 1), lb = cls % (kLmax2c + 1);
            ccost[cls] = class_cost(la, lb, 64);
            cJ[cls] = std::min(la, lb) + 1;
        }
        std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
            const int cx = x / kKbins2c, cy = y / kKbins2c;
            if (cx != cy) {
                if (cJ[cx] != cJ[cy]) return cJ[cx] > cJ[cy];
                return ccost[cx] > ccost[cy] || (ccost[cx] == ccost[cy] && cx < cy);
            }
            return (x % kKbins2c) > (y % kKbins2c);
        });
    }
    for (int r = 0; r < kNBins; ++r) {
        rank[order[r]] = r;
        inv[r] = order[r];
    }
}

// Plans come from a pool of the library: the default pool returns its memory to the system at every synchronisation
// (release threshold 0), and planning synchronises, so a one-shot call on 2,000 pairs spent 200 of its 410 us on mapping its
// 0.9 MB again.  This pool keeps up to kPoolKeep bytes between calls (the plan of 2M pairs takes 22 MB) while the device has
// a basis or a plan, and nothing after the last of them.  Stream-ordered like the default pool, shared by all threads.
constexpr uint64_t kPoolKeep = 256ull << 20;

static cudaError_t make_pool(int dev, cudaMemPool_t *pool)
{
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    return cudaMemPoolCreate(pool, &props);
}

static cudaMemPool_t pool_of(int dev)
{
    std::lock_guard<std::mutex> lk(g_mu);
    return g_dev[dev].pool;
}

// device memory of a plan on the current device, in the order of s (cudaFreeAsync frees it)
static cudaError_t plan_alloc(void **p, size_t bytes, cudaStream_t s)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    return cudaMallocFromPoolAsync(p, bytes, pool_of(dev), s);
}

// A basis or plan of the device was made (+1) or destroyed (-1, after its memory was freed).  Plans may outlive their
// basis, and frees are still queued when the last one goes: from then on the threshold is 0, so the pool returns what the
// trim finds in use at the first synchronisation after those frees.
static void count_user(int dev, int d)
{
    std::lock_guard<std::mutex> lk(g_mu);
    DevState &st = g_dev[dev];
    const bool was = st.users > 0;
    st.users += d;
    if (was == (st.users > 0) || !st.pool) return;
    uint64_t keep = was ? 0 : kPoolKeep;
    cudaMemPoolSetAttribute(st.pool, cudaMemPoolAttrReleaseThreshold, &keep);
    if (was) cudaMemPoolTrimTo(st.pool, 0);
}

const DeviceTables *device_tables_impl(int **ranks, int **rank3 = nullptr)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= 64) {
        fail(SHG_ECUDA, "cudaGetDevice: %s", cudaGetErrorString(e));
        return nullptr;
    }
    std::lock_guard<std::mutex> lk(g_mu);
    DevState &st = g_dev[dev];
    if (!st.ready) {
        int *d_r[2] = {nullptr, nullptr};
        bool ok = (st.pool || make_pool(dev, &st.pool) == cudaSuccess) && cudaMalloc(&d_r[0], 2 * kNBins * sizeof(int)) == cudaSuccess &&
                  cudaMalloc(&d_r[1], 2 * kNBins * sizeof(int)) == cudaSuccess;
        for (int s = 0; s < 2 && ok; ++s) {
            std::vector<int> rank, inv;
            make_ranks(s, rank, inv);
            for (int c = 0; c < kNClass; ++c) g_chunk_class[s][c] = (uint8_t)(inv[(size_t)c * kKbins2c] / kKbins2c);
            rank.insert(rank.end(), inv.begin(), inv.end());
            ok = cudaMemcpy(d_r[s], rank.data(), rank.size() * sizeof(int), cudaMemcpyHostToDevice) == cudaSuccess;
        }
        // three-index bins ordered by estimated cost
        int *d_r3 = nullptr;
        if (ok) {
            // class-major like the two-center ranks (each class one contiguous chunk
            // of kKbins3c ranks, tiled as a whole): classes by decreasing cost of
            // their heaviest bin, Ka*Ka~*Kb descending inside a class
            std::vector<int> order(kNBins3), rank3(2 * kNBins3);
            std::vector<double> ccost(kNClass3);
            for (int cls = 0; cls < kNClass3; ++cls)
                ccost[cls] = class_cost3(cls / 49, (cls / 7) % 7, cls % 7, kKbins3c);
            for (int b = 0; b < kNBins3; ++b) order[b] = b;
            std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
                const int cx = x / kKbins3c, cy = y / kKbins3c;
                if (cx != cy) return ccost[cx] > ccost[cy] || (ccost[cx] == ccost[cy] && cx < cy);
                return (x % kKbins3c) > (y % kKbins3c);
            });
            for (int c = 0; c < kNClass3; ++c) g_chunk_class3[c] = order[(size_t)c * kKbins3c] / kKbins3c;
            for (int r = 0; r < kNBins3; ++r) {
                rank3[order[r]] = r;
                rank3[kNBins3 + r] = order[r];
            }
            ok = cudaMalloc(&d_r3, rank3.size() * sizeof(int)) == cudaSuccess &&
                 cudaMemcpy(d_r3, rank3.data(), rank3.size() * sizeof(int), cudaMemcpyHostToDevice) == cudaSuccess;
        }
        double *d_cg = nullptr, *d_fc = nullptr, *d_ch = nullptr;
        float2 *d_cgm = nullptr;
        int *d_cgb = nullptr;
        if (ok) {
            std::vector<double> cg, ch, fc;
            std::vector<int> cgb;
            make_cg(cg, ch, cgb, fc);
            ok = cudaMalloc(&d_ch, ch.size() * sizeof(double)) == cudaSuccess &&
                 cudaMemcpy(d_ch, ch.data(), ch.size() * sizeof(double), cudaMemcpyHostToDevice) == cudaSuccess;
            std::vector<float2> cgm(cg.size());
            for (size_t i = 0; i < cg.size(); ++i) cgm[i] = split2d(cg[i]);
            ok = ok && cudaMalloc(&d_cg, cg.size() * sizeof(double)) == cudaSuccess &&
                 cudaMalloc(&d_fc, fc.size() * sizeof(double)) == cudaSuccess &&
                 cudaMalloc(&d_cgm, cgm.size() * sizeof(float2)) == cudaSuccess &&
                 cudaMemcpy(d_cgm, cgm.data(), cgm.size() * sizeof(float2), cudaMemcpyHostToDevice) == cudaSuccess &&
                 cudaMalloc(&d_cgb, cgb.size() * sizeof(int)) == cudaSuccess &&
                 cudaMemcpy(d_cg, cg.data(), cg.size() * sizeof(double), cudaMemcpyHostToDevice) == cudaSuccess &&
                 cudaMemcpy(d_fc, fc.data(), fc.size() * sizeof(double), cudaMemcpyHostToDevice) == cudaSuccess &&
                 cudaMemcpy(d_cgb, cgb.data(), cgb.size() * sizeof(int), cudaMemcpyHostToDevice) == cudaSuccess;
        }
        BoysEnt *d_bc = nullptr;
        uint64_t *d_ex = nullptr;
        if (ok) {
            std::vector<BoysEnt> bc;
            make_boys_cells(bc);
            uint64_t ex[kExpTab];
            for (int j = 0; j < kExpTab; ++j) ex[j] = (uint64_t)std::rint(std::ldexp(std::exp((long double)j / 512), 62));
            ok = cudaMalloc(&d_bc, bc.size() * sizeof(BoysEnt)) == cudaSuccess &&
                 cudaMalloc(&d_ex, sizeof ex) == cudaSuccess &&
                 cudaMemcpy(d_bc, bc.data(), bc.size() * sizeof(BoysEnt), cudaMemcpyHostToDevice) == cudaSuccess &&
                 cudaMemcpy(d_ex, ex, sizeof ex, cudaMemcpyHostToDevice) == cudaSuccess;
        }
        if (!ok) {
            fail(SHG_ECUDA, "device tables: upload failed");
            return nullptr;
        }
        st.bin_rank3 = d_r3;
        st.t.cg = CGTab{d_cg, d_cgb, d_fc, d_cgm, d_ch};
        st.t.x = XTab{d_bc, d_ex};
        st.bin_rank[0] = d_r[0];
        st.bin_rank[1] = d_r[1];
        st.ready = true;
    }
    if (ranks) {
        ranks[0] = st.bin_rank[0];
        ranks[1] = st.bin_rank[1];
    }
    if (rank3) *rank3 = st.bin_rank3;
    return &st.t;
}

const DeviceTables *device_tables() { return device_tables_impl(nullptr); }

const DeviceTables *device_tables_if_ready(const int **ranks)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    std::lock_guard<std::mutex> lk(g_mu);
    DevState &st = g_dev[dev];
    if (!st.ready) return nullptr;
    if (ranks) {
        ranks[0] = st.bin_rank[0];
        ranks[1] = st.bin_rank[1];
    }
    return &st.t;
}

const Consts3 &consts3()
{
    static Consts3 k;
    static std::once_flag once;
    std::call_once(once, [] { fill_consts3(k); });
    return k;
}

const Consts &consts()
{
    static Consts k;
    static std::once_flag once;
    std::call_once(once, [] { fill_consts(k); });
    return k;
}

static const KappaMix &kappa_mix()
{
    static KappaMix k;
    static std::once_flag once;
    std::call_once(once, [] {
        for (int n = 0; n < 32; ++n) k.inv[n] = n ? split2(1.0L / n) : make_float2(0, 0);
        for (int l = 0; l < 16; ++l)
            for (int m = 0; m < 16; ++m)
                k.v[l][m] = l && m <= l ? split2((long double)(l * l - m * m) / (4 * l * l - 1)) : make_float2(0, 0);
    });
    return k;
}

static bool is_finite_d(double x) { return std::isfinite(x); }

static int current_device_matches(int dev)
{
    int cur = -1;
    if (cudaGetDevice(&cur) != cudaSuccess) return fail(SHG_ECUDA, "cudaGetDevice failed");
    if (cur != dev) return fail(SHG_EINVAL, "current device %d differs from the basis device %d", cur, dev);
    return SHG_OK;
}

int check_op(int op, double omega, int precision)
{
    if (op < SHG_OP_OVERLAP || op > SHG_OP_RA2N) return fail(SHG_EINVAL, "bad operator %d", op);
    if (op == SHG_OP_RA2N) {
        if (!(omega >= 0 && omega <= kRa2nMax && omega == std::floor(omega)))
            return fail(SHG_EINVAL, "SHG_OP_RA2N takes n = 0..%d in omega (got %g)", kRa2nMax, omega);
        if (precision != SHG_PREC_FP64) return fail(SHG_EINVAL, "SHG_OP_RA2N is available in FP64 only");
    } else if (op != SHG_OP_OVERLAP && op != SHG_OP_COULOMB && !(omega > 0 && std::isfinite(omega))) {
        return fail(SHG_EINVAL, "operator %d needs omega > 0 (got %g)", op, omega);
    }
    if (precision != SHG_PREC_FP64 && precision != SHG_PREC_MIXED)
        return fail(SHG_EINVAL, "precision %d not available", precision);
    return SHG_OK;
}

}  // namespace shg

using namespace shg;

// ------------------------------------------------------------------------- //
// C ABI                                                                      //
// ------------------------------------------------------------------------- //
extern "C" {

const char *shg_last_error(void) { return g_err.c_str(); }

const char *shg_version(void) { return "shg-gb300 0.1 (sm_103a)"; }

int shg_basis_create(int n_shells, const int32_t *l, const int32_t *nprim, const double *exps, const double *coefs,
                     int n_centers, const double *centers, const int32_t *center_of_shell, int normalize,
                     shg_basis_t **out)
{
    Phase phase_("shg:basis_create");
    g_err.clear();
    if (!out) return fail(SHG_EINVAL, "out is NULL");
    *out = nullptr;
    if (n_shells < 1 || n_centers < 1) return fail(SHG_EINVAL, "n_shells and n_centers must be >= 1");
    if (!l || !nprim || !exps || !coefs || !centers || !center_of_shell) return fail(SHG_EINVAL, "NULL input array");
    int64_t n_prims = 0;
    for (int s = 0; s < n_shells; ++s) {
        if (l[s] < 0 || l[s] > kLmax2c) return fail(SHG_EINVAL, "shell %d: l = %d outside 0..%d", s, l[s], kLmax2c);
        if (nprim[s] < 1 || nprim[s] > kKmax) return fail(SHG_EINVAL, "shell %d: K = %d outside 1..%d", s, nprim[s], kKmax);
        if (center_of_shell[s] < 0 || center_of_shell[s] >= n_centers)
            return fail(SHG_EINVAL, "shell %d: center index %d out of range", s, center_of_shell[s]);
        n_prims += nprim[s];
    }
    if (n_prims > (int64_t)INT32_MAX) return fail(SHG_ERANGE, "too many primitives");
    for (int64_t i = 0; i < n_prims; ++i) {
        if (!is_finite_d(exps[i]) || exps[i] <= 0) return fail(SHG_EINVAL, "primitive %lld: exponent %g not > 0", (long long)i, exps[i]);
        if (!is_finite_d(coefs[i])) return fail(SHG_EINVAL, "primitive %lld: coefficient not finite", (long long)i);
    }
    for (int64_t i = 0; i < 3 * (int64_t)n_centers; ++i)
        if (!is_finite_d(centers[i])) return fail(SHG_EINVAL, "center coordinate %lld not finite", (long long)i);

    std::vector<ShellRec> sh(n_shells);
    std::vector<PrimRec> pr(n_prims);
    std::vector<XPrim> xpr(n_prims);
    std::vector<int64_t> first(n_shells + 1, 0);
    for (int s = 0; s < n_shells; ++s) first[s + 1] = first[s] + nprim[s];
    // per-l constants: sqrt(pi) (2l+2)! / (2^{2l+3} (l+1)!) and K_l = sqrt((2l+1)/(4 pi))
    dd pref_l[kLmax2c + 1], K_l[kLmax2c + 1];
    for (int L = 0; L <= kLmax2c; ++L) {
        const long double pi = 3.14159265358979323846264338327950288L;
        pref_l[L] = dd_from(std::sqrt(pi) * lfact(2 * L + 2) / (std::ldexp(1.0L, 2 * L + 3) * lfact(L + 1)));
        K_l[L] = dd_from(std::sqrt((2 * L + 1) / (4 * pi)));
    }
    // sqrt(2 pi^{5/2}) folded into cw: pre = cw_a cw_b / sqrt(c)
    const dd s2p52 = dd_sqrt(dd_from(2.0L * 17.493418327624862846262821679871554L));
    int bad_shell = -1;
#pragma omp parallel for schedule(dynamic, 256)
    for (int s = 0; s < n_shells; ++s) {
        const int L = l[s], K = nprim[s];
        const int64_t off = first[s];
        dd N = {1.0, 0.0};
        if (normalize) {
            // N_l = K_l [sum_ij sqrt(pi) (2l+2)! c_i c_j / (2^{2l+3} (l+1)! (a_i+a_j)^{l+3/2})]^{-1/2}
            dd sum = {0.0, 0.0};
            for (int i = 0; i < K; ++i)
                for (int j = i; j < K; ++j) {
                    const dd sij = dd_two_sum(exps[off + i], exps[off + j]);
                    const dd r = dd_div(dd{1.0, 0.0}, sij);
                    dd pw = r;
                    for (int t = 0; t < L; ++t) pw = dd_mul(pw, r);      // s^-(L+1)
                    dd term = dd_mul(pw, dd_sqrt(r));                    // s^-(L+3/2)
                    term = dd_mul(term, dd_mul(dd{coefs[off + i], 0.0}, dd{coefs[off + j], 0.0}));
                    if (j != i) term = dd{2 * term.hi, 2 * term.lo};
                    sum = dd_add(sum, term);
                }
            sum = dd_mul(sum, pref_l[L]);
            if (!(sum.hi > 0)) {
#pragma omp critical
                bad_shell = s;
                continue;
            }
            N = dd_div(K_l[L], dd_sqrt(sum));
        }
        for (int i = 0; i < K; ++i) {
            const double a = exps[off + i];
            const dd c = dd_mul(N, dd{coefs[off + i], 0.0});
            dd p2 = {1.0, 0.0};
            for (int t = 0; t < L; ++t) p2 = dd_mul(p2, dd{2 * a, 0.0});  // (2a)^l
            PrimRec p;
            const dd ia = dd_div(dd{1.0, 0.0}, dd{a, 0.0});
            const dd w2c = dd_div(c, p2);
            p.alpha = a;
            p.inv_alpha = ia.hi;
            p.w2c = w2c.hi;
            p.wN = c.hi;
            pr[off + i] = p;
            const dd cw = dd_mul(w2c, ia);
            const dd cws = dd_mul(cw, s2p52);
            const xfp::xf xa = xf_of(dd{a, 0.0});
            // a zero weight: a value so small that every term it enters is flushed to 0 (and one that overflowed FP64
            // gives infinities)
            const xfp::xf xw = cws.hi == 0 || !std::isfinite(cws.hi)
                                       ? xfp::xf{1ull << 62, cws.hi == 0 ? -1000000 : 1000000}
                                       : xf_of(cws.hi < 0 ? dd{-cws.hi, -cws.lo} : cws);
            xpr[off + i] = XPrim{xa.m, xw.m | (cws.hi < 0 ? 1ull << 63 : 0), xa.e, xw.e, dd_mul(cw, dd_sqrt(ia)).hi};
        }
        sh[s] = ShellRec{L, K, (int)off, center_of_shell[s]};
    }
    if (bad_shell >= 0) return fail(SHG_EINVAL, "shell %d: contracted function has zero norm", bad_shell);
    // families: shells on one center whose exponent lists are bitwise identical
    std::vector<int32_t> fam(n_shells), fam_prim, fam_k;
    {
        std::unordered_map<std::string, int> ids;
        std::string key;
        for (int s = 0; s < n_shells; ++s) {
            key.assign(reinterpret_cast<const char *>(&center_of_shell[s]), sizeof(int32_t));
            key.append(reinterpret_cast<const char *>(exps + first[s]), sizeof(double) * (size_t)nprim[s]);
            auto it = ids.find(key);
            if (it == ids.end()) {
                it = ids.emplace(key, (int)fam_prim.size()).first;
                fam_prim.push_back((int32_t)first[s]);
                fam_k.push_back(nprim[s]);
            }
            fam[s] = it->second;
        }
    }
    std::vector<ScreenRec> scr(n_shells);
    for (int s = 0; s < n_shells; ++s) {
        double amin = exps[first[s]], sabs = 0;
        for (int64_t i = first[s]; i < first[s + 1]; ++i) {
            amin = std::min(amin, exps[i]);
            sabs += std::fabs(pr[i].wN);
        }
        const int L = l[s];
        const double lfac = L == 0 ? 1.0 : std::pow(L / (amin * 2.718281828459045), 0.5 * L);
        scr[s] = ScreenRec{amin, sabs, lfac, 0.0};
    }
    std::vector<Vec4> ctr(n_centers);
    for (int c = 0; c < n_centers; ++c) ctr[c] = Vec4{centers[3 * c], centers[3 * c + 1], centers[3 * c + 2], 0.0};

    shg_basis_t *b = new (std::nothrow) shg_basis_t;
    if (!b) return fail(SHG_ENOMEM, "host allocation failed");
    BasisDev &d = b->d;
    d.n_shells = n_shells;
    d.n_centers = n_centers;
    d.n_prims = n_prims;
    cudaGetDevice(&d.device);
    d.h_l = new int32_t[n_shells];
    d.h_nprim = new int32_t[n_shells];
    d.h_center = new int32_t[n_shells];
    std::memcpy(d.h_l, l, sizeof(int32_t) * n_shells);
    std::memcpy(d.h_nprim, nprim, sizeof(int32_t) * n_shells);
    std::memcpy(d.h_center, center_of_shell, sizeof(int32_t) * n_shells);
    d.n_fams = (int)fam_prim.size();
    d.h_fam = new int32_t[n_shells];
    d.h_fam_prim = new int32_t[d.n_fams];
    d.h_fam_k = new int32_t[d.n_fams];
    std::memcpy(d.h_fam, fam.data(), sizeof(int32_t) * n_shells);
    std::memcpy(d.h_fam_prim, fam_prim.data(), sizeof(int32_t) * d.n_fams);
    std::memcpy(d.h_fam_k, fam_k.data(), sizeof(int32_t) * d.n_fams);
    if (cudaMalloc(&d.shells, sizeof(ShellRec) * n_shells) != cudaSuccess ||
        cudaMalloc(&d.prims, sizeof(PrimRec) * n_prims) != cudaSuccess ||
        cudaMalloc(&d.centers, sizeof(Vec4) * n_centers) != cudaSuccess ||
        cudaMalloc(&d.xprims, sizeof(XPrim) * n_prims) != cudaSuccess ||
        cudaMalloc(&d.screen, sizeof(ScreenRec) * n_shells) != cudaSuccess) {
        shg_basis_destroy(b);
        return fail(SHG_ENOMEM, "basis: cudaMalloc failed");
    }
    if (cudaMemcpy(d.shells, sh.data(), sizeof(ShellRec) * n_shells, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(d.prims, pr.data(), sizeof(PrimRec) * n_prims, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(d.centers, ctr.data(), sizeof(Vec4) * n_centers, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(d.xprims, xpr.data(), sizeof(XPrim) * n_prims, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(d.screen, scr.data(), sizeof(ScreenRec) * n_shells, cudaMemcpyHostToDevice) != cudaSuccess) {
        shg_basis_destroy(b);
        return fail(SHG_ECUDA, "basis: upload failed");
    }
    if (!device_tables()) {
        shg_basis_destroy(b);
        return SHG_ECUDA;
    }
    count_user(d.device, 1);
    d.counted = true;
    *out = b;
    return SHG_OK;
}

int shg_basis_set_centers(shg_basis_t *b, const double *centers)
{
    Phase phase_("shg:set_centers");
    g_err.clear();
    if (!b || !centers) return fail(SHG_EINVAL, "NULL argument");
    BasisDev &d = b->d;
    const int n = d.n_centers;
    if (n == 0) return SHG_OK;
    if (!d.stage_raw) {
        if (cudaMalloc(&d.stage_raw, sizeof(double) * 3 * n) != cudaSuccess ||
            cudaMalloc(&d.stage_ctr, sizeof(Vec4) * n) != cudaSuccess ||
            cudaMalloc(&d.stage_bad, sizeof(int)) != cudaSuccess) {
            cudaFree(d.stage_raw);
            cudaFree(d.stage_ctr);
            cudaFree(d.stage_bad);
            d.stage_raw = nullptr;
            d.stage_ctr = nullptr;
            d.stage_bad = nullptr;
            return fail(SHG_ENOMEM, "set_centers: cudaMalloc failed");
        }
    }
    // the legacy default stream orders this against work on blocking streams
    const cudaStream_t s = 0;
    SHG_CUDA(cudaMemcpyAsync(d.stage_raw, centers, sizeof(double) * 3 * n, cudaMemcpyHostToDevice, s));
    SHG_CUDA(cudaMemsetAsync(d.stage_bad, 0x7f, sizeof(int), s));
    SHG_CUDA(launch_pack_centers(d.stage_raw, n, d.stage_ctr, d.stage_bad, s));
    int bad = 0;
    SHG_CUDA(cudaMemcpyAsync(&bad, d.stage_bad, sizeof(int), cudaMemcpyDeviceToHost, s));
    SHG_CUDA(cudaStreamSynchronize(s));
    if (bad < n) return fail(SHG_EINVAL, "center %d has a non-finite coordinate", bad);
    SHG_CUDA(cudaMemcpyAsync(d.centers, d.stage_ctr, sizeof(Vec4) * n, cudaMemcpyDeviceToDevice, s));
    SHG_CUDA(cudaStreamSynchronize(s));
    return SHG_OK;
}

void shg_basis_destroy(shg_basis_t *b)
{
    if (!b) return;
    cudaFree(b->d.shells);
    cudaFree(b->d.prims);
    cudaFree(b->d.centers);
    cudaFree(b->d.xprims);
    cudaFree(b->d.screen);
    cudaFree(b->d.stage_raw);
    cudaFree(b->d.stage_ctr);
    cudaFree(b->d.stage_bad);
    if (b->d.counted) count_user(b->d.device, -1);
    delete[] b->d.h_l;
    delete[] b->d.h_nprim;
    delete[] b->d.h_center;
    delete[] b->d.h_fam;
    delete[] b->d.h_fam_prim;
    delete[] b->d.h_fam_k;
    delete b;
}

int64_t shg_basis_nshells(const shg_basis_t *b) { return b ? b->d.n_shells : 0; }
int64_t shg_basis_nprims(const shg_basis_t *b) { return b ? b->d.n_prims : 0; }

int64_t shg_pair_offsets(const shg_basis_t *b, int64_t n, const int32_t *pa, const int32_t *pb, int64_t *offsets)
{
    g_err.clear();
    if (!b || n < 0 || (n > 0 && (!pa || !pb || !offsets))) return fail(SHG_EINVAL, "bad argument");
    int64_t tot = 0;
    for (int64_t p = 0; p < n; ++p) {
        if (pa[p] < 0 || pa[p] >= b->d.n_shells || pb[p] < 0 || pb[p] >= b->d.n_shells)
            return fail(SHG_EINVAL, "pair %lld: shell index out of range", (long long)p);
        offsets[p] = tot;
        tot += (int64_t)(2 * b->d.h_l[pa[p]] + 1) * (2 * b->d.h_l[pb[p]] + 1);
    }
    return tot;
}

int64_t shg_triple_offsets(const shg_basis_t *orb, const shg_basis_t *aux, int64_t n, const int32_t *ta,
                           const int32_t *tt, const int32_t *tb, int64_t *offsets)
{
    g_err.clear();
    if (!orb || !aux || n < 0 || (n > 0 && (!ta || !tt || !tb || !offsets))) return fail(SHG_EINVAL, "bad argument");
    int64_t tot = 0;
    for (int64_t p = 0; p < n; ++p) {
        if (ta[p] < 0 || ta[p] >= orb->d.n_shells || tt[p] < 0 || tt[p] >= orb->d.n_shells || tb[p] < 0 ||
            tb[p] >= aux->d.n_shells)
            return fail(SHG_EINVAL, "triple %lld: shell index out of range", (long long)p);
        offsets[p] = tot;
        tot += (int64_t)(2 * orb->d.h_l[ta[p]] + 1) * (2 * orb->d.h_l[tt[p]] + 1) * (2 * aux->d.h_l[tb[p]] + 1);
    }
    return tot;
}

} // extern "C"
int shg::plan_read(PlanDev &d, const int *summary, int schedule)
{
    if (summary[kNClass + 1])
        return fail(SHG_EINVAL, "pair list holds a shell index outside 0..%d", d.basis->n_shells - 1);
    d.n_tiles = summary[kNClass];
    for (int c = 0; c <= kNClass; ++c) d.class_tile_begin[c] = summary[c];
    const int *first = summary + kNClass + 2;
    TileMap &m = d.map;
    m.tile[0] = 0;
    for (int c = 0; c < kNClass; ++c) {
        m.pair[c] = first[c];
        m.pair[c + 1] = c + 1 < kNClass ? first[c + 1] : (int)d.n_pairs;
        m.tile[c + 1] = m.tile[c] + (m.pair[c + 1] - m.pair[c] + kTile - 1) / kTile;
        m.cls[c] = g_chunk_class[schedule][c];
    }
    // register cap: with more registers per thread the accumulators of high J stay in registers, with fewer more warps
    // hide the latency of the low-J classes (J <= 2), which need few
    int low = 0;
    for (int c = 0; c < kNClass; ++c)
        if (std::min(m.cls[c] / 7, m.cls[c] % 7) <= 1) low += summary[c + 1] - summary[c];
    d.variant = 3 * (int64_t)low > 2 * (int64_t)d.n_tiles ? 1 : 0;
    d.df_begin = d.df_end = 0;
    if (schedule == SHG_SCHED_PERSISTENT) {
        // the persistent rank order is J-major (J descending): the classes with both l >= kMixedFp64MinL are its first
        // chunks, the double-float classes the next
        int n_from[3] = {};
        for (int cls = 0; cls < kNClass; ++cls) {
            n_from[0] += min_l(cls) >= kMixedFp64MinL;
            n_from[1] += min_l(cls) >= kMixedDfMinL;
            n_from[2] += min_l(cls) >= kMixedDfMinLGrad;
        }
        d.df_begin = summary[n_from[0]];
        d.df_end = summary[n_from[1]];
        d.df_end_grad = summary[n_from[2]];
    }
    return SHG_OK;
}
extern "C" {

int shg_plan_2c_create(const shg_basis_t *basis, int64_t n, const int32_t *pa, const int32_t *pb, int schedule,
                       void *stream, shg_plan_t **out)
{
    Phase phase_("shg:plan_2c_create");
    g_err.clear();
    if (!out) return fail(SHG_EINVAL, "out is NULL");
    *out = nullptr;
    if (!basis) return fail(SHG_EINVAL, "basis is NULL");
    if (n < 0 || n > (int64_t)INT32_MAX / 2) return fail(SHG_ERANGE, "n_pairs %lld out of range", (long long)n);
    if (n > 0 && (!pa || !pb)) return fail(SHG_EINVAL, "NULL pair list");
    if (schedule != SHG_SCHED_PER_CLASS && schedule != SHG_SCHED_PERSISTENT)
        return fail(SHG_EINVAL, "bad schedule %d", schedule);
    int r = current_device_matches(basis->d.device);
    if (r) return r;
    int *ranks[2];
    if (!device_tables_impl(ranks)) return SHG_ECUDA;
    cudaStream_t s = (cudaStream_t)stream;

    const int64_t max_tiles = plan_max_tiles(n, kNClass);
    const size_t bytes_perm = sizeof(int32_t) * (size_t)std::max<int64_t>(n, 1);
    const size_t bytes_tiles = sizeof(Tile) * (size_t)max_tiles;
    const size_t bytes_ws = sizeof(int) * plan_ws_ints(n, kNBins, kNClass);
    const size_t bytes = bytes_perm + bytes_tiles + bytes_ws + 256;
    void *blk = nullptr;
    SHG_CUDA(plan_alloc(&blk, bytes, s));

    shg_plan_t *p = new (std::nothrow) shg_plan_t;
    if (!p) {
        cudaFreeAsync(blk, s);
        return fail(SHG_ENOMEM, "host allocation failed");
    }
    PlanDev &d = p->d;
    d.basis = &basis->d;
    d.n_pairs = n;
    d.schedule = schedule;
    d.pair_a = pa;
    d.pair_b = pb;
    d.owner_block = blk;
    d.device = basis->d.device;
    d.stream = s;
    char *c = (char *)blk;
    d.tiles = (Tile *)c;                 c += (bytes_tiles + 15) / 16 * 16;
    d.perm = (int32_t *)c;               c += (bytes_perm + 15) / 16 * 16;
    d.counter = (int *)c;                c += 16;
    int *ws = (int *)c;

    auto cleanup = [&](int code) {
        cudaFreeAsync(blk, s);
        delete p;
        return code;
    };
    cudaError_t e = launch_plan_build(d, ws, kNBins, ranks[schedule], s);
    if (e != cudaSuccess) return cleanup(fail(SHG_ECUDA, "plan build: %s", cudaGetErrorString(e)));
    // first tile and first pair of every class chunk, the tile count and the error flag, in one read-back
    int summary[2 * kNClass + 2];
    if (cudaMemcpyAsync(summary, plan_summary(ws, kNBins), sizeof(summary), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return cleanup(fail(SHG_ECUDA, "plan build: %s", cudaGetErrorString(cudaGetLastError())));
    if ((r = plan_read(d, summary, schedule)) != SHG_OK) return cleanup(r);
    if (schedule == SHG_SCHED_PERSISTENT) {
        p->launches = d.n_tiles > 0 ? 1 : 0;
    } else {
        p->launches = 0;
        for (int cls = 0; cls < kNClass; ++cls) p->launches += d.class_tile_begin[cls + 1] > d.class_tile_begin[cls];
    }
    count_user(d.device, 1);
    *out = p;
    return SHG_OK;
}

int shg_plan_launches(const shg_plan_t *p) { return p ? p->launches : 0; }

int shg_plan_launches_prec(const shg_plan_t *p, int precision)
{
    if (!p || (precision != SHG_PREC_FP64 && precision != SHG_PREC_MIXED)) return -1;
    if (precision == SHG_PREC_FP64 || p->d.schedule != SHG_SCHED_PERSISTENT) return p->launches;
    const int df = p->d.df_end - p->d.df_begin;
    return (df > 0) + (p->d.n_tiles > df);
}

int64_t shg_plan_tiles(const shg_plan_t *p) { return p ? p->d.n_tiles : -1; }

int shg_plan_2c_set_variant(shg_plan_t *p, int variant)
{
    g_err.clear();
    if (!p) return fail(SHG_EINVAL, "plan is NULL");
    if (variant < 0 || variant > 2) return fail(SHG_EINVAL, "kernel variant must be 0, 1 or 2");
    p->d.variant = variant;
    return SHG_OK;
}

int shg_plan_2c_set_launch(shg_plan_t *p, int threads, int ctas_per_sm)
{
    g_err.clear();
    if (!p) return fail(SHG_EINVAL, "plan is NULL");
    if (threads != 32 && threads != 64 && threads != 128) return fail(SHG_EINVAL, "threads per CTA must be 32, 64 or 128");
    if (ctas_per_sm < 0 || ctas_per_sm > 64) return fail(SHG_EINVAL, "ctas_per_sm must be 0..64");
    p->d.threads = threads;
    p->d.ctas_per_sm = ctas_per_sm;
    return SHG_OK;
}

struct shg_graph {
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
};

// Capture the launches `issue` makes on a private stream into an instantiated graph.
extern "C++" {
template <class F>
static int capture_graph(F issue, shg_graph_t **out)
{
    cudaStream_t s = nullptr;
    SHG_CUDA(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
    cudaError_t e = cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) {
        cudaStreamDestroy(s);
        return fail(SHG_ECUDA, "cudaStreamBeginCapture: %s", cudaGetErrorString(e));
    }
    const int rc = issue(s);
    std::string msg = g_err;
    cudaGraph_t graph = nullptr;
    e = cudaStreamEndCapture(s, &graph);
    cudaStreamDestroy(s);
    if (rc != SHG_OK) {
        if (graph) cudaGraphDestroy(graph);
        return fail(rc, "capture: %s", msg.c_str());
    }
    if (e != cudaSuccess) return fail(SHG_ECUDA, "cudaStreamEndCapture: %s", cudaGetErrorString(e));
    cudaGraphExec_t exec = nullptr;
    e = cudaGraphInstantiate(&exec, graph, 0);
    if (e != cudaSuccess) {
        cudaGraphDestroy(graph);
        return fail(SHG_ECUDA, "cudaGraphInstantiate: %s", cudaGetErrorString(e));
    }
    shg_graph_t *g = new (std::nothrow) shg_graph_t;
    if (!g) {
        cudaGraphExecDestroy(exec);
        cudaGraphDestroy(graph);
        return fail(SHG_ENOMEM, "host allocation failed");
    }
    g->graph = graph;
    g->exec = exec;
    *out = g;
    return SHG_OK;
}
}  // extern "C++"

int shg_graph_2c_create(shg_plan_t *p, int n_ops, const int *ops, const double *omegas, int precision,
                        const int64_t *off, double *const *outs, shg_graph_t **out)
{
    g_err.clear();
    if (!out) return fail(SHG_EINVAL, "out is NULL");
    *out = nullptr;
    if (!p || n_ops < 1 || !ops || !omegas || !outs) return fail(SHG_EINVAL, "bad argument");
    for (int i = 0; i < n_ops; ++i) {
        int r = check_op(ops[i], omegas[i], precision);
        if (r) return r;
    }
    return capture_graph(
        [&](cudaStream_t s) {
            int rc = SHG_OK;
            for (int i = 0; i < n_ops && rc == SHG_OK; ++i)
                rc = shg_plan_2c_exec(p, ops[i], omegas[i], 0.0, precision, off, outs[i], s);
            return rc;
        },
        out);
}

int shg_graph_launch(shg_graph_t *g, void *stream)
{
    Phase phase_("shg:graph_launch");
    g_err.clear();
    if (!g) return fail(SHG_EINVAL, "graph is NULL");
    SHG_CUDA(cudaGraphLaunch(g->exec, (cudaStream_t)stream));
    return SHG_OK;
}

void shg_graph_destroy(shg_graph_t *g)
{
    if (!g) return;
    cudaGraphExecDestroy(g->exec);
    cudaGraphDestroy(g->graph);
    delete g;
}

void shg_plan_destroy(shg_plan_t *p)
{
    if (!p) return;
    cudaFreeAsync(p->d.owner_block, p->d.stream);
    count_user(p->d.device, -1);
    delete p;
}


static int exec_fp64(shg_plan_t *p, int op, double omega, double screen, const int64_t *off, double *out,
                     const double *o_pre, cudaStream_t s);
static int exec_fused_fp64(shg_plan_t *p, ArgsFused &a, cudaStream_t s);
static int exec_mixed(shg_plan_t *p, const ArgsFused &f, cudaStream_t s);

int shg_plan_2c_exec(shg_plan_t *p, int op, double omega, double screen, int precision, const int64_t *off,
                     double *out, void *stream)
{
    Phase phase_("shg:plan_2c_exec");
    g_err.clear();
    if (!p) return fail(SHG_EINVAL, "plan is NULL");
    int r = check_op(op, omega, precision);
    if (r) return r;
    if (!(screen >= 0.0) || !std::isfinite(screen)) return fail(SHG_EINVAL, "screening threshold must be >= 0");
    if (p->d.n_pairs == 0 || p->d.n_tiles == 0) return SHG_OK;
    if (!off || !out) return fail(SHG_EINVAL, "NULL output");
    r = current_device_matches(p->d.basis->device);
    if (r) return r;
    const DeviceTables *t = device_tables();
    if (!t) return SHG_ECUDA;
    cudaStream_t s = (cudaStream_t)stream;
    if (precision == SHG_PREC_MIXED) {
        ArgsFused f;
        fused_ops(f, 1, &op, &omega, &out);
        fused_plan(f, *p->d.basis, p->d, *t, off);
        f.screen_thresh = op == SHG_OP_OVERLAP || op == SHG_OP_GAUSS ? screen : 0.0;
        return exec_mixed(p, f, s);
    }
    return exec_fp64(p, op, omega, screen, off, out, nullptr, s);
}

} // extern "C"
namespace shg {
void fused_ops(ArgsFused &a, int n_ops, const int *ops, const double *omegas, double *const *outs)
{
    double w_erf = 0, w_erfc = 0, w_gauss = 0;
    for (int i = 0; i < 6; ++i) a.out[i] = nullptr;
    for (int i = 0; i < n_ops; ++i) {
        a.out[ops[i]] = outs[i];
        if (ops[i] == SHG_OP_ERF) w_erf = omegas[i];
        if (ops[i] == SHG_OP_ERFC) w_erfc = omegas[i];
        if (ops[i] == SHG_OP_GAUSS || ops[i] == SHG_OP_GAUSS_COULOMB) w_gauss = omegas[i];
    }
    a.r.erf = x_omega(w_erf);
    a.r.erfc = x_omega(w_erfc);
    a.r.gauss = x_omega(w_gauss);
    const bool ov = a.out[SHG_OP_OVERLAP], co = a.out[SHG_OP_COULOMB], ec = a.out[SHG_OP_ERFC],
               er = a.out[SHG_OP_ERF], ga = a.out[SHG_OP_GAUSS];
    a.r.want = (ov ? kSumOv : 0) | (co || ec ? kSumCo : 0) | (er ? kSumEr : 0) |
               (ec && !(er && w_erf == w_erfc) ? kSumX : 0) | (ga ? kSumGa : 0) |
               (a.out[SHG_OP_GAUSS_COULOMB] ? kSumGc : 0);
    a.screen_thresh = 0.0;
    a.screen_omega = w_gauss;
}

void fused_plan(ArgsFused &a, const BasisDev &b, const PlanDev &d, const DeviceTables &t, const int64_t *off)
{
    a.shells = b.shells;
    a.centers = b.centers;
    a.pair_a = d.pair_a;
    a.pair_b = d.pair_b;
    a.perm = d.perm;
    a.tiles = d.tiles;
    a.out_off = reinterpret_cast<const long long *>(off);
    a.r.prims = b.xprims;
    a.r.t = t.x;
    a.cg = t.cg;
    a.screen = b.screen;
    a.k = consts();
}
}  // namespace shg
extern "C" {

// FP64 execution of a plan; o_pre != null runs the angular part on
// precomputed contracted radial terms (op = OP_PRE, family path).
static int exec_fp64(shg_plan_t *p, int op, double omega, double screen, const int64_t *off, double *out,
                     const double *o_pre, cudaStream_t s)
{
    const DeviceTables *t = device_tables();
    if (!t) return SHG_ECUDA;
    const int precision = SHG_PREC_FP64;
    if (op <= SHG_OP_GAUSS_COULOMB) {
        ArgsFused f;
        fused_ops(f, 1, &op, &omega, &out);
        fused_plan(f, *p->d.basis, p->d, *t, off);
        f.screen_thresh = op == SHG_OP_OVERLAP || op == SHG_OP_GAUSS ? screen : 0.0;
        return exec_fused_fp64(p, f, s);
    }
    Args2c a;
    a.shells = p->d.basis->shells;
    a.prims = p->d.basis->prims;
    a.centers = p->d.basis->centers;
    a.pair_a = p->d.pair_a;
    a.pair_b = p->d.pair_b;
    a.perm = p->d.perm;
    a.map = p->d.map;
    a.out_off = reinterpret_cast<const long long *>(off);
    a.out = out;
    a.omega = omega;
    a.o_pre = o_pre;
    a.cg = t->cg;
    a.k = consts();
    if (p->d.schedule == SHG_SCHED_PERSISTENT) {
        a.tile_begin = 0;
        a.tile_end = p->d.map.tile[kNClass];
        SHG_CUDA(cudaMemsetAsync(p->d.counter, 0, sizeof(int), s));
        a.counter = p->d.counter;
        SHG_CUDA(launch_2c(a, op, precision, persistent_grid_2c(op, precision, p->d.threads, p->d.ctas_per_sm), true, s,
                           p->d.threads));
    } else {
        a.counter = nullptr;
        for (int c = 0; c < kNClass; ++c) {
            a.tile_begin = p->d.map.tile[c];
            a.tile_end = p->d.map.tile[c + 1];
            if (a.tile_end <= a.tile_begin) continue;
            SHG_CUDA(launch_2c(a, op, precision, 0, false, s, p->d.threads));
        }
    }
    return SHG_OK;
}

// Most tiles that a pass of a persistent plan runs with one CTA each instead of a work counter: all of them are resident at
// once (8 warps or more per SM), spread over the SMs one by one, without the launch that clears the counter (63 tiles of
// 2,000 pairs, overlap and 1/r: 102 us persistent with four-warp CTAs, 95 us with one-warp CTAs)
constexpr int kStaticTiles = SHG_SHORT_LIST_TILES;

// Radial sums of one operator
static unsigned want_of(int op)
{
    switch (op) {
    case SHG_OP_OVERLAP: return kSumOv;
    case SHG_OP_COULOMB: return kSumCo;
    case SHG_OP_ERFC: return kSumCo | kSumX;
    case SHG_OP_ERF: return kSumEr;
    case SHG_OP_GAUSS: return kSumGa;
    default: return kSumGc;
    }
}

// Parts that a pass of a persistent plan over the operators `ops` (bits) is launched in: one per operator (1/r and erfc
// count as one) where all of them take at most kStaticTiles warps, else one
static int pass_parts(const PlanDev &d, unsigned ops)
{
    const unsigned pair = 1u << SHG_OP_COULOMB | 1u << SHG_OP_ERFC;
    int n = (ops & pair) == pair ? -1 : 0;
    for (int op = 0; op < 6; ++op) n += ops >> op & 1;
    return n > 1 && (int64_t)n * d.n_tiles <= kStaticTiles ? n : 1;
}

// Pass over a list of at most kStaticTiles tiles.  With few enough they leave most warp slots empty, so each operator gets
// a launch of its own, all side by side (1/r and erfc, which share their sums, together): 2,000 pairs of short
// contractions, overlap and 1/r, 101 us in one launch, 74 in two; five operators 170 and 107 us.  Beyond the limit the
// common work of one launch tells (10,000 pairs, five operators: 174 and 234 us).  The kernels of one operator and of
// several give the same bits.
static int exec_short(shg_plan_t *p, const ArgsFused &f, bool mixed, cudaStream_t s)
{
    const bool pair = f.out[SHG_OP_COULOMB] && f.out[SHG_OP_ERFC];
    unsigned ops = 0;
    for (int op = 0; op < 6; ++op) ops |= f.out[op] ? 1u << op : 0u;
    const bool split = pass_parts(p->d, ops) > 1;
    ArgsMixFused m;
    if (mixed) m.kappa = kappa_mix();
    bool beside = false;
    for (int op = 0; op < 6; ++op) {
        if (!f.out[op] || (pair && op == SHG_OP_ERFC)) continue;
        ArgsFused a = f;
        if (split) {
            for (int i = 0; i < 6; ++i)
                if (i != op && !(pair && op == SHG_OP_COULOMB && i == SHG_OP_ERFC)) a.out[i] = nullptr;
            a.r.want = want_of(a.out[SHG_OP_ERFC] ? SHG_OP_ERFC : op);
        }
        a.counter = nullptr;
        a.tile_begin = 0;
        a.tile_end = p->d.n_tiles;
        if (mixed && p->d.df_end > p->d.df_begin) {
            m.f = a;
            m.f.tile_begin = p->d.df_begin;
            m.f.tile_end = p->d.df_end;
            m.f.beside = beside;
            SHG_CUDA(launch_2c_mixed(m, s, 32, 0, p->d.variant));
            beside = true;
            a.skip_at = p->d.df_begin;
            a.skip_n = p->d.df_end - p->d.df_begin;
        }
        a.beside = beside;
        if (a.tile_end > a.skip_n) SHG_CUDA(launch_2c_fused(a, s, 32, 0, p->d.variant));
        beside = beside || a.tile_end > a.skip_n;
        if (!split) break;
    }
    return SHG_OK;
}

// FP64 pass over the tiles of a plan
static int exec_fused_fp64(shg_plan_t *p, ArgsFused &a, cudaStream_t s)
{
    if (p->d.schedule == SHG_SCHED_PERSISTENT) {
        a.tile_begin = 0;
        a.tile_end = p->d.n_tiles;
        if (a.tile_end <= kStaticTiles) return exec_short(p, a, false, s);
        SHG_CUDA(cudaMemsetAsync(p->d.counter, 0, sizeof(int), s));
        a.counter = p->d.counter;
        SHG_CUDA(launch_2c_fused(a, s, p->d.threads, p->d.ctas_per_sm, p->d.variant));
        return SHG_OK;
    }
    a.counter = nullptr;
    for (int cls = 0; cls < kNClass; ++cls) {
        a.tile_begin = p->d.class_tile_begin[cls];
        a.tile_end = p->d.class_tile_begin[cls + 1];
        if (a.tile_end <= a.tile_begin) continue;
        SHG_CUDA(launch_2c_fused(a, s, p->d.threads, 0, p->d.variant));
    }
    return SHG_OK;
}

// Leaves the double-float classes of a mixed-precision pass out of an FP64 launch over all tiles of a plan; with a launch
// for them before it, the FP64 one runs beside it
static void skip_df(ArgsFused &f, const PlanDev &d, int df_end, int *counter)
{
    f.tile_begin = 0;
    f.tile_end = d.n_tiles;
    f.skip_at = d.df_begin;
    f.skip_n = df_end - d.df_begin;
    f.beside = f.skip_n > 0;
    f.counter = counter;
}

// Mixed-precision pass: the classes of mixed_runs_fp64 by the FP64 kernel, the others with the double-float angular part.
// A persistent plan starts the double-float launch first (its tiles are among the longest) and the FP64 one beside it.
static int exec_mixed(shg_plan_t *p, const ArgsFused &f, cudaStream_t s)
{
    ArgsMixFused m;
    m.f = f;
    m.kappa = kappa_mix();
    ArgsFused a = f;
    if (p->d.schedule == SHG_SCHED_PERSISTENT) {
        if (p->d.n_tiles <= kStaticTiles) return exec_short(p, f, true, s);
        SHG_CUDA(cudaMemsetAsync(p->d.counter, 0, 2 * sizeof(int), s));
        m.f.tile_begin = p->d.df_begin;
        m.f.tile_end = p->d.df_end;
        m.f.counter = p->d.counter + 1;
        SHG_CUDA(launch_2c_mixed(m, s, p->d.threads, p->d.ctas_per_sm, p->d.variant));
        skip_df(a, p->d, p->d.df_end, p->d.counter);
        SHG_CUDA(launch_2c_fused(a, s, p->d.threads, p->d.ctas_per_sm, p->d.variant));
        return SHG_OK;
    }
    a.counter = m.f.counter = nullptr;
    for (int cls = 0; cls < kNClass; ++cls) {
        a.tile_begin = m.f.tile_begin = p->d.class_tile_begin[cls];
        a.tile_end = m.f.tile_end = p->d.class_tile_begin[cls + 1];
        if (a.tile_end <= a.tile_begin) continue;
        if (mixed_runs_fp64(cls))
            SHG_CUDA(launch_2c_fused(a, s, p->d.threads, 0, p->d.variant));
        else
            SHG_CUDA(launch_2c_mixed(m, s, p->d.threads, 0, p->d.variant));
    }
    return SHG_OK;
}

// Checks of a fused pass: each of overlap, 1/r, erfc, erf and the Gaussian at most once, in the given precision
static int check_fused(shg_plan_t *p, int n_ops, const int *ops, const double *omegas, int precision,
                       const int64_t *off, double *const *outs)
{
    if (!p) return fail(SHG_EINVAL, "plan is NULL");
    if (n_ops < 1 || n_ops > 5) return fail(SHG_EINVAL, "n_ops must be 1..5 (got %d)", n_ops);
    if (!ops || !omegas || !outs) return fail(SHG_EINVAL, "NULL operator, omega or output array");
    unsigned seen = 0;
    for (int i = 0; i < n_ops; ++i) {
        const int op = ops[i];
        if (op < SHG_OP_OVERLAP || op > SHG_OP_GAUSS)
            return fail(SHG_EINVAL, "the fused pass takes overlap, 1/r, erfc, erf and the Gaussian only (got %d)", op);
        int r = check_op(op, omegas[i], precision);
        if (r) return r;
        if (seen >> op & 1) return fail(SHG_EINVAL, "operator %d listed twice", op);
        if (!outs[i]) return fail(SHG_EINVAL, "NULL output for operator %d", op);
        seen |= 1u << op;
    }
    if (!off) return fail(SHG_EINVAL, "NULL output offsets");
    return SHG_OK;
}

int shg_plan_2c_exec_fused(shg_plan_t *p, int n_ops, const int *ops, const double *omegas, int precision,
                           const int64_t *off, double *const *outs, void *stream)
{
    Phase phase_("shg:plan_2c_exec_fused");
    g_err.clear();
    int r = check_fused(p, n_ops, ops, omegas, precision, off, outs);
    if (r) return r;
    if (p->d.n_pairs == 0 || p->d.n_tiles == 0) return SHG_OK;
    r = current_device_matches(p->d.basis->device);
    if (r) return r;
    const DeviceTables *t = device_tables();
    if (!t) return SHG_ECUDA;
    cudaStream_t s = (cudaStream_t)stream;
    ArgsFused a;
    fused_ops(a, n_ops, ops, omegas, outs);
    fused_plan(a, *p->d.basis, p->d, *t, off);
    if (precision == SHG_PREC_MIXED) return exec_mixed(p, a, s);
    return exec_fused_fp64(p, a, s);
}

int shg_plan_launches_fused(const shg_plan_t *p, int n_ops, const int *ops, int precision)
{
    const int one = shg_plan_launches_prec(p, precision);
    if (one < 0 || n_ops < 1 || n_ops > 5 || !ops) return -1;
    unsigned bits = 0;
    for (int i = 0; i < n_ops; ++i) {
        if (ops[i] < SHG_OP_OVERLAP || ops[i] > SHG_OP_GAUSS) return -1;
        bits |= 1u << ops[i];
    }
    return p->d.schedule == SHG_SCHED_PERSISTENT ? one * pass_parts(p->d, bits) : one;
}

int shg_graph_2c_create_fused(shg_plan_t *p, int n_ops, const int *ops, const double *omegas, int precision,
                              const int64_t *off, double *const *outs, shg_graph_t **out)
{
    g_err.clear();
    if (!out) return fail(SHG_EINVAL, "out is NULL");
    *out = nullptr;
    int r = check_fused(p, n_ops, ops, omegas, precision, off, outs);
    if (r) return r;
    return capture_graph(
        [&](cudaStream_t s) { return shg_plan_2c_exec_fused(p, n_ops, ops, omegas, precision, off, outs, s); }, out);
}

int shg_eval_2c(const shg_basis_t *basis, int64_t n, const int32_t *pa, const int32_t *pb, int op, double omega,
                double screen, int precision, const int64_t *off, double *out, void *stream)
{
    g_err.clear();
    int r = check_op(op, omega, precision);
    if (r) return r;
    if (n == 0) return SHG_OK;
    shg_plan_t *p = nullptr;
    r = shg_plan_2c_create(basis, n, pa, pb, SHG_SCHED_PERSISTENT, stream, &p);
    if (r) return r;
    r = shg_plan_2c_exec(p, op, omega, screen, precision, off, out, stream);
    shg_plan_destroy(p);
    return r;
}

static int eval_3c_common(const shg_basis_t *orb, const shg_basis_t *aux, int64_t n, const int32_t *ta,
                          const int32_t *tt, const int32_t *tb, int precision, const int64_t *off, double *out,
                          const double *w, double *grad_a, double *grad_b, void *stream, double screen = 0.0)
{
    Phase phase_("shg:eval_3c");
    if (!orb || !aux) return fail(SHG_EINVAL, "basis is NULL");
    if (precision != SHG_PREC_FP64 && (precision != SHG_PREC_MIXED || grad_a))
        return fail(SHG_EINVAL, "precision %d not available for the (aab) %s", precision,
                    grad_a ? "gradient" : "integrals");
    if (n < 0 || n > (int64_t)INT32_MAX / 2) return fail(SHG_ERANGE, "n_triples %lld out of range", (long long)n);
    if (n == 0) return SHG_OK;
    if (!ta || !tt || !tb || !off || (!out && !grad_a)) return fail(SHG_EINVAL, "NULL device pointer");
    int r = current_device_matches(orb->d.device);
    if (r) return r;
    if (aux->d.device != orb->d.device) return fail(SHG_EINVAL, "orb and aux bases live on different devices");
    int *ranks[2], *rank3 = nullptr;
    const DeviceTables *t = device_tables_impl(ranks, &rank3);
    if (!t) return SHG_ECUDA;
    cudaStream_t s = (cudaStream_t)stream;

    const int64_t max_tiles = plan_max_tiles(n, kNClass3);
    const size_t bytes_perm = sizeof(int32_t) * (size_t)n;
    const size_t bytes_tiles = sizeof(Tile) * (size_t)max_tiles;
    const size_t bytes_ws = sizeof(int) * plan_ws_ints(n, kNBins3, kNClass3);
    const size_t bytes = bytes_perm + bytes_tiles + bytes_ws + 512;
    void *blk = nullptr;
    SHG_CUDA(plan_alloc(&blk, bytes, s));
    PlanDev d;
    d.basis = &orb->d;
    d.aux = &aux->d;
    d.kind = 3;
    d.n_pairs = n;
    d.schedule = SHG_SCHED_PERSISTENT;
    d.pair_a = ta;
    d.trip_t = tt;
    d.pair_b = tb;
    char *c = (char *)blk;
    d.tiles = (Tile *)c;                 c += (bytes_tiles + 15) / 16 * 16;
    d.perm = (int32_t *)c;               c += (bytes_perm + 15) / 16 * 16;
    d.counter = (int *)c;                c += 16;
    int *ws = (int *)c;
    // first tile of every class chunk, tile count and error flags
    int sm[kNClass3 + 2] = {};
    cudaError_t e = launch_plan_build(d, ws, kNBins3, rank3, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(sm, plan_summary(ws, kNBins3), sizeof(sm), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    const int h[2] = {sm[kNClass3 + 1], sm[kNClass3]};              // error flags, tile count
    if (e != cudaSuccess) {
        cudaFreeAsync(blk, s);
        return fail(SHG_ECUDA, "(aab) planning: %s", cudaGetErrorString(e));
    }
    if (h[0]) {
        cudaFreeAsync(blk, s);
        if (h[0] & 1) return fail(SHG_EINVAL, "triple list holds a shell index out of range");
        if (h[0] & 2) return fail(SHG_EINVAL, "a and a~ of a triple are not on the same center");
        return fail(SHG_EINVAL, "la + la~ exceeds %d", kLmaxAabA);
    }
    Args3c a;
    a.orb_shells = orb->d.shells;
    a.aux_shells = aux->d.shells;
    a.orb_prims = orb->d.xprims;
    a.aux_prims = aux->d.xprims;
    a.orb_centers = orb->d.centers;
    a.aux_centers = aux->d.centers;
    a.t_a = ta;
    a.t_t = tt;
    a.t_b = tb;
    a.perm = d.perm;
    a.tiles = d.tiles;
    a.tile_end = h[1];
    a.slot_doubles = 0;
    for (int c = 0; c < kNClass3; ++c)
        if (sm[c + 1] > sm[c])
            a.slot_doubles = std::max(a.slot_doubles,
                                      grad_a ? slot_doubles_3c_grad(g_chunk_class3[c]) : slot_doubles_3c(g_chunk_class3[c]));
    a.counter = d.counter;
    a.out_off = reinterpret_cast<const long long *>(off);
    a.out = out;
    a.w_off = grad_a ? reinterpret_cast<const long long *>(off) : nullptr;
    a.w = w;
    a.grad_a = grad_a;
    a.grad_b = grad_b;
    a.screen_thresh = grad_a ? 0.0 : screen;
    a.orb_screen = orb->d.screen;
    a.aux_screen = aux->d.screen;
    a.exptab = t->x.exp;
    a.cg = t->cg;
    a.k = consts();
    a.k3 = consts3();
    e = cudaMemsetAsync(d.counter, 0, sizeof(int), s);
    if (e == cudaSuccess && h[1] > 0) e = grad_a ? launch_3c_grad(a, s) : launch_3c(a, s);
    cudaFreeAsync(blk, s);
    if (e != cudaSuccess) return fail(SHG_ECUDA, "(aab) launch: %s", cudaGetErrorString(e));
    return SHG_OK;
}

int shg_eval_3c_aab(const shg_basis_t *orb, const shg_basis_t *aux, int64_t n, const int32_t *ta, const int32_t *tt,
                    const int32_t *tb, int precision, double screen, const int64_t *off, double *out, void *stream)
{
    g_err.clear();
    if (!(screen >= 0.0) || !std::isfinite(screen)) return fail(SHG_EINVAL, "screening threshold must be >= 0");
    if (n > 0 && !out) return fail(SHG_EINVAL, "NULL output");
    return eval_3c_common(orb, aux, n, ta, tt, tb, precision, off, out, nullptr, nullptr, nullptr, stream, screen);
}

int shg_eval_2c_grad(const shg_basis_t *basis, int64_t n, const int32_t *pa, const int32_t *pb, int op, double omega,
                     int precision, const int64_t *w_off, const double *w, double *grad_a, double *grad_b,
                     void *stream)
{
    Phase phase_("shg:eval_2c_grad");
    g_err.clear();
    int r = check_op(op, omega, precision);
    if (r) return r;
    if (n == 0) return SHG_OK;
    if (!w_off || !w || !grad_a) return fail(SHG_EINVAL, "NULL device pointer");
    shg_plan_t *p = nullptr;
    r = shg_plan_2c_create(basis, n, pa, pb, SHG_SCHED_PERSISTENT, stream, &p);
    if (r) return r;
    const DeviceTables *t = device_tables();
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = cudaMemsetAsync(p->d.counter, 0, 2 * sizeof(int), s);
    if (op == SHG_OP_RA2N) {
        Args2c a{};
        a.shells = basis->d.shells;
        a.prims = basis->d.prims;
        a.centers = basis->d.centers;
        a.pair_a = pa;
        a.pair_b = pb;
        a.perm = p->d.perm;
        a.map = p->d.map;
        a.tile_begin = 0;
        a.tile_end = p->d.map.tile[kNClass];
        a.counter = p->d.counter;
        a.omega = omega;
        a.w_off = reinterpret_cast<const long long *>(w_off);
        a.w = w;
        a.grad_a = grad_a;
        a.grad_b = grad_b;
        a.cg = t->cg;
        a.k = consts();
        if (e == cudaSuccess) e = launch_2c_grad_ra2n(a, s);
        shg_plan_destroy(p);
        return e == cudaSuccess ? SHG_OK : fail(SHG_ECUDA, "gradient launch: %s", cudaGetErrorString(e));
    }
    ArgsGrad a;
    double *none = nullptr;
    fused_ops(a.f, 1, &op, &omega, &none);
    // fused_ops reads the wanted sums off the outputs
    a.f.r.want = want_of(op);
    fused_plan(a.f, basis->d, p->d, *t, w_off);
    a.kappa = kappa_mix();
    a.w = w;
    a.grad_a = grad_a;
    a.grad_b = grad_b;
    // mixed precision: two launches, as exec_mixed
    if (precision == SHG_PREC_MIXED) {
        a.f.tile_begin = p->d.df_begin;
        a.f.tile_end = p->d.df_end_grad;
        a.f.counter = p->d.counter + 1;
        if (e == cudaSuccess) e = launch_2c_grad_mixed(a, s, 128);
        skip_df(a.f, p->d, p->d.df_end_grad, p->d.counter);
    } else {
        a.f.tile_begin = 0;
        a.f.tile_end = p->d.n_tiles;
        a.f.counter = p->d.counter;
    }
    if (e == cudaSuccess) e = launch_2c_grad(a, s, 128);
    shg_plan_destroy(p);
    if (e != cudaSuccess) return fail(SHG_ECUDA, "gradient launch: %s", cudaGetErrorString(e));
    return SHG_OK;
}

int shg_eval_3c_aab_grad(const shg_basis_t *orb, const shg_basis_t *aux, int64_t n, const int32_t *ta,
                         const int32_t *tt, const int32_t *tb, int precision, const int64_t *w_off, const double *w,
                         double *grad_a, double *grad_b, void *stream)
{
    g_err.clear();
    if (n > 0 && (!w || !w_off || !grad_a)) return fail(SHG_EINVAL, "NULL device pointer");
    return eval_3c_common(orb, aux, n, ta, tt, tb, precision, w_off, nullptr, w, grad_a, grad_b, stream);
}

// ------------------------------------------------------------------------- //
// Family plans                                                               //
// ------------------------------------------------------------------------- //
void shg_family_plan_destroy(shg_family_plan_t *fp)
{
    if (!fp) return;
    if (fp->plan_fam) shg_plan_destroy(fp->plan_fam);
    if (fp->plan_rest) shg_plan_destroy(fp->plan_rest);
    cudaFree(fp->block);
    delete fp;
}

int shg_family_plan_create(const shg_basis_t *basis, int64_t n, const int32_t *d_pa, const int32_t *d_pb, void *stream,
                           shg_family_plan_t **out)
{
    Phase phase_("shg:family_plan_create");
    g_err.clear();
    if (!basis || !out || n < 0 || (n > 0 && (!d_pa || !d_pb))) return fail(SHG_EINVAL, "bad argument");
    if (n > (int64_t)INT32_MAX / 2) return fail(SHG_ERANGE, "n_pairs %lld out of range", (long long)n);
    *out = nullptr;
    int r = current_device_matches(basis->d.device);
    if (r) return r;
    const BasisDev &bd = basis->d;
    std::vector<int32_t> pa(n), pb(n);
    if (n > 0) {
        SHG_CUDA(cudaMemcpy(pa.data(), d_pa, sizeof(int32_t) * n, cudaMemcpyDeviceToHost));
        SHG_CUDA(cudaMemcpy(pb.data(), d_pb, sizeof(int32_t) * n, cudaMemcpyDeviceToHost));
    }
    for (int64_t i = 0; i < n; ++i)
        if (pa[i] < 0 || pa[i] >= bd.n_shells || pb[i] < 0 || pb[i] >= bd.n_shells)
            return fail(SHG_EINVAL, "pair list holds a shell index outside 0..%d", bd.n_shells - 1);
    // family subset, grouped by (family of a, family of b)
    std::vector<std::pair<int64_t, int32_t>> keyed;
    std::vector<int32_t> rest;
    keyed.reserve(n);
    for (int64_t i = 0; i < n; ++i) {
        const int fa = bd.h_fam[pa[i]], fb = bd.h_fam[pb[i]];
        if ((int64_t)bd.h_fam_k[fa] * bd.h_fam_k[fb] <= kFamPP)
            keyed.emplace_back((int64_t)fa * bd.n_fams + fb, (int32_t)i);
        else
            rest.push_back((int32_t)i);
    }
    std::stable_sort(keyed.begin(), keyed.end(), [](const std::pair<int64_t, int32_t> &x,
                                                    const std::pair<int64_t, int32_t> &y) { return x.first < y.first; });
    const int64_t nf = (int64_t)keyed.size(), nr = (int64_t)rest.size();
    std::vector<int32_t> idx_f(nf), pa_f(nf), pb_f(nf), pa_r(nr), pb_r(nr);
    std::vector<FamGroup> groups;
    for (int64_t i = 0; i < nf; ++i) {
        const int32_t o = keyed[i].second;
        idx_f[i] = o;
        pa_f[i] = pa[o];
        pb_f[i] = pb[o];
        const int la = bd.h_l[pa[o]], lb = bd.h_l[pb[o]];
        if (i == 0 || keyed[i].first != keyed[i - 1].first) {
            const int fa = bd.h_fam[pa[o]], fb = bd.h_fam[pb[o]];
            groups.push_back(FamGroup{bd.h_fam_prim[fa], bd.h_fam_k[fa], bd.h_fam_prim[fb], bd.h_fam_k[fb], (int)i, 0,
                                      std::max(la, lb), la + lb, bd.h_center[pa[o]], bd.h_center[pb[o]], 0, 0});
        }
        FamGroup &g = groups.back();
        g.count += 1;
        g.kmin = std::min(g.kmin, std::max(la, lb));
        g.kmax = std::max(g.kmax, la + lb);
    }
    for (int64_t i = 0; i < nr; ++i) {
        pa_r[i] = pa[rest[i]];
        pb_r[i] = pb[rest[i]];
    }
    shg_family_plan_t *fp = new (std::nothrow) shg_family_plan_t;
    if (!fp) return fail(SHG_ENOMEM, "host allocation failed");
    fp->basis = &bd;
    fp->n = n;
    fp->n_fam = nf;
    fp->n_rest = nr;
    fp->n_groups = (int)groups.size();
    auto al = [](size_t b) { return (b + 255) / 256 * 256; };
    const size_t b_i32f = al(sizeof(int32_t) * (size_t)std::max<int64_t>(nf, 1));
    const size_t b_i32r = al(sizeof(int32_t) * (size_t)std::max<int64_t>(nr, 1));
    const size_t b_grp = al(sizeof(FamGroup) * (size_t)std::max(fp->n_groups, 1));
    const size_t b_o = al(sizeof(double) * kJmax * (size_t)std::max<int64_t>(nf, 1));
    const size_t b_offf = al(sizeof(int64_t) * (size_t)std::max<int64_t>(nf, 1));
    const size_t b_offr = al(sizeof(int64_t) * (size_t)std::max<int64_t>(nr, 1));
    const size_t total = 3 * b_i32f + 3 * b_i32r + b_grp + 256 + b_o + b_offf + b_offr;
    if (cudaMalloc(&fp->block, total) != cudaSuccess) {
        delete fp;
        return fail(SHG_ENOMEM, "family plan: cudaMalloc of %zu bytes failed", total);
    }
    char *c = (char *)fp->block;
    fp->d_idx_fam = (int32_t *)c; c += b_i32f;
    fp->d_pa_fam = (int32_t *)c; c += b_i32f;
    fp->d_pb_fam = (int32_t *)c; c += b_i32f;
    fp->d_idx_rest = (int32_t *)c; c += b_i32r;
    fp->d_pa_rest = (int32_t *)c; c += b_i32r;
    fp->d_pb_rest = (int32_t *)c; c += b_i32r;
    fp->d_groups = (FamGroup *)c; c += b_grp;
    fp->d_counter = (int *)c; c += 256;
    fp->d_o = (double *)c; c += b_o;
    fp->d_off_fam = (int64_t *)c; c += b_offf;
    fp->d_off_rest = (int64_t *)c;
    bool ok = true;
    if (nf > 0)
        ok = cudaMemcpy(fp->d_idx_fam, idx_f.data(), sizeof(int32_t) * nf, cudaMemcpyHostToDevice) == cudaSuccess &&
             cudaMemcpy(fp->d_pa_fam, pa_f.data(), sizeof(int32_t) * nf, cudaMemcpyHostToDevice) == cudaSuccess &&
             cudaMemcpy(fp->d_pb_fam, pb_f.data(), sizeof(int32_t) * nf, cudaMemcpyHostToDevice) == cudaSuccess &&
             cudaMemcpy(fp->d_groups, groups.data(), sizeof(FamGroup) * groups.size(), cudaMemcpyHostToDevice) ==
                 cudaSuccess;
    if (ok && nr > 0)
        ok = cudaMemcpy(fp->d_idx_rest, rest.data(), sizeof(int32_t) * nr, cudaMemcpyHostToDevice) == cudaSuccess &&
             cudaMemcpy(fp->d_pa_rest, pa_r.data(), sizeof(int32_t) * nr, cudaMemcpyHostToDevice) == cudaSuccess &&
             cudaMemcpy(fp->d_pb_rest, pb_r.data(), sizeof(int32_t) * nr, cudaMemcpyHostToDevice) == cudaSuccess;
    if (!ok) {
        shg_family_plan_destroy(fp);
        return fail(SHG_ECUDA, "family plan: upload failed");
    }
    if (nf > 0 && (r = shg_plan_2c_create(basis, nf, fp->d_pa_fam, fp->d_pb_fam, SHG_SCHED_PERSISTENT, stream,
                                          &fp->plan_fam)) != SHG_OK) {
        shg_family_plan_destroy(fp);
        return r;
    }
    if (nr > 0 && (r = shg_plan_2c_create(basis, nr, fp->d_pa_rest, fp->d_pb_rest, SHG_SCHED_PERSISTENT, stream,
                                          &fp->plan_rest)) != SHG_OK) {
        shg_family_plan_destroy(fp);
        return r;
    }
    *out = fp;
    return SHG_OK;
}

int64_t shg_family_plan_counts(const shg_family_plan_t *fp, int64_t *n_family_pairs, int64_t *n_groups)
{
    if (!fp) return -1;
    if (n_family_pairs) *n_family_pairs = fp->n_fam;
    if (n_groups) *n_groups = fp->n_groups;
    return fp->n;
}

int shg_family_plan_exec(shg_family_plan_t *fp, int op, double omega, const int64_t *off, double *out, void *stream)
{
    Phase phase_("shg:family_plan_exec");
    g_err.clear();
    if (!fp) return fail(SHG_EINVAL, "plan is NULL");
    int r = check_op(op, omega, SHG_PREC_FP64);
    if (r) return r;
    if (op == SHG_OP_RA2N) return fail(SHG_EINVAL, "SHG_OP_RA2N has no family path (its radial term depends on la)");
    if (fp->n == 0) return SHG_OK;
    if (!off || !out) return fail(SHG_EINVAL, "NULL output");
    r = current_device_matches(fp->basis->device);
    if (r) return r;
    const DeviceTables *t = device_tables();
    if (!t) return SHG_ECUDA;
    cudaStream_t s = (cudaStream_t)stream;
    if (fp->n_fam > 0) {
        SHG_CUDA(launch_gather_i64(off, fp->d_idx_fam, fp->n_fam, fp->d_off_fam, s));
        ArgsFam a;
        a.shells = fp->basis->shells;
        a.prims = fp->basis->prims;
        a.xprims = fp->basis->xprims;
        a.centers = fp->basis->centers;
        a.pair_a = fp->d_pa_fam;
        a.pair_b = fp->d_pb_fam;
        a.groups = fp->d_groups;
        a.n_groups = fp->n_groups;
        a.counter = fp->d_counter;
        a.o_pre = fp->d_o;
        a.omega = x_omega(omega);
        a.t = t->x;
        a.k = consts();
        SHG_CUDA(cudaMemsetAsync(fp->d_counter, 0, sizeof(int), s));
        SHG_CUDA(launch_family_radial(a, op, s));
        r = exec_fp64(fp->plan_fam, 7 /* OP_PRE */, omega, 0.0, fp->d_off_fam, out, fp->d_o, s);
        if (r) return r;
    }
    if (fp->n_rest > 0) {
        SHG_CUDA(launch_gather_i64(off, fp->d_idx_rest, fp->n_rest, fp->d_off_rest, s));
        r = shg_plan_2c_exec(fp->plan_rest, op, omega, 0.0, SHG_PREC_FP64, fp->d_off_rest, out, stream);
        if (r) return r;
    }
    return SHG_OK;
}

int shg_scatter_2c(const shg_basis_t *b, int64_t n, const int32_t *pa, const int32_t *pb, const int64_t *boff,
                   const double *blocks, const int64_t *ao, int64_t ld, int symmetric, double *M, void *stream)
{
    g_err.clear();
    if (!b || n < 0 || ld < 1) return fail(SHG_EINVAL, "bad argument");
    if (n == 0) return SHG_OK;
    if (!pa || !pb || !boff || !blocks || !ao || !M) return fail(SHG_EINVAL, "NULL device pointer");
    int r = current_device_matches(b->d.device);
    if (r) return r;
    SHG_CUDA(launch_scatter_2c(b->d.shells, n, pa, pb, boff, blocks, ao, ld, symmetric, M, (cudaStream_t)stream));
    return SHG_OK;
}

int shg_gather_2c(const shg_basis_t *b, int64_t n, const int32_t *pa, const int32_t *pb, const int64_t *boff,
                  const double *M, const int64_t *ao, int64_t ld, int symmetric, double *blocks, void *stream)
{
    g_err.clear();
    if (!b || n < 0 || ld < 1) return fail(SHG_EINVAL, "bad argument");
    if (n == 0) return SHG_OK;
    if (!pa || !pb || !boff || !blocks || !ao || !M) return fail(SHG_EINVAL, "NULL device pointer");
    int r = current_device_matches(b->d.device);
    if (r) return r;
    SHG_CUDA(launch_gather_2c(b->d.shells, n, pa, pb, boff, M, ao, ld, symmetric, blocks, (cudaStream_t)stream));
    return SHG_OK;
}

int shg_reduce_centers(const shg_basis_t *b, int64_t n, const int32_t *pa, const int32_t *pb, const double *ga,
                       const double *gb, double *out, void *stream)
{
    g_err.clear();
    if (!b || n < 0) return fail(SHG_EINVAL, "bad argument");
    if (n == 0) return SHG_OK;
    if (!pa || !pb || !ga || !gb || !out) return fail(SHG_EINVAL, "NULL device pointer");
    int r = current_device_matches(b->d.device);
    if (r) return r;
    SHG_CUDA(launch_reduce_centers(b->d.shells, n, pa, pb, ga, gb, out, (cudaStream_t)stream));
    return SHG_OK;
}

int shg_debug_boys(int64_t n, const double *T, int nmax, double *F, void *stream)
{
    g_err.clear();
    if (n < 0 || nmax < 0 || nmax >= kBoysOrders) return fail(SHG_EINVAL, "bad n or nmax (nmax <= %d)", kBoysOrders - 1);
    if (n == 0) return SHG_OK;
    if (!T || !F) return fail(SHG_EINVAL, "NULL pointer");
    const DeviceTables *t = device_tables();
    if (!t) return SHG_ECUDA;
    SHG_CUDA(launch_debug_boys(n, T, nmax, F, *t, (cudaStream_t)stream));
    return SHG_OK;
}

int shg_debug_pool(int reset_high, uint64_t *reserved, uint64_t *used, uint64_t *used_high)
{
    g_err.clear();
    if (!reserved || !used || !used_high) return fail(SHG_EINVAL, "NULL pointer");
    int dev = 0;
    SHG_CUDA(cudaGetDevice(&dev));
    *reserved = *used = *used_high = 0;
    cudaMemPool_t pool = dev < 64 ? pool_of(dev) : nullptr;
    if (!pool) return SHG_OK;
    SHG_CUDA(cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, reserved));
    SHG_CUDA(cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemCurrent, used));
    SHG_CUDA(cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemHigh, used_high));
    uint64_t zero = 0;
    if (reset_high) SHG_CUDA(cudaMemPoolSetAttribute(pool, cudaMemPoolAttrUsedMemHigh, &zero));
    return SHG_OK;
}

int shg_measure_alu_peak(int kind, int iters, double *flops, void *stream)
{
    g_err.clear();
    if (kind < 0 || kind > 2 || iters < 1 || !flops) return fail(SHG_EINVAL, "bad argument");
    cudaStream_t s = (cudaStream_t)stream;
    int dev = 0, sms = 0;
    SHG_CUDA(cudaGetDevice(&dev));
    SHG_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int threads = 256, blocks = sms * 8;
    double *sink = nullptr;
    SHG_CUDA(cudaMalloc(&sink, 16));
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    launch_alu_probe(kind, iters, blocks, threads, sink, s);   // warm-up
    cudaEventRecord(e0, s);
    cudaError_t le = launch_alu_probe(kind, iters, blocks, threads, sink, s);
    cudaEventRecord(e1, s);
    cudaError_t se = cudaEventSynchronize(e1);
    float ms = 0;
    cudaEventElapsedTime(&ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(sink);
    if (le != cudaSuccess || se != cudaSuccess) return fail(SHG_ECUDA, "probe failed");
    // flops per thread per chain step: one FMA (2) for kinds 0 and 1; kind 2 a
    // warp-wide m8n8k4 MMA (512 flops) shared by the warp's 32 threads (16)
    const double per = kind == 2 ? 16.0 : 2.0;
    *flops = per * 8.0 * (double)iters * threads * (double)blocks / (ms * 1e-3);
    return SHG_OK;
}

}  // extern "C"
