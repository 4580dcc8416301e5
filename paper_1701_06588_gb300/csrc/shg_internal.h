// Internal declarations shared by the host API (shg_api.cpp) and the CUDA
// kernels (shg_*.cu).  Plain C++: no device code, no torch types.
#pragma once

#include <cstdint>
#include <cstddef>
#include <cuda_runtime.h>

namespace shg {

constexpr int kLmax2c = 6;        // largest l of a two-center shell
constexpr int kLmaxAabA = 10;     // largest la + la~ of an (aab) triple
constexpr int kLmaxR = 10;        // largest l of the scaled solid harmonics table
constexpr int kKmax = 32;         // largest contraction length
constexpr int kJmax = 7;          // min(la, lb) + 1 <= 7
constexpr int kRa2nMax = 5;                // largest n of the (a|r_a^{2n}|b) operator
constexpr int kNClass = (kLmax2c + 1) * (kLmax2c + 1);
constexpr int kTile = 32;         // pairs per warp tile
// Two-center classes whose angular part the mixed-precision passes evaluate in double-float: kMixedDfMinL <= min(la, lb)
// < kMixedFp64MinL (gradients: from kMixedDfMinLGrad).  Above, the angular sums cancel too much (double-float carries 2^-44
// of the largest term); below, the FP64 units, which are otherwise a third busy, take the few sums sooner than the FP32
// pipes take 18 instructions for each: 1M pairs, 1/r and erfc, 2.92 ms with all classes below 4 in double-float, 2.53 ms
// from 2 or from 3 on; 123,000 pairs, erfc, 596, 439 (from 2) and 466 us (from 3); 250,000 gradients of erfc 1.22, 1.16 and
// 1.09 ms.  Between these two limits double-float gains nothing over FP64 for every class either (1M pairs 2.48 ms, the
// 2M-pair step 4.92 against 4.84, 500,000 gradients of erfc 1.97 against 1.93): the classes kept are those where it loses
// least.
constexpr int kMixedDfMinL = 2, kMixedDfMinLGrad = 3, kMixedFp64MinL = 4;
inline int min_l(int cls) { return cls / 7 < cls % 7 ? cls / 7 : cls % 7; }
inline bool mixed_runs_fp64(int cls) { return min_l(cls) < kMixedDfMinL || min_l(cls) >= kMixedFp64MinL; }

// Boys function for the extended-float radial sums: from T = kFarT on the asymptotic form (relative error below 5e-18
// for n <= 13: T^{n-1/2} e^{-T} / Gamma(n+1/2)); below, per order n = 0..kBoysOrders-1 and cell [i, i+1) / 512 of T, the
// Taylor coefficients c_t = F_{n+t}(T_{i+1}) / t! about the upper end of the cell, scaled by 2^s so that c0 < 2^63 (1 - 2^-8): c0, c1 in units 2^-s, c2 likewise with s - 62 in its low 8 bits, c3 in units
// 2^{30-s}, c4 (24 bits) in units 2^{35-s}, c5 (8 bits) in units 2^{49-s}.  y = T_{i+1} - T <= 2^-9, so the dropped
// y^6/720 is below 2^-63.  One 32-byte load per evaluation; 18.9 MB, resident in L2.
constexpr int kFarT = 72;
constexpr int kBoysCells = kFarT * 512;
constexpr int kBoysOrders = 16;
struct alignas(32) BoysEnt {
    uint64_t c0, c1, c2;
    uint32_t c3, c45;
};
constexpr int kExpTab = 356;            // exp(j/512) 2^62, j/512 < 0.6954
struct XTab {
    const BoysEnt *boys;
    const uint64_t *exp;
};
struct XOmega {
    uint64_t w_m, w2_m;                 // omega and omega^2 as extended floats
    int w_e, w2_e;
};
// Sums a radial pass can form (bits of RadialIn::want and of the kernels' masks): overlap, 1/r, the attenuated
// part of erf, that of erfc (not when erf with the same omega is formed), Gaussian, exp(-wr^2)/r (alone)
enum { kSumOv = 1, kSumCo = 2, kSumEr = 4, kSumX = 8, kSumGa = 16, kSumAll = 31, kSumGc = 32 };

// Per-primitive record of the extended-float radial sums (32 bytes): alpha and cw as m 2^e, m in [2^62, 2^63), the sign of cw
// in bit 63 of wm,
//   cw = sqrt(2 pi^{5/2}) w2c / alpha   so that 2 pi^{5/2} w / (alpha beta sqrt(c)) = cw_a cw_b / sqrt(c)
//   fw = w2c alpha^{-3/2}       the far-field weight: for T >= kFarT every order of
//                               w 2 pi^{5/2} / (alpha beta sqrt(c)) (-rho)^n F_n(T) equals
//                               fw_a fw_b pi^3 (-1)^n (2n-1)!! (2R^2)^{-n} / R
struct alignas(32) XPrim {
    uint64_t am, wm;
    int ae, we;
    double fw;
};

// What a radial pass takes beside the pair (by value in the kernel parameters)
struct RadialIn {
    const XPrim *prims;
    XTab t;
    XOmega erf, erfc, gauss;      // gauss: also of exp(-wr^2)/r
    unsigned want;                // sums this launch forms
};

// Per-shell screening data (host-computed): smallest exponent, sum |N c| over
// the primitives, and (l / (alpha_min e))^{l/2} (1 for l = 0).
struct alignas(32) ScreenRec {
    double amin, sabs, lfac, pad;
};

// Per-shell record on the device (16 bytes): l, K, first primitive, center.
struct ShellRec {
    int l, nprim, prim_off, center;
};

// Center coordinates on the device (x, y, z, padding), 32-byte aligned.
struct alignas(32) Vec4 {
    double x, y, z, w;
};

// Per-primitive record on the device (32 bytes).
//   alpha, 1/alpha, w2c = N_l c / (2 alpha)^l (the two-center weight of
//   Eq. O_rab2_deriv), wN = N_l c (normalised coefficient).  Read by the (a|r_a^{2n}|b) kernels and, w2c, by the
//   family contraction.
struct alignas(32) PrimRec {
    double alpha, inv_alpha, w2c, wN;
};

// Small constant tables, passed by value in kernel parameters.
struct Consts {
    double A[kLmaxR + 1][kLmaxR + 1];      // A_{l,mu} of Eq. (A)
    double jB[kJmax][kJmax];               // (2j-1)!! B_{j,kappa}, Eq. (B)
    double pow2[32];                       // 2^k
    double dint[64];                       // (double) n
    double inv_int[192];                   // 1/n (0 for n = 0)
    double dfact[32];                      // (2n-1)!!, (-1)!! = 1
    double binom[kRa2nMax + 1][kRa2nMax + 1];  // C(n, j)
    double ra2n_k[kRa2nMax + 1][kRa2nMax + 1]; // 2^{d-m} (2m+1)!! C(m,d) / (2d+1)!!, [m][d], d <= m
    // low parts of jB and inv_int (value - double(value), from long double) for
    // the double-double (a|r_a^{2n}|b) path
    double jB_lo[kJmax][kJmax];
    double inv_int_lo[64];
    double kappa[16][16];                  // (l^2 - m^2) / (4 l^2 - 1): recursion of the monic Legendre functions
};

void fill_consts(Consts &k);

// Coefficients of the expanded angular part (shg_cg.cuh), per class (la, lb) with la <= kLmaxAabA, lb <= kLmax2c, class
// index c = la (kLmax2c + 1) + lb, J = min(la, lb) + 1:
//   g + gbase[c]: for every (|ma|, |mb|), row-major, J coefficients g1 of |M| = ||ma| - |mb|| and J of |M| = |ma| + |mb|
//   (p = 0..J-1, L = la + lb - 2p; 0 where L < |M|), with the norm nu_{L,M} of p_{L,M} in them
//   fc + 28 c: coefficient of R^{2(p-j)} O^{(la+lb-j)} in F_p at p (p + 1) / 2 + j, with (-1)^lb 2^{la+lb} in it
constexpr int kNClassCG = (kLmaxAabA + 1) * (kLmax2c + 1);
struct CGTab {
    const double *g;
    const int *gbase;
    const double *fc;
    const float2 *gm;             // g as double-float
    const double *h;              // g without nu_{L,M}: coefficients of S_{L,M} in S_{la,ma} S_{lb,mb} (la, lb <= kLmax2c)
};

// kappa of Consts and 1/n as double-float (mixed-precision angular part)
struct KappaMix {
    float2 v[16][16];
    float2 inv[32];
};

// Device-resident tables owned by the library, one set per device.
struct DeviceTables {
    CGTab cg;
    XTab x;
};

// Constants of the three-index kernels (by value).
struct Consts3 {
    double binom[18][18];       // binom(k, i)
    double lag[6][6];           // coefficient of u^j in the Laguerre polynomial L_m^{(1/2)}(-u)
    double K[11][6][6];         // [L][p][m]: binom(p, m) (L)_{p-m} m! (rising factorial, (0)_0 = 1)
};

void fill_consts3(Consts3 &k);

// Returns the tables of the current device (created on first use), or null
// and sets the error message.
const DeviceTables *device_tables();

// Tables of the current device if a basis was already created on it (never
// allocates); ranks[0..1] receive the bin rank tables of both schedules.
const DeviceTables *device_tables_if_ready(const int **ranks);

// Host helpers of shg_api.cpp.
int fail(int code, const char *fmt, ...);          // sets shg_last_error(), returns code
void clear_error();                                // empties shg_last_error() (start of a call)
const Consts &consts();                            // constant tables (host copy)
int check_op(int op, double omega, int precision);  // operator / omega / precision check
struct ArgsFused;
struct BasisDev;
struct PlanDev;
// operators overlap .. Gaussian of a pass (distinct, checked): sums, omegas and outputs
void fused_ops(ArgsFused &a, int n_ops, const int *ops, const double *omegas, double *const *outs);
// basis, plan and table pointers of a pass
void fused_plan(ArgsFused &a, const BasisDev &b, const PlanDev &d, const DeviceTables &t, const int64_t *off);

struct BasisDev {
    int n_shells = 0, n_centers = 0;
    int64_t n_prims = 0;
    int device = 0;
    ShellRec *shells = nullptr;   // device
    PrimRec *prims = nullptr;     // device
    Vec4 *centers = nullptr;      // device
    XPrim *xprims = nullptr;      // device, extended-float primitives (radial sums)
    ScreenRec *screen = nullptr;  // device, per-shell screening data
    // shg_basis_set_centers staging (allocated on its first call): raw
    // coordinates, a packed copy checked before it replaces the live one,
    // and the smallest non-finite center index
    double *stage_raw = nullptr;
    Vec4 *stage_ctr = nullptr;
    int *stage_bad = nullptr;
    // host copies used for validation and offsets
    int32_t *h_l = nullptr, *h_nprim = nullptr, *h_center = nullptr;
    // families: shells on one center with bitwise-identical exponent lists
    int32_t *h_fam = nullptr;                           // family of each shell
    int32_t *h_fam_prim = nullptr, *h_fam_k = nullptr;  // per family: first primitive record, K
    int n_fams = 0;
    bool counted = false;         // among the users of the plan pool of its device
};

// A warp's unit of work: up to kTile / group consecutive entries of the sorted list, all of one class (cls = la*7 + lb, or
// (la*7 + la~)*7 + lb), `group` lanes per entry, which share its primitive pairs.  Two-center pairs get the group by
// their number of primitive pairs, so that a lane sums 32 of them at most (50 beyond 256): with one lane per pair the
// longest tiles (400 one after the other) ran 1.5 ms beyond the end of all others on 200,000 pairs of long contractions
// (2.0 ms in all, 17% of the SMs' time used).  The group follows from the pair alone, so the bits of a block do not
// depend on the list it is evaluated in.
struct Tile {
    int start;
    uint16_t cls;
    uint8_t count, group;
};
constexpr int kNGroups = 4;
constexpr int kGroupOf[kNGroups] = {8, 4, 2, 1};
constexpr int kGroupMinK[kNGroups] = {129, 65, 33, 1};     // fewest primitive pairs of each group

constexpr int kKbins2c = kKmax * kKmax;      // two-center bins per class: Ka*Kb - 1
constexpr int kNBins2c = kNClass * kKbins2c;
constexpr int kNClass3 = 7 * 7 * 7;          // (la, la~, lb) classes
constexpr int kKbins3c = 512;                // three-index bins per class: min(Ka*Ka~*Kb, 512) - 1


// Class chunks of a plan in rank order: first pair of each, first 32-pair tile of each and its class.  The kernels without
// a sum over primitive pairs to share take 32 consecutive pairs of a class per warp whatever the tile list says.
struct TileMap {
    int pair[kNClass + 1] = {};
    int tile[kNClass + 1] = {};
    uint8_t cls[kNClass] = {};
};

struct PlanDev {
    const BasisDev *basis = nullptr;
    const BasisDev *aux = nullptr;  // three-index plans: basis of b
    int kind = 2;                   // 2: pairs, 3: (aab) triples
    int64_t n_pairs = 0;
    int schedule = 0;
    const int32_t *pair_a = nullptr, *pair_b = nullptr;   // device, caller-owned
    const int32_t *trip_t = nullptr;                      // a~ of triples (kind 3)
    int32_t *perm = nullptr;       // device [n_pairs], pairs sorted by bin
    Tile *tiles = nullptr;         // device [n_tiles]
    int *counter = nullptr;        // device, two persistent work counters
    int n_tiles = 0;
    TileMap map;
    int class_tile_begin[kNClass + 1] = {};   // host, per-class tile ranges (class-major)
    int df_begin = 0, df_end = 0, df_end_grad = 0;  // persistent order: tiles of the classes that the mixed-precision
                                                    // passes and gradients run in double-float
    int threads = 128;             // launch shape (autotuned): threads per CTA (32, 64 or 128)
    int ctas_per_sm = 0;           // persistent CTAs per SM, 0 = occupancy limit
    int variant = 1;               // register cap of the kernels (shg_plan_2c_set_variant)
    int device = 0;
    void *owner_block = nullptr;   // device allocation holding all of the above
    cudaStream_t stream = nullptr;
};

// Arguments of the two-center kernels (by value).
struct Args2c {
    const ShellRec *shells;
    const PrimRec *prims;
    const Vec4 *centers;
    const int32_t *pair_a, *pair_b;
    const int32_t *perm;
    TileMap map;                  // 32-pair tiles: tile_begin and tile_end count these
    int tile_begin, tile_end;
    int *counter;                 // persistent schedule (null: static)
    const long long *out_off;
    double *out;
    double omega;
    double screen_thresh;         // > 0: overlap / Gaussian-operator pairs bounded below it write zeros
    const ScreenRec *screen;
    // gradient kernels only: upstream weights W (blocks at w + w_off[p]) and
    // the per-pair outputs dI/dR_a . W and dI/dR_b . W
    const long long *w_off;
    const double *w;
    double *grad_a, *grad_b;
    // family path: contracted radial terms O[j] of pair p precomputed at
    // o_pre[p * kJmax + j] (read by the OP_PRE instantiation only)
    const double *o_pre = nullptr;
    CGTab cg;
    Consts k;
};

// Pass over overlap, 1/r, erfc, erf and the Gaussian operator, one or several of them, or exp(-wr^2)/r: one output per
// requested operator (null = not requested), all with the block offsets out_off.
struct ArgsFused {
    const ShellRec *shells;
    const Vec4 *centers;
    const int32_t *pair_a, *pair_b;
    const int32_t *perm;
    const Tile *tiles;
    int tile_begin, tile_end;
    int skip_at = INT32_MAX, skip_n = 0;  // tiles skip_at .. skip_at + skip_n - 1 are left out (a second launch takes them)
    bool beside = false;          // runs beside the launch before it on the stream, and ends after it
    int *counter;                 // persistent schedule (null: static)
    const long long *out_off;
    double *out[6];               // indexed by OP_OVERLAP .. OP_GCOUL
    RadialIn r;
    CGTab cg;
    double screen_thresh, screen_omega;   // > 0 (one operator, overlap or Gaussian): pairs bounded below it write zeros
    const ScreenRec *screen;
    Consts k;
};

// Family basis sets: a group of shell pairs whose shells a share one
// exponent set (family) on one center, and likewise for b.
constexpr int kFamPP = 100;                // largest K_a * K_b of the family path
constexpr int kFamOrd = 2 * kLmax2c + 1;   // derivative orders 0..la+lb
struct FamGroup {
    int fa_prim, fa_k, fb_prim, fb_k;   // first primitive record and K of each family
    int start, count;                   // range of the group in the grouped pair order
    int kmin, kmax;                     // derivative orders the group's pairs need
    int ca, cb, pad0, pad1;             // centers
};
struct ArgsFam {
    const ShellRec *shells;
    const PrimRec *prims;
    const XPrim *xprims;
    const Vec4 *centers;
    const int32_t *pair_a, *pair_b;     // the family subset of the pair list, in group order
    const FamGroup *groups;
    int n_groups;
    int *counter;
    double *o_pre;                      // [n_subset][kJmax]
    XOmega omega;
    XTab t;
    Consts k;
};

// Mixed-precision pass: radial sums as the FP64 pass, angular part in double-float.
struct ArgsMixFused {
    ArgsFused f;
    KappaMix kappa;
};

// Vector-Jacobian product of one operator: the pass's pair, radial and table arguments (out unused), upstream weights
// (blocks at w + f.out_off[p]) and per-pair results; kappa for the mixed-precision launch.
struct ArgsGrad {
    ArgsFused f;
    KappaMix kappa;
    const double *w;
    double *grad_a, *grad_b;      // grad_b may be null
};

// Arguments of the three-index kernels (by value).
struct Args3c {
    const ShellRec *orb_shells, *aux_shells;
    const XPrim *orb_prims, *aux_prims;
    const Vec4 *orb_centers, *aux_centers;
    const int32_t *t_a, *t_t, *t_b;
    const int32_t *perm;
    const Tile *tiles;            // kGroupOf[0] lanes per triple
    int tile_end;
    int slot_doubles;             // shared memory of a triple: the largest of the list's classes
    int *counter;
    const long long *out_off;
    double *out;
    // gradient kernel
    const long long *w_off;
    const double *w;
    double *grad_a, *grad_b;
    // screening: > 0 writes zeros for a triple whose bound on every element is below it
    double screen_thresh;
    const ScreenRec *orb_screen, *aux_screen;
    const uint64_t *exptab;
    CGTab cg;
    Consts k;
    Consts3 k3;
};

// Kernel launchers (shg_kernels.cu, shg_3c.cu).
// Planning workspace (ints): err, ticket, 2 spare, hist, bin_start, cursor
// (n_bins each), tile_start (n_bins + 1), summary (2 n_chunks + 2), key (n).
// After the build, summary[c] is the first tile of class chunk c
// (c = 0..n_chunks-1), summary[n_chunks] the number of tiles,
// summary[n_chunks + 1] the error flag of the classification and
// summary[n_chunks + 2 + c] the first pair of chunk c.
constexpr size_t plan_ws_ints(int64_t n, int n_bins, int n_chunks)
{
    return 4 + 4 * (size_t)n_bins + 1 + 2 * (size_t)n_chunks + 2 + (size_t)n;
}
// largest number of tiles of n entries: every chunk ends in at most one partial tile per group size
constexpr int64_t plan_max_tiles(int64_t n, int n_chunks)
{
    return n * kGroupOf[0] / kTile + kNGroups * n_chunks + 1;
}
// chunk -> first tile, tile count and error flag (n_chunks + 2 ints of the summary) and the tile map of a two-center plan
int plan_read(PlanDev &d, const int *summary, int schedule);
inline int *plan_summary(int *ws, int n_bins) { return ws + 4 + 4 * (size_t)n_bins + 1; }
cudaError_t launch_plan_build(PlanDev &plan, int *d_ws, int n_bins, const int *d_bin_rank, cudaStream_t s);
cudaError_t launch_3c(const Args3c &args, cudaStream_t s);
cudaError_t launch_3c_grad(const Args3c &args, cudaStream_t s);
// doubles of shared memory that a triple of a class takes
int slot_doubles_3c(int cls);
int slot_doubles_3c_grad(int cls);
// vector-Jacobian products (persistent when the counter is set, else one warp per tile): FP64, mixed precision, and
// (a|r_a^{2n}|b) (32-pair tiles of the map)
cudaError_t launch_2c_grad(const ArgsGrad &args, cudaStream_t s, int threads);
cudaError_t launch_2c_grad_mixed(const ArgsGrad &args, cudaStream_t s, int threads);
cudaError_t launch_2c_grad_ra2n(const Args2c &args, cudaStream_t s);
// double-float part of a mixed-precision pass, kMixedDfMinL <= min(la, lb) < kMixedFp64MinL (arguments as launch_2c_fused)
cudaError_t launch_2c_mixed(const ArgsMixFused &args, cudaStream_t s, int threads, int ctas_per_sm, int variant);
cudaError_t launch_2c_mixed_all(const ArgsMixFused &args, cudaStream_t s, int threads, int ctas_per_sm, int variant);
cudaError_t launch_2c(const Args2c &args, int op, int precision, int n_tiles_or_grid, bool persistent,
                      cudaStream_t s, int threads = 128);
int persistent_grid_2c(int op, int precision, int threads = 128, int ctas_per_sm = 0);
// FP64 pass of the operators in args.r.want; persistent when args.counter is set, else one warp per tile.
// ctas_per_sm: 0 = as many as fit.  variant: register cap (shg_plan_2c_set_variant)
cudaError_t launch_2c_fused(const ArgsFused &args, cudaStream_t s, int threads, int ctas_per_sm, int variant);
cudaError_t launch_2c_all(const ArgsFused &args, cudaStream_t s, int threads, int ctas_per_sm, int variant);
cudaError_t launch_2c_one(const ArgsFused &args, cudaStream_t s, int threads, int ctas_per_sm);
cudaError_t launch_pack_centers(const double *raw, int n, Vec4 *ctr, int *bad, cudaStream_t s);
cudaError_t launch_family_radial(const ArgsFam &a, int op, cudaStream_t s);
cudaError_t launch_gather_i64(const int64_t *src, const int32_t *idx, int64_t n, int64_t *dst, cudaStream_t s);
cudaError_t launch_scatter_2c(const ShellRec *shells, int64_t n, const int32_t *pa, const int32_t *pb,
                              const int64_t *boff, const double *blocks, const int64_t *ao, int64_t ld, int sym,
                              double *M, cudaStream_t s);
cudaError_t launch_gather_2c(const ShellRec *shells, int64_t n, const int32_t *pa, const int32_t *pb,
                             const int64_t *boff, const double *M, const int64_t *ao, int64_t ld, int sym,
                             double *blocks, cudaStream_t s);
cudaError_t launch_reduce_centers(const ShellRec *shells, int64_t n, const int32_t *pa, const int32_t *pb,
                                  const double *ga, const double *gb, double *out, cudaStream_t s);
cudaError_t launch_debug_boys(int64_t n, const double *T, int nmax, double *F, const DeviceTables &t,
                              cudaStream_t s);
cudaError_t launch_alu_probe(int kind, int iters, int blocks, int threads, double *sink, cudaStream_t s);

}  // namespace shg

// Opaque handles of the C ABI.
struct shg_basis {
    shg::BasisDev d;
};

struct shg_plan {
    shg::PlanDev d;
    int launches = 0;
};

// Family plan: the pairs whose shells both belong to families with
// K_a * K_b <= kFamPP, grouped by family pair, plus the rest (regular path).
struct shg_family_plan {
    const shg::BasisDev *basis = nullptr;
    int64_t n = 0, n_fam = 0, n_rest = 0;
    int n_groups = 0;
    int32_t *d_idx_fam = nullptr, *d_idx_rest = nullptr;   // original pair indices
    int32_t *d_pa_fam = nullptr, *d_pb_fam = nullptr, *d_pa_rest = nullptr, *d_pb_rest = nullptr;
    shg::FamGroup *d_groups = nullptr;
    int *d_counter = nullptr;
    double *d_o = nullptr;                                  // [n_fam][kJmax]
    int64_t *d_off_fam = nullptr, *d_off_rest = nullptr;    // offsets gathered at execution
    shg_plan *plan_fam = nullptr, *plan_rest = nullptr;
    void *block = nullptr;
};

