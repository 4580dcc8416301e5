"""Performance cases of the integral library: what a program that uses it has it do.

A case names a path (one public call), the shells it runs on and the operators.  The shell sets follow the recipes of
the package's own workloads (independent pairs; atom clusters with orbital and auxiliary shells; molecules with one
exponent set per element), drawn here from the seed.  `exact` evaluates the same integrals in plain numpy and torch in
64 bits by another route than the library: the product of the two solid harmonics is expanded in solid harmonics
S_LM of the separation, with powers of the Laplacian acting on the radial function of R^2.
"""
import math

import numpy as np
import torch

from paper_1701_06588_gb300 import _lib, api, molecule

OMEGA = {"overlap": 0.0, "coulomb": 0.0, "erfc": 0.11, "erf": 0.11, "gauss": 1.0, "gauss_coulomb": 0.3}

# l distribution, contraction lengths, exponent range and largest separation (bohr) of a pair list
RECIPES = {
    "l3_k4": dict(l="uniform", lmax=3, k=(4, 4), exps=(0.1, 100.0), dmax=6.0),
    "l4_k8": dict(l="uniform", lmax=4, k=(1, 8), exps=(0.05, 500.0), dmax=10.0),
    "l5_k12": dict(l="uniform", lmax=5, k=(1, 12), exps=(0.05, 500.0), dmax=10.0),
    "l6_k20": dict(l="halving", lmax=6, k=None, exps=(0.03, 5000.0), dmax=10.0),
}


def listed():
    return [
        # one call on a short list held in host arrays: the metric of a small molecule, a test, an interactive session
        dict(name="eval_2k", path="eval", recipe="l3_k4", n=2000, ops="coulomb", precision="fp64"),
        # the same size with the plan kept, overlap and Coulomb metric together: one step of a small system
        dict(name="fused_2k", path="fused", recipe="l3_k4", n=2000, ops="overlap,coulomb", precision="fp64"),
        # every operator of a basis-set study over one medium list
        dict(name="fused5_200k", path="fused", recipe="l4_k8", n=200000, ops="overlap,coulomb,erfc,erf,gauss",
             precision="fp64"),
        # long contractions, 1/r and its short-range form, a large system, in both precisions
        dict(name="fused_1m", path="fused", recipe="l6_k20", n=1000000, ops="coulomb,erfc", precision="fp64"),
        dict(name="fused_1m_mixed", path="fused", recipe="l6_k20", n=1000000, ops="coulomb,erfc", precision="mixed"),
        # one operator per call, the range-separated one, on a ragged list with high angular momenta
        dict(name="single_123k_mixed", path="single", recipe="l5_k12", n=123457, ops="erfc", precision="mixed"),
        # forces: the vector-Jacobian product of a pair list, in both precisions
        dict(name="grad_250k", path="grad", recipe="l5_k12", n=250001, ops="coulomb", precision="fp64"),
        dict(name="grad_250k_mixed", path="grad", recipe="l5_k12", n=250001, ops="erfc", precision="mixed"),
        # local RI with an overlap metric: all orbital pairs of an atom with the auxiliary shells of its neighbours
        dict(name="aab_900k", path="aab", layout="orbital_pairs", n=6000, precision="fp64"),
        # the layout with the auxiliary shell on the orbital's atom, large la + la~, mixed precision
        dict(name="aab_375k_mixed", path="aab", layout="aux", n=1501, precision="mixed"),
        # forces of the local RI integrals
        dict(name="aab_grad_300k", path="aab_grad", layout="orbital_pairs", n=2001, precision="fp64"),
        # a molecule with family basis sets: blocks by the family plan, scattered into the dense matrix
        dict(name="molecule_300", path="molecule", n=300, ops="coulomb", precision="fp64"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["eval", "fused", "fused", "single", "grad", "aab", "aab_grad", "molecule"])
    precision = rng.choice(["fp64", "mixed"])
    if path == "molecule":
        return dict(path=path, n=_log_int(rng, 20, 300), ops=rng.choice(sorted(OMEGA)), precision="fp64")
    if path == "aab":
        return dict(path=path, layout=rng.choice(["orbital_pairs", "aux"]), n=_log_int(rng, 40, 1500),
                    precision=precision)
    if path == "aab_grad":
        return dict(path=path, layout=rng.choice(["orbital_pairs", "aux"]), n=_log_int(rng, 40, 900),
                    precision="fp64")
    recipe = rng.choice(sorted(RECIPES))
    if path == "fused":
        ops = rng.sample(["overlap", "coulomb", "erfc", "erf", "gauss"], rng.randint(2, 5))
        return dict(path=path, recipe=recipe, n=_log_int(rng, 1000, 400000), ops=",".join(ops), precision=precision)
    most = {"eval": 60000, "single": 400000, "grad": 250000}[path]
    return dict(path=path, recipe=recipe, n=_log_int(rng, 500, most), ops=rng.choice(sorted(OMEGA)),
                precision=precision)


# ------------------------------------------------------------------------- #
# Inputs: the angular momenta and the index lists belong to the case (they    #
# fix the sizes of the outputs), the rest to the seed                         #
# ------------------------------------------------------------------------- #
LAYOUT_SEED = 1701


def _log_uniform(rng, lo, hi, n):
    return np.exp(rng.uniform(math.log(lo), math.log(hi), n))


def _pairs(case, seed):
    """Shell 2p on center 2p and shell 2p + 1 on center 2p + 1, one geometry per pair."""
    r, n = RECIPES[case["recipe"]], case["n"]
    rng = np.random.default_rng(seed)
    p = np.ones(r["lmax"] + 1) if r["l"] == "uniform" else 2.0 ** -np.arange(r["lmax"] + 1)
    l = np.random.default_rng(LAYOUT_SEED).choice(r["lmax"] + 1, size=2 * n, p=p / p.sum()).astype(np.int32)
    if r["k"]:
        k = rng.integers(r["k"][0], r["k"][1] + 1, 2 * n).astype(np.int32)
    else:                                            # 70% short contractions, 30% of 12 to 20 primitives
        k = np.where(rng.uniform(size=2 * n) < 0.3, rng.integers(12, 21, 2 * n), rng.integers(1, 12, 2 * n))
    d = rng.standard_normal((n, 3))
    d *= (rng.uniform(0.0, r["dmax"], n) / np.linalg.norm(d, axis=1))[:, None]
    centers = np.empty((2 * n, 3))
    centers[0::2] = rng.uniform(-10.0, 10.0, (n, 3))
    centers[1::2] = centers[0::2] + d
    m = int(k.sum())
    shells = dict(l=l, nprim=k.astype(np.int32), exps=_log_uniform(rng, *r["exps"], m), coefs=rng.uniform(-1, 1, m),
                  centers=centers, center_of=np.arange(2 * n, dtype=np.int32))
    return shells, np.arange(0, 2 * n, 2, dtype=np.int32), np.arange(1, 2 * n, 2, dtype=np.int32)


def _cluster(rng, n, box, dmin=1.8):
    pos = np.empty((0, 3))
    while len(pos) < n:
        q = rng.uniform(0.0, box, 3)
        if not len(pos) or ((pos - q) ** 2).sum(1).min() >= dmin * dmin:
            pos = np.vstack([pos, q])
    return pos


def _triples(case, seed):
    """Atom pairs (A, B) of 8 clusters of 32 atoms; 5 orbital and 10 auxiliary shells per atom."""
    rng, lay = np.random.default_rng(seed), np.random.default_rng(LAYOUT_SEED)
    n_cl, n_at, n_orb, n_aux = 8, 32, 5, 10
    per = n_orb + n_aux
    centers = np.concatenate([_cluster(rng, n_at, 12.0) for _ in range(n_cl)])
    n_sh = len(centers) * per
    orb = np.arange(n_sh) % per < n_orb
    l = np.where(orb, lay.integers(0, 5, n_sh), lay.integers(0, 7, n_sh)).astype(np.int32)
    k = np.where(orb, rng.integers(1, 11, n_sh), rng.integers(1, 4, n_sh)).astype(np.int32)
    m = int(k.sum())
    shells = dict(l=l, nprim=k, exps=_log_uniform(rng, 0.1, 200.0, m), coefs=rng.uniform(-1, 1, m), centers=centers,
                  center_of=np.repeat(np.arange(len(centers), dtype=np.int32), per))
    n = case["n"]
    cl, ia = lay.integers(0, n_cl, n), lay.integers(0, n_at, n)
    ib = (ia + lay.integers(1, n_at, n)) % n_at
    if case["layout"] == "orbital_pairs":
        i, j = np.triu_indices(n_orb)
        a, t, b = np.repeat(i, n_aux), np.repeat(j, n_aux), np.tile(n_orb + np.arange(n_aux), len(i))
    else:
        a, t, b = (x.ravel() for x in np.meshgrid(np.arange(n_orb), n_orb + np.arange(n_aux), np.arange(n_orb),
                                                  indexing="ij"))
    first_a, first_b = (cl * n_at + ia)[:, None] * per, (cl * n_at + ib)[:, None] * per
    return shells, *((f + x).ravel().astype(np.int32) for f, x in ((first_a, a), (first_a, t), (first_b, b)))


def _molecule(case, seed):
    """Atoms at 0.1 per cubic bohr; every third has shells (s, s, p, p, d), the others (s, s, p); 7 exponents each."""
    rng = np.random.default_rng(seed)
    n = case["n"]
    coords = _cluster(rng, n, (n / 0.1) ** (1.0 / 3.0))
    sets = {}
    for el, ls in (("H", (0, 0, 1)), ("X", (0, 0, 1, 1, 2))):
        e = np.sort(_log_uniform(rng, 0.05, 60.0, 7))[::-1].copy()
        sets[el] = [(l, e, rng.uniform(-1.0, 1.0, 7)) for l in ls]
    return coords, ["X" if i % 3 == 0 else "H" for i in range(n)], sets


def _cuda(x):
    return torch.from_numpy(x).cuda()


def _weights(total, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 1)
    return torch.randn(total, dtype=torch.float64, device="cuda", generator=g)


def _offsets(l, *lists):
    size = np.prod([2 * l[x].astype(np.int64) + 1 for x in lists], axis=0)
    return np.concatenate([[0], np.cumsum(size)[:-1]]), int(size.sum())


def _ops(case):
    return case["ops"].split(",")


def _precision(case):
    return case["precision"]


# ------------------------------------------------------------------------- #
# The measured calls                                                          #
# ------------------------------------------------------------------------- #
def prepare(case, seed):
    s = dict(case)
    if case["path"] in ("eval", "fused", "single", "grad"):
        shells, pa, pb = _pairs(case, seed)
        s["basis"] = api.Basis(shells)
        if case["path"] == "eval":
            return dict(s, pa=pa, pb=pb)
        off, total = _offsets(shells["l"], pa, pb)
        s.update(pa=_cuda(pa), pb=_cuda(pb), off=_cuda(off))
        if case["path"] == "grad":
            return dict(s, w=_weights(total, seed))
        s["plan"] = api.Plan2c(s["basis"], s["pa"], s["pb"])
        s["outs"] = [torch.empty(total, dtype=torch.float64, device="cuda") for _ in _ops(case)]
        return s
    if case["path"] == "molecule":
        s["mol"] = molecule.Molecule(*_molecule(case, seed))
        pa, pb = s["mol"].shell_pairs()
        off, total = _offsets(s["mol"].shells["l"], pa, pb)
        s.update(pa=_cuda(pa), pb=_cuda(pb), off=_cuda(off))
        s["plan"] = api.FamilyPlan(s["mol"].basis, s["pa"], s["pb"])
        s["blocks"] = torch.empty(total, dtype=torch.float64, device="cuda")
        s["matrix"] = torch.empty((s["mol"].nao, s["mol"].nao), dtype=torch.float64, device="cuda")
        return s
    shells, ta, tt, tb = _triples(case, seed)
    s["basis"] = api.Basis(shells)
    if case["path"] == "aab":
        return dict(s, ta=ta, tt=tt, tb=tb)
    off, total = _offsets(shells["l"], ta, tt, tb)
    return dict(s, ta=_cuda(ta), tt=_cuda(tt), tb=_cuda(tb), off=_cuda(off), w=_weights(total, seed))


def run(s):
    path = s["path"]
    if path == "eval":
        op = s["ops"]
        out, off = api.eval_2c(s["basis"], s["pa"], s["pb"], op, omega=OMEGA[op], precision=_precision(s))
        return [out, off]
    if path == "fused":
        ops = _ops(s)
        return s["plan"].exec_fused(ops, s["off"], s["outs"], omegas=[OMEGA[o] for o in ops], precision=_precision(s))
    if path == "single":
        op = s["ops"]
        return [s["plan"].exec(op, s["off"], s["outs"][0], omega=OMEGA[op], precision=_precision(s))]
    if path == "grad":
        op = s["ops"]
        return api.eval_2c_grad(s["basis"], s["pa"], s["pb"], op, s["w"], offsets=s["off"], omega=OMEGA[op],
                                precision=_precision(s))
    if path == "aab":
        out, off = api.eval_3c_aab(s["basis"], s["basis"], s["ta"], s["tt"], s["tb"], precision=_precision(s))
        return [out, off]
    if path == "aab_grad":
        return api.eval_3c_aab_grad(s["basis"], s["basis"], s["ta"], s["tt"], s["tb"], s["w"], offsets=s["off"])
    mol, op = s["mol"], s["ops"]
    s["plan"].exec(op, s["off"], s["blocks"], omega=OMEGA[op])
    _lib.shg_scatter_2c(mol.basis.handle, len(s["pa"]), s["pa"], s["pb"], s["off"], s["blocks"], mol.d_ao_off,
                        mol.nao, True, s["matrix"], torch.cuda.current_stream().cuda_stream)
    return [s["matrix"]]


# ------------------------------------------------------------------------- #
# Work: bytes in and out once; flops of the contracted sums (a handful per    #
# primitive term and order) and of the angular expansion, leading terms only  #
# ------------------------------------------------------------------------- #
def work(case):
    n = case["n"]
    if case["path"] == "molecule":
        shells, nao = 11 * n / 3, 23 * n / 3
        pairs = shells * (shells + 1) / 2
        return dict(bytes=8.0 * nao * nao + 16 * pairs + 256 * shells, flops=n * n / 2 * 49 * 40 + pairs * 49 * 4)
    if case["path"] in ("aab", "aab_grad"):
        triples = n * (150 if case["layout"] == "orbital_pairs" else 250)
        size = 5 * 5 * 7 if case["layout"] == "orbital_pairs" else 5 * 7 * 5
        prims = 5.5 * 5.5 * 2
        moved = 8.0 * size + 12 + (8 + 48 if case["path"] == "aab_grad" else 8)
        return dict(bytes=triples * moved, flops=triples * (prims * 80 + size * 20.0))
    r = RECIPES[case["recipe"]]
    p = np.ones(r["lmax"] + 1) if r["l"] == "uniform" else 2.0 ** -np.arange(r["lmax"] + 1)
    mean_l = float((p * np.arange(r["lmax"] + 1)).sum() / p.sum())
    mean_k = (r["k"][0] + r["k"][1]) / 2 if r["k"] else 0.7 * 6 + 0.3 * 16
    size, nops = (2 * mean_l + 1) ** 2, len(_ops(case))
    moved = 8.0 * size * nops + 16 + 2 * (24 + 16 + 16 * mean_k) + (48 if case["path"] == "grad" else 0)
    return dict(bytes=n * moved, flops=n * nops * (mean_k ** 2 * 25 + size * (2 * mean_l + 4)))


# ------------------------------------------------------------------------- #
# 64-bit reference                                                            #
# ------------------------------------------------------------------------- #
CHUNK = 4_000_000                                    # primitive terms at a time
_PI = math.pi


def _odd(n):
    return math.prod(range(n, 1, -2))


def _solid(v, lmax):
    """Unit-normalised real solid harmonics S_lm (S_11 = x) as a dict (l, m), v = (x, y, z); orthogonal with
    int S_lm S_l'm' = 4 pi / (2l + 1) on the unit sphere."""
    x, y, z = v
    r2 = x * x + y * y + z * z
    c, s = {(0, 0): torch.ones_like(x)}, {(0, 0): torch.zeros_like(x)}
    out = {}
    for m in range(lmax + 1):
        if m:
            c[m, m] = (2 * m - 1) * (x * c[m - 1, m - 1] - y * s[m - 1, m - 1])
            s[m, m] = (2 * m - 1) * (y * c[m - 1, m - 1] + x * s[m - 1, m - 1])
        for l in range(m, lmax + 1):
            for q in (c, s):
                if l > m:
                    q[l, m] = ((2 * l - 1) * z * q[l - 1, m] - ((l + m - 1) * r2 * q[l - 2, m] if l - 2 >= m else 0)) / (l - m)
            f = math.sqrt((2.0 if m else 1.0) * math.factorial(l - m) / math.factorial(l + m))
            out[l, m] = f * c[l, m]
            if m:
                out[l, -m] = f * s[l, m]
    return out


_GAUNT = {}


def _gaunt(la, lb):
    """[(L, M, ma, mb, c)]: S_la,ma S_lb,mb = sum c r^(la+lb-L) S_LM, by quadrature exact for these degrees."""
    if (la, lb) not in _GAUNT:
        x, w = np.polynomial.legendre.leggauss(la + lb + 1)
        n = 2 * (la + lb) + 2
        ph = 2 * _PI * np.arange(n) / n
        s = np.sqrt(1 - x * x)[:, None]
        v = [torch.from_numpy(np.broadcast_to(q, (len(x), n)).flatten())
             for q in (s * np.cos(ph), s * np.sin(ph), x[:, None])]
        w = torch.from_numpy(np.repeat(w, n) * (2 * _PI / n))
        S = _solid(v, la + lb)
        got = []
        for ma in range(-la, la + 1):
            for mb in range(-lb, lb + 1):
                for L in range(abs(la - lb), la + lb + 1, 2):
                    for M in {s1 * m for m in (abs(ma) + abs(mb), abs(abs(ma) - abs(mb))) for s1 in (1, -1) if m <= L}:
                        c = float((w * S[la, ma] * S[lb, mb] * S[L, M]).sum()) * (2 * L + 1) / (4 * _PI)
                        if abs(c) > 1e-13:
                            got.append((L, M, ma, mb, c))
        _GAUNT[la, lb] = got
    return _GAUNT[la, lb]


def _boys(T, n):
    """[F_0 .. F_n](T): upward from erf for T > 30, else the power series of F_n and downward."""
    T = T.clamp_min(1e-300)
    e, t = torch.exp(-T), T.clamp_max(30.0)
    term = torch.full_like(T, 1.0 / (2 * n + 1))
    low = term.clone()
    for k in range(1, 140):
        term = term * (2 * t) / (2 * n + 2 * k + 1)
        low = low + term
    low = [torch.exp(-t) * low]
    for k in range(n, 0, -1):
        low.append((2 * t * low[-1] + torch.exp(-t)) / (2 * k - 1))
    low.reverse()
    up = [torch.sqrt(_PI / (4 * T)) * torch.erf(torch.sqrt(T))]
    for k in range(n):
        up.append(((2 * k + 1) * up[-1] - e) / (2 * T))
    return [torch.where(T > 30.0, u, lo) for u, lo in zip(up, low)]


def _radial(op, al, be, x, n):
    """d^k/dx^k, k = 0..n, of the integral over two s-type Gaussians, x = R^2."""
    om = OMEGA[op]
    c = al + be
    rho = al * be / c
    T = rho * x
    if op in ("overlap", "gauss"):
        f = rho if op == "overlap" else om * rho / (rho + om)
        g = (_PI / c) ** 1.5 if op == "overlap" else (_PI * _PI / (c * (rho + om))) ** 1.5
        g = g * torch.exp(-f * x)
        return [g * (-f) ** k for k in range(n + 1)]
    pre = 2 * _PI ** 2.5 / (al * be * torch.sqrt(c))
    if op == "gauss_coulomb":
        d = rho + om
        F = _boys(T * rho / d, n)
        g = (_PI / c) ** 1.5 * (2 * _PI / d) * torch.exp(-om * T / d)
        p, q = -om * rho / d, -rho * rho / d
        return [g * sum(math.comb(k, i) * p ** (k - i) * q ** i * F[i] for i in range(k + 1)) for k in range(n + 1)]
    got = [0.0] * (n + 1)
    if op in ("coulomb", "erfc"):
        F = _boys(T, n)
        got = [pre * (-rho) ** k * F[k] for k in range(n + 1)]
    if op in ("erf", "erfc"):
        s = om * om / (om * om + rho)
        F = _boys(s * T, n)
        sign = -1.0 if op == "erfc" else 1.0
        got = [g + sign * pre * torch.sqrt(s) * (-rho * s) ** k * F[k] for k, g in enumerate(got)]
    return got


def _laplace(L, p, x, O):
    """F with Laplacian^p [S_L(grad) G] = S_LM F: 2^L 4^p sum_i C(p,i) (L+3/2+i)...(L+1/2+p) x^i G^(L+p+i)."""
    out = 0.0
    for i in range(p, -1, -1):
        out = out * x + math.comb(p, i) * math.prod(L + 1.5 + q for q in range(i, p)) * O[L + p + i]
    return out * 2.0 ** (L + 2 * p)


def _block(la, lb, v, O):
    """(n, 2la+1, 2lb+1) block (-1)^lb S_la(grad) S_lb(grad) G from the derivatives O[k] of G."""
    x = sum(c * c for c in v)
    S = _solid(v, la + lb)
    F = {L: _laplace(L, (la + lb - L) // 2, x, O) for L in range(abs(la - lb), la + lb + 1, 2)}
    out = [[0.0] * (2 * lb + 1) for _ in range(2 * la + 1)]
    for L, M, ma, mb, c in _gaunt(la, lb):
        out[ma + la][mb + lb] = out[ma + la][mb + lb] + ((-1) ** lb * c) * (S[L, M] * F[L])
    zero = torch.zeros_like(x)
    return torch.stack([torch.stack([e + zero for e in row], -1) for row in out], -2)


class _Shells:
    """The shells on the GPU with normalised coefficients."""

    def __init__(self, sh):
        self.l = torch.from_numpy(sh["l"].astype(np.int64)).cuda()
        self.k = torch.from_numpy(sh["nprim"].astype(np.int64)).cuda()
        self.first = torch.cumsum(self.k, 0) - self.k
        self.e, c = _cuda(np.asarray(sh["exps"])), _cuda(np.asarray(sh["coefs"]))
        self.R = _cuda(np.asarray(sh["centers"]))[_cuda(sh["center_of"].astype(np.int64))]
        kmax = int(self.k.max())
        pad = torch.arange(kmax, device="cuda")
        at = (self.first[:, None] + pad).clamp_max(len(self.e) - 1)
        has = pad < self.k[:, None]
        ex, co = torch.where(has, self.e[at], 1.0), torch.where(has, c[at], 0.0)
        norm = torch.empty(len(self.l), dtype=torch.float64, device="cuda")
        step = max(1, CHUNK // (kmax * kmax))
        for lo in range(0, len(norm), step):
            e_, c_, l_ = ex[lo:lo + step], co[lo:lo + step], self.l[lo:lo + step].double()
            s = (c_[:, :, None] * c_[:, None, :] / (e_[:, :, None] + e_[:, None, :]) ** (l_[:, None, None] + 1.5)).sum((1, 2))
            # int r^(2l+2) exp(-a r^2) = Gamma(l + 3/2) / (2 a^(l+3/2)); angular part 4 pi / (2l + 1)
            norm[lo:lo + step] = torch.rsqrt(s * torch.exp(torch.lgamma(l_ + 1.5)) / 2 * 4 * _PI / (2 * l_ + 1))
        self.c = c * torch.repeat_interleave(norm, self.k)

    def terms(self, *lists):
        """Flat list of the primitive combinations of the entries: entry index and one primitive index per list."""
        ks = [self.k[x] for x in lists]
        total = torch.stack(ks).prod(0)
        ent = torch.repeat_interleave(torch.arange(len(total), device="cuda"), total)
        q = torch.arange(len(ent), device="cuda") - (torch.cumsum(total, 0) - total)[ent]
        prims = []
        for x, k in zip(reversed(lists), reversed(ks)):
            prims.append(self.first[x][ent] + q % k[ent])
            q = q // k[ent]
        return ent, prims[::-1]


def _chunks(sh, lists):
    """Entries grouped by the l of their shells, in chunks of about CHUNK primitive terms."""
    key = 0
    for x in lists:
        key = key * 7 + sh.l[x]
    count = torch.stack([sh.k[x] for x in lists]).prod(0)
    for value in torch.unique(key).tolist():
        idx = torch.nonzero(key == value).ravel()
        part = torch.cumsum(count[idx], 0) // CHUNK
        for q in range(int(part[-1]) + 1):
            sub = idx[part == q]
            if len(sub):
                yield sub, [value // 7 ** (len(lists) - 1 - i) % 7 for i in range(len(lists))]


def _sum(values, ent, n):
    return torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, ent, values)


def _orders_2c(sh, op, a, b, la, lb, x, n):
    ent, (ia, ib) = sh.terms(a, b)
    al, be = sh.e[ia], sh.e[ib]
    w = sh.c[ia] / (2 * al) ** la * sh.c[ib] / (2 * be) ** lb
    return [_sum(w * g, ent, len(a)) for g in _radial(op, al, be, x[ent], n)]


def _orders_aab(sh, a, t, b, L, p, lb, x, n):
    """Orders 0..n of the (L, p) term r^(2p) S_L exp(-(alpha + alpha~) r^2) on A with shell b (overlap)."""
    ent, (ia, it, ib) = sh.terms(a, t, b)
    al, be = sh.e[ia] + sh.e[it], sh.e[ib]
    c = al + be
    rho, g, xe = al * be / c, be * be / c, x[ent]
    w = sh.c[ia] * sh.c[it] * sh.c[ib] * (2 * al) ** -L * (2 * be) ** -lb * (_PI / c) ** 1.5 * torch.exp(-rho * xe)
    poly = [0.0] * (p + 1)                           # polynomial in x before the exponential
    for j in range(p + 1):
        rise = math.prod(L + i for i in range(j))
        if rise:
            m = p - j
            for i in range(m + 1):
                d = 2.0 ** i * _odd(2 * m + 1) * math.comb(m, i) / _odd(2 * i + 1)
                poly[i] = poly[i] + math.comb(p, j) * rise * al ** -j * (2 * c) ** -m * d * g ** i
    got = []
    for k in range(n + 1):
        val = 0.0
        for i in range(p, -1, -1):
            val = val * xe + poly[i]
        got.append(_sum(w * val, ent, len(a)))
        poly = [(i + 1) * (poly[i + 1] if i < p else 0.0) - rho * poly[i] for i in range(p + 1)]
    return got


def _aab_block(la, lt, lb, v, orders):
    """Block [m_a][m_a~][m_b] from the orders of every L of the product expansion of a a~."""
    out = 0.0
    parts = {L: _block(L, lb, v, O) for L, O in orders.items()}
    expand = {}
    for L, M, ma, mt, c in _gaunt(la, lt):
        expand.setdefault(L, torch.zeros(2 * la + 1, 2 * lt + 1, 2 * L + 1, dtype=torch.float64, device="cuda"))
        expand[L][ma + la, mt + lt, M + L] = c
    for L, G in expand.items():
        out = out + torch.einsum("atm,nmb->natb", G, parts[L])
    return out


def _vjp(block, v, tables, w):
    """d/dv of sum w block: the direct part and the part through the orders (dO^(k)/dv = 2 v O^(k+1))."""
    v = [c.detach().requires_grad_() for c in v]
    leaves = {q: [o.detach().requires_grad_() for o in O[:-1]] for q, O in tables.items()}
    flat = [o for q in tables for o in leaves[q]]
    got = torch.autograd.grad((block(v, leaves) * w).sum(), v + flat, allow_unused=True)
    chain = 0.0
    nxt = [O[k + 1] for O in tables.values() for k in range(len(O) - 1)]
    for g, o in zip(got[3:], nxt):
        chain = chain + (g * o if g is not None else 0.0)
    return torch.stack([(g if g is not None else 0.0) + 2 * c.detach() * chain for g, c in zip(got[:3], v)], -1)


def _scatter(out, start, block):
    flat = block.reshape(len(block), -1)
    out[start[:, None] + torch.arange(flat.shape[1], device="cuda")] = flat


def exact(case, seed):
    path = case["path"]
    if path in ("aab", "aab_grad"):
        raw, *lists = _triples(case, seed)
    elif path == "molecule":
        coords, elements, sets = _molecule(case, seed)
        per = [sets[e] for e in elements]
        raw = dict(l=np.array([s[0] for at in per for s in at], np.int32),
                   nprim=np.array([len(s[1]) for at in per for s in at], np.int32),
                   exps=np.concatenate([s[1] for at in per for s in at]),
                   coefs=np.concatenate([s[2] for at in per for s in at]), centers=coords,
                   center_of=np.repeat(np.arange(len(per), dtype=np.int32), [len(at) for at in per]))
        lists = [x.astype(np.int32) for x in np.triu_indices(len(raw["l"]))]
    else:
        raw, *lists = _pairs(case, seed)
    off, total = _offsets(raw["l"], *lists)
    sh = _Shells(raw)
    lists, start = [_cuda(x).long() for x in lists], _cuda(off)
    grad = path in ("grad", "aab_grad")
    w = _weights(total, seed) if grad else None
    ops = ["aab"] if path.startswith("aab") else _ops(case)
    outs = [torch.empty((len(off), 3) if grad else total, dtype=torch.float64, device="cuda") for _ in ops]
    for idx, ls in _chunks(sh, lists):
        sub = [x[idx] for x in lists]
        v = list((sh.R[sub[0]] - sh.R[sub[-1]]).T)
        x = sum(c * c for c in v)
        for op, out in zip(ops, outs):
            if op == "aab":
                la, lt, lb = ls
                tables = {L: _orders_aab(sh, *sub, L, (la + lt - L) // 2, lb, x, L + lb + grad)
                          for L in range(abs(la - lt), la + lt + 1, 2)}

                def block(v, O, la=la, lt=lt, lb=lb):
                    return _aab_block(la, lt, lb, v, O)
            else:
                la, lb = ls
                tables = {0: _orders_2c(sh, op, *sub, la, lb, x, la + lb + grad)}

                def block(v, O, la=la, lb=lb):
                    return _block(la, lb, v, O[0])
            if grad:
                size = math.prod(2 * q + 1 for q in ls)
                wb = w[start[idx][:, None] + torch.arange(size, device="cuda")]
                out[idx] = _vjp(block, v, tables, wb.reshape(len(idx), *(2 * q + 1 for q in ls)))
            else:
                _scatter(out, start[idx], block(v, tables))
    if grad:
        return outs[0], -outs[0]
    if path == "molecule":
        size = 2 * raw["l"].astype(np.int64) + 1
        ao, nao = _cuda(np.cumsum(size) - size), int(size.sum())
        m = torch.empty((nao, nao), dtype=torch.float64, device="cuda")
        for idx, (la, lb) in _chunks(sh, lists):
            a, b = (x[idx] for x in lists)
            na, nb = 2 * la + 1, 2 * lb + 1
            blk = outs[0][start[idx][:, None] + torch.arange(na * nb, device="cuda")].reshape(-1, na, nb)
            row = (ao[a][:, None] + torch.arange(na, device="cuda"))[:, :, None].expand(-1, na, nb)
            col = (ao[b][:, None] + torch.arange(nb, device="cuda"))[:, None, :].expand(-1, na, nb)
            m[row, col] = blk
            m[col, row] = blk
        return [m]
    return [outs[0], None] if path in ("eval", "aab") else outs
