"""Radial sums in extended floats at the sizes where the work mapping changes: primitive pairs per pair around the
group limits (1, 2, 4 and 8 lanes per pair), lists that end inside a tile, R = 0, the far-field limit of T, zero
coefficients and very small and large exponents, against the oracle with the FP64 bar."""
import numpy as np
import pytest

from tests.parity import TOL_FP64, TOL_MIXED, assert_parity, reference_2c

pytestmark = pytest.mark.gpu

OPS = [("overlap", 0, 0.0), ("coulomb", 1, 0.0), ("erfc", 2, 0.11), ("erf", 3, 0.11), ("gauss", 4, 1.0),
       ("gauss_coulomb", 5, 0.3)]


@pytest.fixture(scope="module")
def shg():
    import torch
    from paper_1701_06588_gb300 import api, build
    build.build()
    torch.cuda.init()
    return api


def _shells(n_pairs, ka, kb, seed, exps=(0.05, 500.0), dmax=8.0, ls=(0, 1, 2, 3)):
    rng = np.random.default_rng(seed)
    k = np.tile([ka, kb], n_pairs).astype(np.int32)
    m = int(k.sum())
    centers = rng.uniform(-3, 3, (2 * n_pairs, 3))
    d = rng.standard_normal((n_pairs, 3))
    centers[1::2] = centers[0::2] + d / np.linalg.norm(d, axis=1)[:, None] * rng.uniform(0, dmax, n_pairs)[:, None]
    centers[1] = centers[0]                                    # R = 0
    sh = dict(l=rng.choice(ls, 2 * n_pairs).astype(np.int32), nprim=k,
              exps=np.exp(rng.uniform(np.log(exps[0]), np.log(exps[1]), m)), coefs=rng.uniform(-1, 1, m),
              centers=centers, center_of=np.arange(2 * n_pairs, dtype=np.int32))
    return sh, np.arange(0, 2 * n_pairs, 2, dtype=np.int32), np.arange(1, 2 * n_pairs, 2, dtype=np.int32)


def _check(api, sh, pa, pb, ops, precision="fp64"):
    import torch
    b = api.Basis(sh)
    off, total = b.pair_offsets(pa, pb)
    plan = api.Plan2c(b, pa, pb)
    for name, op, om in ops:
        out = torch.full((total,), float("nan"), dtype=torch.float64, device="cuda")
        plan.exec(name, torch.from_numpy(off).cuda(), out, omega=om, precision=precision)
        ref, scale = reference_2c(sh, pa, pb, op, om)
        assert_parity(out.cpu().numpy(), ref, TOL_MIXED if precision == "mixed" else TOL_FP64, name, scale)
    plan.close()
    b.close()


@pytest.mark.parametrize("ka,kb", [(1, 1), (4, 8), (3, 11), (8, 8), (5, 13), (8, 16), (3, 32), (32, 32)])
def test_group_limits(shg, ka, kb):
    _check(shg, *_shells(19, ka, kb, 100 * ka + kb), OPS)


def test_mixed_group_limits(shg):
    for ka, kb in ((2, 2), (6, 7), (9, 9), (13, 12)):
        _check(shg, *_shells(11, ka, kb, 7 * ka + kb), OPS, precision="mixed")


@pytest.mark.parametrize("n", [1, 31, 32, 33])
def test_list_lengths_and_zero_coefficients(shg, n):
    sh, pa, pb = _shells(n, 3, 2, 40 + n)
    sh["coefs"][::5] = 0.0                                     # every shell keeps a primitive: 5 does not divide 3 + 2 twice
    sh["coefs"][0:5] = [0.0, 0.7, -0.2, 0.0, 1.0]
    _check(shg, sh, pa, pb, OPS[:3])


def test_far_field_limit_and_exponent_range(shg):
    """One s-type pair per T = rho R^2 around the table's end, and exponents from 1e-6 to 1e8."""
    T = np.concatenate([np.linspace(71.9, 72.1, 21), np.linspace(119.9, 120.1, 5), [0.0, 1e-30, 1 / 512, 2 / 512, 700.0]])
    n = len(T)
    sh, pa, pb = _shells(n, 1, 1, 5, ls=(0, 2, 6))
    sh["exps"][:] = 2.0                                        # rho = 1
    sh["centers"][1::2] = sh["centers"][0::2] + np.sqrt(T)[:, None] * np.array([[0.6, 0.0, 0.8]])
    _check(shg, sh, pa, pb, OPS[1:4])
    sh, pa, pb = _shells(40, 2, 3, 6, exps=(1e-6, 1e8), dmax=3.0, ls=(0, 1, 2))
    _check(shg, sh, pa, pb, [("coulomb", 1, 0.0), ("erf", 3, 40.0), ("erfc", 2, 1e-3)])
