"""The inverse square root of the extended floats on the GPU where its FP32 seed reaches the ends of its binade: arguments
at and just below powers of four."""
import numpy as np
import pytest

from tests.parity import TOL_FP64, assert_parity, reference_2c

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def shg():
    import torch
    from paper_1701_06588_gb300 import api, build
    build.build()
    torch.cuda.init()
    return api


def test_far_boys_function_below_powers_of_four(shg):
    """F_0(T) = sqrt(pi / T) / 2 beyond the tables.  The library rounds once (2^-53), the reference three times."""
    import torch
    from paper_1701_06588_gb300 import _lib as L
    b = shg.Basis(dict(l=[0], nprim=[1], exps=[1.0], coefs=[1.0], centers=np.zeros((1, 3)), center_of=[0]))
    below = np.concatenate([np.arange(0, 200), 2.0 ** np.arange(8, 51)]) * 2.0 ** -53
    base = 4.0 ** np.arange(4, 400, 3)
    T = np.concatenate([(base[:, None] * (1 - below)).ravel(), (base[:, None] * (1 + 2 * below[:64])).ravel()])
    d_T = torch.from_numpy(T).cuda()
    F = torch.empty(len(T), dtype=torch.float64, device="cuda")
    L.shg_debug_boys(len(T), d_T, 0, F, torch.cuda.current_stream().cuda_stream)
    ref = np.sqrt(np.pi / T) / 2
    assert np.abs(F.cpu().numpy() / ref - 1).max() <= 4.5 * 2.0 ** -53
    b.close()


@pytest.mark.parametrize("l", [0, 2])
def test_exponent_sums_below_powers_of_four(shg, l):
    """alpha + beta = 4^k (1 - j 2^-53) exactly, against the oracle."""
    import torch
    c = np.repeat(4.0 ** np.arange(-4, 8), 8)
    n = len(c)
    a = 0.3125 * c
    sh = dict(l=np.full(2 * n, l, np.int32), nprim=np.ones(2 * n, np.int32),
              exps=np.stack([a, c * (1 - np.tile(np.arange(8), n // 8) * 2.0 ** -53) - a], 1).ravel(),
              coefs=np.ones(2 * n), centers=np.zeros((2 * n, 3)), center_of=np.arange(2 * n, dtype=np.int32))
    sh["centers"][1::2] = (0.7 / np.sqrt(c))[:, None] * np.array([0.48, 0.6, 0.64])
    pa, pb = np.arange(0, 2 * n, 2, dtype=np.int32), np.arange(1, 2 * n, 2, dtype=np.int32)
    b = shg.Basis(sh)
    for name, op, om in (("overlap", 0, 0.0), ("coulomb", 1, 0.0), ("erfc", 2, 0.3), ("gauss", 4, 1.0)):
        out, _ = shg.eval_2c(b, pa, pb, name, omega=om)
        ref, scale = reference_2c(sh, pa, pb, op, om)
        assert_parity(out.cpu().numpy(), ref, TOL_FP64, name, scale)
    b.close()
