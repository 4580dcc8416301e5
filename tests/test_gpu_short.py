"""Short lists run one launch per operator and tile; the bits of a block do not depend on the list it is evaluated in."""
import numpy as np
import pytest

from paper_1701_06588_gb300 import workloads as W

pytestmark = pytest.mark.gpu

@pytest.fixture(scope="module")
def shg():
    import torch
    from paper_1701_06588_gb300 import api, build
    build.build()
    torch.cuda.init()
    return api


OPS = [("overlap", 0.0), ("coulomb", 0.0), ("erfc", 0.3), ("erf", 0.3), ("gauss", 0.7)]


def _blocks(shg, b, pa, pb, ops, precision, schedule):
    import torch
    off, total = b.pair_offsets(pa, pb)
    d_off = torch.from_numpy(off).cuda()
    outs = [torch.full((total,), float("nan"), dtype=torch.float64, device="cuda") for _ in ops]
    plan = shg.Plan2c(b, pa, pb, schedule=schedule)
    if len(ops) == 1:
        plan.exec(ops[0][0], d_off, outs[0], omega=ops[0][1], precision=precision)
    else:
        plan.exec_fused([o for o, _ in ops], d_off, outs, omegas=[w for _, w in ops], precision=precision)
    torch.cuda.synchronize()
    plan.close()
    return off, [o.cpu().numpy() for o in outs]


@pytest.mark.parametrize("schedule", ["persistent", "per_class"])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("ops", [[o] for o in OPS] + [[("gauss_coulomb", 0.7)], OPS[1:3], OPS])
def test_short_list_has_the_bits_of_a_long_one(shg, ops, precision, schedule):
    """Contractions of 1 to 20 primitives (1 to 400 primitive pairs: one to eight lanes per pair), l <= 6, tiles that are not
    full.  401 pairs: a launch per operator; 1501 pairs: one launch of all, without a work counter."""
    sh, pa, pb = W.make("c3_2m_l6_k20", n=70000)
    b = shg.Basis(sh)
    off, long = _blocks(shg, b, pa, pb, ops, precision, schedule)
    for n_short in (401, 1501):
        pick = np.random.default_rng(4).permutation(len(pa))[:n_short]
        npp = sh["nprim"][pa[pick]] * sh["nprim"][pb[pick]]
        assert npp.min() < 8 and npp.max() > 129
        off1, short = _blocks(shg, b, pa[pick], pb[pick], ops, precision, schedule)
        n = (2 * sh["l"][pa[pick]] + 1) * (2 * sh["l"][pb[pick]] + 1)
        at = np.concatenate([np.arange(o, o + k) for o, k in zip(off[pick], n)])
        for x, y in zip(long, short):
            assert np.isfinite(y).all()
            np.testing.assert_array_equal(x[at], y)
    b.close()
