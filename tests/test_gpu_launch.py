"""Launch shapes and register caps on lists that run with a work counter (more than SHG_SHORT_LIST_TILES tiles): the same
operations in the same order, so the same bits as a short list of the same pairs."""
import numpy as np
import pytest

from paper_1701_06588_gb300 import _lib as L
from paper_1701_06588_gb300 import workloads as W

pytestmark = pytest.mark.gpu

ALL = [("overlap", 0.0), ("coulomb", 0.0), ("erfc", 0.3), ("erf", 0.3), ("gauss", 0.7)]
SETS = [[o] for o in ALL] + [[("gauss_coulomb", 0.7)], ALL[1:3], ALL]


@pytest.fixture(scope="module")
def case():
    import torch
    from paper_1701_06588_gb300 import api, build
    build.build()
    torch.cuda.init()
    sh, pa, pb = W.make("c3_2m_l6_k20", n=24000)
    b = api.Basis(sh)
    off, total = b.pair_offsets(pa, pb)
    plan = api.Plan2c(b, pa, pb)
    assert plan.tiles > 2 * L.SHG_SHORT_LIST_TILES
    yield api, b, pa, pb, torch.from_numpy(off).cuda(), total, plan
    plan.close()
    b.close()


def _run(plan, d_off, total, ops, precision):
    import torch
    outs = [torch.full((total,), float("nan"), dtype=torch.float64, device="cuda") for _ in ops]
    if len(ops) == 1:
        plan.exec(ops[0][0], d_off, outs[0], omega=ops[0][1], precision=precision)
    else:
        plan.exec_fused([o for o, _ in ops], d_off, outs, omegas=[w for _, w in ops], precision=precision)
    torch.cuda.synchronize()
    assert all(bool(torch.isfinite(o).all()) for o in outs)
    return outs


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("ops", SETS, ids=lambda s: "+".join(o for o, _ in s))
def test_register_caps_give_the_same_bits(case, ops, precision):
    import torch
    api, b, pa, pb, d_off, total, plan = case
    ref = None
    for variant in (0, 1, 2):
        api.set_launch(plan, 128, 0, variant)
        outs = _run(plan, d_off, total, ops, precision)
        ref = ref or outs
        for o, r in zip(outs, ref):
            assert torch.equal(o, r), variant
    # the same pairs in pieces of at most the short-list limit: no work counter, one warp per CTA
    n = len(pa)
    for lo in range(0, n, n // 8):
        hi = min(n, lo + n // 8)
        p = api.Plan2c(b, pa[lo:hi], pb[lo:hi])
        assert p.tiles <= L.SHG_SHORT_LIST_TILES
        end = int(d_off[hi]) if hi < n else total
        short = _run(p, d_off[lo:hi] - d_off[lo], end - int(d_off[lo]), ops, precision)
        for o, r in zip(short, ref):
            assert torch.equal(o, r[int(d_off[lo]):end])
        p.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_launch_shapes_give_the_same_bits(case, precision):
    import torch
    from paper_1701_06588_gb300 import autotune
    api, b, pa, pb, d_off, total, plan = case
    api.set_launch(plan, 128, 0, 1)
    ref = _run(plan, d_off, total, ALL[1:3], precision)
    for sched, threads, ctas in autotune.CANDIDATES:
        p = autotune.tuned_plan(b, pa, pb, {"schedule": sched, "threads_per_cta": threads, "ctas_per_sm": ctas})
        for o, r in zip(_run(p, d_off, total, ALL[1:3], precision), ref):
            assert torch.equal(o, r), (sched, threads, ctas)
        p.close()
