"""Host time of a planned call: a mixed-precision pass issues two launches instead of one and computes nothing on the host."""
import statistics
import time

import pytest

from paper_1701_06588_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_mixed_pass_costs_the_host_its_second_launch_only():
    """Two launches cost at most twice one; the bound leaves half of that again for the other arguments (measured 1.6; 4.7
    while every call recomputed the constants of the double-float launch)."""
    import torch
    from paper_1701_06588_gb300 import api, build
    build.build()
    sh, pa, pb = W.make("c1_2k_l3_k4", n=256)
    b = api.Basis(sh)
    off, total = b.pair_offsets(pa, pb)
    d_off = torch.from_numpy(off).cuda()
    out = torch.zeros(total, dtype=torch.float64, device="cuda")
    plan = api.Plan2c(b, pa, pb)
    assert (plan.launches_for("fp64"), plan.launches_for("mixed")) == (1, 2)

    def host(precision):
        t = []
        for _ in range(200):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            plan.exec("coulomb", d_off, out, precision=precision)
            t.append(time.perf_counter() - t0)
        return statistics.median(t)

    ratio = min(host("mixed") / host("fp64") for _ in range(5))
    assert ratio < 3
    plan.close()
    b.close()
