"""The library's pool of plan memory: shg_eval_2c draws on it and shg_eval_2c_noalloc does not, and nothing of it is kept
after the last basis and plan."""
import os
import subprocess
import sys

import pytest

from paper_1701_06588_gb300 import _lib as L
from paper_1701_06588_gb300 import workloads as W

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_noalloc_calls_do_not_draw_on_the_plan_pool():
    import torch
    from paper_1701_06588_gb300 import api, build
    build.build()
    shells, pa, pb = W.make("c2_200k_l4_k8", n=6000)
    basis = api.Basis(shells)
    off, total = basis.pair_offsets(pa, pb)
    d_pa, d_pb, d_off = (torch.from_numpy(x).cuda() for x in (pa, pb, off))
    out = torch.empty(total, dtype=torch.float64, device="cuda")
    st = torch.cuda.current_stream().cuda_stream

    def peak(call):
        torch.cuda.synchronize()
        _, used, _ = L.shg_debug_pool(reset_high=True)
        reserved, _, _ = L.shg_debug_pool()
        call()
        torch.cuda.synchronize()
        r1, u1, high = L.shg_debug_pool()
        assert u1 == used
        return high - used, r1 - reserved

    def plain():
        L.shg_eval_2c(basis.handle, len(pa), d_pa, d_pb, L.SHG_OP_COULOMB, 0.0, 0.0, L.SHG_PREC_FP64, d_off, out, st)

    def noalloc():
        L.shg_eval_2c_noalloc(basis.handle, len(pa), d_pa, d_pb, L.SHG_OP_COULOMB, 0.0, L.SHG_PREC_FP64, d_off, out, st)

    noalloc()                                              # the first call looks the array's address up
    assert peak(plain)[0] >= 8 * len(pa)                   # the plan: order and keys of the pairs, 4 bytes each, and more
    assert peak(noalloc) == (0, 0)
    basis.close()


PROGRAM = """
import torch
from paper_1701_06588_gb300 import _lib as L, api, workloads as W
shells, pa, pb = W.make("c2_200k_l4_k8", n=20000)
for last in ("basis", "plan", "pending"):
    basis = api.Basis(shells)
    plan = api.Plan2c(basis, pa, pb)
    assert L.shg_debug_pool()[1] > 0
    if last == "basis":
        plan.close()
        torch.cuda.synchronize()
        assert L.shg_debug_pool()[0] > 0                   # kept for the next plan
        basis.close()
    elif last == "plan":
        basis.close()
        assert L.shg_debug_pool()[0] > 0                   # in use
        plan.close()
    else:                                                  # the free waits behind work on the stream
        x = torch.randn(8192, 8192, device="cuda")
        for _ in range(20):
            x = x @ x * 1e-4
        basis.close()
        plan.close()
    torch.cuda.synchronize()
    print(last, *L.shg_debug_pool()[:2])
"""


def test_the_pool_is_given_back_after_the_last_basis_and_plan():
    """In a process of its own: no other test's basis keeps the pool."""
    from paper_1701_06588_gb300 import build
    build.build()
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    assert r.stdout.split() == ["basis", "0", "0", "plan", "0", "0", "pending", "0", "0"], r.stdout
