"""The launch counts that a plan states are the kernels that its passes put on the stream, counted under capture."""
import ctypes

import pytest

from paper_1701_06588_gb300 import _lib as L
from paper_1701_06588_gb300 import workloads as W

pytestmark = pytest.mark.gpu

ALL = [("overlap", 0.0), ("coulomb", 0.0), ("erfc", 0.3), ("erf", 0.3), ("gauss", 0.7)]


@pytest.fixture(scope="module")
def shg():
    import torch
    from paper_1701_06588_gb300 import api, build
    build.build()
    torch.cuda.init()
    return api


def _kernels(issue):
    """Kernel nodes of what issue(stream) puts on a capturing stream (driver API)."""
    import torch
    cu = ctypes.CDLL("libcuda.so.1")
    s = torch.cuda.Stream()
    h = ctypes.c_void_p(s.cuda_stream)
    assert cu.cuStreamBeginCapture_v2(h, 1) == 0                     # thread-local
    graph = ctypes.c_void_p()
    try:
        issue(s)
    finally:
        assert cu.cuStreamEndCapture(h, ctypes.byref(graph)) == 0
    n = ctypes.c_size_t()
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    kernels = 0
    for node in nodes:
        t = ctypes.c_int()
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(t)) == 0
        kernels += t.value == 0                                      # CU_GRAPH_NODE_TYPE_KERNEL
    cu.cuGraphDestroy(graph)
    return kernels


@pytest.mark.parametrize("schedule", ["persistent", "per_class"])
@pytest.mark.parametrize("n,lmax", [(300, 6), (300, 1), (1500, 6), (24000, 6)])
def test_stated_launches_are_issued(shg, n, lmax, schedule):
    """One launch per operator, one of all, with and without a work counter; lists with and without double-float classes."""
    import torch
    sh, pa, pb = W.make("c3_2m_l6_k20", n=n)
    sh = dict(sh, l=sh["l"].clip(max=lmax))
    b = shg.Basis(sh)
    off, total = b.pair_offsets(pa, pb)
    d_off = torch.from_numpy(off).cuda()
    plan = shg.Plan2c(b, pa, pb, schedule=schedule)
    outs = [torch.zeros(total, dtype=torch.float64, device="cuda") for _ in ALL]
    torch.cuda.synchronize()
    seen = set()
    for precision in ("fp64", "mixed"):
        for op, om in ALL:
            got = _kernels(lambda s: plan.exec(op, d_off, outs[0], omega=om, precision=precision, stream=s))
            assert got == plan.launches_for(precision), (op, precision)
            assert precision == "mixed" or got == plan.launches
        for ops in (ALL[:1], ALL[:2], ALL[1:3], ALL):
            names, oms = [o for o, _ in ops], [w for _, w in ops]
            got = _kernels(lambda s: plan.exec_fused(names, d_off, outs[:len(ops)], omegas=oms, precision=precision,
                                                     stream=s))
            assert got == plan.launches_for(precision, names), (names, precision)
            seen.add(got)
    if schedule == "persistent":
        parts = max(k for k in (4, 2, 1) if k == 1 or k * plan.tiles <= L.SHG_SHORT_LIST_TILES)
        assert max(seen) == parts * (2 if lmax > 1 else 1)
    plan.close()
    b.close()


def test_bad_arguments_have_no_count(shg):
    sh, pa, pb = W.make("c1_2k_l3_k4", n=8)
    b = shg.Basis(sh)
    plan = shg.Plan2c(b, pa, pb)
    for ops in ([], ["gauss_coulomb"], ["ra2n"]):
        with pytest.raises(L.ShgError):
            plan.launches_for("fp64", ops)
    plan.close()
    b.close()
