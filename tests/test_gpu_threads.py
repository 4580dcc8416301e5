"""Calls from several host threads at once, each on a stream of its own, give what they give alone."""
import threading

import numpy as np
import pytest

from paper_1701_06588_gb300 import _lib as L

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def shg():
    import torch
    from paper_1701_06588_gb300 import api, build
    build.build()
    torch.cuda.init()
    return api


def _triples(api, la, lt, lb, n, seed):
    """n triples of one class: shells 2i, 2i+1 on center i (a, a~), shell 2n+i on center n+i (b)."""
    import torch
    rng = np.random.default_rng(seed)
    l = np.concatenate([np.tile([la, lt], n), np.full(n, lb)]).astype(np.int32)
    k = np.full(3 * n, 2, np.int32)
    sh = dict(l=l, nprim=k, exps=rng.uniform(0.2, 3.0, 6 * n), coefs=rng.uniform(0.2, 1.0, 6 * n),
              centers=rng.uniform(-1, 1, (2 * n, 3)),
              center_of=np.concatenate([np.repeat(np.arange(n), 2), np.arange(n, 2 * n)]).astype(np.int32))
    b = api.Basis(sh)
    t = [np.arange(0, 2 * n, 2, dtype=np.int32), np.arange(1, 2 * n, 2, dtype=np.int32),
         np.arange(2 * n, 3 * n, dtype=np.int32)]
    off, total = b.triple_offsets(b, *t)
    dev = [torch.from_numpy(x).cuda() for x in (*t, off)]
    return b, dev, total


def test_three_index_calls_of_different_classes_from_several_threads(shg):
    """The longest class (5, 5, 6), 20 and 43 KB of shared memory a warp, and the shortest, 0.4 and 0.7 KB.  No call may
    change what another one's launch is allowed."""
    import torch
    n, calls = 8, 1500
    work = []
    for la, lt, lb, seed in ((5, 5, 6, 1), (0, 0, 0, 2), (0, 0, 0, 3), (0, 0, 0, 4)):
        b, dev, total = _triples(shg, la, lt, lb, n, seed)
        w = torch.linspace(-1, 1, total, dtype=torch.float64, device="cuda")
        out = torch.zeros(total, dtype=torch.float64, device="cuda")
        ga = torch.zeros((n, 3), dtype=torch.float64, device="cuda")

        def run(stream, b=b, dev=dev, w=w, out=out, ga=ga):
            L.shg_eval_3c_aab(b.handle, b.handle, n, *dev[:3], L.SHG_PREC_FP64, 0.0, dev[3], out, stream)
            L.shg_eval_3c_aab_grad(b.handle, b.handle, n, *dev[:3], L.SHG_PREC_FP64, dev[3], w, ga, None, stream)

        run(torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        work.append((run, out, ga, out.clone(), ga.clone()))
    start = threading.Barrier(len(work))
    errors = []

    def loop(run, out, ga, ref, gref):
        s = torch.cuda.Stream()
        start.wait()
        for _ in range(calls):
            try:
                run(s.cuda_stream)
            except L.ShgError as e:
                errors.append(str(e))
        s.synchronize()

    threads = [threading.Thread(target=loop, args=x) for x in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, (len(errors), errors[0])
    for _, out, ga, ref, gref in work:
        assert torch.equal(out, ref) and torch.equal(ga, gref)
