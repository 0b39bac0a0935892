"""Products called from several threads on one geometry, the first calls (plans, choices) among them."""
import threading

import pytest
import torch

import paper_2002_07704_gb300 as lsq
from gpu_common import gpu_geometry, si

pytestmark = pytest.mark.gpu

# (b, precision, ranges of A, B and C); the second operand transposed, so that no call needs scratch for that
CALLS = [(4, lsq.F64, 1, 1, 1), (4, lsq.F64, 2, 1, 2), (4, lsq.F32, 2, 2, 2), (4, lsq.TF32X3, 1, 2, 1), (4, lsq.F32, 0, 1, 1),
         (4, lsq.F64, 0, 2, 2), (13, lsq.F64, 0, 0, 0), (13, lsq.F32, 0, 1, 0)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    lsq.build()
    lsq.load()


def _operands(g, call, seed):
    b, prec, ra, rb, rc = call
    t = torch.float64 if prec == lsq.F64 else torch.float32
    gen = torch.Generator(device="cuda").manual_seed(seed)
    A, B = (torch.randn((g.nnzb(r), b, b), generator=gen, device="cuda", dtype=t) for r in (ra, rb))
    return A, B


def _run(g, call, A, B):
    b, prec, ra, rb, rc = call
    C = torch.zeros((g.nnzb(rc), b, b), dtype=A.dtype, device="cuda")
    n = lsq.block_matmul(g, b, A, ra, B, rb, C, rc, precision=prec, trans_b=True)
    return n, C


def test_threads_share_a_geometry():
    pos, cell = si(3, 0.1, 89)
    alone = gpu_geometry(pos, cell, [3.0, 6.6, 10.0])
    ops = [_operands(alone, c, k) for k, c in enumerate(CALLS)]
    want = [_run(alone, c, *o) for c, o in zip(CALLS, ops)]
    torch.cuda.synchronize()
    for _ in range(3):
        g = gpu_geometry(pos, cell, [3.0, 6.6, 10.0])
        start, wrong = threading.Barrier(len(CALLS)), []

        def work(k):
            s = torch.cuda.Stream()
            start.wait()
            with torch.cuda.stream(s):
                for _ in range(4):
                    # each thread meets every product, in an order of its own
                    for m in range(len(CALLS)):
                        c = (k + m) % len(CALLS)
                        n, C = _run(g, CALLS[c], *ops[c])
                        s.synchronize()
                        # FMA schedules are picked by timing and sum in different orders
                        err = float((C - want[c][1]).abs().max() / want[c][1].abs().max())
                        if n != want[c][0] or err > (1e-13 if C.dtype == torch.float64 else 1e-5):
                            wrong.append((k, c, n, err))

        threads = [threading.Thread(target=work, args=(k,)) for k in range(len(CALLS))]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert not wrong
        g.device_status()
