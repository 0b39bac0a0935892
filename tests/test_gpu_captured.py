"""Captured products own the memory of their operand copies.

A CUDA graph that captured a product on the tensor cores is replayed after the geometry's own buffers
have been replaced by larger ones, on several streams at once, and beside calls on other streams.
Results are compared with the same product run outside the graph (the same kernels: equal bits).
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2002_07704_gb300 as lsq
from gpu_common import cuda, gpu_geometry, si, si_hs

pytestmark = pytest.mark.gpu

RANGES = [4.0, 6.6, 10.0]
PREC = {"f64": (lsq.F64, torch.float64), "f32": (lsq.F32, torch.float32), "mixed": (lsq.TF32X3, torch.float32)}


@pytest.fixture(scope="module", autouse=True)
def _built():
    lsq.build()
    lsq.load()


@pytest.fixture(autouse=True)
def _forced(monkeypatch):
    monkeypatch.setenv("LSQ_F64_SLICED", "1")
    monkeypatch.setenv("LSQ_F32_SPLIT", "1")


class Product:
    """C = A.B^T on ranges (ra, rb, rc), in buffers that a graph can hold on to."""

    def __init__(self, g, b, prec, ra, rb, rc):
        self.g, self.b, self.prec, self.r = g, b, PREC[prec][0], (ra, rb, rc)
        new = lambda r: torch.empty((g.nnzb(r), b, b), dtype=PREC[prec][1], device="cuda")
        self.A, self.B, self.C = new(ra), new(rb), new(rc)

    def fill(self, seed):
        gen = torch.Generator(device="cuda").manual_seed(seed)
        for X in (self.A, self.B):
            X.copy_(torch.randn(X.shape, generator=gen, device="cuda", dtype=X.dtype))

    def run(self):
        lsq.block_matmul(self.g, self.b, self.A, self.r[0], self.B, self.r[1], self.C, self.r[2], precision=self.prec,
                         trans_b=True)

    def expected(self, seed):
        self.fill(seed)
        self.run()
        torch.cuda.synchronize()
        return self.C.clone()

    def capture(self):
        self.run()  # plans and choices are made outside a capture
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            self.run()
        return graph


@pytest.mark.parametrize("b,prec", [(4, "f64"), (13, "f64"), (4, "f32"), (13, "f32"), (4, "mixed")])
def test_graph_outlives_the_geometrys_buffers(b, prec):
    pos, cell = si(2, 0.1, 85)
    g = gpu_geometry(pos, cell, RANGES)
    p = Product(g, b, prec, 0, 0, 0)
    graph = p.capture()
    want = [p.expected(s) for s in (1, 2)]
    big = Product(g, b, prec, 2, 2, 2)  # replaces the geometry's buffers by larger ones
    big_want = big.expected(3)
    # whatever takes their place has to stay as it is
    room = [torch.full((n,), 0x5a, dtype=torch.uint8, device="cuda") for n in (1 << 12, 1 << 16, 1 << 20, 1 << 22) for _ in range(8)]
    for seed, w in ((1, want[0]), (2, want[1])):
        p.fill(seed)
        p.C.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(p.C, w)
    assert all(bool((x == 0x5a).all()) for x in room)
    big.run()
    assert torch.equal(big.C, big_want)
    g.device_status()


@pytest.mark.parametrize("b,prec", [(4, "f64"), (4, "f32"), (13, "f64")])
def test_graphs_and_calls_on_several_streams(b, prec):
    pos, cell = si(3 if b == 4 else 2, 0.1, 86)
    g = gpu_geometry(pos, cell, RANGES)
    ps = [Product(g, b, prec, 1, 2, 1), Product(g, b, prec, 1, 2, 1), Product(g, b, prec, 2, 1, 2)]
    want = [p.expected(10 + k) for k, p in enumerate(ps)]
    graphs = [p.capture() for p in ps[:2]]
    streams = [torch.cuda.Stream() for _ in ps]
    for p in ps:
        p.C.zero_()
    torch.cuda.synchronize()
    for _ in range(6):
        for k, s in enumerate(streams):
            with torch.cuda.stream(s):
                if k < 2:
                    graphs[k].replay()
                else:
                    ps[2].run()
        # each round has to come out right, not only the last
    torch.cuda.synchronize()
    for p, w in zip(ps, want):
        assert torch.equal(p.C, w)
    g.device_status()


def test_a_replay_with_odd_values_leaves_no_trace():
    """Float32: values that the split does not take go to FMA in that replay, and in no later one."""
    pos, cell = si(2, 0.1, 87)
    g = gpu_geometry(pos, cell, RANGES)
    p = Product(g, 4, "f32", 1, 1, 1)
    graph = p.capture()
    want = p.expected(1)
    p.A[7, 1, 2] = float("inf")
    graph.replay()
    torch.cuda.synchronize()
    assert not bool(torch.isfinite(p.C).all())
    p.fill(1)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(p.C, want)


def test_batch_steps_beside_larger_products():
    """A batch minimisation replays captured steps while another thread's product replaces buffers."""
    import threading
    pos, cell = si(2, 0.05, 88)
    ranges = lsq.lnv_required_ranges(6.6, 6.6, 8.0)
    one = gpu_geometry(pos, cell, ranges)
    g = lsq.concat_geometries([one, one])
    pat = oracle.neighbour_list(pos, cell, 6.6)
    H, S = si_hs(pos, cell, pat)
    two = lambda x: torch.cat([cuda(x), cuda(x)])
    def minimise(busy):
        ctx = lsq.Lnv(g, 4, 6.6, 6.6, 8.0)
        L = torch.zeros((g.nnzb(g.range_id(8.0)), 4, 4), dtype=torch.float64, device="cuda")
        ctx.init_L(two(S), L)
        stop = threading.Event()
        def other():
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                while not stop.is_set():
                    for p in products:
                        p.run()
                    s.synchronize()
        t = threading.Thread(target=other) if busy else None
        if t:
            t.start()
        try:
            rep = ctx.minimise_batch(L, two(S), two(H), [-2.0, -2.0], max_iter=12, precision=lsq.F64)
        finally:
            stop.set()
            if t:
                t.join()
        return L, [r["omega_ev"] for r in rep]
    products = []
    alone, om = minimise(False)
    n = len(ranges) - 1
    products = [Product(g, 4, "f64", 0, 0, 0), Product(g, 4, "f64", n, n, 0)]
    for p in products:
        p.fill(5)
        p.run()
    torch.cuda.synchronize()
    beside, om2 = minimise(True)
    assert om == om2 and torch.equal(alone, beside)
