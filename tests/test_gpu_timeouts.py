"""An expired wait of a product is an error of the call that waits for its results.

With the bound of the pipeline waits set to 0 ns a wait that does not succeed at once expires (the
kernel then drains, frees its tensor memory and returns), so blocks of a result are missing.
"""
import pytest
import torch

import oracle
import paper_2002_07704_gb300 as lsq
from gpu_common import cuda, gpu_geometry, si, si_hs

pytestmark = pytest.mark.gpu

TIMEOUT = 8


@pytest.fixture(scope="module", autouse=True)
def _built():
    lsq.build()
    lsq.load()


@pytest.fixture
def system(monkeypatch):
    monkeypatch.setenv("LSQ_F64_SLICED", "1")
    monkeypatch.setenv("LSQ_F32_SPLIT", "1")
    monkeypatch.setenv("LSQ_TC_CHOICE", "all=1")
    pos, cell = si(2, 0.05, 90)
    g = gpu_geometry(pos, cell, lsq.lnv_required_ranges(6.6, 6.6, 8.0))
    pat = oracle.neighbour_list(pos, cell, 6.6)
    H, S = si_hs(pos, cell, pat)
    ctx = lsq.Lnv(g, 4, 6.6, 6.6, 8.0)
    L = torch.zeros((g.nnzb(g.range_id(8.0)), 4, 4), dtype=torch.float64, device="cuda")
    ctx.init_L(cuda(S), L)
    return g, ctx, L, cuda(S), cuda(H)


def _expires(monkeypatch, g, call):
    want = call()
    monkeypatch.setenv("LSQ_TC_WAIT_NS", "0")
    with pytest.raises(lsq.LsqError) as e:
        call()
    assert e.value.code == TIMEOUT
    monkeypatch.delenv("LSQ_TC_WAIT_NS")
    g.device_status()  # reported once
    assert call() == want


@pytest.mark.parametrize("precision", [lsq.F64, lsq.F32, lsq.TF32X3])
def test_energy(system, monkeypatch, precision):
    g, ctx, L, S, H = system
    _expires(monkeypatch, g, lambda: ctx.energy_gradient(L, S, H, -2.0, precision=precision))


def test_minimisation(system, monkeypatch):
    g, ctx, L, S, H = system
    _expires(monkeypatch, g, lambda: ctx.minimise(L.clone(), S, H, -2.0, max_iter=3, precision=lsq.F64)["omega_ev"])


@pytest.mark.parametrize("graph", [False, True])
def test_batch(system, monkeypatch, graph):
    one, _, L, S, H = system
    g = lsq.concat_geometries([one, one])
    ctx = lsq.Lnv(g, 4, 6.6, 6.6, 8.0)
    two = lambda x: torch.cat([x, x])
    L2, S2, H2 = two(L), two(S), two(H)
    _expires(monkeypatch, g, lambda: [r["omega_ev"] for r in ctx.minimise_batch(L2.clone(), S2, H2, [-2.0, -2.0], max_iter=4,
                                                                              graph=graph)])


def test_inverse_and_trace(system, monkeypatch):
    g, ctx, L, S, H = system
    rs, rl = g.range_id(6.6), g.range_id(8.0)
    X = torch.zeros_like(L)
    inv = lambda: lsq.hotelling_inverse(g, 4, S, rs, X, rl, g.range_id(8.0 + 6.6), 3, precision=lsq.F64)
    _expires(monkeypatch, g, lambda: (inv(), X.sum().item())[1])
    C = torch.zeros_like(L)

    def product_then_trace():
        lsq.block_matmul(g, 4, L, rl, S, rs, C, rl, precision=lsq.F64, trans_b=True)
        return lsq.trace(g, 4, C, rl, S, rs)
    _expires(monkeypatch, g, product_then_trace)
