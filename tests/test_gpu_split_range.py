"""Float32 products split on the tensor cores where values are small, large or no numbers.

Every element is held to what an FMA sum of n terms keeps: n 2^-24 of the sum of absolute values (with
2^-22 for the parts of the operands and their short sums), and half the smallest subnormal a term.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2002_07704_gb300 as lsq
from gpu_common import cuda, gpu_geometry, si

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    lsq.build()
    lsq.load()


@pytest.fixture(autouse=True)
def _forced(monkeypatch):
    monkeypatch.setenv("LSQ_F32_SPLIT", "1")


def _operands(b, seed):
    pos, cell = si(2 if b == 4 else 1, 0.1, 92)
    pos = pos[:-1]
    ra, rb = (6.6, 4.0) if b == 4 else (4.0, 2.6)
    g = gpu_geometry(pos, cell, [rb, ra])
    pa, pb = oracle.neighbour_list(pos, cell, ra), oracle.neighbour_list(pos, cell, rb)
    rng = np.random.default_rng(seed)
    A, B = (oracle.Bsr(p, b, rng.standard_normal((p.nnzb, b, b)).astype(np.float32)) for p in (pa, pb))
    return g, A, B, rng


def _check(g, A, B, sums=None):
    """C = A.B on A's pattern against the oracle; returns C."""
    f = torch.float32
    with np.errstate(over="ignore", under="ignore", invalid="ignore"):
        ref, _ = oracle.matmul(A, B, A.pat)
        absx = lambda X: oracle.Bsr(X.pat, X.b, np.abs(X.val))
        bound, _ = oracle.matmul(absx(A), absx(B), A.pat)
    C = cuda(np.full(ref.val.shape, 7.0), f)
    lsq.block_matmul(g, A.b, cuda(A.val, f), 1, cuda(B.val, f), 0, C, 1, precision=lsq.F32)
    g.device_status()
    got = C.double().cpu().numpy()
    n = A.b * 17
    top = np.finfo(np.float32).max
    fine = np.isfinite(ref.val) & (bound.val < top / 2)
    assert np.array_equal(np.isnan(got), np.isnan(ref.val)) or not np.isfinite(bound.val).all()
    with np.errstate(invalid="ignore"):
        err = np.abs(got - ref.val)
    assert np.all(err[fine] <= (n * 2.0 ** -24 + 2.0 ** -22) * bound.val[fine] + n * 2.0 ** -149)
    return got, ref.val


@pytest.mark.parametrize("b", [4, 13])
# the two operands' scales: small times small (parts below the normal range), small times large, subnormal
@pytest.mark.parametrize("ea,eb", [(0, 0), (-60, -60), (-62, -64), (-75, -40), (-100, 30), (-118, 0), (-118, 60), (-140, 90),
                                   (60, 60), (-30, -100)])
def test_scaled_operands(b, ea, eb):
    g, A, B, _ = _operands(b, 11)
    A.val = (A.val.astype(np.float64) * 2.0 ** ea).astype(np.float32).astype(np.float64)
    B.val = (B.val.astype(np.float64) * 2.0 ** eb).astype(np.float32).astype(np.float64)
    _check(g, A, B)


@pytest.mark.parametrize("b", [4, 13])
@pytest.mark.parametrize("low", [40, 149])
def test_tails_in_every_row(b, low):
    """Values of all sizes down to the subnormal ones, zeros among them."""
    g, A, B, rng = _operands(b, 12)
    for X in (A, B):
        X.val = X.val * 2.0 ** -rng.integers(0, low, size=X.val.shape).astype(np.float64)
        X.val[rng.random(X.val.shape) < 0.2] = 0.0
        X.val = X.val.astype(np.float32).astype(np.float64)
    _check(g, A, B)


@pytest.mark.parametrize("b", [4, 13])
@pytest.mark.parametrize("bits", [0x7f800000, 0xff800000, 0x7fc00000, 0x7fffffff, 0xffffffff, 0x7f800001])
def test_infinities_and_nans_reach_only_their_sums(b, bits):
    g, A, B, _ = _operands(b, 13)
    bad = np.array([bits], dtype=np.uint32).view(np.float32)[0]
    A.val[3, 1, 2] = bad
    B.val[5, b - 1, 0] = bad
    with np.errstate(invalid="ignore"):
        got, ref = _check(g, A, B)
    assert np.array_equal(np.isfinite(got), np.isfinite(ref))
    inf = np.isinf(ref)
    assert np.array_equal(got[inf], ref[inf])


def test_products_run_on_fma_where_the_copies_do_not_fit():
    """Without memory for the operand copies a float32 product still runs."""
    pos, cell = si(4, 0.1, 93)
    ranges = [2.6, 0.95 * 3 ** 0.5 * cell[0]]
    gen = torch.Generator(device="cuda").manual_seed(1)
    g = gpu_geometry(pos, cell, ranges)
    A = torch.randn((g.nnzb(1), 16, 16), generator=gen, device="cuda")   # 268 MB; its copy takes 537 MB
    C = torch.zeros((g.nnzb(0), 16, 16), device="cuda")
    rp, col = g.pattern(0)
    rows = A.view(g.n_atoms, g.n_atoms, 16, 16).permute(0, 2, 1, 3).reshape(g.n_atoms * 16, -1)
    picked = torch.arange(40, device="cuda")
    left = rows.view(g.n_atoms, 16, -1)[torch.repeat_interleave(torch.arange(g.n_atoms, device="cuda"), rp.diff())[picked]].double()
    right = rows.view(g.n_atoms, 16, -1)[col[:40].long()].double()
    want, bound = left @ right.transpose(1, 2), left.abs() @ right.abs().transpose(1, 2)
    del rows, left, right
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    rest = torch.empty(torch.cuda.mem_get_info()[0] - (400 << 20), dtype=torch.uint8, device="cuda")
    try:
        lsq.block_matmul(g, 16, A, 1, A, 1, C, 0, precision=lsq.F32, trans_b=True)
        torch.cuda.synchronize()
    finally:
        del rest
        torch.cuda.empty_cache()
    # what a float32 sum of 8192 terms keeps in the worst case
    assert bool(((C[:40].double() - want).abs() <= 8192 * 2.0 ** -24 * bound).all())


@pytest.mark.parametrize("b", [4, 13])
@pytest.mark.parametrize("low", [20, 100, 149])
def test_stored_zero_blocks_meet_infinities(b, low):
    """A stored zero block adds nothing, except to a block with an infinity or a NaN."""
    g, A, B, rng = _operands(b, 14)
    for X in (A, B):
        X.val = X.val * 2.0 ** -rng.integers(0, low, size=(X.pat.nnzb, 1, 1)).astype(np.float64)
    A.val[rng.random(A.pat.nnzb) < 0.9] = 0.0
    A.val[:, b - 1, :] = 0.0
    for X in (A, B):
        X.val = X.val.astype(np.float32).astype(np.float64)
    for bad in (None, np.inf, np.nan):
        if bad is not None:
            B.val[7, 1, 2] = bad
        with np.errstate(invalid="ignore"):
            got, ref = _check(g, A, B)
        assert np.array_equal(np.isnan(got), np.isnan(ref))
        inf = np.isinf(ref)
        assert np.array_equal(got[inf], ref[inf])
