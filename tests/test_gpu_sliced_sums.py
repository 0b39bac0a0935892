"""Long sums of the float64 products from integer slices.

Constant operands and sums of squares make the digit products of every order pile up with one sign
instead of cancelling, so the integer sums of a long list of atoms k are as large as they can be.
The slices drop at most 2^-70 of the largest entries of the two rows a term, and a result is rounded
once: sums of terms of one size are within 2^-52 of themselves.
"""
from fractions import Fraction

import numpy as np
import pytest
import torch

import paper_2002_07704_gb300 as lsq
from gpu_common import cuda, si

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    lsq.build()
    lsq.load()


@pytest.fixture(autouse=True)
def _forced(monkeypatch):
    monkeypatch.setenv("LSQ_F64_SLICED", "1")


def _all_pairs(cells, drop):
    """A crystal, less `drop` atoms, whose rows hold every atom on range 1, and a short range 0."""
    pos, cell = si(cells, 0.1, 80)
    pos = np.ascontiguousarray(pos[:pos.shape[0] - drop])
    g = lsq.Geometry(torch.from_numpy(pos).cuda(), cell, [2.6, 0.95 * 3 ** 0.5 * cell[0]])
    assert g.nnzb(1) == pos.shape[0] ** 2
    return g, pos.shape[0]


# lists of 11 groups of 16 atoms k and more (a group is 4 atoms for b > 4), whole and ragged
@pytest.mark.parametrize("b,cells,drop", [(4, 3, 41), (4, 3, 0), (4, 4, 1), (4, 6, 0), (13, 2, 0), (13, 3, 5), (13, 4, 0)])
@pytest.mark.parametrize("value", [0.1, 1 / 3, (256 / 511) * (1 + 2.0 ** -52)])
def test_constant_operands(b, cells, drop, value):
    g, n = _all_pairs(cells, drop)
    A = torch.full((n * n, b, b), value, dtype=torch.float64, device="cuda")
    B = torch.full_like(A, -value)
    C = torch.zeros((g.nnzb(0), b, b), dtype=torch.float64, device="cuda")
    lsq.block_matmul(g, b, A, 1, B, 1, C, 0, precision=lsq.F64, trans_b=1)
    g.device_status()
    want = float(-n * b * Fraction(value) ** 2)
    assert float((C - want).abs().max()) <= 2.0 ** -52 * abs(want)


@pytest.mark.parametrize("b,cells", [(4, 3), (4, 6), (13, 3)])
def test_sums_of_squares(b, cells):
    g, n = _all_pairs(cells, 0)
    x = np.random.default_rng(b).standard_normal((n, n, b, b))
    A = cuda(x.reshape(n * n, b, b))
    C = torch.zeros((g.nnzb(0), b, b), dtype=torch.float64, device="cuda")
    lsq.block_matmul(g, b, A, 1, A, 1, C, 0, precision=lsq.F64, trans_b=1)
    g.device_status()
    rp, col = (t.cpu().numpy() for t in g.pattern(0))
    for i in (0, n // 2, n - 1):
        q = rp[i] + int(np.nonzero(col[rp[i]:rp[i + 1]] == i)[0][0])
        want = (x[i].astype(np.longdouble) ** 2).sum(axis=(0, 2))
        got = np.diagonal(C[q].cpu().numpy())
        assert np.all(np.abs(got - want) <= 2.0 ** -52 * want)
