"""Float32 products split on the tensor cores (LSQ_F32 where its rule takes them) against float64.

Each operand is held to 2^-22 by its hi and lo parts, a tensor-core sum of 8 atoms k truncates its
32 additions (a few units of 2^-23 of the sum's size), and the sums are added in float32: for the
lists of at most 64 atoms here an element is within 2^-19 of the sum of |a| |b| over its terms.
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


def _run(g, A, ra, B, rb, pc, rc, ta, tb, triangle=0, alpha=1.0, beta=0.0, C0=None):
    f = torch.float32
    C = cuda(np.zeros((pc.nnzb, A.b, A.b)) if C0 is None else C0, f)
    lsq.block_matmul(g, A.b, cuda(A.val, f), g.range_id(ra), cuda(B.val, f), g.range_id(rb), C, g.range_id(rc),
                     precision=lsq.F32, trans_a=ta, trans_b=tb, triangle=triangle, alpha=alpha, beta=beta)
    g.device_status()
    return C.double().cpu().numpy()


def _operands(n, drop, b, ra, rb, rc, ta, tb, seed):
    pos, cell = si(n, 0.1, 91)
    pos = pos[:pos.shape[0] - drop]
    ranges = sorted({ra, rb, rc})
    g = gpu_geometry(pos, cell, ranges)
    P = {R: oracle.neighbour_list(pos, cell, R) for R in ranges}
    rng = np.random.default_rng(seed)
    A, B = (oracle.Bsr(P[R], b, rng.standard_normal((P[R].nnzb, b, b)).astype(np.float32)) for R in (ra, rb))
    return g, P, A, B


def _reference(A, B, ta, tb, pc):
    opA = oracle.transpose(A, A.pat) if ta else A
    opB = oracle.transpose(B, B.pat) if tb else B
    absx = lambda X: oracle.Bsr(X.pat, X.b, np.abs(X.val))
    return oracle.matmul(opA, opB, pc)[0].val, oracle.matmul(absx(opA), absx(opB), pc)[0].val


# ragged groups of 16 and tiles of 32 (61 and 7 atoms), k-lists shorter than a stage; larger blocks
@pytest.mark.parametrize("n,drop,b,ra,rb,rc", [(2, 3, 4, 6.6, 8.0, 8.0), (2, 0, 4, 2.5, 2.5, 4.0), (1, 7, 4, 3.0, 3.0, 3.0),
                                               (1, 1, 9, 4.0, 2.6, 4.0), (2, 3, 13, 2.6, 4.0, 4.0), (1, 0, 16, 4.0, 4.0, 2.6)])
@pytest.mark.parametrize("ta,tb", [(0, 0), (0, 1), (1, 0), (1, 1)])
def test_split_product(n, drop, b, ra, rb, rc, ta, tb):
    g, P, A, B = _operands(n, drop, b, ra, rb, rc, ta, tb, b)
    ref, bound = _reference(A, B, ta, tb, P[rc])
    C0 = np.random.default_rng(1).standard_normal(ref.shape).astype(np.float32)
    for alpha, beta in ((1.0, 0.0), (-0.75, 0.5)):
        got = _run(g, A, ra, B, rb, P[rc], rc, ta, tb, alpha=alpha, beta=beta, C0=C0)
        assert np.all(np.abs(got - (alpha * ref + beta * C0)) <= 2.0 ** -19 * (bound + np.abs(C0)))
    rows = np.repeat(np.arange(P[rc].n), np.diff(P[rc].ptr))
    up, low, off = P[rc].col >= rows, P[rc].col <= rows, P[rc].col != rows
    for tri, sel in ((1, up), (2, up), (3, low)):
        got = _run(g, A, ra, B, rb, P[rc], rc, ta, tb, triangle=tri)
        assert np.all(np.abs(got - ref)[sel] <= 2.0 ** -19 * bound[sel])
        if tri == 1:
            assert np.array_equal(got[off], oracle.transpose(oracle.Bsr(P[rc], b, got), P[rc]).val[off])


@pytest.mark.parametrize("b", [4, 13])
@pytest.mark.parametrize("ta,tb", [(0, 1), (1, 0)])
@pytest.mark.parametrize("case", ["inf_nan", "huge", "tiny"])
def test_split_product_leaves_odd_values_to_fma(b, ta, tb, case):
    """Infinities, NaN and values whose parts would leave float32's range: as the FMA kernels."""
    g, P, A, B = _operands(1, 1, b, 4.0, 2.6, 4.0, ta, tb, 2)
    if case == "inf_nan":
        A.val[5, 1, 2], A.val[20, 0, 0], B.val[7, 3, 3] = np.inf, np.nan, -np.inf
    elif case == "huge":
        A.val *= np.float32(2.0 ** 120)
        A.val[3, 0, 0] = np.finfo(np.float32).max
        B.val *= np.float32(2.0 ** -4)
    else:
        A.val *= np.float32(2.0 ** -118)
    with np.errstate(invalid="ignore", over="ignore"):
        ref, bound = _reference(A, B, ta, tb, P[4.0])
    C0 = np.random.default_rng(1).standard_normal(ref.shape).astype(np.float32) * (0.0 if case == "tiny" else 1.0)
    for beta in (0.0, 0.5):
        got = _run(g, A, 4.0, B, 2.6, P[4.0], 4.0, ta, tb, beta=beta, C0=C0)
        want = ref + beta * C0
        fine = np.isfinite(want)
        assert np.array_equal(np.isnan(want), np.isnan(got))
        assert np.array_equal(want[~fine & ~np.isnan(want)], got[~fine & ~np.isnan(want)])
        assert np.all(np.abs(got - want)[fine] <= 2.0 ** -19 * (bound + np.abs(C0))[fine])


@pytest.mark.parametrize("triangle", [0, 2])
def test_internal_precision_codes_are_refused(triangle):
    """The library's own code for FMA products is not a precision of the ABI."""
    g, P, A, B = _operands(1, 0, 4, 2.6, 2.6, 2.6, 0, 0, 3)
    C = cuda(np.zeros((P[2.6].nnzb, 4, 4)), torch.float32)
    with pytest.raises(lsq.LsqError):
        lsq.block_matmul(g, 4, cuda(A.val, torch.float32), g.range_id(2.6), cuda(B.val, torch.float32), g.range_id(2.6), C,
                         g.range_id(2.6), precision=101, triangle=triangle)
