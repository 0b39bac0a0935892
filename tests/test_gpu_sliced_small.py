"""Float64 products from integer slices where results lie far below the largest entries of their rows.

A float64 sum of n terms is within n 2^-53 of the sum of their absolute values, element by element.
The products from slices keep that bound: a sum that is too short for the digits it was made of is
taken in FP64 instead.  (16 more units for short sums: the digits left out are below 2^-54 of a sum
when they have random signs, 2^-50 when all have one.)
"""
import numpy as np
import pytest

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
    monkeypatch.setenv("LSQ_F64_SLICED", "1")


def _sums(A, B, pc):
    """A.B over the stored blocks in extended precision, the same of absolute values, and the terms."""
    C = np.zeros((pc.nnzb, A.b, A.b), dtype=np.longdouble)
    S, terms = np.zeros_like(C), np.zeros(pc.nnzb, dtype=int)
    for i in range(pc.n):
        at = {int(j): q for q, j in zip(range(pc.ptr[i], pc.ptr[i + 1]), pc.col[pc.ptr[i]:pc.ptr[i + 1]])}
        for pa in range(A.pat.ptr[i], A.pat.ptr[i + 1]):
            k = A.pat.col[pa]
            x = A.val[pa].astype(np.longdouble)
            for pb in range(B.pat.ptr[k], B.pat.ptr[k + 1]):
                q = at.get(int(B.pat.col[pb]))
                if q is not None:
                    y = B.val[pb].astype(np.longdouble)
                    C[q] += x @ y
                    S[q] += np.abs(x) @ np.abs(y)
                    terms[q] += A.b
    return C, S, terms


def _product(b, A, ra, B, rb, pc, rc, g, **kw):
    C = cuda(np.zeros((pc.nnzb, b, b)))
    lsq.block_matmul(g, b, cuda(A.val), g.range_id(ra), cuda(B.val), g.range_id(rb), C, g.range_id(rc),
                     precision=lsq.F64, **kw)
    g.device_status()
    return C.cpu().numpy()


# blocks: each block of the operands at a level of its own, like the far blocks of decaying matrices.
# entries: each scalar (a small sum beside a large one in the same block).  rows: whole scalar rows of a
# block.  sparse: most scalars zero, so that many sums have no terms or a few.
@pytest.mark.parametrize("b,n,ra,rb,rc", [(4, 2, 6.6, 8.0, 8.0), (4, 2, 3.0, 6.6, 6.6), (13, 1, 4.0, 2.6, 4.0)])
@pytest.mark.parametrize("kind", ["blocks", "entries", "rows", "sparse"])
@pytest.mark.parametrize("low", [10, 17, 40, 80])
def test_small_sums(b, n, ra, rb, rc, kind, low):
    pos, cell = si(n, 0.1, 81)
    pos = pos[:pos.shape[0] - 1]
    ranges = sorted({ra, rb, rc})
    g = gpu_geometry(pos, cell, ranges)
    P = {R: oracle.neighbour_list(pos, cell, R) for R in ranges}
    rng = np.random.default_rng(low)
    A, B = (oracle.Bsr(P[R], b, rng.standard_normal((P[R].nnzb, b, b))) for R in (ra, rb))
    for X in (A, B):
        shape = {"blocks": (1, 1), "rows": (b, 1)}.get(kind, (b, b))
        X.val *= 2.0 ** -rng.integers(0, low, size=(X.pat.nnzb, *shape))
        if kind == "sparse":
            X.val[rng.random(X.val.shape) < 0.9] = 0.0
    ref, bound, terms = _sums(A, B, P[rc])
    got = _product(b, A, ra, B, rb, P[rc], rc, g)
    assert np.all(np.abs(got - ref) <= (terms[:, None, None] + 16) * 2.0 ** -53 * bound)


@pytest.mark.parametrize("b,n", [(4, 2), (13, 1)])
@pytest.mark.parametrize("side", ["left", "right"])
def test_product_with_the_identity_returns_the_operand(b, n, side):
    pos, cell = si(n, 0.1, 82)
    ra, rb = 4.0, 2.6
    g = gpu_geometry(pos, cell, [rb, ra])
    pa, pb = oracle.neighbour_list(pos, cell, ra), oracle.neighbour_list(pos, cell, rb)
    rng = np.random.default_rng(5)
    X = oracle.Bsr(pa, b, rng.standard_normal((pa.nnzb, b, b)) * 2.0 ** -rng.integers(0, 90, size=(pa.nnzb, b, b)))
    one = np.zeros((pb.nnzb, b, b))
    one[pb.col == np.repeat(np.arange(pb.n), np.diff(pb.ptr))] = np.eye(b)
    E = oracle.Bsr(pb, b, one)
    got = _product(b, E, rb, X, ra, pa, ra, g) if side == "left" else _product(b, X, ra, E, rb, pa, ra, g)
    assert np.array_equal(got, X.val)


def test_blocks_without_terms_are_zero_or_scaled():
    """C's range reaches beyond the product's: blocks with no stored pair are beta C."""
    pos, cell = si(3, 0.1, 83)
    g = gpu_geometry(pos, cell, [2.6, 8.0])
    p, pc = oracle.neighbour_list(pos, cell, 2.6), oracle.neighbour_list(pos, cell, 8.0)
    rng = np.random.default_rng(6)
    A = oracle.Bsr(p, 4, rng.standard_normal((p.nnzb, 4, 4)) * 1e-9 ** rng.integers(0, 2, size=(p.nnzb, 4, 4)))
    ref, bound, terms = _sums(A, A, pc)
    assert (terms == 0).any() and (terms > 0).any()
    C0 = rng.standard_normal((pc.nnzb, 4, 4))
    for beta in (0.0, 0.5):
        C = cuda(C0)
        lsq.block_matmul(g, 4, cuda(A.val), 0, cuda(A.val), 0, C, 1, precision=lsq.F64, beta=beta)
        got = C.cpu().numpy()
        assert np.array_equal(got[terms == 0], beta * C0[terms == 0])
        assert np.all(np.abs(got - (ref + beta * C0)) <= (terms[:, None, None] + 16) * 2.0 ** -53 * (bound + np.abs(beta * C0)))


@pytest.mark.parametrize("b,n", [(4, 2), (13, 1)])
def test_stored_zero_blocks_meet_infinities(b, n):
    """A stored zero block adds nothing, except to a block with an infinity or a NaN."""
    pos, cell = si(n, 0.1, 84)
    ra, rb = (6.6, 4.0) if b == 4 else (4.0, 2.6)
    g = gpu_geometry(pos, cell, [rb, ra])
    pa, pb = oracle.neighbour_list(pos, cell, ra), oracle.neighbour_list(pos, cell, rb)
    rng = np.random.default_rng(8)
    # the first operand nearly all zeros, small entries in every row of both
    A, B = (oracle.Bsr(p, b, rng.standard_normal((p.nnzb, b, b)) * 2.0 ** -rng.integers(0, 60, size=(p.nnzb, 1, 1)))
            for p in (pa, pb))
    A.val[rng.random(pa.nnzb) < 0.9] = 0.0
    A.val[:, b - 1, :] = 0.0
    for bad in (None, np.inf, np.nan):
        if bad is not None:
            B.val[7, 1, 2] = bad
        with np.errstate(invalid="ignore"):
            ref, bound, terms = _sums(A, B, pa)
        got = _product(b, A, ra, B, rb, pa, ra, g)
        assert np.array_equal(np.isnan(got), np.isnan(ref.astype(float)))
        inf = np.isinf(ref.astype(float))
        assert np.array_equal(got[inf], ref.astype(float)[inf])
        fine = np.isfinite(ref.astype(float))
        with np.errstate(invalid="ignore"):
            ok = np.abs(got - ref) <= (terms[:, None, None] + 16) * 2.0 ** -53 * bound
        assert ok[fine].all()


@pytest.mark.parametrize("b", [4, 13])
def test_small_sums_of_a_symmetric_result(b):
    """Triangle 1: a block left to FP64 is mirrored like the others, and scaled."""
    pos, cell = si(2 if b == 4 else 1, 0.1, 95)
    ra = 6.6 if b == 4 else 4.0
    g = gpu_geometry(pos, cell, [ra])
    pa = oracle.neighbour_list(pos, cell, ra)
    rng = np.random.default_rng(9)
    A = oracle.Bsr(pa, b, rng.standard_normal((pa.nnzb, b, b)) * 2.0 ** -rng.integers(0, 40, size=(pa.nnzb, 1, 1)))
    At = oracle.transpose(A, pa)
    ref, bound, terms = _sums(A, At, pa)
    C = cuda(np.zeros((pa.nnzb, b, b)))
    lsq.block_matmul(g, b, cuda(A.val), 0, cuda(A.val), 0, C, 0, precision=lsq.F64, trans_b=1, triangle=1, alpha=-0.5)
    got = C.cpu().numpy()
    assert np.all(np.abs(got + 0.5 * ref) <= (terms[:, None, None] + 16) * 2.0 ** -53 * bound)
    rows = np.repeat(np.arange(pa.n), np.diff(pa.ptr))
    off = pa.col != rows
    assert np.array_equal(got[off], oracle.transpose(oracle.Bsr(pa, b, got), pa).val[off])
