"""Float64 products from integer slices on the tensor cores against exact sums.

The reference is the sum of the float64 products in extended precision (numpy longdouble, 64 bits
or more).  A result is off by its last rounding (2^-53 of itself) and by what the slices drop, at
most 2^-70 of the largest entries of its row of A and column of B per term: together less than
2^-50 of max |A| max |B| for the sums of up to 2^11 terms here, and for a block that lies far
below that, 1e-9 of its own largest entry (blocks 2^34 below it are summed in FP64).
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


def _reference(A, B, pc, atoms):
    """Blocks of (A.B)|pc in the rows `atoms`, in extended precision, the same of the absolute
    values, and their positions in pc."""
    n = pc.n
    sel = np.concatenate([np.arange(pc.ptr[i], pc.ptr[i + 1]) for i in atoms])
    at = np.repeat(np.arange(len(atoms)), [pc.ptr[i + 1] - pc.ptr[i] for i in atoms])

    def dense(X, rows):
        out = np.zeros((len(rows), 4, n, 4), dtype=np.longdouble)
        for k, i in enumerate(rows):
            q = slice(X.pat.ptr[i], X.pat.ptr[i + 1])
            out[k][:, X.pat.col[q], :] = X.val[q].transpose(1, 0, 2)
        return out.reshape(len(rows) * 4, n * 4)

    dA, dB = dense(A, atoms), dense(B, range(n))
    with np.errstate(invalid="ignore", over="ignore"):
        C, S = dA @ dB, np.abs(dA) @ np.abs(dB)
    pick = lambda X: X.reshape(len(atoms), 4, n, 4)[at, :, pc.col[sel], :]
    return pick(C), pick(S), sel


def _sums(A, B, pc):
    """As _reference, over the stored blocks only, block by block."""
    C = np.zeros((pc.nnzb, A.b, A.b), dtype=np.longdouble)
    S = np.zeros_like(C)
    with np.errstate(invalid="ignore", over="ignore"):
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
    return C, S


def _run(g, A, ra, B, rb, pc, rc, ta=0, tb=0, triangle=0, alpha=1.0, beta=0.0, C0=None):
    C = cuda(np.zeros((pc.nnzb, A.b, A.b)) if C0 is None else C0)
    lsq.block_matmul(g, A.b, cuda(A.val), g.range_id(ra), cuda(B.val), g.range_id(rb), C, g.range_id(rc),
                     precision=lsq.F64, trans_a=ta, trans_b=tb, triangle=triangle, alpha=alpha, beta=beta)
    g.device_status()
    return C.cpu().numpy()


# ragged groups and tiles (61 atoms), one atom, lists of less than 16 atoms k
@pytest.mark.parametrize("n,drop,ra,rb,rc", [(2, 3, 6.6, 8.0, 8.0), (2, 0, 2.5, 2.5, 4.0), (1, 7, 3.0, 3.0, 3.0),
                                             (3, 1, 10.0, 6.6, 14.0)])
@pytest.mark.parametrize("ta,tb", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("kind", ["normal", "decaying", "full"])
def test_sliced_product(n, drop, ra, rb, rc, ta, tb, kind, monkeypatch):
    monkeypatch.setenv("LSQ_F64_SLICED", "1")
    pos, cell = si(n, 0.1, 77)
    pos = pos[:pos.shape[0] - drop]
    ranges = sorted({ra, rb, rc})
    g = gpu_geometry(pos, cell, ranges)
    P = {R: oracle.neighbour_list(pos, cell, R) for R in ranges}
    rng = np.random.default_rng(3)

    def mat(R):
        p = P[R]
        x = rng.standard_normal((p.nnzb, 4, 4))
        if kind == "decaying":
            x *= np.exp(-5.0 * rng.random((p.nnzb, 1, 1)))
        if kind == "full":  # every digit of every entry -256 or so: the largest sums
            x = np.full_like(x, -(256 / 511) * (1 + 2.0 ** -52)) * rng.choice([1.0, 1.0, 1.0, -1.0], size=x.shape)
        return oracle.Bsr(p, 4, x)

    A, B = mat(ra), mat(rb)
    opA = oracle.transpose(A, P[ra]) if ta else A
    opB = oracle.transpose(B, P[rb]) if tb else B
    ref, _, sel = _reference(opA, opB, P[rc], sorted(rng.choice(P[rc].n, size=min(4, P[rc].n), replace=False)))
    C0 = rng.standard_normal((P[rc].nnzb, 4, 4))
    scale = np.abs(A.val).max() * np.abs(B.val).max()
    for alpha, beta in ((1.0, 0.0), (-0.75, 0.5)):
        got = _run(g, A, ra, B, rb, P[rc], rc, ta, tb, alpha=alpha, beta=beta, C0=C0)
        want = alpha * ref + beta * C0[sel]
        assert np.abs(got[sel] - want).max() <= 2.0 ** -50 * max(scale, np.abs(want).max())
    # triangles: those blocks as in the whole product, and the mirrored half of a symmetric one
    rows = np.repeat(np.arange(P[rc].n), np.diff(P[rc].ptr))
    up = P[rc].col >= rows
    full = _run(g, A, ra, B, rb, P[rc], rc, ta, tb)
    assert np.array_equal(_run(g, A, ra, B, rb, P[rc], rc, ta, tb, triangle=2)[up], full[up])
    assert np.array_equal(_run(g, A, ra, B, rb, P[rc], rc, ta, tb, triangle=3)[P[rc].col <= rows], full[P[rc].col <= rows])
    sym = _run(g, A, ra, B, rb, P[rc], rc, ta, tb, triangle=1)
    mirrored = oracle.transpose(oracle.Bsr(P[rc], 4, sym), P[rc]).val
    off = P[rc].col != rows
    assert np.array_equal(sym[up], full[up]) and np.array_equal(sym[off], mirrored[off])


@pytest.mark.parametrize("case", ["range", "inf_nan", "zero_rows", "huge", "tiny"])
def test_sliced_product_falls_back_where_slices_do_not_reach(case, monkeypatch):
    monkeypatch.setenv("LSQ_F64_SLICED", "1")
    pos, cell = si(2, 0.1, 78)
    g = gpu_geometry(pos, cell, [6.6, 8.0])
    pa, pb = oracle.neighbour_list(pos, cell, 6.6), oracle.neighbour_list(pos, cell, 8.0)
    rng = np.random.default_rng(4)
    a, b = rng.standard_normal((pa.nnzb, 4, 4)), rng.standard_normal((pb.nnzb, 4, 4))
    if case == "range":  # blocks of very different size in a row: each C block has its own scale
        a *= 10.0 ** rng.integers(-30, 30, size=(pa.nnzb, 1, 1))
        b *= 10.0 ** rng.integers(-30, 30, size=(pb.nnzb, 1, 1))
        b[rng.random(pb.nnzb) < 0.7] = 0.0
    if case == "inf_nan":
        a[5, 1, 2], a[100, 0, 0], b[40, 3, 3] = np.inf, np.nan, -np.inf
    if case == "zero_rows":
        a[pa.ptr[3]:pa.ptr[5]] = 0.0
        b[:] = 0.0
        b[::7] = 1e-300
    if case == "huge":
        a *= 1e200
        b *= 1e107
    if case == "tiny":
        a *= 1e-200
        b *= 1e-115
    A, B = oracle.Bsr(pa, 4, a), oracle.Bsr(pb, 4, b)
    # nothing stored reaches blocks outside the patterns, so a dense sum would let 0 x inf in there
    ref, bound = _sums(A, B, pb)
    got = _run(g, A, 6.6, B, 8.0, pb, 8.0)
    with np.errstate(over="ignore"):
        want = ref.astype(np.float64)
    fine = np.isfinite(want)
    assert np.array_equal(np.isnan(want), np.isnan(got)) and np.array_equal(want[~fine & ~np.isnan(want)], got[~fine & ~np.isnan(want)])
    # relative to the block's largest sum of absolute values: what an FP64 sum keeps
    err = np.where(fine, np.abs(got - want), 0.0).max(axis=(1, 2))
    top = np.where(fine, bound, 0.0).max(axis=(1, 2)).astype(np.float64)
    assert np.all(err <= 1e-9 * top + 1e-322)


# larger blocks in 4 x 4 units: the smallest, an odd and the largest size; one atom in a ragged group of two
@pytest.mark.parametrize("b", [9, 13, 16])
@pytest.mark.parametrize("ta,tb", [(0, 0), (0, 1), (1, 0), (1, 1)])
def test_sliced_product_large_blocks(b, ta, tb, monkeypatch):
    monkeypatch.setenv("LSQ_F64_SLICED", "1")
    pos, cell = si(1, 0.1, 79)
    pos = pos[:7]
    g = gpu_geometry(pos, cell, [2.6, 4.0])
    pa, pb = oracle.neighbour_list(pos, cell, 4.0), oracle.neighbour_list(pos, cell, 2.6)
    rng = np.random.default_rng(b)
    A, B = (oracle.Bsr(p, b, rng.standard_normal((p.nnzb, b, b))) for p in (pa, pb))
    opA = oracle.transpose(A, pa) if ta else A
    opB = oracle.transpose(B, pb) if tb else B
    ref, _ = _sums(opA, opB, pa)
    C0 = rng.standard_normal((pa.nnzb, b, b))
    scale = np.abs(A.val).max() * np.abs(B.val).max()
    for alpha, beta in ((1.0, 0.0), (-0.75, 0.5)):
        got = _run(g, A, 4.0, B, 2.6, pa, 4.0, ta, tb, alpha=alpha, beta=beta, C0=C0)
        assert np.abs(got - (alpha * ref + beta * C0)).max() <= 2.0 ** -50 * max(scale, np.abs(ref).max())
    rows = np.repeat(np.arange(pa.n), np.diff(pa.ptr))
    full = _run(g, A, 4.0, B, 2.6, pa, 4.0, ta, tb)
    sym = _run(g, A, 4.0, B, 2.6, pa, 4.0, ta, tb, triangle=1)
    mirrored = oracle.transpose(oracle.Bsr(pa, b, sym), pa).val
    off, up = pa.col != rows, pa.col >= rows
    assert np.array_equal(sym[up], full[up]) and np.array_equal(sym[off], mirrored[off])
    # entries out of the slices' reach, and ones that are no numbers
    A.val *= 10.0 ** rng.integers(-30, 30, size=(pa.nnzb, 1, 1))
    A.val[3, b - 1, 0], B.val[2, 0, b - 1] = np.inf, np.nan
    opA = oracle.transpose(A, pa) if ta else A
    opB = oracle.transpose(B, pb) if tb else B
    ref, bound = _sums(opA, opB, pa)
    got, want = _run(g, A, 4.0, B, 2.6, pa, 4.0, ta, tb), ref.astype(np.float64)
    fine = np.isfinite(want)
    assert np.array_equal(np.isnan(want), np.isnan(got))
    assert np.array_equal(want[~fine & ~np.isnan(want)], got[~fine & ~np.isnan(want)])
    with np.errstate(invalid="ignore"):
        err = np.where(fine, np.abs(got - want), 0.0)
    # per 4 x 4 unit of a block, against its largest sum of absolute values
    for R in range(0, b, 4):
        for K in range(0, b, 4):
            u = (slice(None), slice(R, R + 4), slice(K, K + 4))
            top = np.where(fine[u], bound[u], 0.0).max(axis=(1, 2)).astype(np.float64)
            assert np.all(err[u].max(axis=(1, 2)) <= 1e-9 * top)
