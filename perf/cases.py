"""What this library is timed on: its public entry points over the sizes its users run.

Every case is diamond silicon (8 atoms a cell of 5.431 Angstrom, Gaussian displacements, some
atoms left out where a case says so, which makes the counts odd) in a two-centre sp3 model, the
workload of this repository's tests and benchmark: overlap and Hamiltonian reach 6.6 Angstrom,
the density matrix 8 or 10.  Sizes run from 64 atoms, where launches and latency count, to 4096.

`exact` forms the same results with dense float64 algebra, pairs beyond a range masked to zero.
"""
import math

import numpy as np
import torch

import paper_2002_07704_gb300 as lsq
from paper_2002_07704_gb300.autograd import lnv_omega

A_SI = 5.431
R_BOND = 2.35
R_S = R_H = 6.6
MU = -2.0
PREC = {"f64": lsq.F64, "f32": lsq.F32, "mixed": lsq.TF32X3}
BASIS = np.array([[0, 0, 0], [0, .5, .5], [.5, 0, .5], [.5, .5, 0],
                  [.25, .25, .25], [.25, .75, .75], [.75, .25, .75], [.75, .75, .25]])


def listed():
    return [
        # one energy and gradient of a 64-atom cell: the smallest call a user makes (a geometry
        # optimiser or a test loop calls it over and over); latency and launches
        dict(name="gradient_f64_64", kind="gradient", cells=2, vacancies=0, b=4, r_l=8.0, prec="f64"),
        # the float64 energy and gradient that ends and refines every minimisation
        dict(name="gradient_f64_1728", kind="gradient", cells=6, vacancies=0, b=4, r_l=10.0, prec="f64"),
        # the energy and gradient of the mixed mode at the benchmark's size
        dict(name="gradient_mixed_4096", kind="gradient", cells=8, vacancies=0, b=4, r_l=10.0, prec="mixed"),
        # float32 arithmetic on a crystal with vacancies: an odd number of atoms, ragged rows
        dict(name="gradient_f32_989", kind="gradient", cells=5, vacancies=11, b=4, r_l=10.0, prec="f32"),
        # the 13-orbital model of the batched workload, float64
        dict(name="gradient_f64_b13_64", kind="gradient", cells=2, vacancies=0, b=13, r_l=8.0, prec="f64"),
        # a whole minimisation in the mixed mode with its default float64 refinement and result
        dict(name="minimise_mixed_1000", kind="minimise", cells=5, vacancies=0, b=4, r_l=10.0, prec="mixed",
             steps=6),
        # many small independent systems minimised in one call
        dict(name="batch_f32_16", kind="batch", systems=16, cells=2, cells_max=3, b=4, r_l=8.0, prec="f32",
             steps=6),
        # LS.L on its natural range, float64: the plain product call on a large system
        dict(name="product_f64_2744", kind="product", cells=7, vacancies=0, b=4, ra=16.6, rb=10.0, rc=16.6,
             trans_a=False, trans_b=False, prec="f64"),
        # SL.Q^T truncated to the density matrix's range, split TF32: the product that takes most
        # of a mixed step
        dict(name="product_mixed_4096", kind="product", cells=8, vacancies=0, b=4, ra=16.6, rb=23.2, rc=10.0,
             trans_a=False, trans_b=True, prec="mixed"),
        # LS.L of the 13-orbital model in float32, one operand transposed
        dict(name="product_f32_b13_493", kind="product", cells=4, vacancies=19, b=13, ra=14.6, rb=8.0, rc=14.6,
             trans_a=True, trans_b=False, prec="f32"),
        # Omega and its derivatives in L, S and H through autograd (forces need them)
        dict(name="autograd_f32_512", kind="autograd", cells=4, vacancies=0, b=4, r_l=10.0, prec="f32"),
        # what an MD step does to the density matrix before its minimisation: the history of X
        # moves to the new geometry's patterns, propagates, S^-1 is refined and gives the next L
        dict(name="md_step_1720", kind="md", cells=6, vacancies=8, b=4, r_l=10.0, prec="f32", steps=3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["gradient", "gradient", "minimise", "batch", "product", "product", "autograd", "md"])
    b = 13 if kind in ("gradient", "product") and rng.random() < 0.3 else 4
    prec = rng.choice(["f64", "f32", "mixed"])
    if kind in ("autograd", "md", "batch") and prec == "mixed":
        prec = "f32"
    most = {"gradient": 1728 if prec == "f64" else 4096, "minimise": 1000, "autograd": 1000, "md": 1728,
            "product": 2744 if prec == "f64" else 4096, "batch": 216}[kind]
    if b == 13:
        most = 64 if prec == "f64" else 343
    atoms = _log(rng, 64, most)
    cells = max(2, math.ceil((atoms / 8) ** (1 / 3) - 1e-9))
    # up to a tenth of the atoms is left out
    c = dict(kind=kind, cells=cells, vacancies=min(8 * cells ** 3 - atoms, 8 * cells ** 3 // 10), b=b, prec=prec)
    if kind == "product":
        c["ra"], c["rb"], c["rc"] = (rng.choice([6.6, 10.0, 16.6]), rng.choice([6.6, 10.0, 16.6]),
                                     rng.choice([6.6, 10.0, 16.6]))
        c["trans_a"], c["trans_b"] = rng.random() < 0.5, rng.random() < 0.5
        return c
    c["r_l"] = rng.choice([8.0, 9.0, 10.0])
    if kind == "minimise":
        c["steps"] = rng.randint(3, 6)
    if kind == "md":
        c["steps"] = rng.randint(2, 4)
    if kind == "batch":
        c.update(systems=rng.randint(3, 16), cells=2, cells_max=rng.randint(2, 3), steps=rng.randint(3, 6))
        del c["vacancies"]
    return c


# ---- inputs ------------------------------------------------------------------------------------
def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _gen(seed, part):
    g = torch.Generator(device=_dev())
    g.manual_seed((int(seed) * 1000003 + part) & 0x7fffffffffff)
    return g


def _positions(n, vacancies, part=0):
    """n x n x n cells with displacements of 0.05 Angstrom, `vacancies` random atoms left out.

    The atoms of a case stay where they are: in use, one geometry is met by many Hamiltonians and
    density matrices (the iterations of a self-consistent field), and these come from the seed.
    """
    rng = np.random.default_rng([n, vacancies, part])
    ax = np.arange(n)
    cells = np.stack(np.meshgrid(ax, ax, ax, indexing="ij"), axis=-1).reshape(-1, 3)
    pos = (cells[:, None, :] + BASIS[None]).reshape(-1, 3) * A_SI
    pos = pos + rng.normal(0.0, 0.05, size=pos.shape)
    if vacancies:
        pos = pos[np.sort(rng.permutation(pos.shape[0])[vacancies:])]
    L = n * A_SI
    pos = np.mod(pos, L)
    pos[pos >= L] = 0.0
    return torch.from_numpy(np.ascontiguousarray(pos)).to(_dev()), [float(L)] * 3


class Pairs:
    """The atom pairs within R of each other (nearest images), row by row, and their distances."""

    def __init__(self, pos, cell, R):
        d2 = None
        for k in range(3):
            s = pos[None, :, k] - pos[:, None, k]
            s = s - cell[k] * torch.round(s / cell[k])
            d2 = s * s if d2 is None else d2 + s * s
        self.n = pos.shape[0]
        self.rows, self.cols = torch.nonzero(d2 <= R * R, as_tuple=True)
        self.dist = torch.sqrt(d2[self.rows, self.cols])
        key = self.rows * self.n + self.cols
        self.mirror = torch.searchsorted(key, self.cols * self.n + self.rows)

    def __len__(self):
        return int(self.rows.numel())


def _symmetrised(pairs, x):
    """(x + x^T) / 2; the same two numbers are added on both sides, so it is exactly symmetric."""
    return 0.5 * (x + x[pairs.mirror].transpose(1, 2))


def _decaying(pairs, b, gen, size, length, symmetric):
    """Random blocks that fall off with the distance of their atoms, as those of a gapped system do."""
    x = torch.randn((len(pairs), b, b), generator=gen, device=pairs.rows.device, dtype=torch.float64)
    x *= (size * torch.exp(-pairs.dist / length))[:, None, None]
    return _symmetrised(pairs, x) if symmetric else x


def _sk(pos, cell, pairs, b, gen):
    """H and S of the two-centre sp3 model, summed over periodic images, with a small symmetric
    perturbation of H; three copies of it and a d-like orbital for b = 13."""
    n = len(pairs)
    H = torch.zeros((n, 4, 4), dtype=torch.float64, device=pos.device)
    S = torch.zeros_like(H)
    d = pos[pairs.cols] - pos[pairs.rows]
    cl = torch.tensor(cell, dtype=torch.float64, device=pos.device)
    d = d - cl * torch.round(d / cl)
    eye3 = torch.eye(3, dtype=torch.float64, device=pos.device)
    reach = 1 if min(cell) < 2 * R_S + A_SI else 0
    for sx in range(-reach, reach + 1):
        for sy in range(-reach, reach + 1):
            for sz in range(-reach, reach + 1):
                v = d + cl * torch.tensor([sx, sy, sz], dtype=torch.float64, device=pos.device)
                r = torch.linalg.vector_norm(v, dim=1)
                cut = 0.5 * (1.0 + torch.cos(math.pi * torch.clamp(r - 5.6, 0.0, 1.0)))
                cut = torch.where((r < R_S) & (r > 1e-6), cut, torch.zeros_like(cut))
                r = torch.clamp(r, min=0.1)
                u = v / r[:, None]
                fh, fs = (R_BOND / r) ** 2 * cut, torch.exp(-2.0 * (r / R_BOND - 1.0)) * cut
                for M, f, (sss, sps, pps, ppp) in ((H, fh, (-1.94, 1.75, 3.05, -1.08)),
                                                   (S, fs, (0.10, -0.08, -0.12, 0.04))):
                    M[:, 0, 0] += sss * f
                    M[:, 0, 1:] += sps * f[:, None] * u
                    M[:, 1:, 0] -= sps * f[:, None] * u
                    M[:, 1:, 1:] += f[:, None, None] * ((pps - ppp) * u[:, :, None] * u[:, None, :] + ppp * eye3)
    on = pairs.rows == pairs.cols
    H[on] += torch.diag(torch.tensor([-5.25, 1.20, 1.20, 1.20], dtype=torch.float64, device=pos.device))
    S[on] += torch.eye(4, dtype=torch.float64, device=pos.device)
    noise = torch.rand((n, b, b), generator=gen, device=pos.device, dtype=torch.float64) - 0.5
    if b == 4:
        H += 0.02 * noise * torch.exp(-pairs.dist / R_BOND)[:, None, None]
    else:
        H4, S4 = H, S
        H = 0.2 * noise
        S = torch.zeros_like(H)
        for k in range(0, 12, 4):
            H[:, k:k + 4, k:k + 4] += H4
            S[:, k:k + 4, k:k + 4] = S4
        H[on, 12, 12] += 8.0
        S[on, 12, 12] = 1.0
    return _symmetrised(pairs, H), _symmetrised(pairs, S)


def _start_L(pairs, b, gen):
    """An L on its way to the minimum: half an inverse overlap on the atoms, decaying blocks around."""
    L = _decaying(pairs, b, gen, 0.02, 2.5, True)
    L[pairs.rows == pairs.cols] += 0.5 * torch.eye(b, dtype=torch.float64, device=L.device)
    return L


def _system(case, seed, part=0, cells=None):
    pos, cell = _positions(cells or case["cells"], case.get("vacancies", 0), part)
    gen = _gen(seed, part)
    ps, pl = Pairs(pos, cell, R_S), Pairs(pos, cell, case["r_l"])
    H, S = _sk(pos, cell, ps, case["b"], gen)
    return dict(pos=pos, cell=cell, ps=ps, pl=pl, H=H, S=S, L=_start_L(pl, case["b"], gen))


def _product_operands(case, seed):
    pos, cell = _positions(case["cells"], case["vacancies"])
    gen = _gen(seed, 0)
    pa, pb, pc = (Pairs(pos, cell, case[k]) for k in ("ra", "rb", "rc"))
    A, B = (_decaying(p, case["b"], gen, 1.0, 3.0, False) for p in (pa, pb))
    if case["prec"] != "f64":
        A, B = A.float(), B.float()
    return pos, cell, (pa, pb, pc), A, B


def _history(case, seed):
    """The MD history: geometry t, the one a step later, X(t), X(t - dt), ... and L S on R_L + R_S."""
    pos, cell = _positions(case["cells"], case["vacancies"])
    gen = _gen(seed, 0)
    moved = pos + 0.01 * torch.randn(pos.shape, generator=_gen(0, 1), device=pos.device, dtype=torch.float64)
    L = torch.tensor(cell, dtype=torch.float64, device=pos.device)
    moved = torch.remainder(moved, L)
    moved = torch.where(moved >= L, torch.zeros_like(moved), moved).contiguous()
    px = Pairs(pos, cell, case["r_l"] + R_S)
    X0 = _decaying(px, case["b"], gen, 0.05, 3.0, False)
    X0[px.rows == px.cols] += 0.5 * torch.eye(case["b"], dtype=torch.float64, device=pos.device)
    hist = [X0 + _decaying(px, case["b"], gen, 1e-3, 3.0, False) for _ in range(6)]
    return pos, moved, cell, px, hist, X0, gen


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind in ("gradient", "minimise", "autograd"):
        sys = _system(case, seed)
        ranges = lsq.lnv_required_ranges(R_S, R_H, case["r_l"])
        geom = lsq.Geometry(sys["pos"], sys["cell"], ranges)
        st.update(geom=geom, L=sys["L"], S=sys["S"], H=sys["H"])
        if kind == "autograd":
            dt = torch.float64 if case["prec"] == "f64" else torch.float32
            st.update({k: st[k].to(dt).requires_grad_(True) for k in ("L", "S", "H")})
        else:
            st.update(ctx=lsq.Lnv(geom, case["b"], R_S, R_H, case["r_l"]), G=torch.empty_like(sys["L"]))
        if kind == "minimise":
            st["ctx"].init_L(st["S"], st["L"].zero_())
    elif kind == "batch":
        cells = _batch_cells(case)
        parts = [_system(case, seed, k + 1, n) for k, n in enumerate(cells)]
        ranges = lsq.lnv_required_ranges(R_S, R_H, case["r_l"])
        geoms = [lsq.Geometry(p["pos"], p["cell"], ranges) for p in parts]
        geom = lsq.concat_geometries(geoms)
        st.update(geom=geom, ctx=lsq.Lnv(geom, case["b"], R_S, R_H, case["r_l"]),
                  S=torch.cat([p["S"] for p in parts]), H=torch.cat([p["H"] for p in parts]),
                  L=torch.zeros_like(torch.cat([p["L"] for p in parts])), mu=[MU] * len(parts))
        st["ctx"].init_L(st["S"], st["L"])
    elif kind == "product":
        pos, cell, pairs, A, B = _product_operands(case, seed)
        ranges = sorted({case["ra"], case["rb"], case["rc"]})
        geom = lsq.Geometry(pos, cell, ranges)
        C = torch.empty((len(pairs[2]), case["b"], case["b"]), dtype=A.dtype, device=A.device)
        st.update(geom=geom, A=A, B=B, C=C)
    elif kind == "md":
        pos, moved, cell, px, hist, X0, gen = _history(case, seed)
        r_l, b = case["r_l"], case["b"]
        ranges = [R_S, r_l, r_l + R_S]
        g0, g1 = lsq.Geometry(pos, cell, ranges), lsq.Geometry(moved, cell, ranges)
        ps = Pairs(moved, cell, R_S)
        _, S = _sk(moved, cell, ps, b, gen)
        blocks = lambda r: torch.empty((g1.nnzb(r), b, b), dtype=torch.float64, device=pos.device)
        # a start of S^-1 carried from the step before: a few refinements away from the new one
        Xi = blocks(1).zero_()
        lsq.hotelling_inverse(g1, b, S, 0, Xi, 1, 2, 6, precision=lsq.F64)
        st.update(geom=g0, geom_to=g1, hist=hist, LS=X0, S=S, Xi0=Xi, Xi=torch.empty_like(Xi),
                  X_next=torch.empty_like(X0), moved=[blocks(2) for _ in hist], L=blocks(1))
    if "ctx" in st and kind != "gradient":
        st["L_work"] = torch.empty_like(st["L"])
    return st


def _batch_cells(case):
    """Cells per edge of each system: small and larger ones in turn."""
    return [case["cells"] + k % (case["cells_max"] - case["cells"] + 1) for k in range(case["systems"])]


def run(st):
    case, geom = st["case"], st["geom"]
    kind, b, prec = case["kind"], case["b"], PREC[case["prec"]]
    if kind == "gradient":
        om, ne = st["ctx"].energy_gradient(st["L"], st["S"], st["H"], MU, precision=prec, G=st["G"])
        return {"omega": om, "ne": ne, "G": _held(case, st["G"])}
    if kind == "minimise":
        L = st["L_work"].copy_(st["L"])
        rep = st["ctx"].minimise(L, st["S"], st["H"], MU, max_iter=case["steps"], precision=prec)
        return {"omega": rep["omega_ev"], "ne": rep["ne"], "L": _held(case, L)}
    if kind == "batch":
        L = st["L_work"].copy_(st["L"])
        reps = st["ctx"].minimise_batch(L, st["S"], st["H"], st["mu"], max_iter=case["steps"], precision=prec)
        return {"omega": np.array([r["omega_ev"] for r in reps], dtype=np.float32),
                "ne": np.array([r["ne"] for r in reps], dtype=np.float32), "L": _held(case, L)}
    if kind == "product":
        r = [geom.range_id(case[k]) for k in ("ra", "rb", "rc")]
        n = lsq.block_matmul(geom, b, st["A"], r[0], st["B"], r[1], st["C"], r[2], precision=prec,
                             trans_a=case["trans_a"], trans_b=case["trans_b"])
        return {"triples": n, "C": st["C"]}
    if kind == "autograd":
        args = [st[k] for k in ("L", "S", "H")]
        om = lnv_omega(geom, b, *args, MU, (0, 1, 2, 3, 5))
        dL, dS, dH = torch.autograd.grad(om, args)
        return {"omega": om.detach().float(), "dL": dL, "dS": dS, "dH": dH}
    # md
    kappa, alpha, c = lsq.XL_DISSIPATION_K5
    g1 = st["geom_to"]
    lsq.xl_propagate(geom, b, 2, st["hist"], st["LS"], st["X_next"], kappa, alpha, c)
    for src, dst in zip([st["X_next"]] + st["hist"][:-1], st["moved"]):
        lsq.pattern_remap(geom, 2, g1, 2, b, src, dst)
    Xi = st["Xi"].copy_(st["Xi0"])
    lsq.hotelling_inverse(g1, b, st["S"], 0, Xi, 1, 2, case["steps"], precision=prec, start=False)
    lsq.xl_initial_L(g1, b, 2, st["moved"][0], 1, Xi, 1, st["L"], precision=prec)
    return {"X": st["moved"], "Sinv": _held(case, Xi), "L": _held(case, st["L"])}


def _held(case, x):
    """A result in the precision that it was computed in (the library hands every gradient and
    density matrix back in float64 arrays)."""
    return x if case["prec"] == "f64" else x.float()


# ---- the work a pass cannot do without ----------------------------------------------------------
def _triples(ma, mb, mc):
    """Block products (i, k, j) of C = A.B with pairs masked by ma, mb and mc (float32 0/1)."""
    return float(((ma @ mb) * mc).double().sum())


def work(case):
    b, kind = case["b"], case["kind"]
    es = 8 if case["prec"] == "f64" else 4
    total = {"bytes": 0.0, "flops": 0.0}
    # TF32 would round the counts
    torch.backends.cuda.matmul.allow_tf32 = False

    def add(nbytes, triples):
        total["bytes"] += nbytes
        total["flops"] += 2.0 * b ** 3 * triples

    sizes = _batch_cells(case) if kind == "batch" else [case["cells"]]
    for n in sizes:
        pos, cell = _positions(n, case.get("vacancies", 0))
        memo = {}

        def m(R):
            if R not in memo:
                p = Pairs(pos, cell, R)
                x = torch.zeros((p.n, p.n), dtype=torch.float32, device=pos.device)
                x[p.rows, p.cols] = 1.0
                memo[R] = (x, float(len(p)))
            return memo[R]

        bb = b * b
        if kind == "product":
            ra, rb, rc = case["ra"], case["rb"], case["rc"]
            add(es * bb * (m(ra)[1] + m(rb)[1] + m(rc)[1]), _triples(m(ra)[0], m(rb)[0], m(rc)[0]))
            continue
        rl = case["r_l"]
        r1, r3 = rl + R_S, R_H + rl + R_S
        # the products of one energy and gradient; symmetric results and triangles count half
        t_ls = _triples(m(rl)[0], m(R_S)[0], m(r1)[0])
        if kind == "md":
            x, s, l = m(r1)[1], m(R_S)[1], m(rl)[1]
            t_u = _triples(m(r1)[0], m(rl)[0], m(rl)[0])
            add(8 * bb * (8 * x + 2 * 6 * x), 0.0)
            add(8 * bb * (s + 3 * l), case["steps"] * (t_ls + 0.5 * t_u) + t_u)
            continue
        t_lsl = _triples(m(r1)[0], m(rl)[0], m(r3)[0])
        t_q = _triples(m(R_H)[0], m(r1)[0], m(r3)[0])
        t_m = _triples(m(r1)[0], m(r3)[0], m(rl)[0])
        grad = t_ls + t_q + t_m
        energy = 0.5 * t_lsl + 0.5 * t_q  # LSL, SLS
        line = t_ls + 0.5 * t_lsl + t_q + 0.5 * t_m  # P, F, QD, Z
        inputs = bb * (m(rl)[1] + m(R_S)[1] + m(R_H)[1])
        if kind == "gradient":
            add(8 * (inputs + bb * m(rl)[1]), grad + energy)
        elif kind == "autograd":
            t_k = _triples(m(r3)[0], m(r1)[0], m(R_H)[0])
            fwd = 2 * t_ls + t_lsl + t_k
            add(es * 2 * inputs, 3 * fwd)
        else:  # minimise, batch: mixed steps, two float64 ones in a mixed run, the result in float64
            steps = case["steps"] + (0 if case["prec"] == "f64" else 2)
            fresh = 1 + (0 if case["prec"] == "f64" else 1)
            add(8 * (inputs + bb * m(rl)[1]), steps * (t_ls + t_m + line) + fresh * t_q + t_ls + t_q + energy)
    return total


# ---- the same results in dense float64 ----------------------------------------------------------
def _dense(pairs, x):
    b = x.shape[1]
    out = torch.zeros((pairs.n, b, pairs.n, b), dtype=torch.float64, device=x.device)
    out[pairs.rows, :, pairs.cols, :] = x.double()
    return out.reshape(pairs.n * b, pairs.n * b)


def _blocks(pairs, X):
    b = X.shape[0] // pairs.n
    return X.reshape(pairs.n, b, pairs.n, b)[pairs.rows, :, pairs.cols, :].contiguous()




def exact(case, seed):
    kind, b = case["kind"], case["b"]
    n = 8 * case["cells"] ** 3 - case.get("vacancies", 0)
    if kind == "product":
        if n * b > 17000:
            return None
        _, _, (pa, pb, pc), A, B = _product_operands(case, seed)
        triples = _triples(*((_dense(p, torch.ones((len(p), 1, 1), device=A.device)).float()) for p in (pa, pb, pc)))
        dA, dB = _dense(pa, A), _dense(pb, B)
        dA, dB = dA.t() if case["trans_a"] else dA, dB.t() if case["trans_b"] else dB
        return {"triples": int(triples), "C": _blocks(pc, dA @ dB)}
    if kind in ("gradient", "autograd"):
        if n * b > 8000:
            return None
        sys = _system(case, seed)
        if kind == "autograd" and case["prec"] != "f64":
            sys.update({k: sys[k].float() for k in ("L", "S", "H")})
        L, S, H = _dense(sys["pl"], sys["L"]), _dense(sys["ps"], sys["S"]), _dense(sys["ps"], sys["H"])
        if kind == "gradient":
            Hp = H - MU * S
            LS = L @ S
            LSL = LS @ L
            Q = Hp @ LS
            SLS = S @ LS
            G1 = Q @ LS
            M = G1 + G1.t() + Q.t() @ LS
            # N_e sums LSL over the pairs within R_H + R_L + R_S, which hold all of S and S L S
            omega = 2.0 * (3.0 * (L * Q).sum() - 2.0 / 3.0 * (L * M).sum())
            ne = 2.0 * (3.0 * (S * LSL).sum() - 2.0 * (LSL * SLS).sum())
            G = 2.0 * (3.0 * (Q + Q.t()) - 2.0 * M)
            return {"omega": float(omega), "ne": float(ne), "G": _blocks(sys["pl"], G)}
        L, S, H = (x.requires_grad_(True) for x in (L, S, H))
        LSL = L @ S @ L
        Hp = H - MU * S
        om = 2.0 * (3.0 * (Hp.t() * LSL).sum() - 2.0 * (Hp.t() * (LSL @ (S @ L))).sum())
        dL, dS, dH = torch.autograd.grad(om, (L, S, H))
        return {"omega": om.detach(), "dL": _blocks(sys["pl"], dL), "dS": _blocks(sys["ps"], dS),
                "dH": _blocks(sys["ps"], dH)}
    if kind == "md":
        if n * b > 8000:
            return None
        pos, moved, cell, px, hist, X0, gen = _history(case, seed)
        qx, ql, ps = (Pairs(moved, cell, R) for R in (case["r_l"] + R_S, case["r_l"], R_S))
        _, S = _sk(moved, cell, ps, b, gen)
        kappa, alpha, c = lsq.XL_DISSIPATION_K5
        nxt = 2.0 * hist[0] - hist[1] + kappa * (X0 - hist[0])
        for ck, x in zip(c, hist):
            nxt = nxt + alpha * ck * x
        out = [_blocks(qx, _dense(px, x)) for x in [nxt] + hist[:-1]]
        Sd = _dense(ps, S)
        mask = _dense(ql, torch.ones((len(ql), b, b), device=pos.device))
        X = Sd / Sd.abs().sum(1).max() ** 2 * mask
        for _ in range(6 + case["steps"]):
            X = 2.0 * X - (X @ Sd @ X) * mask
        P = _dense(qx, out[0]) @ X
        return {"X": out, "Sinv": _blocks(ql, X), "L": _blocks(ql, 0.5 * (P + P.t()))}
    return None  # a minimisation's path is its own
