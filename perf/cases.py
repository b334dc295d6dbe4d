"""What a user of this framework has it do, as measurable cases: solves of
cracked XFEM systems (K u = f to a relative residual of 1e-8) and the single
operations that a solve consists of, through the package's public entry
points.

A case's mesh, crack and subdomain boxes come from the case alone (they are the
set-up system); the loads and vectors come from the seed.  The listed sizes are
those of the repository's own workloads: 8^3 (the parity cube), 12^3 and 36^3
(iterations against system size), 24^3, 32^3 (propagation sweep) and 48^3 (the
benchmark).  draw() spreads over the same range, odd mesh sizes included.
"""
import functools
import hashlib
import json

import numpy as np
import torch

import xfem_inputs as X
from paper_2111_09294_gb300 import Elements, Solver
from paper_2111_09294_gb300 import sweep
from paper_2111_09294_gb300.autograd import solve as differentiable_solve
from xfem_inputs import cracks as C

TOL = 1e-8


def _ellipse(name, do, m, n_box, a, b, tilt, warp, r_e, its, **kw):
    return dict(name=name, do=do, m=m, n_box=n_box, crack="ellipse", a=a, b=b, tilt=tilt,
                warp=warp, r_e=r_e, its=its, **kw)


def _two_cracks(name, do, its, **kw):
    return dict(name=name, do=do, m=48, n_box=8, crack="two", r_e=0.05, its=its, **kw)


def listed():
    """its: the iterations that the method takes on that system (for work())."""
    edge8 = dict(m=8, n_box=2, crack="edge", z0=0.5, front=0.45, r_e=0.15)
    ell = dict(a=0.30, b=0.20, tilt=30.0, warp=0.03)
    swp = dict(m=32, n_box=8, a=0.25, b=0.25, tilt=30.0, warp=0.0, r_e=0.07)
    return [
        # a small component or a coarse study: launches and latency decide
        dict(name="solve_fp64_8", do="solve", precision="fp64", its=57, **edge8),
        # the same in mixed precision, on the smallest system of the scalability study
        _ellipse("solve_mixed_12", "solve", 12, 2, r_e=2.0 / 12, its=72, precision="mixed", **ell),
        # an ordinary model in plain FP64
        _ellipse("solve_fp64_24", "solve", 24, 4, r_e=0.08, its=68, precision="fp64", **ell),
        # the paper's own preconditioner blocks, one per subdomain
        _ellipse("solve_blocks_24", "blocks", 24, 4, r_e=0.08, its=50, precision="mixed", **ell),
        # the benchmark system, in both precisions: the largest solves
        _two_cracks("solve_mixed_48", "solve", 115, precision="mixed"),
        _two_cracks("solve_fp64_48", "solve", 110, precision="fp64"),
        # eight load cases of one crack front, as one batch
        _ellipse("batch8_32", "batch", its=100, loads=8, precision="mixed", **swp),
        # successive crack fronts of a sweep solved together, uneven load counts
        _ellipse("sweep_32", "sweep", its=100, fronts=3, step=0.04, loads=5, precision="mixed",
                 **swp),
        # a differentiable solve: compliance, its gradient in the load and in every modulus
        _ellipse("adjoint_32", "adjoint", its=130, sigma=0.3, precision="mixed", **swp),
        # the next crack front of a propagation: set-up from host arrays, then the solve
        _ellipse("front_32", "front", its=100, step=0.0133, precision="mixed", **swp),
        # one application of the preconditioner (Algorithm 3) in FP64
        _ellipse("precond_36", "precond", 36, 6, r_e=2.0 / 36, its=1, precision="fp64", **ell),
        # one product with the block-scaled FP32 operator
        _two_cracks("spmv_mixed_48", "spmv", 1, precision="mixed"),
    ]


def draw(rng):
    do = rng.choice(["solve", "solve", "precond", "spmv", "batch", "adjoint", "front", "sweep",
                     "blocks"])
    lo, hi = {"solve": (8, 44), "precond": (8, 44), "spmv": (8, 44), "batch": (10, 32),
              "adjoint": (10, 30), "front": (12, 28), "sweep": (10, 24), "blocks": (8, 20)}[do]
    m = int(round(lo * (hi / lo) ** rng.random()))
    c = dict(do=do, m=m, n_box=max(2, min(8, round(m / rng.uniform(4.0, 6.5)))), its=80)
    c["precision"] = (rng.choice(["fp64", "mixed"]) if do in ("solve", "spmv") else
                      "fp64" if do == "precond" else "mixed")
    if m < 14:
        c.update(crack="edge", z0=0.5, front=round(rng.uniform(0.3, 0.6), 3),
                 r_e=round(rng.uniform(1.1, 1.4) / m, 4))
    else:
        a = round(rng.uniform(0.18, 0.31), 3)
        c.update(crack="ellipse", a=a, b=round(a * rng.uniform(0.6, 1.0), 3),
                 tilt=round(rng.uniform(0.0, 35.0), 1), warp=round(rng.uniform(0.0, 0.03), 3),
                 r_e=round(rng.uniform(1.8, 2.3) / m, 4))
    if do == "batch":
        c["loads"] = rng.randint(2, 8)
    if do == "sweep":
        c.update(fronts=2, loads=rng.randint(2, 8))
    if do in ("front", "sweep"):
        c["step"] = round(rng.uniform(0.3, 1.2) / m, 4)
    if do == "adjoint":
        c["sigma"] = 0.3
    return c


# ---- the systems -------------------------------------------------------------

def _cracks(c, i):
    """The crack of front i (each front is `step` further than the one before)."""
    grow = i * c.get("step", 0.0)
    if c["crack"] == "edge":
        return [C.PlanarEdgeCrack(c["z0"], c["front"] + grow, c["r_e"])]
    if c["crack"] == "two":
        return [C.WarpedPennyCrack((0.5, 0.5, 0.3), 0.2, 0.02, c["r_e"]),
                C.WarpedEdgeCrack(0.7, 0.25, 0.02, c["r_e"])]
    return [C.TiltedEllipticalCrack((0.5, 0.5, 0.5), c["a"] + grow, c["b"] + grow,
                                    np.deg2rad(c["tilt"]), c["warp"], c["r_e"])]


GEOMETRY = ("m", "n_box", "crack", "z0", "front", "a", "b", "tilt", "warp", "r_e", "step", "sigma")


@functools.lru_cache(maxsize=4)
def _system(text, i):
    c = json.loads(text)
    name = "case_" + hashlib.sha256(f"{text} {i}".encode()).hexdigest()[:16]
    X.CONFIGS[name] = dict(m=c["m"], n_box=c["n_box"], cracks=lambda: _cracks(c, i))
    if c.get("sigma"):
        X.CONFIGS[name]["young"] = lambda m: np.random.default_rng(0).lognormal(
            0.0, c["sigma"], m ** 3)
    P = X.make(name)
    return X.by_subdomain(P) if c["do"] == "blocks" else (P, None)


def _problem(case, i=0):
    """The system of front i and the caller's blocks (or None), kept per geometry."""
    geometry = {k: case[k] for k in GEOMETRY if k in case}
    geometry["do"] = "blocks" if case["do"] == "blocks" else ""
    return _system(json.dumps(geometry, sort_keys=True), i)


def _loads(case, i, seed):
    """Seeded tractions on the loaded face: (load cases, n), every front another set."""
    P, blocks = _problem(case, i)
    m = case.get("loads", 1)
    if case["do"] == "sweep":
        m = max(1, m - i)
    if blocks is not None:        # the generator's numbering first, then box by box
        F = X.load_cases(_problem(dict(case, do="solve"))[0], m, seed)
        out = np.empty_like(F)
        out[:, P.dof_map_from] = F
        return out
    return X.load_cases(P, m, seed=seed + 1000 * i)


def _vector(case, seed):
    dt = np.float32 if case["precision"] == "mixed" else np.float64
    return np.random.default_rng(seed).standard_normal(int(_problem(case)[0].n)).astype(dt)


# ---- what a user's program does ------------------------------------------------

def prepare(case, seed):
    do = case["do"]
    P, blocks = _problem(case)
    s = {"do": do, "precision": case["precision"]}
    kw = {"precision": case["precision"]}
    if do == "sweep":
        Ps = [_problem(case, i)[0] for i in range(case["fronts"])]
        s["solvers"] = sweep.make_solvers(Ps)
        s["F"] = [torch.tensor(_loads(case, i, seed), device="cuda")
                  for i in range(case["fronts"])]
        return s
    if do == "batch":
        kw["max_batch"] = case["loads"]
    if do == "blocks":
        kw["blocks"] = blocks
    s["solver"] = Solver.from_problem(P, **kw)
    if do in ("precond", "spmv"):
        s["x"] = torch.tensor(_vector(case, seed), device="cuda")
        return s
    if do == "front":
        s["next"] = _problem(case, 1)[0]
        s["f"] = torch.tensor(_loads(case, 1, seed)[0], device="cuda")
        return s
    F = torch.tensor(_loads(case, 0, seed), device="cuda")
    if do == "batch":
        s["F"] = F
        return s
    s["f"] = F[0].contiguous()
    if do == "adjoint":
        s["f"].requires_grad_(True)
        s["young"] = torch.tensor(P.young, device="cuda", requires_grad=True)
        s["elements"] = Elements.from_dict(X.element_data(P), "cuda")
    return s


def run(s):
    do = s["do"]
    if do in ("solve", "blocks"):
        return s["solver"].solve(s["f"], tol=TOL)[0]
    if do == "batch":
        return s["solver"].solve_batch(s["F"], tol=TOL)[0]
    if do == "sweep":
        return [U for U, _ in sweep.solve_systems(s["solvers"], s["F"], TOL)]
    if do == "adjoint":
        u = differentiable_solve(s["solver"], s["f"], TOL, young=s["young"],
                                 elements=s["elements"])
        J = (s["f"] * u).sum()
        df, dE = torch.autograd.grad(J, (s["f"], s["young"]))
        return {"J": J, "df": df, "dE": dE}
    if do == "front":
        solver = Solver.from_problem(s["next"], precision=s["precision"], prev=s["solver"])
        u = solver.solve(s["f"], tol=TOL)[0]
        solver.close()
        return u
    if do == "precond":
        return s["solver"].precond(s["x"])
    y, xty = s["solver"].spmv(s["x"], precision=s["precision"])
    return {"y": y, "xty": xty}


# ---- what it cannot do without ---------------------------------------------------

def _modes(P):
    """Coarse columns of each box: 6 rigid modes, and 6 more where its
    jump-enriched nodes are not all on one line."""
    cols = np.full(P.n_sub, 6)
    jump = np.asarray(P.kind) == 1
    for b in np.unique(np.asarray(P.sub_of_node)[jump]):
        x = P.coords[jump & (np.asarray(P.sub_of_node) == b)]
        if len(x) >= 3:
            d = x[np.argmax(((x - x[0]) ** 2).sum(1))] - x[0]
            off = np.cross(x - x[0], d)
            if ((off * off).sum(1) > 1e-12 * (d @ d) ** 2).any():
                cols[b] = 12
    return cols


def work(case):
    """One pass: the product, the coarse solve and the vectors of every
    iteration (the matrix is read again in each: it is larger than the caches
    on the systems that matter); the gradient and the set-up on top."""
    size = 4 if case["precision"] == "mixed" else 8
    total = {"bytes": 0.0, "flops": 0.0}
    for i in range(case.get("fronts", 1)):
        P = _problem(case, 1 if case["do"] == "front" else i)[0]
        n, nnz, nnzb = int(P.n), len(P.val), len(P.col)
        k = int(_modes(P).sum())
        loads = max(1, case.get("loads", 1) - (i if case["do"] == "sweep" else 0))
        if case["do"] == "spmv":
            b, f = size * (nnz + 2 * n) + 4 * nnzb, 2.0 * nnz
        elif case["do"] == "precond":
            b, f = size * (k * k + 4 * n), 2.0 * k * k + 60.0 * n
        else:
            b = size * (nnz + k * k + 10 * n * loads) + 4 * nnzb
            f = 2.0 * loads * (nnz + k * k + 20 * n)
            if case["do"] == "blocks":
                sq = float((np.diff(_problem(case)[1].astype(np.int64)) ** 2).sum())
                b, f = b + size * sq, f + 2.0 * sq
            runs = case["its"] * (2 if case["do"] == "adjoint" else 1)
            b, f = b * runs, f * runs
        if case["do"] == "front":
            b, f = b + 8.0 * (nnz + 2 * k * k), f + float(k) ** 3
        total["bytes"] += b
        total["flops"] += f
    return total


# ---- the same in 64 bits, by torch alone -------------------------------------------

class _Exact:
    """K as a scalar CSR matrix, its node-block (or given block) Cholesky
    factors and the deflation basis, in FP64."""

    def __init__(self, P, blocks=None, coarse=True):
        dev = lambda a, t=torch.int64: torch.as_tensor(np.asarray(a), device="cuda").to(t)
        dof, rowp, col, vp = (dev(a) for a in (P.dof_ptr, P.row_ptr, P.col, P.val_ptr))
        val = dev(P.val, torch.float64)
        self.n, self.dof, n_nodes = int(P.n), dof, int(P.n_nodes)
        bsz = dof.diff()
        node = torch.repeat_interleave(torch.arange(n_nodes, device="cuda"), rowp.diff())
        bJ = bsz[col]
        before = torch.cumsum(bJ, 0) - bJ                     # columns before block p
        total = torch.cat([before, (before[-1:] + bJ[-1:])])
        length = total[rowp[1:]] - total[rowp[:-1]]           # scalar row length
        p = torch.repeat_interleave(torch.arange(len(col), device="cuda"), vp.diff())
        w = torch.arange(len(val), device="cuda") - vp[p]
        a, b = w // bJ[p], w % bJ[p]
        at = vp[rowp[node[p]]] + a * length[node[p]] + before[p] - before[rowp[node[p]]] + b
        cols, vals = torch.empty_like(at), torch.empty_like(val)
        cols[at], vals[at] = dof[col[p]] + b, val
        own = torch.repeat_interleave(torch.arange(n_nodes, device="cuda"), bsz)
        crow = vp[rowp[own]] + (torch.arange(self.n, device="cuda") - dof[own]) * length[own]
        crow = torch.cat([crow, crow.new_tensor([len(val)])])
        self.K = torch.sparse_csr_tensor(crow, cols, vals, (self.n, self.n))
        diag = torch.nonzero(col == node)[:, 0]
        self.blocks = []
        for size in (3, 6, 15):
            I = torch.nonzero(bsz == size)[:, 0]
            if len(I):
                e = torch.arange(size * size, device="cuda")
                D = val[vp[diag[I]][:, None] + e].reshape(-1, size, size)
                d = dof[I][:, None] + torch.arange(size, device="cuda")
                self.blocks.append((d, torch.linalg.cholesky(D)))
        if coarse:
            self._coarse(P, dev)

    def _coarse(self, P, dev):
        cols = _modes(P)
        first = np.concatenate([[0], np.cumsum(cols)])
        sub, kind = np.asarray(P.sub_of_node), np.asarray(P.kind)
        x = P.coords - P.centres[sub]
        o, z = np.ones(len(x)), np.zeros(len(x))
        R = [[o, z, z, z, x[:, 2], -x[:, 1]], [z, o, z, -x[:, 2], z, x[:, 0]],
             [z, z, o, x[:, 1], -x[:, 0], z]]
        d = np.asarray(P.dof_ptr, dtype=np.int64)[:-1]
        more = (cols == 12)[sub]
        jump = more & (kind == 1)
        i, j, v = [], [], []
        for r in range(3):
            for c in range(6):
                for rows, shift, scale, sel in ((d + r, 0, o, o > 0),
                                                (d + r, 6, P.hsign.astype(float), more),
                                                (d + 3 + r, 6, o, jump)):
                    i.append(rows[sel])
                    j.append((first[:-1][sub] + shift + c)[sel])
                    v.append((scale * R[r][c])[sel])
        ij, v = dev(np.stack([np.concatenate(i), np.concatenate(j)])), dev(
            np.concatenate(v), torch.float64)
        shape = (self.n, int(first[-1]))
        Z = torch.sparse_coo_tensor(ij, v, shape).coalesce()
        self.Z = Z.to_sparse_csr()
        self.Zt = Z.t().coalesce().to_sparse_csr()
        E = self.Zt @ (self.K @ Z.to_dense())
        self.E = torch.linalg.cholesky(0.5 * (E + E.t()))

    def coarse(self, g):
        return self.Z @ torch.cholesky_solve(g[:, None], self.E)[:, 0]

    def jacobi(self, r):
        y = torch.empty_like(r)
        for d, L in self.blocks:
            y[d] = torch.cholesky_solve(r[d][:, :, None], L)[:, :, 0]
        return y

    def precond(self, r):
        y = self.jacobi(r)
        return y + self.coarse(self.Zt @ (r - self.K @ y))

    def solve(self, f):
        """Preconditioned CG, restarted on the residual until it is as small as FP64 gives."""
        u = torch.zeros_like(f)
        for _ in range(3):
            r = f - self.K @ u
            d = self.coarse(self.Zt @ r)
            r = r - self.K @ d
            stop = 1e-9 * float(r.norm())
            z = self.precond(r)
            p, rz = z, torch.dot(r, z)
            for it in range(1000):
                q = self.K @ p
                alpha = rz / torch.dot(p, q)
                d, r = d + alpha * p, r - alpha * q
                if it % 10 == 9 and float(r.norm()) <= stop:
                    break
                z = self.precond(r)
                rz, old = torch.dot(r, z), rz
                p = z + (rz / old) * p
            u = u + d
        return u

    def scaled(self, x):
        """L^-1 K L^-T x, L the node blocks' Cholesky factors."""
        t = torch.empty_like(x)
        for d, L in self.blocks:
            t[d] = torch.linalg.solve_triangular(L.mT, x[d][:, :, None], upper=True)[:, :, 0]
        t = self.K @ t
        y = torch.empty_like(x)
        for d, L in self.blocks:
            y[d] = torch.linalg.solve_triangular(L, t[d][:, :, None], upper=False)[:, :, 0]
        return y


def _modulus_gradient(P, u):
    """-u_e^T Khat_e u_e of every element."""
    D = X.element_data(P)
    size = np.diff(D["dof_ptr"])
    mats = torch.tensor(D["mats"], device="cuda")
    uz = torch.cat([u, u.new_zeros(1)])
    out = u.new_zeros(len(size))
    for d in np.unique(size):
        for e in np.array_split(np.nonzero(size == d)[0], max(1, (size == d).sum() // 4096)):
            ue = uz[torch.as_tensor(D["dofs"][D["dof_ptr"][e][:, None] + np.arange(d)].astype(
                np.int64), device="cuda")]
            at = torch.as_tensor(D["mat_off"][e][:, None] + np.arange(d * d), device="cuda")
            K = mats[at].reshape(-1, d, d)
            out[torch.as_tensor(e, device="cuda")] = -torch.einsum("ei,eij,ej->e", ue, K, ue)
    return out


def exact(case, seed):
    do = case["do"]
    if do == "sweep":
        return [torch.stack([S.solve(f) for f in torch.tensor(_loads(case, i, seed), device="cuda")])
                for i, S in ((i, _Exact(_problem(case, i)[0])) for i in range(case["fronts"]))]
    P = _problem(case, 1 if do == "front" else 0)[0]
    S = _Exact(P, coarse=do != "spmv")
    if do in ("precond", "spmv"):
        x = torch.tensor(_vector(case, seed), device="cuda").double()
        if do == "precond":
            return S.precond(x)
        y = S.scaled(x) if case["precision"] == "mixed" else S.K @ x
        return {"y": y, "xty": torch.dot(x, y)}
    F = torch.tensor(_loads(case, 1 if do == "front" else 0, seed), device="cuda")
    U = torch.stack([S.solve(f) for f in F])
    if do == "batch":
        return U
    if do == "adjoint":
        return {"J": torch.dot(F[0], U[0]), "df": 2.0 * U[0], "dE": _modulus_gradient(P, U[0])}
    return U[0]
