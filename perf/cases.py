"""The workloads by which this library's speed is followed.

A user of the library sets up one mesh (host set-up, then bind: what a program
keeps) and solves on it for one source after another; so the handle of a case
is kept for the process and every seed gives new sources, new vectors.  Most
cases are that solve in its different forms: the smallest mesh, where launches
and latency count, up to operators several times the L2; odd block sizes (n_p =
3), even ones (6, 10), tetrahedra; FP64 and FP32 V-cycles; the p-multigrid front
end; GMRES as in the paper; many meshes; many right-hand sides; forward and
adjoint with gradients.  Two are single operations that programs with their own
outer method call.  Outputs are solutions, gradients and vectors.
"""
import functools
import itertools
import math

import numpy as np
import torch

from paper_2012_08024_gb300 import BatchSolver, Solver
from paper_2012_08024_gb300.autograd import CDGSolve, SolverCache
from synthetic import batched_squares, face_neighbors, jittered_square, kuhn_cube, smoothed_lognormal_kappa

DEV = "cuda:0"


def listed():
    return [
        # the default options on a small mesh: a solve inside someone's loop, all latency
        dict(name="tri32_p2", kind="solve", dim=2, n=32, p=2, levels=4, nu=1, precision="fp64"),
        # p = 1 (n_p = 3, the paper's degree), a ragged mid-size mesh, host arrays in and out
        dict(name="tri101_p1_host", kind="solve", dim=2, n=101, p=1, levels=5, nu=1, precision="fp64", host=True),
        # the benchmark's discretisation, V(2,2) in FP64; level 0 is several times the L2
        dict(name="tri256_p3", kind="solve", dim=2, n=256, p=3, levels=6, nu=2, precision="fp64"),
        # the same hierarchy with the FP32 V-cycle inside FP64 CG
        dict(name="tri256_p3_fp32", kind="solve", dim=2, n=256, p=3, levels=6, nu=2, precision="fp32"),
        # tetrahedra: flux coarsening behind the p-multigrid front end, FP32 V-cycle
        dict(name="tet24_p2_pmg_fp32", kind="solve", dim=3, n=24, p=2, levels=5, nu=2, precision="fp32", pmg=True),
        # the paper's solver, GMRES(50) with V(0,3), its mixed boundary, hierarchy to one element
        dict(name="tri128_p1_gmres", kind="gmres", dim=2, n=128, p=1, levels=16, nu=3, precision="fp64", beta=0.0),
        # 64 meshes of 500 to 20000 triangles in one handle
        dict(name="batch64_p2", kind="batch", count=64, tmin=500, tmax=20000, p=2, levels=4, nu=1, precision="fp64"),
        # many right-hand sides: FP32 V-cycle blocks, the FP64 apply by exact splitting
        dict(name="multi256_tri100_p3", kind="multi", dim=2, n=100, p=3, levels=5, nu=2, precision="fp32", nrhs=256,
             split=True),
        # a small ragged number of columns, n_p = 6, FP64 apply on CUDA cores
        dict(name="multi40_tri50_p2", kind="multi", dim=2, n=50, p=2, levels=4, nu=1, precision="fp32", nrhs=40,
             split=False),
        # a differentiable solve with variable kappa on tetrahedra: forward and backward
        dict(name="adjoint_tet16_p2", kind="adjoint", dim=3, n=16, p=2, levels=5, nu=1, precision="fp64"),
        # one V-cycle as the preconditioner of a caller's own Krylov method
        dict(name="vcycle_tri128_p3", kind="vcycle", dim=2, n=128, p=3, levels=5, nu=2, precision="fp64"),
        # one product with the level-0 operator
        dict(name="apply_tri256_p3", kind="apply", dim=2, n=256, p=3, levels=6, nu=2, precision="fp64"),
    ]


def n_basis(dim, p):
    return math.comb(p + dim, dim)


def log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["solve"] * 6 + ["multi"] * 2 + ["gmres", "batch", "adjoint", "vcycle", "apply"])
    dim = 2 if kind in ("batch", "multi", "gmres") else 3 if kind == "adjoint" else rng.choice([2, 2, 3])
    p = rng.choice([1, 2, 2, 3, 3, 4] if dim == 2 else [1, 2])
    nu = rng.choice([1, 2])
    if kind == "batch":
        tmin = int(log_uniform(rng, 100, 1000))
        return dict(kind=kind, count=int(log_uniform(rng, 2, 64)), tmin=tmin,
                    tmax=int(tmin * log_uniform(rng, 2, 20)), p=min(p, 3), levels=3, nu=nu, precision="fp64")
    if kind == "multi":
        p, nrhs = min(p, 3), int(log_uniform(rng, 3, 256))
        n = max(9, int(math.sqrt(log_uniform(rng, 3e5, 5e7) / nrhs / (2 * n_basis(2, p)))))
        return dict(kind=kind, dim=2, n=min(n, 120), p=p, levels=levels_for(2, min(n, 120)), nu=nu,
                    precision=rng.choice(["fp32", "fp32", "bf16"]), nrhs=nrhs, split=rng.random() < 0.5)
    per = 2 if dim == 2 else 6
    elements = log_uniform(rng, 3e3, {"adjoint": 2.5e5, "gmres": 4e5}.get(kind, 1.3e6)) / n_basis(dim, p)
    n = max(5, round((elements / per) ** (1 / dim)))
    if kind == "gmres":
        return dict(kind=kind, dim=2, n=n, p=min(p, 2), levels=16, nu=3, precision="fp64",
                    beta=rng.choice([0.0, 1.0, 10.0]))
    case = dict(kind=kind, dim=dim, n=n, p=p, levels=levels_for(dim, n), nu=nu, precision="fp64")
    if kind == "solve":
        if dim == 3 or p in (2, 3):
            case["precision"] = rng.choice(["fp64", "fp32"])
        if p > 1 and rng.random() < 0.4:
            case["pmg"] = True
        elif dim == 3:
            case["coarsen"] = "primal"
        case["host"] = rng.random() < 0.2
    elif kind != "adjoint" and dim == 3:
        case["coarsen"] = "primal"
    return case


def levels_for(dim, n):
    """Agglomeration levels down to some 60 elements (a factor 8 or 17, then 4 to 5)."""
    ne = (2 * n * n / 8) if dim == 2 else (6 * n ** 3 / 17)
    return max(2, 2 + round(math.log(max(ne, 64) / 64) / math.log(4.0 if dim == 2 else 4.7)))


# ------------------------------------------------------------------ what a program keeps
def mesh_of(c):
    if c["kind"] == "gmres":
        return jittered_square(c["n"], neumann_axes=(0,))
    return jittered_square(c["n"]) if c["dim"] == 2 else kuhn_cube(c["n"])


@functools.lru_cache(maxsize=16)
def handle(key):
    """The bound handle of a case, its quadrature points on the device and its kappa."""
    c = dict(key)
    kappa = None
    kw = dict(p=c["p"], max_levels=c["levels"], nu_pre=c["nu"], nu_post=c["nu"], precision=c["precision"])
    if c["kind"] == "batch":
        S = BatchSolver(batched_squares(c["count"], c["tmin"], c["tmax"]), **kw).bind(DEV)
        cache = None
    elif c["kind"] == "adjoint":
        mesh = mesh_of(c)
        kappa = torch.tensor(smoothed_lognormal_kappa(face_neighbors(mesh)), device=DEV)
        cache = SolverCache(mesh, coarsen="primal", tol=1e-12, **kw)
        S = cache.get(kappa, DEV)
    else:
        if c["kind"] == "gmres":
            kw.update(nu_pre=0, krylov="gmres", beta=c["beta"], velocity=(1.0, 0.0))
        if c["kind"] == "multi":
            kw.update(nrhs=c["nrhs"], tc_fp64_apply=c["split"])
        kw.update(pmg=bool(c.get("pmg")), coarsen=c.get("coarsen", "flux"), maxit=1000)
        S = Solver(mesh_of(c), **kw).bind(DEV)
        cache = None
    xq = torch.tensor(S.quadrature_points()[0], device=DEV)
    return S, xq, kappa, cache


def key_of(case):
    return tuple(sorted((k, v) for k, v in case.items() if k not in ("name", "host")))


# ------------------------------------------------------------------ inputs of a seed
def sources(xq, seed, count=None):
    """Sine combinations f = sum c_mn sin(m pi x) sin(n pi y) (times a z profile on
    cubes), c ~ N(0, 1), m, n <= 8, at the quadrature points."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    m = torch.arange(1, 9, device=DEV, dtype=torch.float64) * math.pi
    s = [torch.sin(xq[..., k, None] * m) for k in range(xq.shape[-1])]
    out = torch.empty((count or 1,) + xq.shape[:-1], dtype=torch.float64, device=DEV)
    for k in range(count or 1):
        f = ((s[0] @ torch.randn(8, 8, generator=g, device=DEV, dtype=torch.float64)) * s[1]).sum(-1)
        if len(s) == 3:
            f = f * (s[2] @ torch.randn(8, generator=g, device=DEV, dtype=torch.float64))
        out[k] = f
    return out if count else out[0]


def vector(S, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    return torch.randn(S.info["n_dofs"], generator=g, device=DEV, dtype=torch.float64)


def prepare(case, seed):
    S, xq, kappa, cache = handle(key_of(case))
    kind = case["kind"]
    state = dict(kind=kind, S=S)
    if kind in ("vcycle", "apply"):
        state.update(x=vector(S, seed), y=torch.empty(S.info["n_dofs"], dtype=torch.float64, device=DEV))
    elif kind == "multi":
        state.update(f=sources(xq, seed, case["nrhs"]))
    elif kind == "adjoint":
        # the gradient of <w, u> with respect to the source and to kappa
        state.update(f=sources(xq, seed).requires_grad_(True), kappa=kappa.clone().requires_grad_(True),
                     w=vector(S, seed + 1).reshape(S.ne, S.np_), cache=cache)
    elif case.get("host"):
        state.update(kind="host", f=sources(xq, seed).cpu().numpy())
    else:
        state.update(f=sources(xq, seed))
    return state


def converged(rc):
    if rc:
        raise RuntimeError("the solve did not converge (code %d)" % rc)


def run(state):
    S, kind = state["S"], state["kind"]
    if kind == "vcycle":
        S.vcycle(state["x"], state["y"])
        return state["y"]
    if kind == "apply":
        S.apply(0, state["x"], state["y"])
        return state["y"]
    if kind == "adjoint":
        f, kappa = state["f"], state["kappa"]
        u = CDGSolve.apply(f, kappa, state["cache"])
        df, dkappa = torch.autograd.grad(u, (f, kappa), state["w"])
        return dict(u=u.detach(), df=df, dkappa=dkappa)
    solve = {"multi": S.solve_multi, "host": S.solve_host}.get(kind, S.solve)
    u, _, _, rc = solve(state["f"])
    converged(rc)
    return u


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    """The operator of each level read once for every application that the method
    makes (CG or GMRES apply, smoothing steps, V-cycle residual) in 60 outer steps,
    the sources and the solution once."""
    kind, nu = case["kind"], case["nu"]
    s = 8 if case["precision"] == "fp64" else 4 if case["precision"] == "fp32" else 2
    if kind == "batch":
        rng = np.random.default_rng(1)
        ne = sum(np.exp(rng.uniform(np.log(case["tmin"]), np.log(case["tmax"]), size=case["count"])))
        dim = 2
    else:
        dim = case["dim"]
        ne = (2 if dim == 2 else 6) * float(case["n"]) ** dim
    npb = n_basis(dim, case["p"])
    level0 = ne * (dim + 2) * npb * npb
    cycle = (level0 if not case.get("pmg") else 1.3 * level0) * 1.3 * (nu + 1 if kind == "gmres" else 2 * nu + 1)
    vec = ne * npb
    if kind == "apply":
        return {"bytes": 8 * (level0 + 2 * vec), "flops": 2 * level0}
    if kind == "vcycle":
        return {"bytes": s * cycle + 16 * vec, "flops": 2 * cycle}
    cols = case.get("nrhs", 1)
    solves = 2 if kind == "adjoint" else 1
    steps = 60 * solves
    # with many columns the vectors, not the blocks, are what each application moves
    per_step = 8 * level0 + s * cycle + (cols > 1) * cols * vec * (8 * 10 + 4 * 3 * (2 * nu + 1))
    return {"bytes": steps * per_step + 24 * solves * vec * cols, "flops": 2 * steps * cols * (level0 + cycle)}


# ------------------------------------------------------------------ the same in plain 64-bit torch
def load_vector(mesh, p, f):
    """b[K][i] = int_K f phi_i with the collapsed Gauss-Legendre rule of degree 2p and
    the orthonormalised scaled monomials, user order (f at the rule's points)."""
    d = mesh.dim
    ref, w = [], []
    one = [np.polynomial.legendre.leggauss(math.ceil((2 * p + k) / 2)) for k in range(1, d + 1)]
    one = [(0.5 * (x + 1.0), 0.5 * v) for x, v in one]
    for ids in itertools.product(*(range(len(x)) for x, _ in one)):
        t = [one[k][0][i] for k, i in enumerate(ids)]
        pt, wt = [], float(np.prod([one[k][1][i] for k, i in enumerate(ids)]))
        for k in range(d):
            pt.append(t[k] * float(np.prod([1 - t[j] for j in range(k + 1, d)])))
            wt *= (1 - t[k]) ** k
        ref.append(pt)
        w.append(wt)
    ref, w = torch.tensor(ref, device=DEV, dtype=torch.float64), torch.tensor(w, device=DEV, dtype=torch.float64)
    v = torch.tensor(mesh.xyz, device=DEV)[torch.tensor(mesh.elem, device=DEV)]
    E = v[:, 1:] - v[:, :1]
    x = v[:, :1] + ref @ E
    c = v.mean(1, keepdim=True)
    h = (v - c).norm(dim=2).amax(1)
    y = (x - c) / h[:, None, None]
    exps = [a for t in range(p + 1)
            for a in sorted((a for a in itertools.product(range(t + 1), repeat=d) if sum(a) == t), reverse=True)]
    mono = torch.stack([torch.stack([y[..., k] ** a[k] for k in range(d)]).prod(0) for a in exps], -1)
    wq = w * torch.linalg.det(E).abs()[:, None]
    R = torch.linalg.cholesky(torch.einsum("kqi,kq,kqj->kij", mono, wq, mono))
    phi = torch.linalg.solve_triangular(R, mono.transpose(1, 2), upper=False)
    return torch.einsum("kiq,kq,...kq->...ki", phi, wq, f), phi * wq[:, None, :]


def operator(row, col, val, n):
    """CSR of a matrix given by square blocks."""
    b = val.shape[1]
    counts = np.diff(row)
    crow = np.zeros(n * b + 1, dtype=np.int64)
    crow[1:] = np.cumsum(np.repeat(counts * b, b))
    blockrow = torch.tensor(np.repeat(np.arange(n), counts), device=DEV)
    v = torch.tensor(val, device=DEV)
    order = torch.argsort(((blockrow[:, None] * b + torch.arange(b, device=DEV)).reshape(-1)), stable=True)
    cols = (torch.tensor(col, device=DEV).long()[:, None] * b + torch.arange(b, device=DEV))
    cols = cols[:, None, :].expand(-1, b, -1).reshape(-1, b)[order].reshape(-1)
    A = torch.sparse_csr_tensor(torch.tensor(crow, device=DEV), cols, v.reshape(-1, b)[order].reshape(-1),
                                size=(n * b, n * b))
    on_diagonal = torch.tensor(col, device=DEV) == blockrow
    return A, torch.linalg.inv(v[on_diagonal])


class Plain:
    """V-cycle and conjugate gradients on the exported level operators, tree order."""

    def __init__(self, S, nu_pre, nu_post):
        self.nu, self.lev = (nu_pre, nu_post), []
        for l in range(S.n_levels):
            e = S.export_level(l)
            A, Dinv = operator(e["rowptr"], e["col"], e["val"], len(e["perm"]))
            self.lev.append((A, Dinv, torch.tensor(e["L"], device=DEV), torch.tensor(e["parent"], device=DEV).long()))
            if l == 0:
                self.perm = torch.tensor(e["perm"], device=DEV)
        self.last = torch.linalg.inv(self.lev[-1][0].to_dense())

    def smooth(self, l, x, b, times):
        A, Dinv = self.lev[l][:2]
        for _ in range(times):
            r = b - A @ x
            x = x + 2.0 / 3.0 * torch.bmm(Dinv, r.reshape(Dinv.shape[0], Dinv.shape[1], -1)).reshape(x.shape)
        return x

    def cycle(self, b, l=0):
        if l + 1 == len(self.lev):
            x = self.last @ b
            return x + self.last @ (b - self.lev[l][0] @ x)
        A, Dinv, L, parent = self.lev[l]
        x = self.smooth(l, torch.zeros_like(b), b, self.nu[0])
        r = torch.bmm(L.transpose(1, 2), (b - A @ x).reshape(L.shape[0], L.shape[1], -1))
        nc = self.lev[l + 1][1].shape[0]
        bc = torch.zeros(nc, r.shape[1], r.shape[2], dtype=b.dtype, device=DEV).index_add_(0, parent, r)
        xc = self.cycle(bc.reshape(-1, b.shape[1]), l + 1).reshape(bc.shape)
        x = x + torch.bmm(L, xc[parent]).reshape(x.shape)
        return self.smooth(l, x, b, self.nu[1])

    def solve(self, b):
        """b [n][columns]: conjugate gradients to 1e-14 of each column."""
        x, r = torch.zeros_like(b), b.clone()
        z = self.cycle(r)
        p, rz, stop = z.clone(), (r * z).sum(0), 1e-14 * b.norm(dim=0)
        for _ in range(400):
            q = self.lev[0][0] @ p
            a = rz / (p * q).sum(0)
            x, r = x + a * p, r - a * q
            if bool((r.norm(dim=0) <= stop).all()):
                break
            z = self.cycle(r)
            rz, old = (r * z).sum(0), rz
            p = z + rz / old * p
        return x


def exact(case, seed):
    kind = case["kind"]
    unknowns = n_basis(case.get("dim", 2), case["p"]) * case.get("nrhs", 1) * float(case.get("n", 0)) ** case.get("dim", 2)
    if kind == "batch" or case.get("beta") or unknowns > 3e6:
        return None   # several meshes, a non-symmetric operator, hundreds of columns: over 20 s
    state = prepare(case, seed)
    S = state["S"]
    H = Plain(S, case["nu"], case["nu"])   # symmetric, as conjugate gradients need (GMRES solves with V(0, nu))
    if kind == "apply":
        return H.lev[0][0] @ state["x"]
    if kind == "vcycle":
        return H.cycle(state["x"][:, None])[:, 0]
    f = state["f"]
    f = torch.tensor(f, device=DEV) if isinstance(f, np.ndarray) else f.detach()
    b, weights = load_vector(mesh_of(case), case["p"], f)
    b = b[None] if b.dim() == 2 else b

    def solved(b):   # [columns][element][i], user order
        u = torch.empty_like(b)
        x = H.solve(b[:, H.perm].reshape(b.shape[0], -1).T.contiguous())
        u[:, H.perm] = x.T.reshape(b.shape)
        return u

    u = solved(b)
    if kind == "adjoint":
        lam = solved(state["w"][None])[0]
        return dict(u=u[0], df=torch.einsum("kiq,ki->kq", weights, lam), dkappa=None)
    return u if kind == "multi" else u[0]
