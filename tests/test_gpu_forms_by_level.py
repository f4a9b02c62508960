"""FP64 handles at n_p = 3 and 4, whose levels of many rows hold FP64 blocks and whose smaller ones digits, through
the calls that meet both: V-cycles against the oracle's (1e-9, as elsewhere), the CG and GMRES solves, a batch, the
p-multigrid front end (whose level of degree 1 has as many rows as the mesh), vectors that are not 16-byte
aligned, and many columns (whose level 0 is in digits whatever its n_p)."""
import numpy as np
import pytest

from synthetic import jittered_square, kuhn_cube, sin_source
from tests.gpu_common import OracleCase, rel

pytestmark = pytest.mark.gpu


def _t(x):
    import torch
    return torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("make", [lambda: jittered_square(50), lambda: kuhn_cube(10)])
@pytest.mark.parametrize("nu", [1, 2])
def test_vcycle_matches_oracle(make, nu):
    import torch
    from paper_2012_08024_gb300 import Solver
    mesh = make()
    S, oc = Solver(mesh, p=1, max_levels=4, nu_pre=nu, nu_post=nu).bind(), OracleCase(mesh, 1, 4, nu=nu)
    r = np.random.default_rng(nu).standard_normal(S.info["n_dofs"])
    want = oc.to_tree(0, oc.V.apply(oc.to_work(0, r)))
    for shift in (0, 1):   # vectors on 16-byte boundaries, and 8 bytes behind one
        buf = torch.zeros(2, S.info["n_dofs"] + 1, dtype=torch.float64, device="cuda")
        src, dst = buf.view(-1)[shift:shift + S.info["n_dofs"]], torch.zeros(S.info["n_dofs"] + 1, dtype=torch.float64,
                                                                            device="cuda")[shift:][:S.info["n_dofs"]]
        src.copy_(torch.tensor(r, device="cuda"))
        S.vcycle(src, dst)
        assert rel(dst.cpu().numpy(), want) <= 1e-9
        y = torch.zeros(S.info["n_dofs"] + 1, dtype=torch.float64, device="cuda")[shift:][:S.info["n_dofs"]]
        S.apply(0, src, y)
        assert rel(y.cpu().numpy(), oc.to_tree(0, oc.H.A[0] @ oc.to_work(0, r))) <= 1e-13


@pytest.mark.parametrize("make,p,kw", [
    (lambda: jittered_square(60), 1, {}), (lambda: jittered_square(60), 1, dict(precision="fp32")),
    (lambda: jittered_square(60), 1, dict(single_graph=False)), (lambda: kuhn_cube(10), 1, dict(coarsen="primal")),
    (lambda: jittered_square(60), 1, dict(krylov="gmres", nu_pre=0, nu_post=3)),
    (lambda: jittered_square(60), 3, dict(pmg=True)), (lambda: kuhn_cube(10), 2, dict(pmg=True))])
def test_solves_reach_the_tolerance(make, p, kw):
    from scipy.sparse import bsr_matrix
    from paper_2012_08024_gb300 import Solver
    S = Solver(make(), p=p, max_levels=4, **kw).bind()
    b = np.random.default_rng(p).standard_normal((S.ne, S.np_))
    u, hist, it, rc = S.solve_b(_t(b))
    assert rc == 0
    e = S.export_level(0)
    A = bsr_matrix((e["val"], e["col"], e["rowptr"]), shape=(S.info["n_dofs"],) * 2).tocsr()
    x, b = u.cpu().numpy()[e["perm"]].ravel(), b[e["perm"]].ravel()
    size = np.linalg.norm(abs(A) @ np.abs(x))
    assert np.linalg.norm(b - A @ x) <= 1e-10 * np.linalg.norm(b) + it * 2.0 ** -53 * size


def test_batch_matches_single_solves():
    from paper_2012_08024_gb300 import BatchSolver, Solver
    meshes = [jittered_square(n, seed=k) for k, n in enumerate((41, 30, 43))]
    B = BatchSolver(meshes, p=1, max_levels=4).bind()
    u, hists, its, rc = B.solve(_t(sin_source(B.quadrature_points()[0])))
    assert rc == 0
    for m, mesh in enumerate(meshes):
        S = Solver(mesh, p=1, max_levels=4).bind()
        us, _, it, rcs = S.solve(_t(sin_source(S.quadrature_points()[0])))
        assert rcs == 0 and abs(int(its[m]) - it) <= 1
        assert rel(u[B.elem_offsets[m]:B.elem_offsets[m + 1]].cpu().numpy(), us.cpu().numpy()) <= 1e-10


@pytest.mark.parametrize("make,p", [(lambda: jittered_square(50), 1), (lambda: kuhn_cube(10), 1)])
def test_many_columns(make, p):
    import torch
    from paper_2012_08024_gb300 import Solver
    mesh, R = make(), 5
    S, S1 = Solver(mesh, p=p, max_levels=4, precision="fp32", nrhs=R).bind(), Solver(mesh, p=p, max_levels=4).bind()
    n = S.info["n_dofs"]
    x = torch.tensor(np.random.default_rng(p).standard_normal((n, R)), device="cuda")
    y, y1 = torch.empty_like(x), torch.empty(n, dtype=torch.float64, device="cuda")
    S.apply_multi(x, y)
    for r in range(R):
        S1.apply(0, x[:, r].contiguous(), y1)
        assert rel(y[:, r].cpu().numpy(), y1.cpu().numpy()) <= 1e-14
    S.apply(0, x[:, 0].contiguous(), y1)
    assert rel(y[:, 0].cpu().numpy(), y1.cpu().numpy()) <= 1e-15
