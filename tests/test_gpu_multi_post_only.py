"""Many right-hand sides with V(0, nu) cycles, whose first kernels differ from those of V(nu, nu) (D^-1 b without
a first step, the restriction taken from the right-hand side itself, the prolongation without an addition): every
column has to converge and to agree with its own single solve.  In exact arithmetic these solves take 65 to 90
iterations (V(0, 2), V(0, 3), meshes of this kind), far below the limit of 500, which a wrong cycle does not meet.
Both solves end at 1e-12, so the solutions differ by far less than 1e-9."""
import pytest

from synthetic import jittered_square, sine_combination_sources

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R", [3, 34, 132])
@pytest.mark.parametrize("p,nu_post", [(1, 3), (2, 2), (2, 3), (3, 2)])
@pytest.mark.parametrize("tune", [True, False])
def test_columns_converge(R, p, nu_post, tune):
    import torch
    from paper_2012_08024_gb300 import Solver
    mesh = jittered_square(14)
    S1 = Solver(mesh, p=p, max_levels=3, tol=1e-12).bind()
    f = torch.tensor(sine_combination_sources(S1.quadrature_points()[0], R, mmax=4), device="cuda")
    S = Solver(mesh, p=p, max_levels=3, tol=1e-12, nu_pre=0, nu_post=nu_post, precision="fp32", nrhs=R,
               autotune=tune).bind()
    u, _, its, rc = S.solve_multi(f)
    assert rc == 0, its
    for r in sorted({0, R // 2, R - 1}):
        want = S1.solve(f[r].contiguous())[0]
        assert float((u[r] - want).norm() / want.norm()) <= 1e-9, r
