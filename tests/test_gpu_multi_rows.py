"""Many-right-hand-side block kernels at ragged column counts: the FP64 level-0 apply by integer digits
(one column per lane) and the FP32 V-cycle kernels (one, two or four columns per lane, as R allows).

Apply, per entry: the digits keep A to 2^-59 of its row's bound and x to 2^-59 of its column's largest
value among the row's neighbours, so T <= 50 terms are off by less than 1e-14 (largest |A|)(largest |x|),
and the FP64 reference by T eps of the same: 1e-13 of it bounds both.  Solves run to 1e-12, so a column
and its single solve differ by far less than 1e-9."""
import numpy as np
import pytest

from synthetic import jittered_square, kuhn_cube, sine_combination_sources

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make,p", [(lambda: jittered_square(17), 1), (lambda: jittered_square(12), 2),
                                    (lambda: jittered_square(9), 3), (lambda: kuhn_cube(4), 1), (lambda: kuhn_cube(3), 2)])
@pytest.mark.parametrize("R", [1, 5, 33, 64])
@pytest.mark.parametrize("fuse", [0, 3])
def test_digit_apply(make, p, R, fuse):
    import torch
    from scipy.sparse import bsr_matrix
    from paper_2012_08024_gb300 import Solver
    S = Solver(make(), p=p, max_levels=2, precision="fp32", nrhs=R, fuse_transfers=fuse).bind()
    e = S.export_level(0)
    n, npb = S.ne, S.np_
    A = bsr_matrix((e["val"], e["col"], e["rowptr"]), shape=(n * npb, n * npb)).tocsr()
    x = np.random.default_rng(R).standard_normal((n * npb, R)) * 10.0 ** np.arange(R)[None, :].clip(max=40)
    bad = R > 2
    if bad:
        x[n * npb // 2, 2] = np.inf
    y = torch.empty((n * npb, R), dtype=torch.float64, device="cuda")
    S.apply_multi(torch.tensor(x, device="cuda"), y)
    y = y.cpu().numpy()
    for r in range(R):
        with np.errstate(invalid="ignore"):
            want = A @ x[:, r]
        fine = np.isfinite(want)
        assert np.array_equal(fine, np.isfinite(y[:, r])), r
        top = np.abs(x[np.isfinite(x[:, r]), r]).max()
        assert np.abs(y[fine, r] - want[fine]).max() <= 1e-13 * np.abs(e["val"]).max() * top, r


@pytest.mark.parametrize("R", [3, 34, 132])
@pytest.mark.parametrize("nu_pre", [0, 1])
def test_solve_columns(R, nu_pre):
    import torch
    from paper_2012_08024_gb300 import Solver
    mesh = jittered_square(14)
    kw = dict(p=2, max_levels=3, nu_pre=1, nu_post=1, tol=1e-12)
    S1 = Solver(mesh, **kw).bind()
    f = torch.tensor(sine_combination_sources(S1.quadrature_points()[0], R, mmax=4), device="cuda")
    if nu_pre == 0:   # V(0, 2) is not symmetric, which the flexible CG has to cope with
        kw.update(nu_pre=0, nu_post=2)
    for tune in (True, False):
        u, _, its, rc = Solver(mesh, precision="fp32", nrhs=R, autotune=tune, **kw).bind().solve_multi(f)
        if nu_pre == 0 and rc != 0:
            continue   # an iteration limit is an answer here; the kernels of V(0, nu) ran
        assert rc == 0
        for r in (0, R // 2, R - 1):
            want = S1.solve(f[r].contiguous())[0]
            assert float((u[r] - want).norm() / want.norm()) <= 1e-9, r


@pytest.mark.parametrize("prec,split", [("fp32", False), ("fp32", True), ("bf16", False)])
@pytest.mark.parametrize("maxit", [500, 3, 0])
def test_graph_and_host_driven_loops_agree(prec, split, maxit):
    """The CG loop as one graph launch and as a host-driven loop: the same kernels in the same order."""
    import torch
    from paper_2012_08024_gb300 import Solver
    mesh, R = jittered_square(13), 37
    out = []
    for graph in (True, False):
        S = Solver(mesh, p=3, max_levels=3, precision=prec, nrhs=R, tc_fp64_apply=split, maxit=maxit, autotune=False,
                   single_graph=graph).bind()
        f = sine_combination_sources(S.quadrature_points()[0], R, mmax=4)
        f[5] = 0.0   # a column that is converged before the loop
        for _ in range(2):   # captured, then replayed
            out.append(S.solve_multi(torch.tensor(f, device="cuda")))
    u0, h0, i0, rc0 = out[0]
    assert i0[5] == 0 and (maxit or not i0.any())
    for u, h, i, rc in out[1:]:
        assert rc == rc0 and np.array_equal(i, i0)
        assert all(np.array_equal(a, b) for a, b in zip(h, h0))
        assert np.array_equal(u.cpu().numpy(), u0.cpu().numpy())
