"""FP64 products in integer digits, row by row, where the blocks of a row or the values that meet them
differ in size by many orders: contrasts of kappa, vectors that jump between elements.

Bound of a scalar row (NumPy's long double is the exact reference: 64 bits and more): within one block an
entry a of A is off by at most 2^-58 M, M the largest |a| of its scalar row in the block (2^-59 of the power
of two above it), and a value of x by at most 2^-58 X, X the largest |x| of the neighbour; so the n_p products of
the block by 2^-57 n_p M X; what the blocks' sums lose when they are added is below 2^-90 of that, and the
result is rounded once.  Levels of many rows at n_p = 3 and 4 hold FP64 blocks: T fused multiply-adds in a row
are off by at most T 2^-53 sum |a| |x| to first order."""
import numpy as np
import pytest

from synthetic import jittered_square, kuhn_cube

pytestmark = pytest.mark.gpu

# more than 4,864 rows on level 0 (2,432 above n_p = 10): packed there, a warp per row below
CASES = [(lambda: jittered_square(50), 1, {}), (lambda: jittered_square(50), 2, {}), (lambda: jittered_square(50), 3, {}),
         (lambda: jittered_square(36), 4, {}), (lambda: jittered_square(9), 6, {}), (lambda: kuhn_cube(10), 1, {}),
         (lambda: kuhn_cube(10), 2, dict(coarsen="primal")), (lambda: kuhn_cube(5), 3, dict(coarsen="primal"))]


def contrast(mesh, seed=0):
    return 10.0 ** np.random.default_rng(seed).integers(-4, 5, len(mesh.elem))


def vectors(rng, n, npb):
    base = rng.standard_normal((n, npb))
    yield base
    yield base * 10.0 ** rng.integers(0, 13, (n, 1)).astype(float)
    yield base * 10.0 ** rng.integers(-120, 121, (n, 1)).astype(float)
    yield base * 10.0 ** -np.arange(npb)   # the higher modes of smooth functions are small


def exact_rows(e, x):
    """A x of the exported blocks in long double, its error bound in digits, sum |a| |x|."""
    npb = x.shape[1]
    xs = x[e["col"]]
    sums = lambda t: np.add.reduceat(t, np.asarray(e["rowptr"][:-1]), axis=0)   # no row is empty
    y = sums(np.einsum("bij,bj->bi", e["val"].astype(np.longdouble), xs.astype(np.longdouble)))
    bound = sums(2.0 ** -57 * npb * np.abs(e["val"]).max(2) * np.abs(xs).max(1)[:, None])
    return y, bound + 1.001 * 2.0 ** -53 * np.abs(y).astype(float), sums(np.einsum("bij,bj->bi", np.abs(e["val"]), np.abs(xs)))


@pytest.mark.parametrize("k", range(len(CASES)))
@pytest.mark.parametrize("kappa", [False, True])
def test_rows_of_the_operators(k, kappa):
    import torch
    from paper_2012_08024_gb300 import Solver
    make, p, kw = CASES[k]
    mesh = make()
    S = Solver(mesh, p=p, max_levels=4, kappa=contrast(mesh) if kappa else None, **kw).bind()
    rng = np.random.default_rng(k)
    for level in range(S.n_levels):
        e = S.export_level(level)
        n, npb = S.info["n_l"][level], S.np_
        for v, x in enumerate(vectors(rng, n, npb)):
            y = torch.empty(n * npb, dtype=torch.float64, device="cuda")
            S.apply(level, torch.tensor(x.reshape(-1), device="cuda"), y)
            want, bound, size = exact_rows(e, x)
            off = np.abs(y.cpu().numpy().reshape(n, npb) - want).astype(float)
            if npb < 6 and n > 4864:
                bound = (npb * np.diff(e["rowptr"])[:, None] + 1) * 2.0 ** -53 * size
            assert np.all(off <= bound), (level, v, (off / bound).max())


@pytest.mark.parametrize("make,p", [(lambda: jittered_square(17), 1), (lambda: jittered_square(12), 2),
                                    (lambda: jittered_square(9), 3), (lambda: kuhn_cube(4), 1), (lambda: kuhn_cube(3), 2)])
@pytest.mark.parametrize("R", [4, 37])
def test_rows_of_the_many_column_apply(make, p, R):
    import torch
    from paper_2012_08024_gb300 import Solver
    mesh = make()
    S = Solver(mesh, p=p, max_levels=2, precision="fp32", nrhs=R, kappa=contrast(mesh)).bind()
    e = S.export_level(0)
    rng = np.random.default_rng(R)
    cols = [v for _ in range((R + 3) // 4) for v in vectors(rng, S.ne, S.np_)][:R]
    x = np.stack(cols, axis=-1)
    y = torch.empty((S.ne * S.np_, R), dtype=torch.float64, device="cuda")
    S.apply_multi(torch.tensor(x.reshape(-1, R), device="cuda"), y)
    y = y.cpu().numpy().reshape(S.ne, S.np_, R)
    for r in range(R):
        want, bound, size = exact_rows(e, x[..., r])
        off = np.abs(y[..., r] - want).astype(float)
        assert np.all(off <= bound), (r, (off / bound).max())


@pytest.mark.parametrize("kw", [dict(fuse_transfers=1), dict(), dict(precision="fp32"), dict(persistent_vcycle=True)])
def test_solve_with_a_contrast_of_kappa(kw):
    """The recurrence ends at 1e-10; the true residual differs from it by rounding, which FP64 bounds by some
    (iterations) 2^-53 || |A| |u| ||; kappa from 1e-2 to 1e2 at random (with FP64 blocks, fuse_transfers = 1,
    683 iterations; from 1e-4 to 1e4 no form converges in 2,000)."""
    import torch
    from paper_2012_08024_gb300 import Solver
    mesh = jittered_square(40)
    kappa = 10.0 ** np.random.default_rng(0).integers(-2, 3, len(mesh.elem))
    S = Solver(mesh, p=2, max_levels=4, kappa=kappa, maxit=2000, coarsen="primal", **kw).bind()
    e = S.export_level(0)
    n, npb = S.ne, S.np_
    b = np.random.default_rng(2).standard_normal((n, npb))
    u, hist, it, rc = S.solve_b(torch.tensor(b, device="cuda"))
    assert rc == 0
    u = u.cpu().numpy()[e["perm"]]
    want, _, size = exact_rows(e, u)
    off = np.linalg.norm((b[e["perm"]] - want).astype(float))
    assert off <= 1e-10 * np.linalg.norm(b) + it * 2.0 ** -53 * np.linalg.norm(size)
