"""FP64 block products in integer digits (device_fixed.cu) against FP64 products of the
exported operators: every level of hierarchies whose levels take both the packed and the
row-per-warp mapping, all block sizes, rows of one step and of several, vectors whose
magnitude jumps between elements, subnormal values, infinities and NaN.

Tolerance: an entry of A is kept to 2^-59 of its row's bound and a value of x to 2^-59 of
the largest the warp gathers, so a row of T terms is off by at most 2 T 2^-58 (row bound)
(gathered maximum); with at most 60 blocks of n_p terms per row that is below 1e-14 times
the product of the largest entry and the largest value.  FP64 summation on the reference's
side adds T eps of the same product."""
import numpy as np
import pytest

from synthetic import jittered_square, kuhn_cube

pytestmark = pytest.mark.gpu

CASES = [(lambda: jittered_square(60), 1, {}), (lambda: jittered_square(72), 2, {}), (lambda: jittered_square(40), 3, {}),
         (lambda: jittered_square(14), 4, {}), (lambda: jittered_square(9), 6, {}), (lambda: kuhn_cube(9), 1, {}),
         (lambda: kuhn_cube(10), 2, dict(coarsen="primal")), (lambda: kuhn_cube(5), 3, dict(coarsen="primal"))]


def product(e, x, npb):
    from scipy.sparse import bsr_matrix
    n = len(e["perm"])
    A = bsr_matrix((e["val"], e["col"], e["rowptr"]), shape=(n * npb, n * npb))
    A.sort_indices()
    return A.tocsr() @ x


def vectors(rng, n, npb):
    base = rng.standard_normal(n * npb)
    yield base
    yield base * np.repeat(10.0 ** rng.integers(-200, 200, n).astype(float), npb)   # from element to element
    yield np.zeros(n * npb)
    yield base * 1e-310                                                          # subnormal


@pytest.mark.parametrize("k", range(len(CASES)))
def test_level_products(k):
    import torch
    from paper_2012_08024_gb300 import Solver
    make, p, kw = CASES[k]
    S = Solver(make(), p=p, max_levels=4, **kw).bind()
    rng = np.random.default_rng(k)
    for level in range(S.n_levels):
        e = S.export_level(level)
        n, npb = S.info["n_l"][level], S.np_
        big = np.abs(e["val"]).max()
        for x in vectors(rng, n, npb):
            y = torch.empty(n * npb, dtype=torch.float64, device="cuda")
            S.apply(level, torch.tensor(x, device="cuda"), y)
            diff = np.abs(y.cpu().numpy() - product(e, x, npb))
            # the maximum over the whole vector bounds what a warp gathers
            assert diff.max() <= 1e-13 * big * np.abs(x).max() + 1e-318, (level, diff.max())


@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_non_finite_values_spread_like_ieee(bad):
    import torch
    from paper_2012_08024_gb300 import Solver
    S = Solver(jittered_square(40), p=2, max_levels=3).bind()
    for level in range(S.n_levels):
        e = S.export_level(level)
        n, npb = S.info["n_l"][level], S.np_
        x = np.random.default_rng(3).standard_normal(n * npb)
        x[(n // 2) * npb + 1] = bad
        y = torch.empty(n * npb, dtype=torch.float64, device="cuda")
        S.apply(level, torch.tensor(x, device="cuda"), y)
        y = y.cpu().numpy()
        with np.errstate(invalid="ignore"):
            want = product(e, x, npb)
        assert np.array_equal(np.isfinite(y), np.isfinite(want))
        fine = np.isfinite(want)
        assert np.allclose(y[fine], want[fine], rtol=0, atol=1e-13 * np.abs(e["val"]).max() * 10)
