"""The FP32 apply on levels of every size (few rows: a warp per block row, its blocks shared by the
groups of the warp; many rows: packed) against FP64 products of the exported operators.

Tolerance, per entry: T products of FP32-rounded A with FP32 x, summed in FP32 in any order, are off by
at most (T + 2) 2^-24 (|A| |x|) to first order; T is the longest row's number of terms."""
import numpy as np
import pytest

from synthetic import jittered_square, kuhn_cube

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make,p,kw", [
    (lambda: jittered_square(110), 1, {}), (lambda: jittered_square(60), 2, {}), (lambda: jittered_square(50), 3, {}),
    (lambda: jittered_square(12), 4, {}), (lambda: jittered_square(7), 5, {}),
    (lambda: kuhn_cube(9), 1, {}), (lambda: kuhn_cube(8), 2, dict(pmg=True))])
def test_fp32_apply_on_every_level(make, p, kw):
    import torch
    from scipy.sparse import bsr_matrix
    from paper_2012_08024_gb300 import Solver
    S = Solver(make(), p=p, max_levels=4, precision="fp32", **kw).bind()
    rng = np.random.default_rng(p)
    for level in range(S.n_levels - 1):
        e = S.export_level(level)
        n, npb = S.info["n_l"][level], S.info["np_l"][level]
        A = bsr_matrix((e["val"], e["col"], e["rowptr"]), shape=(n * npb, n * npb)).tocsr()
        x = rng.standard_normal(n * npb).astype(np.float32)
        y = torch.empty(n * npb, dtype=torch.float32, device="cuda")
        S.apply_f32(level, torch.tensor(x, device="cuda"), y)
        terms = int(np.diff(e["rowptr"]).max()) * npb
        bound = (terms + 2) * 2.0 ** -24 * (abs(A) @ np.abs(x.astype(np.float64)))
        assert np.all(np.abs(y.cpu().numpy() - A @ x.astype(np.float64)) <= bound), level
