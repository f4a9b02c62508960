"""cdg_restrict and cdg_prolong of FP64 handles run the kernels of the V-cycle, the products with L_K^T and
L_K in integer digits: every row against the bound of those, on levels whose coarse rows share a warp
and on levels whose rows have one each.

Bound, as for the operators' rows: a block with largest entry M in the scalar row and largest value X of the
vector it meets contributes at most 2^-57 n_p M X, and the sum is rounded once (the prolongation's
addition to x once more).  FP64 sums of a row's products do not keep to it; levels of many rows at n_p = 3 hold
FP64 blocks, and their T fused multiply-adds are off by at most T 2^-53 sum |L| |r| to first order."""
import numpy as np
import pytest

from synthetic import jittered_square, kuhn_cube

pytestmark = pytest.mark.gpu

CASES = [(lambda: jittered_square(150), 1, {}), (lambda: jittered_square(150), 2, {}), (lambda: jittered_square(50), 3, {}),
         (lambda: jittered_square(20), 4, {}), (lambda: kuhn_cube(8), 2, dict(coarsen="primal"))]


@pytest.mark.parametrize("k", range(len(CASES)))
def test_rows_of_the_transfers(k):
    import torch
    from paper_2012_08024_gb300 import Solver
    make, p, kw = CASES[k]
    S = Solver(make(), p=p, max_levels=6, **kw).bind()
    rng = np.random.default_rng(k)
    npb = S.np_
    for l in range(S.n_levels - 1):
        e = S.export_level(l)
        n, nc = S.info["n_l"][l], S.info["n_l"][l + 1]
        L, parent = e["L"], e["parent"]
        first = np.searchsorted(parent, np.arange(nc))   # children of an agglomerate are consecutive
        for jumps in (False, True):
            r = rng.standard_normal((n, npb))
            xc, x = rng.standard_normal((nc, npb)), rng.standard_normal((n, npb))
            if jumps:
                r *= 10.0 ** rng.integers(0, 13, (n, 1)).astype(float)
                xc *= 10.0 ** rng.integers(0, 13, (nc, 1)).astype(float)
            ext = np.longdouble
            want = np.add.reduceat(np.einsum("kji,kj->ki", L.astype(ext), r.astype(ext)), first, axis=0)
            bound = np.add.reduceat(2.0 ** -57 * npb * np.abs(L).max(1) * np.abs(r).max(1)[:, None], first, axis=0)
            bc = torch.empty(nc * npb, dtype=torch.float64, device="cuda")
            S.restrict(l, torch.tensor(r.reshape(-1), device="cuda"), bc)
            off = np.abs(bc.cpu().numpy().reshape(nc, npb) - want).astype(float)
            bound = bound + 1.001 * 2.0 ** -53 * np.abs(want).astype(float)
            blocks = npb < 6 and n > 4864   # FP64 blocks
            if blocks:
                terms = npb * np.diff(np.append(first, n))[:, None] + 1
                bound = terms * 2.0 ** -53 * np.add.reduceat(np.einsum("kji,kj->ki", np.abs(L), np.abs(r)), first, axis=0)
            assert np.all(off <= bound), (l, "restrict", (off / bound).max())

            add = np.einsum("kij,kj->ki", L.astype(ext), xc[parent].astype(ext))
            want = x + add
            y = torch.tensor(x.reshape(-1), device="cuda")
            S.prolong(l, torch.tensor(xc.reshape(-1), device="cuda"), y)
            off = np.abs(y.cpu().numpy().reshape(n, npb) - want).astype(float)
            bound = 2.0 ** -57 * npb * np.abs(L).max(2) * np.abs(xc[parent]).max(1)[:, None]
            if blocks:
                bound = (npb + 1) * 2.0 ** -53 * np.einsum("kij,kj->ki", np.abs(L), np.abs(xc[parent]))
            bound = bound + 1.001 * 2.0 ** -53 * (np.abs(add) + np.abs(want)).astype(float)
            assert np.all(off <= bound), (l, "prolong", (off / bound).max())
