"""The meshes of a batched handle are independent whatever the scales of their data: operations and
solves of one mesh do not depend on what another mesh holds.

The meshes' element counts are no multiples of the block rows that a warp takes (10, 5 and 3 at
n_p = 3, 6 and 10) and exceed the 4,864 rows up to which a row has a warp of its own, so that warps
hold rows of two meshes.  Operations: every step is linear and scaling by a power of two is exact
(no overflow, no subnormal values), so results have to agree bit for bit.  Solves: as in the tests of
batches of one scale, 1e-10 between a mesh and its own single solve; the true residual is within the
tolerance and the gap between it and the recurrence (well below 1e-10 at 1e-10)."""
import numpy as np
import pytest

from synthetic import jittered_square, sin_source
from tests.gpu_common import rel

pytestmark = pytest.mark.gpu

SIZES = (41, 42)


def _batch(p, sizes=SIZES, **kw):
    from paper_2012_08024_gb300 import BatchSolver
    return BatchSolver([jittered_square(n, seed=k) for k, n in enumerate(sizes)], p=p, max_levels=4, **kw).bind()


@pytest.mark.parametrize("p", [1, 2, 3])
@pytest.mark.parametrize("kw", [dict(), dict(persistent_vcycle=True), dict(nu_pre=0, nu_post=2), dict(precision="fp32")])
@pytest.mark.parametrize("exponent", [100, -100, None])
def test_operations_of_a_mesh_do_not_see_its_neighbours(p, kw, exponent):
    import torch
    if kw.get("precision") == "fp32" and exponent:
        exponent //= 4   # inside the range of the FP32 V-cycle
    scale = 0.0 if exponent is None else 2.0 ** exponent   # of the first mesh
    B = _batch(p, **kw)
    cut, n = int(B.elem_offsets[1]) * B.np_, B.info["n_dofs"]
    rng = np.random.default_rng(p)
    x, b = rng.standard_normal((2, n))
    ops = [lambda x, b, y: B.apply(0, x, y), lambda x, b, y: B.residual(0, x, b, y), lambda x, b, y: B.vcycle(b, y)]
    if kw.get("precision") != "fp32":
        ops.append(lambda x, b, y: B.smooth(0, x, b, y))
    for k, op in enumerate(ops):
        y = []
        for s in (1.0, scale):
            xs, bs = x.copy(), b.copy()
            xs[:cut] *= s
            bs[:cut] *= s
            out = torch.empty(n, dtype=torch.float64, device="cuda")
            op(torch.tensor(xs, device="cuda"), torch.tensor(bs, device="cuda"), out)
            y.append(out.cpu().numpy())
        assert np.array_equal(y[1][cut:], y[0][cut:]), k
        assert np.array_equal(y[1][:cut], scale * y[0][:cut]), k


@pytest.mark.parametrize("kw", [dict(), dict(precision="fp32"), dict(persistent_vcycle=True)])
def test_solves_of_meshes_of_different_scale(kw):
    import torch
    from scipy.sparse import bsr_matrix
    from paper_2012_08024_gb300 import Solver
    sizes, scales = (41, 42, 43, 39), (1.0, 1e10, 1e-10, 1e18)
    B = _batch(2, sizes, **kw)
    f = sin_source(B.quadrature_points()[0])
    for m, s in enumerate(scales):
        f[B.elem_offsets[m]:B.elem_offsets[m + 1]] *= s
    u, hists, its, rc = B.solve(torch.tensor(f, device="cuda"))
    assert rc == 0
    for m, n in enumerate(sizes):
        S = Solver(jittered_square(n, seed=m), p=2, max_levels=4, **kw).bind()
        fm = torch.tensor(f[B.elem_offsets[m]:B.elem_offsets[m + 1]], device="cuda")
        um = u[B.elem_offsets[m]:B.elem_offsets[m + 1]].contiguous()
        us, _, it, rcs = S.solve(fm)
        assert rcs == 0 and abs(int(its[m]) - it) <= 1, m
        assert rel(um.cpu().numpy(), us.cpu().numpy()) <= 1e-10, m
        e = S.export_level(0)
        A = bsr_matrix((e["val"], e["col"], e["rowptr"]), shape=(S.info["n_dofs"],) * 2).tocsr()
        b, x = torch.empty(S.info["n_dofs"], dtype=torch.float64, device="cuda"), fm.new_empty(S.info["n_dofs"])
        S.to_tree(S.rhs(fm).reshape(-1), b)
        S.to_tree(um.reshape(-1), x)
        b, x = b.cpu().numpy(), x.cpu().numpy()
        assert np.linalg.norm(b - A @ x) <= 2e-10 * np.linalg.norm(b), m


@pytest.mark.parametrize("p", [1, 2])
@pytest.mark.parametrize("scale", [2.0 ** 100, 2.0 ** -100, 0.0])
def test_persistent_cycle_on_fp64_blocks(p, scale):
    """More than 20,000 elements: the persistent kernel on FP64 blocks."""
    import torch
    B = _batch(p, (105, 106), persistent_vcycle=True)
    cut, n = int(B.elem_offsets[1]) * B.np_, B.info["n_dofs"]
    r = np.random.default_rng(p).standard_normal(n)
    z = []
    for s in (1.0, scale):
        rs = r.copy()
        rs[:cut] *= s
        out = torch.empty(n, dtype=torch.float64, device="cuda")
        B.vcycle(torch.tensor(rs, device="cuda"), out)
        z.append(out.cpu().numpy())
    assert np.array_equal(z[1][cut:], z[0][cut:])
    assert np.array_equal(z[1][:cut], scale * z[0][:cut])
