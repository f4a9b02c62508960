"""persistent_vcycle and fuse_transfers together: the persistent kernel runs (it fuses no transfers), as it
does without the second option."""
import numpy as np
import pytest

from synthetic import jittered_square, kuhn_cube, sin_source

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fuse", [1, 2, 3])
@pytest.mark.parametrize("precision,p", [("fp64", 1), ("fp64", 3), ("fp32", 2)])
def test_persistent_kernel_runs(fuse, precision, p):
    import torch
    from paper_2012_08024_gb300 import CdgError, Solver
    mesh = jittered_square(20)
    kw = dict(p=p, max_levels=3, persistent_vcycle=True, precision=precision)
    S, S0 = Solver(mesh, fuse_transfers=fuse, **kw).bind(), Solver(mesh, **kw).bind()
    f = torch.tensor(sin_source(S.quadrature_points()[0]), device="cuda")
    S.set_wait_limit(0)   # only the persistent kernel has a wait to give up
    with pytest.raises(CdgError) as e:
        S.solve(f)
    assert e.value.code == 6 and "grid barrier" in str(e.value)
    S.set_wait_limit(-1)
    r = torch.tensor(np.random.default_rng(p).standard_normal(S.info["n_dofs"]), device="cuda")
    z, z0 = torch.empty_like(r), torch.empty_like(r)
    S.vcycle(r, z)
    S0.vcycle(r, z0)
    assert torch.equal(z, z0)
    u, _, it, rc = S.solve(f)
    u0, _, it0, rc0 = S0.solve(f)
    assert rc == rc0 == 0 and it == it0 and float((u - u0).norm() / u0.norm()) <= 1e-12


@pytest.mark.parametrize("kw", [dict(p=4), dict(p=3, pmg=True)])
def test_per_phase_kernels_where_the_persistent_one_does_not_apply(kw):
    import torch
    from paper_2012_08024_gb300 import Solver
    mesh = jittered_square(12)
    out = []
    for more in (dict(), dict(persistent_vcycle=True)):
        S = Solver(mesh, max_levels=3, fuse_transfers=3, **kw, **more).bind()
        out.append(S.solve(torch.tensor(sin_source(S.quadrature_points()[0]), device="cuda")))
    assert out[0][3] == out[1][3] == 0 and out[0][2] == out[1][2] and torch.equal(out[0][0], out[1][0])


@pytest.mark.parametrize("make,p,kw", [(lambda: jittered_square(104), 1, {}), (lambda: jittered_square(104), 2, {}),
                                       (lambda: jittered_square(96), 2, {}),
                                       (lambda: kuhn_cube(15), 1, dict(coarsen="primal"))])
def test_persistent_kernel_on_fp64_blocks_and_in_digits(make, p, kw):
    """Below n_p = 10 the persistent kernel keeps FP64 blocks above 20,000 elements, digits up to there.  Its
    V-cycle agrees with that of the per-phase kernels to 1e-9, as the V-cycle with the oracle's."""
    import torch
    from paper_2012_08024_gb300 import Solver
    mesh = make()
    kw = dict(p=p, max_levels=5, nu_pre=2, nu_post=2, **kw)
    S, S0 = Solver(mesh, persistent_vcycle=True, **kw).bind(), Solver(mesh, **kw).bind()
    digits = S.info["device_bytes"] == S0.info["device_bytes"]
    assert digits == (len(mesh.elem) <= 20000)
    r = torch.tensor(np.random.default_rng(p).standard_normal(S.info["n_dofs"]), device="cuda")
    z, z0 = torch.empty_like(r), torch.empty_like(r)
    S.vcycle(r, z)
    S0.vcycle(r, z0)
    assert float((z - z0).norm() / z0.norm()) <= (1e-14 if digits else 1e-9)
    f = torch.tensor(sin_source(S.quadrature_points()[0]), device="cuda")
    u, _, it, rc = S.solve(f)
    u0, _, it0, rc0 = S0.solve(f)
    assert rc == rc0 == 0 and abs(it - it0) <= 1 and float((u - u0).norm() / u0.norm()) <= 1e-9
