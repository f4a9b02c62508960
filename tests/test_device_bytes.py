"""Device memory that a handle asks for (CPU only)."""
import numpy as np
import pytest

from synthetic import jittered_square


@pytest.mark.parametrize("p", [1, 2, 3])
def test_digit_form_holds_the_transfer_blocks_twice(p):
    """An FP64 handle with its operators in digits needs, beside what one with FP64 blocks needs, the blocks of
    the restriction (one n_p x n_p block per element below the coarsest level), 16-bit exponents and
    padded column tables; the FP64 transfer blocks it does not hold."""
    from paper_2012_08024_gb300 import Solver
    mesh = jittered_square(40)
    digits, fp64 = Solver(mesh, p=p, max_levels=4), Solver(mesh, p=p, max_levels=4, fuse_transfers=1)
    more = 0
    for l in range(digits.n_levels):
        n, nnzb, npb = digits.info["n_l"][l], digits.info["nnzb_l"][l], digits.np_
        width = int(np.diff(digits.export_level(l)["rowptr"]).max())
        last = l + 1 == digits.n_levels
        more += 2 * npb * nnzb + 4 * n * width
        if not last:
            more += 8 * n * npb ** 2 + 2 * npb * (nnzb + 3 * n) + 4 * n * width
        more += 256 * 12   # alignment
    assert digits.info["device_bytes"] <= fp64.info["device_bytes"] + more
