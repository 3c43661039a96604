"""Where the refinement's conjugate gradients stop early (a step length that is
not positive and finite), the direction it returns is one direction: A'dy + ds =
0 to the rounding of the FP64 pass.  The steps are driven there by scaling x and
s by powers of two (D, and so M and its factor, stay the same): r, and with it
rho'P^-1 rho and p'M p, slide through the subnormal range to zero within a few
steps.  The tolerances are out of reach, so that nothing but the step itself ends the
refinement; the last rows of A are nearly dependent, so that each step moves dy
by far more than the bound."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.mark.parametrize("m", [96, 300])  # the double-float and the digit factor of the FP64 tier
@pytest.mark.parametrize("first", range(440, 512, 12))
def test_direction_is_consistent(m, first):
    import paper_1502_03543_gb300 as P
    n = 2 * m + 8
    rng = np.random.default_rng(m)
    A = rng.standard_normal((m, n)).astype(np.float32)
    for r in (m - 1, m - 2):
        A[r] = A[r - 2] + np.float32(2.0 ** -14) * A[r]
    x, s = rng.uniform(0.5, 1.5, n), rng.uniform(0.5, 1.5, n)
    dev = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()
    Ad, A64 = dev(A), dev(A.astype(np.float64))
    with P.Solver(m, n, "fp32_ir", torch.float32, dspread_refactor=1e-300, refine_tol=1e-300, refine_be=0.0) as S:
        for k in range(first, first + 12):
            dx, dy, ds, info = S.direction(Ad, dev(x * 2.0 ** -k), dev(s * 2.0 ** -k))
            assert info["used_fp64"] == 1
            assert bool(torch.isfinite(dy).all()), k
            # (dy / 2^-k is of order one: scaled back, nothing of the check itself is subnormal)
            dy, ds = dy * 2.0 ** k, ds * 2.0 ** k
            bound = 2 * m * U / (1 - m * U) * (A64.abs().T @ dy.abs())
            assert bool(((A64.T @ dy + ds).abs() <= bound + 1e-290).all()), (k, info["refine_sweeps"])
