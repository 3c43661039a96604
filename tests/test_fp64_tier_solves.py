"""The FP64 tier's triangular solves with inverted 64 x 64 diagonal blocks, at
block edges and ragged ends, against numpy.  Each solve's backward error is at
most (m + 2 64) u cond(L_bb) in norm (the product with an inverse whose own
error is 64 u cond), the factor's m u, and cond(L_bb)^2 <= cond(M): the
solution is within 3 (m + 200) u cond(M)^1.5."""
import numpy as np
import pytest
import torch

import lpgen

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("tc", [0, 1])
@pytest.mark.parametrize("m", [2, 63, 64, 65, 130, 511, 1030])
def test_inverted_block_solves(m, tc):
    import paper_1502_03543_gb300 as P
    rng = np.random.default_rng(m)
    lp = lpgen.generate(m, 2 * m + 1, seed=3, storage="f32")
    G = rng.standard_normal((m, 2 * m + 3))
    M = G @ G.T / (2 * m + 3) + np.eye(m)
    M = M * np.outer(d := 2.0 ** rng.integers(-8, 9, m), d)  # (an exact scaling: the bound holds for the scaled system)
    b = rng.standard_normal(m) * d
    with P.Solver(m, 2 * m + 1, "fp32_ir", torch.float32, dspread_refactor=1e-300, fp64_tier_tc=tc) as S:
        info = S.direction(gpu(lp.A64.astype(np.float32)), gpu(lp.x0), gpu(lp.s0))[3]
        assert info["used_fp64"] == 1
        S.load_matrix(gpu(M))
        S.factor()
        x = S.factor_solve(gpu(b)).cpu().numpy()
        y = S.factor_solve(gpu(b)).cpu().numpy()
    assert np.array_equal(x, y)
    Ms = M / np.outer(d, d)
    ref = np.linalg.solve(Ms, b / d)
    tol = 3 * (m + 200) * U * np.linalg.cond(Ms) ** 1.5
    # (the double-float factor, without fp64_tier_tc or up to m = 256, has 46 bits)
    tol *= 2.0 ** 7 if tc == 0 or m <= 256 else 1.0
    assert np.linalg.norm(x * d - ref) <= tol * np.linalg.norm(ref)
