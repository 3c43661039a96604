"""The plain FP64 form's factor with tensor-core trailing updates: its backward
error beside the SIMT factor's (both are FP64 factorisations, whose error is at
most gamma_{m+1}(u) |L||L'| elementwise), at one panel, panel edges and ragged
tiles; and a matrix that is not positive definite, which goes through both."""
import numpy as np
import pytest
import torch

import lpgen

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("m", [3, 64, 65, 129, 192, 300, 700])
def test_backward_error(m):
    import paper_1502_03543_gb300 as P
    rng = np.random.default_rng(m)
    G = rng.standard_normal((m, 2 * m + 3))
    M = (G * rng.uniform(0.01, 100.0, G.shape[1])) @ G.T
    for tc in (1, 0):
        with P.Solver(m, m + 1, "fp64", fp64_tier_tc=tc) as S:
            S.load_matrix(gpu(M))
            S.factor()
            L = np.tril(S.copy_matrix().cpu().numpy())
        bound = (m + 1) * U / (1 - (m + 1) * U) * (np.abs(L) @ np.abs(L).T)
        # (the library reads the lower triangle; M's two triangles differ by rounding)
        assert np.all(np.tril(np.abs(L @ L.T - M)) <= 2 * bound), tc


def test_not_positive_definite_then_good():
    import paper_1502_03543_gb300 as P
    m, n = 300, 700
    lp = lpgen.generate(m, n, seed=4)
    A, x, s = gpu(lp.A64), gpu(lp.x0), gpu(lp.s0)
    bad = A.clone()
    bad[170] = 0.0  # a zero row: pivot 170 of M is zero
    with P.Solver(m, n, "fp64") as S:
        dy0 = S.direction(A, x, s)[1]
        with pytest.raises(P.PdasError):
            S.direction(bad, x, s)
        assert S.last_error_index() == 170
        dx, dy, ds, info = S.direction(A, x, s)
        assert info["factor_form"] == 4 and torch.equal(dy, dy0)
    with P.Solver(m, n, "fp64", fp64_tier_tc=0) as S:
        dy1, info = S.direction(A, x, s)[1::2]
        assert info["factor_form"] == 3
    assert float((dy1 - dy0).norm()) <= 1e-11 * float(dy1.norm())
