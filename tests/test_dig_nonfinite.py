"""An infinity or a NaN below the diagonal fails the factor with digit-plane
updates at that row's pivot, as it fails the SIMT factor: in the first panel, in
a later one, next to a panel's edge and in the last row; plain FP64 form and the
FP64 tier of the mixed forms."""
import numpy as np
import pytest
import torch

import lpgen

pytestmark = pytest.mark.gpu


def gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("form", ["fp64", "fp32_ir"])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("p,q", [(64, 0), (150, 3), (150, 70), (128, 127), (299, 255), (299, 20)])
def test_off_diagonal(form, value, p, q):
    import paper_1502_03543_gb300 as P
    m, n = 300, 640
    rng = np.random.default_rng(p)
    G = rng.standard_normal((m, 2 * m))
    M = G @ G.T
    M[p, q] = M[q, p] = value
    opts = {} if form == "fp64" else dict(dspread_refactor=1e-300)
    with P.Solver(m, n, form, torch.float64, **opts) as S:
        if form != "fp64":  # into the FP64 tier first
            lp = lpgen.generate(m, n, seed=1)
            info = S.direction(gpu(lp.A64), gpu(lp.x0), gpu(lp.s0))[3]
            assert info["factor_form"] == 4
        S.load_matrix(gpu(M))
        assert S.factor(raise_on_error=False) == -3
        assert S.last_error_index() == p
        M[p, q] = M[q, p] = 0.0
        S.load_matrix(gpu(M))
        assert S.factor(raise_on_error=False) == 0
