"""The FP32 tile factor where its fast 8 x 8 pivot blocks hand over to the
full-range ones: pivots that are subnormal, or so large that their reciprocal
is; and panel edges.  Bound: the backward error of an FP32 factorisation plus
the rounding of subnormal results."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [2.0 ** 127, 2.0 ** -127, 1.0])
@pytest.mark.parametrize("m", [1, 8, 33, 100, 128])
def test_pivot_range(m, scale):
    import paper_1502_03543_gb300 as P
    G = np.random.default_rng(m).standard_normal((m, 2 * m + 4))
    M = G @ G.T
    M = (M / M.diagonal().max() * scale).astype(np.float32).astype(np.float64)
    with P.Solver(m, m + 1, "fp32_ir", torch.float32) as S:
        S.load_matrix(torch.from_numpy(M).cuda())
        S.factor()
        L = np.tril(S.copy_matrix().cpu().numpy().astype(np.float64))
    assert np.abs(L @ L.T - M).max() <= 4 * m * 2.0 ** -24 * np.abs(M).max() + 8 * m * 2.0 ** -149


@pytest.mark.parametrize("m,bad", [(40, 7), (40, 8), (128, 127), (300, 128), (300, 160), (300, 299)])
def test_failed_pivot_index(m, bad):
    import paper_1502_03543_gb300 as P
    M = np.eye(m)
    M[bad, bad] = -1.0
    with P.Solver(m, m + 1, "fp32_ir", torch.float32) as S:
        S.load_matrix(torch.from_numpy(M).cuda())
        assert S.factor(raise_on_error=False) == -3 and S.last_error_index() == bad
