"""The error of the plain FP64 form's factors on matrices whose panel rows are
strongly graded, in opposite directions from row to row.  A row of a panel is held
to 2^-56 of its largest entry's binade by the digit planes, so the tensor-core
factor has no elementwise bound gamma |L||L'| (two rows (1, 1e-10) and (1e-10, 1)
have a product of 2e-10); what both factors satisfy is the bound that governs the
solve's accuracy after symmetric scaling,
    |L L' - M|_pq <= c u sqrt(M_pp M_qq).
c of the tensor-core factor: 65 for the FP64 factor of a panel; its digits are off
by u/4 of the row's largest entry, so 64 columns by 2 8 u/4 |P_p||P_q|, and what
the products leave out by u/2 max max: 5 over all panels (Cauchy-Schwarz); the
conversion and the subtraction of each of m / 64 updates 2: m / 32 + 71 in all.  The
SIMT factor's is m + 1."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def graded(m, decades, seed):
    rng = np.random.default_rng(seed)
    k = np.arange(m) % 64 / 64.0
    up, down = 10.0 ** (-decades * k), 10.0 ** (-decades * (1 - k))
    L = np.tril(rng.standard_normal((m, m)), -1)
    L[0::2] *= up
    L[1::2] *= down
    L[1:] *= (0.5 / np.linalg.norm(L[1:], axis=1))[:, None]  # a quarter of M_pp: M is safely positive definite
    L[np.arange(m), np.arange(m)] = 1.0
    L *= (10.0 ** rng.uniform(-2, 0, m))[:, None]
    M = L @ L.T
    return np.tril(M) + np.tril(M, -1).T


@pytest.mark.parametrize("decades", [0, 4, 10, 14])
@pytest.mark.parametrize("m", [65, 130, 200])
def test_scaled_backward_error(m, decades):
    import paper_1502_03543_gb300 as P
    M = graded(m, decades, m + decades)
    d = np.sqrt(M.diagonal())
    for tc, c in ((1, m / 32 + 71), (0, m + 1)):
        with P.Solver(m, m + 1, "fp64", fp64_tier_tc=tc) as S:
            S.load_matrix(torch.from_numpy(M).cuda())
            S.factor()
            L = np.tril(S.copy_matrix().cpu().numpy()).astype(np.longdouble)
        E = np.tril(np.abs(np.matmul(L, L.T) - M)) / np.outer(d, d)
        assert E.max() <= c * U, (tc, float(E.max() / U))
