"""pdas_factor on the plain FP64 form accepts what the SIMT factor accepts: a
pivot that the tensor-core factor finds not positive is confirmed by the SIMT
factor on the matrix as it was loaded, with its index; and a call that was done
over leaves nothing behind for the next one."""
import numpy as np
import pytest
import torch

import lpgen

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("m", [40, 200, 333])
def test_matrices_at_the_edge(m):
    """The last row of G depends on the others but for a part whose square is
    near the rounding of M = G G'."""
    import paper_1502_03543_gb300 as P
    both = 0
    with P.Solver(m, m + 1, "fp64") as S, P.Solver(m, m + 1, "fp64", fp64_tier_tc=0) as T:
        for seed in range(60):
            rng = np.random.default_rng(seed)
            G = rng.standard_normal((m, m + 20))
            G[m - 1] = G[: m - 1].T @ rng.standard_normal(m - 1) / np.sqrt(m) + 2.0 ** rng.uniform(
                -27, -22) * rng.standard_normal(m + 20)
            M = np.tril(G @ G.T)
            M += np.tril(M, -1).T
            T.load_matrix(gpu(M))
            simt = T.factor(raise_on_error=False)
            S.load_matrix(gpu(M))
            st = S.factor(raise_on_error=False)
            assert st in (0, -3) and (st == 0 or (simt == -3 and S.last_error_index() == T.last_error_index())), seed
            if st == 0:
                L = np.tril(S.copy_matrix().cpu().numpy())
                d = np.sqrt(M.diagonal())
                assert np.tril(np.abs(L @ L.T - M) / np.outer(d, d)).max() <= 2 * (m + 1) * U, seed
            both += st == simt == 0
    assert both >= 20


def test_a_call_done_over_leaves_nothing_behind():
    import paper_1502_03543_gb300 as P
    m, n = 300, 700
    lp = lpgen.generate(m, n, seed=4)
    A, x, s = gpu(lp.A64), gpu(lp.x0), gpu(lp.s0)
    bad = A.clone()
    bad[170] = 0.0
    G = np.random.default_rng(1).standard_normal((m, m + 9))
    M = gpu(G @ G.T)
    with P.Solver(m, n, "fp64") as S:
        def factored():
            S.load_matrix(M)
            S.factor()
            return S.copy_matrix().tril()
        L = factored()
        with pytest.raises(P.PdasError):
            S.direction(bad, x, s)
        assert torch.equal(factored(), L)
        S.load_matrix(gpu(-np.eye(m)))
        assert S.factor(raise_on_error=False) == -3 and S.last_error_index() == 0
        assert torch.equal(factored(), L)
