"""The fused passes over A and the clustered triangular solves at the sizes
where their cut changes: one and several row chunks of A'u, chunks at the cap of
512 rows, ragged column blocks, rows that are not 16-byte aligned; solves of one
cluster of 8 blocks, of a cluster and one block, and ragged last blocks.
Bounds as in test_gpu_parity.py."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

U64, U32 = 2.0 ** -53, 2.0 ** -24
DT = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}


def gamma(n, u):
    return n * u / (1 - n * u)


@pytest.mark.parametrize("form", ["fp64", "fp32_ir"])
@pytest.mark.parametrize("dt", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("m,n", [(31, 33), (257, 264), (600, 6000), (1100, 20001), (5000, 5008)])
def test_passes(m, n, dt, form):
    import paper_1502_03543_gb300 as P
    g = torch.Generator(device="cuda").manual_seed(m + n)
    A = torch.randn(m, n, device="cuda", generator=g, dtype=torch.float32).to(DT[dt])
    v = torch.randn(n, device="cuda", generator=g, dtype=torch.float64)
    u = torch.randn(m, device="cuda", generator=g, dtype=torch.float64)
    with P.Solver(m, n, form, DT[dt]) as S:
        for _ in range(2):  # the second call finds the tickets as the first left them
            r, w = S.gemv(A, v), S.gemv_t(A, u)
    Ad = A.double()
    mr, mw = Ad.abs() @ v.abs(), Ad.abs().T @ u.abs()
    extra = 2.0 ** -41 if form != "fp64" and dt != "f64" else 0.0
    # (the reference is torch's FP64 product: as accurate as the pass, so twice the bound)
    assert bool(((r - Ad @ v).abs() <= (extra + 2 * gamma(n, U64)) * mr + 1e-300).all())
    assert bool(((w - Ad.T @ u).abs() <= (extra + 2 * gamma(m, U64)) * mw + 1e-300).all())


@pytest.mark.parametrize("m", [128, 129, 1024, 1025, 1300, 2176])
def test_clustered_solves(m):
    import paper_1502_03543_gb300 as P
    rng = np.random.default_rng(m)
    G = rng.standard_normal((m, m + 50))
    M = G @ G.T / m + np.eye(m)
    rhs = rng.standard_normal(m)
    with P.Solver(m, m + 1, "fp32_ir", torch.float32) as S:
        S.load_matrix(torch.from_numpy(M).cuda())
        S.factor()
        L = np.tril(S.copy_matrix().cpu().numpy().astype(np.float64))
        x = [S.factor_solve(torch.from_numpy(rhs).cuda()).cpu().numpy() for _ in range(3)]
    assert np.array_equal(x[0], x[1]) and np.array_equal(x[0], x[2])
    xo = oracle.backward(L, oracle.forward(L, rhs))
    assert np.linalg.norm(x[0] - xo) <= 2 * np.linalg.cond(L) ** 2 * gamma(m, U32) * np.linalg.norm(xo)
