"""The SIMT normal matrices (FP64, FP32) where their cut into tiles and K
slices changes: 16 x 16 and 32 x 32 tiles, one slice and many, ragged edges of
both, sizes whose rows are not 16-byte aligned; against the oracle, within the
elementwise bound of the arithmetic (as in test_gpu_parity.py)."""
import numpy as np
import pytest
import torch

import lpgen
import oracle

pytestmark = pytest.mark.gpu


def gamma(n, u):
    return n * u / (1 - n * u)


def formed(m, n, form, storage, dtype):
    import paper_1502_03543_gb300 as P
    lp = lpgen.generate(m, n, seed=m + n, storage=storage)
    rng = np.random.default_rng(m)
    x, s = rng.uniform(0.01, 10, n), rng.uniform(0.01, 10, n)
    dv = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    A = dv(lp.A_store) if storage != "bf16" else dv(lp.A_store.view(np.int16)).view(torch.bfloat16)
    with P.Solver(m, n, form, dtype) as S:
        for _ in range(2):  # the second call finds the tickets as the first left them
            S.form_normal(A, dv(x), dv(s))
        M = S.copy_matrix().cpu().numpy().astype(np.float64)
    D = oracle.scaling(x, s)
    low = np.tril_indices(m)
    return M[low], oracle.normal_matrix(lp.A64, D)[low], ((np.abs(lp.A64) * D) @ np.abs(lp.A64).T)[low]


@pytest.mark.parametrize("storage", ["f64", "bf16"])
@pytest.mark.parametrize("m,n", [(15, 17), (33, 500), (64, 130), (100, 3001), (513, 700), (1570, 1601)])
def test_fp64(m, n, storage):
    M, ref, mag = formed(m, n, "fp64", storage, {"f64": torch.float64, "bf16": torch.bfloat16}[storage])
    assert np.all(np.abs(M - ref) <= 2 * gamma(n + 2, 2.0 ** -53) * mag)


@pytest.mark.parametrize("storage", ["f32", "f64"])
@pytest.mark.parametrize("m,n", [(127, 129), (129, 2000), (300, 5003), (1001, 1030), (2200, 2203)])
def test_fp32(m, n, storage):
    M, ref, mag = formed(m, n, "fp32_ir", storage, {"f32": torch.float32, "f64": torch.float64}[storage])
    assert np.all(np.abs(M - ref) <= 2 * gamma(n + 3, 2.0 ** -24) * mag)
