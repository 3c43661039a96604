"""The FP64 normal matrix of an A stored in FP32 or BF16 has the bits of the same
A stored in FP64: the widening is exact, for zeros, subnormals and the largest
values too.  (Its columns hold values of one magnitude, scaled back by D, so that
no sum overflows.)"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("m,n", [(20, 47), (130, 300)])  # 16 x 16 and 32 x 32 tiles
def test_same_bits_as_fp64_storage(m, n, dtype):
    import paper_1502_03543_gb300 as P
    rng = np.random.default_rng(m)
    e = rng.integers(-133, 128, n)  # from below the smallest normal to the largest exponent
    e[:2] = -133, 127
    A64 = rng.uniform(1.0, 2.0, (m, n)) * rng.choice([-1.0, 1.0], (m, n)) * 2.0 ** e
    A64[rng.random((m, n)) < 0.05] = 0.0
    A64[0, :4] = -0.0
    A = torch.from_numpy(A64).cuda().to(dtype)
    A = torch.where(torch.isfinite(A), A, torch.ones_like(A))
    x = torch.from_numpy(rng.uniform(0.5, 1.5, n) * 2.0 ** (-2.0 * e)).cuda()
    s = torch.from_numpy(rng.uniform(0.5, 1.5, n)).cuda()
    M = []
    for a in (A, A.double()):
        with P.Solver(m, n, "fp64", a.dtype) as S:
            S.form_normal(a, x, s)
            M.append(S.copy_matrix().tril())
    assert bool(torch.isfinite(M[0]).all()) and torch.equal(M[0], M[1])
