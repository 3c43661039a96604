"""The operand fl32(A_pk D_k) of the FP32 normal matrix is the FP64 product rounded
once: D next to the midpoints of FP32 numbers, on either side by its last bits,
must round to its own side.  One nonzero entry, a power of two, per row of A: M_pp
is that operand times the entry, exactly."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16, torch.float64])
def test_rounding_next_to_midpoints(dtype):
    import paper_1502_03543_gb300 as P
    m, n = 200, 201
    rng = np.random.default_rng(0)
    f = 1.0 + rng.integers(0, 1 << 23, n) * 2.0 ** -23  # an FP32 number, its midpoint to the next, and 1 to 8 last bits off
    D = (f + 2.0 ** -24 + rng.choice([-1, 1], n) * rng.integers(1, 9, n) * 2.0 ** -52) * 2.0 ** rng.integers(-20, 21, n)
    a = rng.choice([-1.0, 1.0], m) * 2.0 ** rng.integers(-8, 9, m)
    A = np.zeros((m, n))
    A[np.arange(m), np.arange(m)] = a
    dev = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()
    with P.Solver(m, n, "fp32_ir", dtype) as S:
        S.form_normal(dev(A).to(dtype), dev(D), dev(np.ones(n)))
        got = S.copy_matrix().cpu().numpy().diagonal()
    assert np.array_equal(got, (a * D[:m]).astype(np.float32) * a.astype(np.float32))
