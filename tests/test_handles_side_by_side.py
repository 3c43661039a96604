"""Handles of different sizes side by side: the shared-memory limit of a
kernel belongs to the function, so a small handle made later must not take it
away from a larger one (batches, Woodbury solvers)."""
import numpy as np
import pytest
import torch

import lpgen

pytestmark = pytest.mark.gpu


def batch(m, n, count):
    lps = [lpgen.generate(m, n, seed=i, storage="f32") for i in range(count)]
    d = lpgen.pack(lps)
    t = {k: torch.from_numpy(d[k]).cuda() for k in ("A", "b", "c", "x0", "y0", "s0")}
    return d, t


def test_a_small_batch_after_a_large_one():
    import paper_1502_03543_gb300 as P
    out = []
    for later in (False, True):
        d, t = batch(128, 1024, 3)
        g = torch.from_numpy(np.random.default_rng(0).standard_normal(int(d["n"].sum()))).cuda()
        make = lambda d, t: P.BatchSolver(d["m"], d["n"], t["A"], t["b"], t["c"], t["x0"], t["y0"], t["s0"], tol=0.3,
                                          autotune=False)
        with make(d, t) as S:
            small = make(*batch(16, 40, 2)) if later else None
            r = S.solve()
            out.append([t["x0"].clone(), *S.backward(g)[:3], torch.from_numpy(r["iters"])])
            if small:
                small.solve()
                small.close()
    assert all(torch.equal(a, b) for a, b in zip(*out))


def test_a_small_woodbury_handle_after_a_large_one():
    import paper_1502_03543_gb300 as P
    m, n = 3200, 3210  # 2 m doubles of shared memory: more than a kernel has without asking
    g = torch.Generator(device="cuda").manual_seed(0)
    A = torch.randn(m, n, device="cuda", generator=g, dtype=torch.float64)
    D = torch.rand(n, device="cuda", generator=g, dtype=torch.float64) + 1.0
    r = torch.randn(m, device="cuda", generator=g, dtype=torch.float64)
    with P.WoodburySolver(m, n) as W:
        W.prepare(A)
        x = W.solve(A, D, r)[0]
        with P.WoodburySolver(20, 40):
            assert torch.equal(W.solve(A, D, r)[0], x)
