"""The batch kernel's FP32 normal matrix and factor carry an LP as far as their
arithmetic allows: M is summed by 32-column partial sums, and the factor
subtracts a pivot column at a time from the stored entry, both replayed here in
FP32.  The kernel moves an LP to the FP64 tier at the first pivot that is not
positive; replayed at the oracle's iterates, that factor must fail at the same
iteration or the next: the device's iterates differ from the oracle's by less
than an FP32 rounding, and from one iteration to the next M's smallest scaled
eigenvalue falls several-fold, where another set of roundings moves it by a
small factor.  (Summed over all columns in one chain, M broke down one to four
iterations sooner.)"""
import numpy as np
import pytest
import torch

import lpgen
import oracle

SIZES = [(33, 132), (60, 240), (100, 400), (128, 384), (129, 516), (180, 720), (200, 800), (225, 900), (240, 960),
         (256, 1024)]
F = np.float32


def fp32_factor_fails(A, x, s):
    """True if the FP32 Cholesky of (A D^1/2)(A D^1/2)' meets a pivot <= 0."""
    B = (A * np.sqrt(x / s).astype(F)).astype(F)
    m, n = B.shape
    M = np.zeros((m, m), F)
    for k0 in range(0, n, 32):
        acc = np.zeros((m, m))  # (FP32 values; FP64 holds each product exactly)
        for k in range(k0, min(n, k0 + 32)):
            c = B[:, k].astype(np.float64)
            acc = (acc + np.outer(c, c)).astype(F).astype(np.float64)
        M += acc.astype(F)
    for k in range(m):
        d = M[k, k]
        if not (d > 0 and np.isfinite(d)):
            return True
        col = (M[k + 1:, k] * F(1 / np.sqrt(np.float64(d)))).astype(np.float64)
        M[k + 1:, k + 1:] = (M[k + 1:, k + 1:] - np.outer(col, col)).astype(F)
    return False


def test_the_replay_on_exact_cases():
    A = np.array([[1, 2, 0], [0, 1, 1]], F)
    assert not fp32_factor_fails(A, np.ones(3), np.ones(3))
    assert fp32_factor_fails(np.array([[1, 2, 0], [2, 4, 0]], F), np.ones(3), np.ones(3))


@pytest.mark.gpu
def test_iterations_until_the_fp64_tier():
    import paper_1502_03543_gb300 as P
    lps = [lpgen.generate(m, n, seed=700 + m, storage="f32") for m, n in SIZES]
    d = lpgen.pack(lps)
    t = {k: torch.from_numpy(d[k]).cuda() for k in ("A", "b", "c", "x0", "y0", "s0")}
    with P.BatchSolver(d["m"], d["n"], t["A"], t["b"], t["c"], t["x0"], t["y0"], t["s0"], autotune=False) as S:
        r = S.solve()
    checked = 0
    for i, lp in enumerate(lps):
        f = int(r["iters"][i] - r["fp64_iters"][i])  # FP32 iterations: the first FP64 one starts at iterate f
        if r["fp64_iters"][i] == 0:
            continue  # the FP32 factor lasted to the end
        checked += 1
        ref = oracle.solve(lp.A64, lp.b, lp.c, lp.x0, lp.y0, lp.s0, tol=1e-7, keep_iterates=True)
        it = ref["iterates"]
        fails = [fp32_factor_fails(lp.A_store, it[k - 1][:lp.n], it[k - 1][lp.n + lp.m:])
                 for k in (f, f + 1) if k <= len(it)]
        assert any(fails), (lp.m, lp.n, f, ref["iters"])
    assert checked >= len(lps) - 2
