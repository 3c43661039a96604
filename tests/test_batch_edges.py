"""The batch kernel at the sizes where its blocks change: 8 x 8 units and 32-row
blocks with remainders, one to four columns per thread, every bucket and its
edges, odd row lengths.  A few iterations from the start, where two correct
64-bit codes agree to 1e-13 and the directions are accurate to a backward error
of 1e-14: iterates within 1e-9 of the oracle's."""
import numpy as np
import pytest
import torch

import lpgen
import oracle

pytestmark = pytest.mark.gpu

SIZES = [(1, 2), (7, 16), (8, 33), (31, 70), (33, 67), (63, 300), (64, 129), (65, 1024), (97, 260), (127, 513),
         (128, 384), (129, 1000), (160, 321), (192, 768), (193, 777), (240, 961), (255, 511), (256, 1024)]


@pytest.mark.parametrize("autotune", [False, True])
def test_iterates(autotune):
    import paper_1502_03543_gb300 as P
    lps = [lpgen.generate(m, n, seed=50 + m, storage="f32") for m, n in SIZES]
    d = lpgen.pack(lps)
    t = {k: torch.from_numpy(d[k]).cuda() for k in ("A", "b", "c", "x0", "y0", "s0")}
    with P.BatchSolver(d["m"], d["n"], t["A"], t["b"], t["c"], t["x0"], t["y0"], t["s0"], tol=1e-30, max_iter=4,
                       autotune=autotune) as S:
        r = S.solve()
        x, y, s = (t[k].cpu().numpy() for k in ("x0", "y0", "s0"))
    on = om = 0
    for i, lp in enumerate(lps):
        ref = oracle.solve(lp.A64, lp.b, lp.c, lp.x0, lp.y0, lp.s0, tol=1e-30, max_iter=4)
        for got, want in ((x[on:on + lp.n], ref["x"]), (y[om:om + lp.m], ref["y"]), (s[on:on + lp.n], ref["s"])):
            assert np.linalg.norm(got - want) <= 1e-9 * np.linalg.norm(want), (lp.m, lp.n)
        assert r["iters"][i] == ref["iters"] and r["status"][i] == ref["status"]
        on, om = on + lp.n, om + lp.m
