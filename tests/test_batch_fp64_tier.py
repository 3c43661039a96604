"""One direction of the batch kernel in its FP64 tier at ragged sizes on both sides
of its switch (row-by-row solves up to 64 rows of capacity, blocked ones with
inverted diagonal blocks beyond).  From an iterate where nine tenths of m columns have
D ~ 1 and the others 1e-9, M has a condition number of 1e9 and more: the FP32 factor
fails, the FP64 one holds.  After one step from y = 0, y = theta dy, and theta
follows from x: the direction's backward error is that of the refinement's
acceptance (1e-14) plus what the recovery of dy and the check itself round, 4e-14
in all."""
import numpy as np
import pytest
import torch

import lpgen

pytestmark = pytest.mark.gpu

SIZES = [(20, 45), (40, 83), (63, 130), (65, 140), (97, 200), (127, 260), (129, 263), (161, 330), (193, 400),
         (224, 451), (255, 513), (256, 1024)]


def test_direction():
    import paper_1502_03543_gb300 as P
    lps = [lpgen.generate(m, n, seed=900 + m, storage="f32") for m, n in SIZES]
    for lp in lps:
        rng = np.random.default_rng(lp.m)
        big = np.zeros(lp.n, dtype=bool)
        big[rng.permutation(lp.n)[: (9 * lp.m) // 10]] = True
        lp.x0[:] = np.where(big, rng.uniform(0.5, 1.5, lp.n), 1e-5 * rng.uniform(0.5, 1.5, lp.n))
        lp.s0[:] = np.where(big, rng.uniform(0.5, 1.5, lp.n), 1e4 * rng.uniform(0.5, 1.5, lp.n))
        lp.y0[:] = 0.0
    d = lpgen.pack(lps)
    t = {k: torch.from_numpy(d[k]).cuda() for k in ("A", "b", "c", "x0", "y0", "s0")}
    with P.BatchSolver(d["m"], d["n"], t["A"], t["b"], t["c"], t["x0"], t["y0"], t["s0"], tol=1e-300, max_iter=1,
                       autotune=False) as S:
        r = S.solve()
        x, y, s = (t[k].cpu().numpy() for k in ("x0", "y0", "s0"))
    on = om = 0
    for i, lp in enumerate(lps):
        x1, y1, s1 = x[on:on + lp.n], y[om:om + lp.m], s[on:on + lp.n]
        on, om = on + lp.n, om + lp.m
        assert r["fp64_iters"][i] == 1 and r["unrefined"][i] == 0 and r["iters"][i] == 1, (lp.m, lp.n)
        A, D = lp.A64, lp.x0 / lp.s0
        w = A.T @ y1
        assert np.abs(s1 - (lp.s0 - w)).max() <= 1e-13 * (np.abs(lp.s0).max() + np.abs(w).max())
        theta = float(lp.x0 @ (lp.x0 + D * w - x1)) / float(lp.x0 @ lp.x0)
        rhs, Mdy = theta * (A @ lp.x0), A @ (D * w)
        scale = ((A * A) @ D).max() * np.abs(y1).max() + np.abs(rhs).max()
        assert np.abs(rhs - Mdy).max() <= 4e-14 * scale, (lp.m, lp.n)
