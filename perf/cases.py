"""Timing cases of the PDAS solver: the calls its users make, over the sizes,
storage types and precision forms they make them with.

A user of this library either drives a solve themselves (one Newton direction
or one step per iteration), hands over a whole solve, solves and differentiates
a batch of small LPs, or uses single passes over A.  The cases are those calls.
The data is synthetic, drawn on the GPU from the seed: dense Gaussian A, columns
scaled by U(0.1, 10) where A is stored in BF16, as in the repository's
workloads.

Directions are taken at a mid-solve iterate: complementary pairs x_j s_j ~ mu,
one and a half times m columns with large D = x/s and the others graded down to
mu.  There M = A D A' is well conditioned although max D / min D is large, so
that results of correct codes agree closely.  For the same reason whole solves
stop at a rough relative gap, and the batch is differentiated at a rougher one:
the refined directions are accurate to a backward error of 1e-14, and the
iterates drift from those of a 64-bit code as M grows ill-conditioned (about
2e-10 at a gap of 3e-2, 1e-9 at 1e-2, 1e-7 and more at the end).
"""
import math

import numpy as np
import torch

import paper_1502_03543_gb300 as P

DTYPES = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
ALPHA = 0.95


def listed():
    return [
        # the smallest LP: latency of the launches and of the host loop (the parity workload's size)
        dict(name="direction_fp64_64x128", kind="direction", form="fp64", dtype="f64", m=64, n=128, mu=1e-2, tier=False),
        # the plain FP64 form at an ordinary size, off the tile grid
        dict(name="direction_fp64_1000x2500", kind="direction", form="fp64", dtype="f64", m=1000, n=2500, mu=1e-2,
             tier=False),
        # FP64-stored A through the TF32 tensor-core form (the mid-size dense workload)
        dict(name="direction_tf32_2048x8192", kind="direction", form="tf32_ir", dtype="f64", m=2048, n=8192, mu=1e-3,
             tier=False),
        # the BF16 form at a small size: launches and dependency chains
        dict(name="direction_bf16_512x2048", kind="direction", form="bf16_ir", dtype="bf16", m=512, n=2048, mu=1e-3,
             tier=False),
        # the benchmark's LP, an iteration with the FP32 factor
        dict(name="direction_bf16_8192x32768", kind="direction", form="bf16_ir", dtype="bf16", m=8192, n=32768,
             mu=1e-3, tier=False),
        # late iterations of the BF16 form: M formed and factored at FP64 grade from the significant columns
        dict(name="direction_bf16_late_4096x16384", kind="direction", form="bf16_ir", dtype="bf16", m=4096, n=16384,
             mu=1e-6, tier=True),
        # FP32-stored A with odd, ragged sizes (rows are not 16-byte aligned)
        dict(name="direction_fp32_1001x3003", kind="direction", form="fp32_ir", dtype="f32", m=1001, n=3003, mu=1e-3,
             tier=False),
        # one differentiable LP: the sensitivities to A, b and c after a step
        dict(name="backward_tf32_1024x4096", kind="backward", form="tf32_ir", dtype="f32", m=1024, n=4096, mu=1e-2),
        # single passes over A: A v and A' u
        dict(name="passes_bf16_4096x16384", kind="passes", form="bf16_ir", dtype="bf16", m=4096, n=16384),
        # a whole solve from an infeasible start, to a rough gap
        dict(name="solve_bf16_infeasible_700x2800", kind="solve", form="bf16_ir", dtype="bf16", m=700, n=2800,
             infeasible=True),
        # many small LPs of uneven sizes, solved together to a rough gap
        dict(name="batch_solve_512", kind="batch_solve", count=512, m_lo=16, m_hi=256),
        # the differentiable batch: the sensitivities of every LP of equal size
        dict(name="batch_backward_256", kind="batch_backward", count=256, m_lo=128, m_hi=128),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["direction", "direction", "direction", "direction", "late", "backward", "passes", "solve",
                       "batch_solve", "batch_backward"])
    if kind.startswith("batch"):
        lo = rng.randint(16, 128)
        return dict(kind=kind, count=_log_int(rng, 32, 512 if kind == "batch_solve" else 256), m_lo=lo,
                    m_hi=rng.randint(lo, 256 if kind == "batch_solve" else 160))
    form, dtype, hi = rng.choice([("fp64", "f64", 1200), ("tf32_ir", "f64", 2500), ("tf32_ir", "f32", 2500),
                                  ("fp32_ir", "f32", 2000), ("bf16_ir", "bf16", 6000), ("bf16_ir", "bf16", 6000)])
    if kind == "late" and form == "fp64":
        form, dtype, hi = "bf16_ir", "bf16", 6000
    if kind == "late" and dtype != "bf16":
        hi = 1200
    if kind in ("backward", "solve"):
        hi = min(hi, 1500)
    m = _log_int(rng, 64, hi)
    n = int(m * rng.uniform(2.0, 4.0))
    if rng.random() < 0.5:  # aligned sizes as often as odd ones
        m, n = (m + 15) // 16 * 16, (n + 63) // 64 * 64
    case = dict(kind="direction" if kind == "late" else kind, form=form, dtype=dtype, m=m, n=n)
    if kind in ("direction", "late"):
        case.update(mu=1e-6 if kind == "late" else 10.0 ** rng.uniform(-3.0, -1.0), tier=kind == "late")
    elif kind == "backward":
        case.update(mu=1e-2)
    elif kind == "solve":
        case.update(infeasible=rng.random() < 0.5)
    return case


# ---- inputs ------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) + 1)


def _uniform(g, n, lo=0.5, hi=1.5):
    return torch.rand(n, dtype=torch.float64, device="cuda", generator=g) * (hi - lo) + lo


def _normal(g, n):
    return torch.randn(n, dtype=torch.float64, device="cuda", generator=g)


def _matrix(g, m, n, dtype):
    A = torch.randn(m, n, dtype=torch.float32 if dtype != "f64" else torch.float64, device="cuda", generator=g)
    if dtype == "bf16":
        A *= _uniform(g, n, 0.1, 10.0).to(A.dtype)
    return A.to(DTYPES[dtype])


def _iterate(g, m, n, mu):
    """(x, s) with x_j s_j ~ mu: large D on 1.5 m random columns (at most n - 1), graded on the others."""
    large = torch.zeros(n, dtype=torch.bool, device="cuda")
    large[torch.randperm(n, device="cuda", generator=g)[: min(n - 1, m + m // 2)]] = True
    u, v = _uniform(g, n), _uniform(g, n)
    small = mu ** _uniform(g, n, 0.3, 1.0)
    return torch.where(large, u, small * u), torch.where(large, mu * v, v)


def _times(A, v, transpose=False):
    """A v or A' v in 64 bits, a block of rows at a time (A may be stored in 16 or 32 bits)."""
    step = max(1, (1 << 26) // A.shape[1])
    if not transpose:
        return torch.cat([A[i:i + step].double() @ v for i in range(0, A.shape[0], step)])
    out = torch.zeros(A.shape[1], dtype=torch.float64, device="cuda")
    for i in range(0, A.shape[0], step):
        out += A[i:i + step].double().T @ v[i:i + step]
    return out


def _lp(case, seed):
    """One LP: A, b, c and an interior point (x, y, s), feasible unless the case says otherwise."""
    g = _gen(seed)
    m, n = case["m"], case["n"]
    A = _matrix(g, m, n, case["dtype"])
    x, s = _iterate(g, m, n, case["mu"]) if "mu" in case else (_uniform(g, n), _uniform(g, n))
    y = _normal(g, m)
    xf, yf, sf = (_uniform(g, n), _normal(g, m), _uniform(g, n)) if case.get("infeasible") else (x, y, s)
    return dict(A=A, b=_times(A, xf), c=_times(A, yf, True) + sf, x=x, y=y, s=s)


def _batch(case, seed):
    """A batch of LPs with feasible interior starts, packed one after another; n_i = 2 to 4 times m_i
    (3 times where the batch is differentiated)."""
    g, sizes = _gen(seed), np.random.default_rng(case["count"])  # the sizes do not depend on the seed
    m = sizes.integers(case["m_lo"], case["m_hi"] + 1, case["count"])
    n = m * (sizes.integers(2, 5, case["count"]) if case["kind"] == "batch_solve" else 3)
    A = torch.randn(int((m * n).sum()), dtype=torch.float32, device="cuda", generator=g)
    x, s = _uniform(g, int(n.sum())), _uniform(g, int(n.sum()))
    y = _normal(g, int(m.sum()))
    b, c = torch.empty_like(y), s.clone()
    at = mt = nt = 0
    for mi, ni in zip(m.tolist(), n.tolist()):
        Ai = A[at:at + mi * ni].view(mi, ni).double()
        b[mt:mt + mi] = Ai @ x[nt:nt + ni]
        c[nt:nt + ni] += Ai.T @ y[mt:mt + mi]
        at, mt, nt = at + mi * ni, mt + mi, nt + ni
    return dict(m=m, n=n, A=A, b=b, c=c, x=x, y=y, s=s)


TOL = {"solve": 3e-2, "batch_solve": 3e-2, "batch_backward": 0.3}


def prepare(case, seed):
    kind = case["kind"]
    if kind.startswith("batch"):
        d = _batch(case, seed)
        d["start"] = [d[k].clone() for k in ("x", "y", "s")]
        # no autotuning: a program that makes many handles does without it
        d["solver"] = P.BatchSolver(d["m"], d["n"], *(d[k] for k in ("A", "b", "c", "x", "y", "s")), alpha=ALPHA,
                                    tol=TOL[kind], autotune=False)
        if kind == "batch_backward":
            d["g"] = _normal(_gen(seed + 7919), int(d["n"].sum()))
            torch.cuda.synchronize()
            d["solver"].solve()
        return dict(d, kind=kind)
    opts = {}
    if case.get("tier"):
        opts["dspread_refactor"] = 1e8  # the rule that moves a late iteration to the FP64-grade factor
    if kind == "solve":
        opts["infeasible"] = int(case["infeasible"])
    d = _lp(case, seed) if kind != "passes" else dict(A=_matrix(_gen(seed), case["m"], case["n"], case["dtype"]))
    d["solver"] = P.Solver(case["m"], case["n"], case["form"], DTYPES[case["dtype"]], **opts)
    if kind == "passes":
        g = _gen(seed + 7919)
        d.update(v=_normal(g, case["n"]), u=_normal(g, case["m"]))
    elif kind == "backward":
        d["solver"].step(d["A"], d["b"], d["c"], d["x"], d["y"], d["s"], alpha=ALPHA)
        d["g"] = _normal(_gen(seed + 7919), case["n"])
    return dict(d, kind=kind)


def run(state):
    d, kind = state, state["kind"]
    S = d["solver"]
    if kind == "direction":
        dx, dy, ds, _ = S.direction(d["A"], d["x"], d["s"])
        return {"dx": dx, "dy": dy, "ds": ds}
    if kind == "backward":
        dA, db, dc = S.backward(d["A"], d["x"], d["y"], d["s"], d["g"])
        return {"dA": dA, "db": db, "dc": dc}
    if kind == "passes":
        return {"Av": S.gemv(d["A"], d["v"]), "Atu": S.gemv_t(d["A"], d["u"])}
    if kind == "solve":
        x, y, s = d["x"].clone(), d["y"].clone(), d["s"].clone()
        r = S.solve(d["A"], d["b"], d["c"], x, y, s, alpha=ALPHA, tol=TOL[kind])
        return {"x": x, "y": y, "s": s, "iters": r["iters"], "status": r["status"]}
    if kind == "batch_backward":
        dA, db, dc, status = S.backward(d["g"])
        return {"dA": dA, "db": db, "dc": dc, "status": status}
    for t, t0 in zip((d["x"], d["y"], d["s"]), d["start"]):
        t.copy_(t0)
    # the handle runs on a stream of its own, which does not wait for the copies
    torch.cuda.current_stream().synchronize()
    r = S.solve()
    return {"x": d["x"], "y": d["y"], "s": d["s"], "iters": r["iters"], "status": r["status"]}


# ---- what a pass cannot do without ---------------------------------------------
def work(case):
    kind = case["kind"]
    if kind.startswith("batch"):
        m = 0.5 * (case["m_lo"] + case["m_hi"])
        m2, m3 = (sum(k ** p for k in range(case["m_lo"], case["m_hi"] + 1)) / (case["m_hi"] - case["m_lo"] + 1)
                  for p in (2, 3))
        # one direction per LP iteration (about 8 iterations to the gap): M, its factor, six products with A
        direction = 3 * m3 + m3 / 3 + 6 * 2 * 3 * m2
        if kind == "batch_solve":
            return {"bytes": case["count"] * (4 * 3 * m2 + 8 * (2 * m + 4 * 3 * m)), "flops": case["count"] * 8 * direction}
        return {"bytes": case["count"] * (12 * 3 * m2 + 8 * (3 * m + 5 * 3 * m)),
                "flops": case["count"] * (direction + 3 * 3 * m2)}
    m, n = case["m"], case["n"]
    a = m * n * {"f64": 8, "f32": 4, "bf16": 2}[case["dtype"]]
    if kind == "passes":
        return {"bytes": a + 8 * 2 * (m + n), "flops": 4.0 * m * n}
    direction = 1.0 * m * (m + 1) * n + m ** 3 / 3.0 + 4.0 * m * n
    if kind == "backward":  # the factor is there: products with A and solves with it, and dL/dA
        return {"bytes": a + 8.0 * m * n + 8 * (3 * m + 5 * n), "flops": 7.0 * m * n + 4.0 * m * m}
    if kind == "solve":  # about 8 iterations to the gap
        return {"bytes": a + 8 * (2 * m + 5 * n), "flops": 8 * direction}
    return {"bytes": a + 8 * (m + 4 * n), "flops": direction}


# ---- the same in plain 64 bits ---------------------------------------------------
def _normal_equations(A, D, r):
    """M = A D A' by its Cholesky factor, in 64 bits, refined; A in 64 bits."""
    L = torch.linalg.cholesky((A * D) @ A.T)
    solve = lambda v: torch.cholesky_solve(v[:, None], L)[:, 0]  # noqa: E731
    z = solve(r)
    for _ in range(2):
        z = z + solve(r - A @ (D * (A.T @ z)))
    return z, solve


def _direction(A, x, s, rd=None, r=None):
    D = x / s
    dy, _ = _normal_equations(A, D, A @ x if r is None else r)
    ds = -(A.T @ dy) if rd is None else rd - A.T @ dy
    return D * (-ds) - x, dy, ds


def _step(A, x, y, s, dx, dy, ds, capped=False):
    psi = max(float((-dx / x).max()), float((-ds / s).max()))
    theta = (1.0 if psi <= ALPHA else ALPHA / psi) if capped else (1.0 if psi <= 1.0 else ALPHA / psi)
    return x + theta * dx, y + theta * dy, s + theta * ds


def _solve(A, b, c, x, y, s, infeasible, tol):
    for _ in range(500):
        if infeasible:
            rd = c - A.T @ y - s
            dx, dy, ds = _direction(A, x, s, rd, b + A @ ((x / s) * rd))
        else:
            dx, dy, ds = _direction(A, x, s)
        x, y, s = _step(A, x, y, s, dx, dy, ds, infeasible)
        cx = float(c @ x)
        gap = (cx - float(b @ y)) / (1.0 + abs(cx))
        if infeasible:
            pres = float((b - A @ x).abs().max() / (1.0 + b.abs().max()))
            dres = float((c - A.T @ y - s).abs().max() / (1.0 + c.abs().max()))
            gap = max(abs(gap), pres, dres)
        if gap < tol:
            break
    return x, y, s


def _adjoint(A, x, y, s, g):
    """The adjoint of F = [A x - b; A'y + s - c; x s - sigma] at (x, y, s), refined on the full system."""
    D = x / s
    la, lb, lc, wt = 0.0, 0.0, 0.0, 0.0
    r1, r3, t, solve = g, torch.zeros_like(g), D * g, None
    for k in range(4):
        if solve is None:
            da, solve = _normal_equations(A, D, A @ t)
        else:
            rhs = A @ t
            da = solve(rhs)
            for _ in range(2):
                da = da + solve(rhs - A @ (D * (A.T @ da)))
        w = A.T @ da
        db = D * (w - r1) + r3
        la, lb, lc, wt = la + da, lb + db, lc + (r3 - db) / x, wt + w
        r1, r3 = g - wt - s * lc, -lb - x * lc
        t = D * r1 - r3 - lb
    return -(torch.outer(la, x) + torch.outer(y, lb)), la, lb


def exact(case, seed):
    kind = case["kind"]
    if kind.startswith("batch"):
        d = _batch(case, seed)
        g = _normal(_gen(seed + 7919), int(d["n"].sum()))
        got, at, mt, nt = [], 0, 0, 0
        for mi, ni in zip(d["m"].tolist(), d["n"].tolist()):
            A = d["A"][at:at + mi * ni].view(mi, ni).double()
            m_, n_ = slice(mt, mt + mi), slice(nt, nt + ni)
            x, y, s = _solve(A, d["b"][m_], d["c"][n_], d["x"][n_], d["y"][m_], d["s"][n_], False,
                             TOL[kind])
            got.append((x, y, s) if kind == "batch_solve" else _adjoint(A, x, y, s, g[n_]))
            at, mt, nt = at + mi * ni, mt + mi, nt + ni
        a, b, c = (torch.cat([t[k].reshape(-1) for t in got]) for k in range(3))
        if kind == "batch_solve":
            return {"x": a, "y": b, "s": c, "iters": None, "status": None}
        return {"dA": a, "db": b, "dc": c, "status": None}
    if kind == "passes":
        A, g = _matrix(_gen(seed), case["m"], case["n"], case["dtype"]), _gen(seed + 7919)
        v, u = _normal(g, case["n"]), _normal(g, case["m"])
        return {"Av": _times(A, v), "Atu": _times(A, u, True)}
    d = _lp(case, seed)
    A, x, y, s = d["A"].double(), d["x"], d["y"], d["s"]
    if kind == "solve":
        x, y, s = _solve(A, d["b"], d["c"], x, y, s, case["infeasible"], TOL[kind])
        return {"x": x, "y": y, "s": s, "iters": None, "status": None}
    dx, dy, ds = _direction(A, x, s)
    if kind == "direction":
        return {"dx": dx, "dy": dy, "ds": ds}
    x, y, s = _step(A, x, y, s, dx, dy, ds)
    dA, db, dc = _adjoint(A, x, y, s, _normal(_gen(seed + 7919), case["n"]))
    return {"dA": dA, "db": db, "dc": dc}
