"""What a user of the MGWR library has it do: whole solves through the public entry points.

Every case is a solve (or a few) of a time-fractional problem with a manufactured source, a sum of
sine modes whose time profiles are t^2 or t^alpha.  A sine mode is an eigenvector of the discrete
Laplacian, so the exact solution of the discrete problem is one scalar L1 recurrence per mode;
`exact` marches it in 64 bits.  Right-hand sides are on the device where a program keeps them there,
and numpy arrays where it calls with host data.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1608_05400_gb300 import mgwr

PRECISION = {"fp64": mgwr.MGWR_FP64, "mixed": mgwr.MGWR_MIXED, "mixed_dd": mgwr.MGWR_MIXED_DD,
             "auto": mgwr.MGWR_AUTO}
MODES = 3
T_END = 1.0


def _solve(name, d, n, M, alpha, kind, precision, tol, **more):
    return dict(name=name, path="solve", d=d, n=n, M=M, alpha=alpha, kind=kind, precision=precision,
                tol=tol, cycle=1, nu1=1, nu2=1, order="text", tuned=False, **more)


def listed():
    return [
        # the smallest problem: a plain FP64 solve of a short 1-D grid, bound by latency
        _solve("fp64-1d-63x64", 1, 63, 64, 0.5, "t2", "fp64", 1e-10),
        # plain FP64 on a 2-D grid, the accuracy reference that mixed solves are held against
        _solve("fp64-2d-255x1024", 2, 255, 1024, 0.5, "t2", "fp64", 1e-10),
        # the paper's 1-D iteration study: V(0,1) from a non-zero initial value
        dict(_solve("fp64-1d-511x512-v01", 1, 511, 512, 0.7, "t2", "fp64", 1e-10), nu1=0,
             order="table", path="initial"),
        # the large mixed-precision solve, on a handle tuned once and kept
        dict(_solve("mixed-2d-511x4096", 2, 511, 4096, 0.5, "talpha", "mixed", 1e-8), tuned=True),
        # a medium 2-D solve whose program leaves the precision and launch shapes to the library
        _solve("auto-2d-255x1024", 2, 255, 1024, 0.3, "talpha", "auto", 1e-8),
        # a medium 1-D solve called with host arrays
        dict(_solve("auto-1d-1023x2048-host", 1, 1023, 2048, 0.8, "t2", "auto", 1e-8), path="host"),
        # long memory: 65536 steps on the finest 1-D grid
        _solve("long-1d-4095x65536", 1, 4095, 65536, 0.2, "talpha", "auto", 1e-8),
        # many small problems with their own orders in one handle
        dict(_solve("batch512-2d-63x256", 2, 63, 256, 0.0, "t2", "mixed", 1e-8), path="batch",
             batch=512, tuned=True),
        # a study over the order on one handle, W(1,1) cycles in FP64
        dict(_solve("study-2d-127x512-w11", 2, 127, 512, 0.0, "t2", "fp64", 1e-10), path="study",
             cycle=2, count=3),
        # one problem, once: create, solve with host data, destroy
        dict(_solve("once-2d-63x128", 2, 63, 128, 0.5, "t2", "fp64", 1e-10), path="once"),
        # the nonlinear problem by waveform relaxation FAS
        dict(name="fas-1d-255x256", path="fas", n=255, M=256, alpha=0.4, c=1.0, tol=1e-10),
        # a burst of requests of mixed sizes through the server
        dict(name="serve-12", path="serve", count=12, shapes=1608, tol=1e-8),
    ]


def draw(rng):
    path = rng.choice(("solve", "solve", "solve", "solve", "initial", "host", "long", "batch", "study",
                       "once", "fas", "serve"))
    alpha = round(rng.uniform(0.1, 0.9), 3)
    kind = rng.choice(("t2", "talpha"))
    d = rng.choice((1, 2))
    if path == "fas":
        # any number of steps: powers of two from 128 take the whole-line smoother, others march
        M = rng.choice((64, 100, 128, 200, 256, 333, 512))
        return dict(path=path, n=2 ** rng.randint(5, 8) - 1, M=M, alpha=alpha,
                    c=rng.choice((-1.0, 1.0, 2.0)), tol=1e-10)
    if path == "serve":
        return dict(path=path, count=rng.randint(3, 16), shapes=rng.randrange(10000), tol=1e-8)
    if path == "long":
        return dict(pick(d=1, n=2 ** rng.randint(8, 11) - 1, M=2 ** rng.randint(13, 15), alpha=alpha,
                         kind=kind, precision=rng.choice(("auto", "mixed_dd", "fp64"))), path="solve")
    if path == "initial":
        return dict(pick(d=1, n=2 ** rng.randint(5, 9) - 1, M=2 ** rng.randint(5, 10),
                         alpha=round(rng.uniform(0.4, 0.9), 3), kind="t2", precision="fp64"),
                    nu1=0, order="table", path=path, cycle=rng.choice((1, 2)))
    if path == "batch":
        return dict(pick(d=d, n=2 ** rng.randint(3, 6) - 1, M=2 ** rng.randint(6, 9), alpha=0.0,
                         kind=kind, precision=rng.choice(("mixed", "mixed_dd", "fp64"))), path=path,
                    batch=rng.randint(3, 150), tuned=rng.random() < 0.5)
    if path == "study":
        return dict(pick(d=d, n=2 ** rng.randint(4, 7) - 1, M=2 ** rng.randint(6, 10), alpha=0.0,
                         kind=kind, precision=rng.choice(("fp64", "auto"))), path=path, count=3,
                    cycle=rng.choice((1, 2)))
    if path in ("once", "host"):
        n = 2 ** (rng.randint(5, 11) if d == 1 else rng.randint(4, 7)) - 1
        return dict(pick(d=d, n=n, M=2 ** rng.randint(5, 10), alpha=alpha, kind=kind,
                         precision=rng.choice(("fp64", "auto"))), path=path)
    precision = rng.choice(("fp64", "mixed", "mixed_dd", "auto"))
    while True:  # log-uniform over the supported grids up to the size of the large case
        n = 2 ** (rng.randint(5, 12) if d == 1 else rng.randint(4, 9)) - 1
        M = 2 ** rng.randint(5, 12)
        if n ** d * M <= (1 << 26 if precision == "fp64" else 1 << 28):
            break
    if precision != "fp64" and n > 2047:
        precision = "auto"  # FP32 cycles stall there; the library's own choice
    return dict(pick(d=d, n=n, M=M, alpha=alpha, kind=kind, precision=precision),
                tuned=rng.random() < 0.3, nu1=rng.choice((1, 1, 1, 2)))


def pick(d, n, M, alpha, kind, precision):
    # FP64 solves stop at 1e-10 where the grid's rounding floor is well below it
    tol = 1e-10 if precision == "fp64" and n <= 511 else 1e-8
    case = _solve("", d, n, M, alpha, kind, precision, tol)
    del case["name"]
    return case


# ---- the manufactured problems ------------------------------------------------------------------


def problem(d, n, M, alpha, kind, seed):
    """(phi (N, MODES), mode eigenvalues of A_h, F (MODES, M)): f = phi F."""
    rng = np.random.default_rng(seed)
    x = np.arange(1, n + 1) / (n + 1)
    t = np.arange(1, M + 1) * (T_END / M)
    top = max(2, min(6, (n + 1) // 4))
    phi, lam, F = [], [], []
    for j in range(MODES):
        k = [1] * d if j == 0 else [int(v) for v in rng.integers(1, top + 1, d)]
        amp = (1.0 if j == 0 else 0.3) * rng.uniform(0.5, 1.5) * (1 if rng.random() < 0.5 else -1)
        sines = [np.sin(math.pi * kk * x) for kk in k]
        phi.append(sines[0] if d == 1 else np.outer(sines[1], sines[0]).reshape(-1))
        lam.append(4.0 * (n + 1) ** 2 * sum(math.sin(math.pi * kk / (2 * (n + 1))) ** 2 for kk in k))
        w = t * t if kind == "t2" else t ** alpha
        dw = (2.0 * t ** (2.0 - alpha) / math.gamma(3.0 - alpha) if kind == "t2"
              else np.full(M, math.gamma(1.0 + alpha)))
        F.append(amp * (dw + math.pi ** 2 * sum(kk * kk for kk in k) * w))
    return np.stack(phi, 1), np.array(lam), np.stack(F)


def l1_weights(alpha, M):
    """c and d_1..d_M of the L1 scheme: c (d_1 u_m - sum_k (d_k - d_{k+1}) u_{m-k} - d_m u_0)."""
    k = np.arange(2, M + 1, dtype=np.float64)
    dk = np.concatenate([[1.0], (k - 1) ** (1 - alpha) * np.expm1((1 - alpha) * np.log1p(1 / (k - 1)))])
    return (T_END / M) ** -alpha / math.gamma(2.0 - alpha), dk


def discrete_modes(alpha, M, lam, F, g=None):
    """(MODES, M): the time coefficient of every mode of the discrete solution."""
    c, dk = l1_weights(alpha, M)
    drop = np.ascontiguousarray((dk[:-1] - dk[1:])[::-1])  # drop[-k] = d_k - d_{k+1}
    U = np.zeros((len(lam), M))
    for m in range(M):
        r = F[:, m] + (c * dk[m] * g if g is not None else 0.0)
        if m:
            r = r + c * (U[:, :m] @ drop[M - 1 - m:])
        U[:, m] = r / (c + lam)
    return U


def on_gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def field(phi, F):
    return on_gpu(phi) @ on_gpu(F)


def host_field(phi, F):
    return np.ascontiguousarray(phi @ F)


def alphas_of(case, seed):
    count = case["batch"] if case["path"] == "batch" else case["count"]
    return np.random.default_rng(seed).uniform(0.1, 0.9, count)


def requests(case, seed):
    """The burst's shapes (from the case) and problems (from the seed): dicts with f on the host."""
    shapes = np.random.default_rng(case["shapes"])
    rng = np.random.default_rng(seed)
    got = []
    while len(got) < case["count"]:
        d = int(shapes.integers(1, 3))
        n = 2 ** int(shapes.integers(5, 13) if d == 1 else shapes.integers(5, 10)) - 1
        M = 2 ** int(shapes.integers(7, 13))
        if n ** d * M > 1 << 23:
            continue  # the burst holds the stream's smaller requests
        got.append(dict(d=d, n=n, M=M, alpha=float(rng.uniform(0.1, 0.9)),
                        kind="t2" if rng.integers(0, 2) == 0 else "talpha",
                        seed=int(rng.integers(1 << 30))))
    return got


def initial_modes(seed):
    return np.random.default_rng(seed + 1).uniform(0.5, 1.5, MODES)


# ---- passes -------------------------------------------------------------------------------------


def solver(case, alpha):
    s = mgwr.Solver(case["d"], case["n"], case["M"], T_END, alpha)
    s.set_precision(PRECISION[case["precision"]])
    if case["order"] == "table":
        s.set_order(mgwr.MGWR_ORDER_TABLE)
    if case["path"] == "batch" and case["precision"] != "fp64":
        s.set_inner_cycles(3)
    return s


def on_stream(s):
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    s.set_stream(stream.cuda_stream)
    return stream


def prepare(case, seed):
    path = case["path"]
    if path == "fas":
        n, M = case["n"], case["M"]
        x, t = np.arange(1, n + 1) / (n + 1), np.arange(1, M + 1) / M
        a = np.random.default_rng(seed).uniform(0.3, 1.0, 3)
        s = mgwr.FAS(n, M, T_END, case["alpha"], c=case["c"])
        s.set_order(mgwr.MGWR_ORDER_TABLE)
        f = a[0] + a[1] * np.outer(np.sin(math.pi * x), t) + a[2] * np.outer(np.sin(2 * math.pi * x), t * t)
        return dict(case=case, solver=s, f=f)
    if path == "serve":
        rqs = requests(case, seed)
        for q in rqs:
            phi, _, F = problem(q["d"], q["n"], q["M"], q["alpha"], q["kind"], q["seed"])
            q["f"] = host_field(phi, F)
        return dict(case=case, server=mgwr.Server(64 << 30, slots=8), requests=rqs)
    if path in ("batch", "study"):
        alphas = alphas_of(case, seed)
        fs = [problem(case["d"], case["n"], case["M"], a, case["kind"], seed + k)
              for k, a in enumerate(alphas)]
        s = solver(case, alphas if path == "batch" else float(alphas[0]))
        f = [field(phi, F) for phi, _, F in fs]
        f = torch.stack(f) if path == "batch" else f
        u = torch.empty_like(f) if path == "batch" else [torch.empty_like(v) for v in f]
        state = dict(case=case, solver=s, f=f, u=u, alphas=[float(a) for a in alphas])
    else:
        phi, _, F = problem(case["d"], case["n"], case["M"], case["alpha"], case["kind"], seed)
        if path in ("host", "once", "initial"):
            state = dict(case=case, f=host_field(phi, F), alpha=case["alpha"])
            if path == "initial":
                state["g"] = phi @ initial_modes(seed)
            if path != "once":
                state["solver"] = solver(case, case["alpha"])
            return state
        f = field(phi, F)
        state = dict(case=case, solver=solver(case, case["alpha"]), f=f, u=torch.empty_like(f))
    state["stream"] = on_stream(state["solver"])
    if case["tuned"]:
        state["solver"].set_rhs_dev((state["f"] if path != "study" else state["f"][0]).data_ptr())
        state["solver"].autotune()
    return state


def solve(s, case):
    s.solve(cycle=case["cycle"], nu1=case["nu1"], nu2=case["nu2"], tol=case["tol"], max_cycles=200)


def run(state):
    case = state["case"]
    path = case["path"]
    if path == "serve":
        srv = state["server"]
        tickets = [srv.submit(q["d"], q["n"], q["M"], T_END, q["alpha"], q["f"],
                              precision=mgwr.MGWR_AUTO, tol=case["tol"]) for q in state["requests"]]
        out = []
        for t in tickets:
            r = None
            while r is None:
                r = srv.poll(t, timeout_us=100000)
            out.append(r.u)
        return out
    if path == "once":
        with solver(case, state["alpha"]) as s:
            s.set_rhs(state["f"])
            solve(s, case)
            return s.solution()
    s = state["solver"]
    if path == "fas":
        s.set_rhs(state["f"])
        s.solve(cycle=1, nu1=0, nu2=1, tol=case["tol"], max_cycles=100)
        return s.solution()
    if path in ("host", "initial"):
        s.set_rhs(state["f"], state.get("g"))
        solve(s, case)
        return s.solution()
    if path == "study":
        for alpha, f, u in zip(state["alphas"], state["f"], state["u"]):
            s.set_problem(T_END, alpha)
            s.set_rhs_dev(f.data_ptr())
            solve(s, case)
            s.solution_dev(u.data_ptr())
        return state["u"]
    s.set_rhs_dev(state["f"].data_ptr())
    solve(s, case)
    s.solution_dev(state["u"].data_ptr())
    return state["u"]


# ---- what a pass needs, and what it gives ----------------------------------------------------------


def unknowns(case):
    if case["path"] == "serve":
        return sum(q["n"] ** q["d"] * q["M"] for q in requests(case, 0))
    per = case["n"] ** case.get("d", 1) * case["M"]
    return per * (case.get("batch") or case.get("count") or 1)


def work(case):
    """The right-hand side in, the solution out; two time convolutions of every line (the fewest a
    defect and a smoothing step of one cycle can take) by transforms of twice its length."""
    N = unknowns(case)
    M = case.get("M", 1024)
    return {"bytes": 16.0 * N, "flops": 2.0 * N * 20.0 * math.log2(2 * M)}


def exact(case, seed):
    path = case["path"]
    if path == "fas":
        return exact_fas(case, seed)

    def one(d, n, M, alpha, kind, sd, host, g=None):
        phi, lam, F = problem(d, n, M, alpha, kind, sd)
        U = discrete_modes(alpha, M, lam, F, g)
        return host_field(phi, U) if host else field(phi, U)

    if path == "serve":
        return [one(q["d"], q["n"], q["M"], q["alpha"], q["kind"], q["seed"], True)
                for q in requests(case, seed)]
    if path in ("batch", "study"):
        got = [one(case["d"], case["n"], case["M"], float(a), case["kind"], seed + k, False)
               for k, a in enumerate(alphas_of(case, seed))]
        return torch.stack(got) if path == "batch" else got
    return one(case["d"], case["n"], case["M"], case["alpha"], case["kind"], seed,
               path in ("host", "once", "initial"), initial_modes(seed) if path == "initial" else None)


def exact_fas(case, seed):
    """Time marching of the nonlinear scheme, Newton's method on the whole grid at every step."""
    n, M, conv = case["n"], case["M"], case["c"]
    x, t = np.arange(1, n + 1) / (n + 1), np.arange(1, M + 1) / M
    a = np.random.default_rng(seed).uniform(0.3, 1.0, 3)
    f = a[0] + a[1] * np.outer(np.sin(math.pi * x), t) + a[2] * np.outer(np.sin(2 * math.pi * x), t * t)
    c, dk = l1_weights(case["alpha"], M)
    drop = np.ascontiguousarray((dk[:-1] - dk[1:])[::-1])
    h2, h = (n + 1.0) ** -2, 1.0 / (n + 1)
    U = np.zeros((n, M))
    i = np.arange(n)
    for m in range(M):
        known = f[:, m] + (c * (U[:, :m] @ drop[M - 1 - m:]) if m else 0.0)
        v = U[:, m - 1].copy() if m else np.zeros(n)
        for _ in range(50):
            w = np.concatenate([[0.0], v, [0.0]])
            D = 1.0 + w * w
            ap, am = 0.5 * (D[2:] + D[1:-1]), 0.5 * (D[:-2] + D[1:-1])
            up, dn = w[2:] - w[1:-1], w[1:-1] - w[:-2]
            res = c * v - (ap * up - am * dn) / h2 - conv * (up if conv >= 0 else dn) / h - known
            J = np.zeros((n, n))
            J[i, i] = c + (ap + am - v * up + v * dn) / h2 + abs(conv) / h
            J[i[:-1], i[1:]] = -(ap[:-1] + w[2:-1] * up[:-1]) / h2 - (conv / h if conv >= 0 else 0.0)
            J[i[1:], i[:-1]] = -(am[1:] - w[1:-2] * dn[1:]) / h2 + (conv / h if conv < 0 else 0.0)
            step = np.linalg.solve(J, res)
            v = v - step
            if np.abs(step).max() <= 1e-14 * max(1e-3, np.abs(v).max()):
                break
        U[:, m] = v
    return U
