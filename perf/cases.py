"""Performance cases: what a user of the library has it solve, through the Python binding of its C ABI.

Every pass is a whole call sequence as a program makes it: a single LP is loaded, solved and read back on a handle that the
program keeps; a batch is one ``lp_solve_batch`` call; a served burst is submitted to a running server and waited for; a product
is one ``lp_dgemm_emulated`` call.  Inputs are seeded LPs of the families that this repository's tests and benchmark use
(integer dense LPs, real ones of the paper's distribution, LPs with >= rows that need Phase I), in device memory where a
program would generate or keep them there, in host memory where it would read them from elsewhere.
"""
import math

import numpy as np
import torch

from paper_1804_04737_gb300 import capi, lpgen

DEV = "cuda"


# ------------------------------------------------------------------ cases --

def _lp(name, m, n, family="dense", form="primal", precision="fp64", memory="device"):
    return {"name": name, "kind": "lp", "family": family, "m": m, "n": n, "form": form, "precision": precision,
            "memory": memory}


def listed():
    return [
        # the smallest call: one little LP from host arrays, where latency and launches count
        _lp("lp_64", 64, 64, memory="host"),
        # an ordinary LP of the paper's distribution (real data, many pivots), odd sizes
        _lp("lp_paper_500x700", 501, 703, family="paper"),
        # a mid-size LP that the origin does not satisfy: Phase I (dual rule, then primal)
        _lp("lp_phase1_200x300", 200, 301, family="phase1"),
        # many variables, few constraints, and the reverse (the two flat shapes of the benchmark's set)
        _lp("lp_512x4096", 512, 4096),
        _lp("lp_4096x512", 4096, 512),
        # the square mid-size LP in both formulations; the dual one comes from pinned host memory
        _lp("lp_2048", 2048, 2048),
        _lp("lp_2048_dual", 2048, 2048, form="dual", memory="pinned"),
        # the largest single LP, FP64 and the FP32 tableau with FP64 reinversion
        _lp("lp_8192", 8192, 8192),
        _lp("lp_8192_fp32", 8192, 8192, precision="fp32"),
        # many uneven LPs at once
        {"name": "batch_1024", "kind": "batch", "count": 1024, "lo": 32, "hi": 1024, "shapes": 0, "precision": "fp64"},
        # a burst of requests of mixed sizes to a running server
        {"name": "serve_64", "kind": "serve", "count": 64, "lo": 64, "hi": 4096, "shapes": 1, "precision": "fp64"},
        # the FP32 mode's body-refresh product as a library call
        {"name": "product", "kind": "product", "m": 7858, "n": 16385, "k": 334},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["lp", "batch", "serve", "product"], [8, 2, 1, 1])[0]
    if kind == "lp":
        family = rng.choices(["dense", "paper", "phase1"], [6, 2, 1])[0]
        lo, hi = {"dense": (48, 8192), "paper": (48, 720), "phase1": (48, 320)}[family]
        form = "primal" if family == "phase1" else rng.choice(["primal", "primal", "dual"])
        precision = "fp64" if family == "phase1" else rng.choice(["fp64", "fp64", "fp32"])
        return {"kind": "lp", "family": family, "m": _log(rng, lo, hi), "n": _log(rng, lo, hi), "form": form,
                "precision": precision, "memory": rng.choice(["device", "host", "pinned"])}
    if kind == "batch":
        return {"kind": "batch", "count": _log(rng, 16, 1024), "lo": 32, "hi": rng.randint(256, 1024),
                "shapes": rng.randrange(1 << 20), "precision": rng.choice(["fp64", "fp32"])}
    if kind == "serve":
        return {"kind": "serve", "count": rng.randint(8, 64), "lo": 64, "hi": rng.randint(512, 3000),
                "shapes": rng.randrange(1 << 20), "precision": rng.choice(["fp64", "fp32"])}
    return {"kind": "product", "m": _log(rng, 500, 7858), "n": _log(rng, 500, 16385), "k": _log(rng, 16, 334)}


# ----------------------------------------------------------------- inputs --

def _gen(seed, *more):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(np.random.SeedSequence([seed, *more]).generate_state(1)[0]))
    return g


def _dense(m, n, g):
    """Integer data: A in [1, 1000], b in [1000, 100000], c in [1, 100]."""
    def ints(lo, hi, shape):
        return torch.randint(lo, hi + 1, shape, generator=g, device=DEV).to(torch.float64)
    return ints(1, 1000, (m, n)), ints(1000, 100000, (m,)), ints(1, 100, (n,))


def _paper(m, n, g):
    """The paper's distribution: density 0.9, nonzeros uniform on (0, 50), a feasible point, objective row A'u."""
    def uni(*shape):
        return torch.rand(shape, generator=g, device=DEV, dtype=torch.float64)
    while True:
        A = torch.where(uni(m, n) < 0.9, 50.0 * uni(m, n), 0.0)
        b = A @ (10.0 * uni(n))
        r1, r2, r3, r4 = uni(m), uni(m), uni(m), uni(m)
        c = -(A.T @ torch.where(r1 > r2, r3 - r4, 0.0))
        if bool((c > 0).any()):
            return A, b, c


def _phase1(m, n, g):
    """A dense LP with a tenth of its rows turned into >= rows that the origin violates."""
    A, b, c = _dense(m, n, g)
    rs = A.sum(1)
    t = 0.5 * float((b / rs).min())
    rows = torch.randperm(m, generator=g, device=DEV)[:max(1, round(0.1 * m))]
    b[rows] = -0.5 * t * rs[rows]
    A[rows] = -A[rows]
    return A, b, c


def _data(case, seed):
    """(A, b, c) of the max form, on the device."""
    g = _gen(seed, 1)
    return {"dense": _dense, "paper": _paper, "phase1": _phase1}[case["family"]](case["m"], case["n"], g)


def _many(case, seed):
    shapes = lpgen.log_uniform_shapes(case["count"], case["lo"], case["hi"], case["shapes"])
    g = _gen(seed, 2)
    return [_dense(m, n, g) for m, n in shapes]


def _factors(case, seed):
    """The body refresh's factors: rows of the LP's own data, and the rows of the product X."""
    g = _gen(seed, 3)
    A = torch.randint(1, 1001, (case["m"], case["k"]), generator=g, device=DEV).to(torch.float64)
    return A, torch.randn((case["k"], case["n"]), generator=g, device=DEV, dtype=torch.float64)


class _Held:
    """A handle or a server that lives as long as the state that holds it."""

    def __init__(self, ptr, destroy):
        self.ptr, self.destroy = ptr, destroy

    def __del__(self):
        self.destroy(self.ptr)


def _opts(case):
    if case["precision"] == "fp32":
        return capi.lp_options_default(precision=capi.LP_FP32_REINV)
    return capi.lp_options_default()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "product":
        A, B = _factors(case, seed)
        return {"kind": kind, "A": A, "B": B, "C": torch.empty((case["m"], case["n"]), dtype=torch.float64, device=DEV)}
    if kind == "lp":
        A, b, c = _data(case, seed)
        if case["form"] == "dual":
            A, b, c = A.T.contiguous(), c, b
        if case["memory"] != "device":
            A, b, c = A.cpu(), b.cpu(), c.cpu()
            if case["memory"] == "pinned":
                A, b, c = A.pin_memory(), b.pin_memory(), c.pin_memory()
        torch.cuda.synchronize()  # the handle works on a stream of its own
        h = _Held(capi.lp_create(_opts(case)), capi.lp_destroy)
        return {"kind": kind, "h": h, "A": A, "b": b, "c": c,
                "sense": capi.LP_MIN_GE if case["form"] == "dual" else capi.LP_MAX_LE}
    lps = _many(case, seed)
    torch.cuda.synchronize()
    if kind == "batch":
        return {"kind": kind, "lps": [(A, b, c, capi.LP_MAX_LE) for A, b, c in lps], "opt": _opts(case)}
    lps = [tuple(t.cpu().numpy() for t in lp) for lp in lps]
    srv = _Held(capi.lp_server_create(_opts(case), hbm_budget_bytes=16 << 30, max_slots=256), capi.lp_server_destroy)
    return {"kind": kind, "srv": srv, "lps": lps}


# -------------------------------------------------------------------- run --

def run(s):
    if s["kind"] == "product":
        capi.lp_dgemm_emulated(s["A"], s["B"], s["C"])
        return {"C": s["C"]}
    if s["kind"] == "lp":
        h = s["h"].ptr
        capi.lp_load(h, s["A"], s["b"], s["c"], s["sense"])
        capi.lp_solve(h)
        x, y = np.empty(s["A"].shape[1]), np.empty(s["A"].shape[0])
        obj, status, iters = capi.lp_result(h, x, y)
        return {"x": x, "y": y, "obj": obj, "status": status, "iters": iters}
    if s["kind"] == "batch":
        obj, status, iters, xs, ys = capi.lp_solve_batch(s["lps"], s["opt"], want_xy=True)
    else:
        tickets = [capi.lp_server_submit(s["srv"].ptr, *lp) for lp in s["lps"]]
        got = [capi.lp_server_wait(s["srv"].ptr, t, lp[0].shape[0], lp[0].shape[1]) for t, lp in zip(tickets, s["lps"])]
        obj, status, iters = (np.array([r[k] for r in got]) for k in range(3))
        xs, ys = [r[3] for r in got], [r[4] for r in got]
    return {"x": np.concatenate(xs), "y": np.concatenate(ys), "obj": obj, "status": status, "iters": iters}


# ------------------------------------------------------------------- work --

def _pivots(m, n, family):
    """About how many pivots the family's LPs take (the method needs them; their number depends on the data)."""
    s = math.sqrt(m * n)
    return {"dense": 15.0 * (s / 64.0) ** 0.55, "paper": 1.4 * s, "phase1": 5.0 * s}[family]


def _lp_work(m, n, family):
    """Inputs read and results written once; per pivot one multiply-add for each entry of the rows' structural columns and
    the rhs (the columns of the slacks that stay basic never change)."""
    return 8.0 * (m * n + 2 * m + 2 * n + 1), 2.0 * _pivots(m, n, family) * (m + 1) * (n + 1)


def work(case):
    if case["kind"] == "product":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": 8.0 * (m * k + k * n + m * n), "flops": 2.0 * m * n * k}
    if case["kind"] == "lp":
        every = [_lp_work(case["m"], case["n"], case["family"])]
    else:
        every = [_lp_work(m, n, "dense")
                 for m, n in lpgen.log_uniform_shapes(case["count"], case["lo"], case["hi"], case["shapes"])]
    return {"bytes": sum(w[0] for w in every), "flops": sum(w[1] for w in every)}


# ------------------------------------------------------------------ exact --

def _rule(T, basis, dual, eps_d, eps_p, eps_r):
    """Pivot the tableau T in place to the end of the primal or the dual rule."""
    m = T.shape[0] - 1
    for _ in range(20 * (T.shape[1] + 50)):
        if dual:
            p = int(torch.argmin(T[:m, -1]))
            if float(T[p, -1]) >= -eps_r:
                return
            row = T[p, :-1]
            q = int(torch.argmin(torch.where(row < -eps_p, T[m, :-1].clamp_min(0.0) / -row, math.inf)))
        else:
            q = int(torch.argmin(T[m, :-1]))
            if float(T[m, q]) >= -eps_d:
                return
            col = T[:m, q]
            p = int(torch.argmin(torch.where(col > eps_p, T[:m, -1].clamp_min(0.0) / col, math.inf)))
        prow = T[p] / T[p, q]
        T.addr_(T[:, q].clone(), prow, alpha=-1.0)
        T[p] = prow
        basis[p] = q
    raise RuntimeError("no end of the pivots")


def _optimum(A, b, c):
    """(x, y, obj) of max c'x, Ax <= b, x >= 0 in 64 bits: tableau pivots find the basis, two solves and a refinement step
    give its solution."""
    m, n = A.shape
    T = torch.zeros((m + 1, n + m + 1), dtype=torch.float64, device=A.device)
    T[:m, :n], T[:m, -1] = A, b
    T[:m, n:n + m].fill_diagonal_(1.0)
    eps = [1e-9 * max(1.0, float(v.abs().max())) for v in (c, A, b)]
    basis = torch.arange(n, n + m, device=A.device)
    if bool((b < 0).any()):
        # any objective row >= 0 steers Phase 1 to a feasible basis: one without ties
        T[m, :n] = torch.linspace(1.0, 2.0, n, dtype=torch.float64, device=A.device)
        _rule(T, basis, True, *eps)
        cb = torch.where(basis < n, c[basis.clamp_max(n - 1)], 0.0)
        T[m] = cb @ T[:m]
        T[m, :n] -= c
    else:
        T[m, :n] = -c
    _rule(T, basis, False, *eps)
    del T
    # the structural basics S over the rows R whose slack is not basic
    S = basis[basis < n]
    free = torch.ones(m, dtype=torch.bool, device=A.device)
    free[basis[basis >= n] - n] = False
    x, y = torch.zeros_like(c), torch.zeros_like(b)
    if S.numel():
        K = A[free][:, S]

        def solve(M, r):
            v = torch.linalg.solve(M, r)
            return v + torch.linalg.solve(M, r - M @ v)
        x[S] = solve(K, b[free])
        y[free] = solve(K.T.contiguous(), c[S])
    return x.cpu().numpy(), y.cpu().numpy(), float(c @ x)


def exact(case, seed):
    if case["kind"] == "product":
        A, B = _factors(case, seed)
        return {"C": A @ B}
    if case["kind"] == "lp":
        x, y, obj = _optimum(*_data(case, seed))
        if case["form"] == "dual":
            x, y = y, x
    else:
        got = [_optimum(*lp) for lp in _many(case, seed)]
        x, y, obj = np.concatenate([r[0] for r in got]), np.concatenate([r[1] for r in got]), np.array([r[2] for r in got])
    return {"x": x, "y": y, "obj": obj, "status": None, "iters": None}
