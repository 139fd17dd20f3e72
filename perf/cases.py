"""The work that this solver's users have it do, as cases that can be timed and compared.

Each case is one call (or the few calls that belong together) through the public entry points:
``capi.Solver``, ``capi.admm_solve_noalloc``, ``capi.Batch`` with the C ABI's ``admm_batch_wait``,
``capi.Server`` and ``capi.quartic_min``.  Sizes and settings are those of the repository's
configurations, tests and benchmark: the plain n = 100 instance, the PHEV-shaped n = 1000, q = 50
instance, the plain n = 1e5, m = 4, q = 20 instance, batches and served controllers with n
log-uniform in [50, 5000], m in {2, 3, 4}, q in [1, 20], and the quartic benchmark of Sec. III-C.

Most solves run a fixed number of iterations (``max_iter`` below the count to convergence), as a
controller with a fixed time slot does; the smallest instance, the large batch and the served
requests run to the stop test.  Mixed-precision solves hold x in FP32, so their x is returned in
FP32 (the cast from the FP64 buffer of the interface is exact); FP64 solves return FP64.

``exact`` is the iteration (a)-(i) of App. A in plain torch FP64.
"""
import ctypes
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1903_10041_gb300 import capi
from paper_1903_10041_gb300 import workloads as W

ABI = ctypes.CDLL(capi.LIB_PATH)
ABI.admm_batch_wait.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.POINTER(capi.admm_result)]
ABI.admm_batch_wait.restype = ctypes.c_int


def listed():
    return [
        # One small controller solved to the stop test, over and over: launches and latency count.
        {"name": "plain_n100_fp64", "kind": "single", "recipe": "plain", "n": 100, "m": 2, "q": 1,
         "precision": "fp64", "iters": 5000, "rho2": 1.0, "adapt": False},
        # The paper's robust PHEV problem in the reference precision.
        {"name": "phev_n1000_q50_fp64", "kind": "single", "recipe": "phev", "n": 1000, "m": 2, "q": 50,
         "precision": "fp64", "iters": 300, "rho2": 0.001, "adapt": False},
        # A control loop that may not allocate: odd sizes, the state in the caller's buffers, penalties adapted.
        {"name": "noalloc_n4099_q7_fp64", "kind": "noalloc", "recipe": "plain", "n": 4099, "m": 3, "q": 7,
         "precision": "fp64", "iters": 200, "rho2": 1.0 / 4099, "adapt": True},
        # The same PHEV problem in mixed precision: little work per iteration, so what is around it counts.
        {"name": "phev_n1000_q50_mixed", "kind": "single", "recipe": "phev", "n": 1000, "m": 2, "q": 50,
         "precision": "mixed", "iters": 400, "rho2": 0.001, "adapt": False},
        # The large single instance (8e6 elements), larger than the caches.
        {"name": "plain_n1e5_q20_mixed", "kind": "single", "recipe": "plain", "n": 100000, "m": 4, "q": 20,
         "precision": "mixed", "iters": 60, "rho2": 1e-5, "adapt": False},
        # More sources than four, odd sizes, cost and loss maps shared by the scenarios.
        {"name": "shared_n10007_m6_mixed", "kind": "single", "recipe": "shared", "n": 10007, "m": 6, "q": 11,
         "precision": "mixed", "iters": 100, "rho2": 1.0 / 10007, "adapt": True},
        # A batch with the default launch configuration (8 warps per CTA, no clusters) and a fixed iteration budget.
        {"name": "batch_600", "kind": "batch", "count": 600, "shapes": 7, "iters": 100, "adapt": False, "warps": 8,
         "cluster": 1, "cluster_min": 131072},
        # The benchmark's batch, solved to the stop test with the launch configuration its autotuner picks.
        {"name": "batch_4096", "kind": "batch", "count": 4096, "shapes": 1903, "iters": 5000, "adapt": True, "warps": 16,
         "cluster": 2, "cluster_min": 250000},
        # A burst of one-off requests to the server, each solved to the stop test; host data in, x out.
        {"name": "serve_48", "kind": "serve", "count": 48, "shapes": 5, "n_max": 600, "warps": 16},
        # The quartic benchmark (Sec. III-C): a call that is all latency, FP64, and the large FP32 one.
        {"name": "quartic_1000_f32", "kind": "quartic", "count": 1000, "precision": "fp32", "mode": "exact"},
        {"name": "quartic_1e6_f64", "kind": "quartic", "count": 1000003, "precision": "fp64", "mode": "exact"},
        {"name": "quartic_2p26_f32", "kind": "quartic", "count": 1 << 26, "precision": "fp32", "mode": "exact"},
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(["single", "single", "single", "noalloc", "batch", "batch", "serve", "quartic", "quartic"])
    if kind == "quartic":
        prec = rng.choice(["fp32", "fp64"])
        return {"kind": kind, "count": _log(rng, 1, 1 << (26 if prec == "fp32" else 23)), "precision": prec,
                "mode": rng.choice(["exact", "exact", "paper"])}
    if kind == "batch":
        return {"kind": kind, "count": _log(rng, 2, 1024), "shapes": rng.randrange(10000), "iters": rng.randint(40, 160),
                "adapt": rng.random() < 0.5, "warps": rng.choice([8, 16]), "cluster": rng.choice([1, 2, 8]),
                "cluster_min": rng.choice([32768, 250000])}
    if kind == "serve":
        return {"kind": kind, "count": rng.randint(4, 64), "shapes": rng.randrange(10000),
                "n_max": _log(rng, 100, 1000), "warps": rng.choice([8, 16])}
    recipe = rng.choice(["plain", "plain", "phev", "shared"]) if kind == "single" else rng.choice(["plain", "phev"])
    prec = rng.choice(["fp64", "mixed"]) if kind == "single" else "fp64"
    m = 2 if recipe == "phev" else rng.choice([1, 2, 2, 3, 4, 4, 6, 8])
    q = _log(rng, 1, 100)
    most = 8_000_000 if prec == "mixed" else 1_000_000
    n = _log(rng, 30, max(40, min(100_000, most // (m * q))))
    return {"kind": kind, "recipe": recipe, "n": n, "m": m, "q": q, "precision": prec, "iters": rng.randint(40, 120),
            "rho2": 1.0 / n, "adapt": rng.random() < 0.5}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(1903 + 7919 * int(seed) + salt)
    return g


def _uniform(g, shape, a, b):
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) * (b - a) + a


def _problem(case, seed):
    """One instance on the GPU, drawn by the recipes of the repository's workloads."""
    g = _gen(seed)
    n, m, q, recipe = case["n"], case["m"], case["q"], case["recipe"]
    sh = (m, n) if recipe == "shared" else (m, q, n)
    zero = torch.zeros(sh, device="cuda", dtype=torch.float64)
    if recipe == "phev":
        f2, f1, g2, g1 = zero.clone(), zero.clone(), zero.clone(), zero.clone()
        f2[0] = _uniform(g, (q, n), 0.1, 1.0)
        f1[0] = _uniform(g, (q, n), -1.0, 1.0)
        g2[1] = _uniform(g, (q, n), 0.01, 0.1)
        g1[1] = 1.0
        lo = torch.tensor([[0.0], [-1.0]], device="cuda", dtype=torch.float64).expand(2, n).contiguous()
        hi = torch.tensor([[3.0], [1.0]], device="cuda", dtype=torch.float64).expand(2, n).contiguous()
        k = torch.arange(n, device="cuda", dtype=torch.float64)
        amp, per, pha = _uniform(g, (3, 1), 0.0, 0.8 / 3), _uniform(g, (3, 1), 50.0, 500.0), _uniform(g, (3, 1), 0.0, 2 * math.pi)
        y = 1.0 + (amp * torch.sin(2 * math.pi * k / per + pha)).sum(0) + 0.1 * torch.randn(
            (q, n), generator=g, device="cuda", dtype=torch.float64)
        c = torch.tensor([math.inf, 0.3 * n], device="cuda", dtype=torch.float64)
    else:
        f2, f1, g2 = _uniform(g, sh, 0.1, 1.0), _uniform(g, sh, -1.0, 1.0), _uniform(g, sh, 0.01, 0.1)
        g1 = torch.ones_like(zero)
        lo = torch.full((m, n), -1.0, device="cuda", dtype=torch.float64)
        hi = torch.full((m, n), 2.0, device="cuda", dtype=torch.float64)
        y = _uniform(g, (q, n), 0.5, 2.0)
        tot = (4.0 * g2 + 2.0 * g1).sum(-1)
        c = 0.6 * (tot if recipe == "shared" else tot.amin(1))
    return SimpleNamespace(n=n, m=m, q=q, f2=f2, f1=f1, f0=zero, g2=g2, g1=g1, g0=zero.clone(), lo=lo, hi=hi,
                           y=y.contiguous(), c=c.contiguous(), coef_shared=recipe == "shared")


def _shapes(case):
    """(n, m, q) of the instances: n log-uniform in [50, n_max], m in {2, 3, 4}, q in [1, 20]."""
    rs = np.random.RandomState(case["shapes"])
    top = case.get("n_max", 5000)
    return [(int(round(math.exp(rs.uniform(math.log(50.0), math.log(top))))), 2 + rs.randint(3), 1 + rs.randint(20))
            for _ in range(case["count"])]


def _many(case, seed):
    """Instances of the batched recipe in host memory, with the per-element distributions of the
    repository's batched workload; the data of an instance are ranges of one random pool per array
    (quick to make however many there are)."""
    shapes = _shapes(case)
    rs = np.random.RandomState((1903 + 7919 * int(seed)) % (1 << 32))
    most = max(n * m * q for n, m, q in shapes)
    pool = most + most // 2 + 1000
    f2, f1, g2, y = rs.uniform(0.1, 1.0, pool), rs.uniform(-1.0, 1.0, pool), rs.uniform(0.01, 0.1, pool), rs.uniform(0.5, 2.0, pool)
    zero, one = np.zeros(most), np.ones(most)
    lo, hi = np.full(most, -1.0), np.full(most, 2.0)
    cum = np.concatenate([[0.0], np.cumsum(g2)])
    out = []
    for n, m, q in shapes:
        el = m * q * n
        o = [int(v) for v in rs.randint(0, pool - el + 1, 4)]
        rows = o[2] + n * np.arange(m * q + 1)
        tot = (4.0 * np.diff(cum[rows]) + 2.0 * n).reshape(m, q)
        out.append(SimpleNamespace(
            n=n, m=m, q=q, f2=f2[o[0]:o[0] + el].reshape(m, q, n), f1=f1[o[1]:o[1] + el].reshape(m, q, n),
            g2=g2[o[2]:o[2] + el].reshape(m, q, n), f0=zero[:el].reshape(m, q, n), g0=zero[:el].reshape(m, q, n),
            g1=one[:el].reshape(m, q, n), lo=lo[:m * n].reshape(m, n), hi=hi[:m * n].reshape(m, n),
            y=y[o[3]:o[3] + q * n].reshape(q, n), c=0.6 * tot.min(1), coef_shared=False))
    return out


def _quartics(case, seed):
    g = _gen(seed, 1)
    dt = torch.float32 if case["precision"] == "fp32" else torch.float64

    def u(a, b):
        return torch.rand(case["count"], generator=g, device="cuda", dtype=dt) * (b - a) + a

    A, B, C, D, mid, half = u(0.01, 2.0), u(-2.0, 2.0), u(-3.0, 3.0), u(-2.0, 2.0), u(-2.0, 2.0), u(0.0, 3.0)
    return A, B, C, D, mid - half, mid + half


def _params(case):
    return W.Params(rho=(1.0, case["rho2"], 1.0, 1.0), max_iter=case["iters"], precision=case["precision"],
                    adapt_rho=case["adapt"])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "quartic":
        a = _quartics(case, seed)
        return {"kind": kind, "case": case, "args": a, "out": torch.empty_like(a[0])}
    if kind == "batch":
        P = _many(case, seed)
        b = capi.Batch(P, W.Params(rho2_over_n=True, precision="mixed", adapt_rho=case["adapt"], max_iter=case["iters"]))
        b.set_config(warps_per_cta=case["warps"], cluster_size=case["cluster"], cluster_min_elements=case["cluster_min"])
        x = torch.zeros(sum(p.n * p.m * p.q for p in P), device="cuda", dtype=torch.float64)
        x1 = torch.zeros(sum(p.m for p in P), device="cuda", dtype=torch.float64)
        res = (capi.admm_result * len(P))()
        at = at1 = 0
        dp = ctypes.POINTER(ctypes.c_double)
        for r, p in zip(res, P):
            r.x = ctypes.cast(ctypes.c_void_p(x.data_ptr() + 8 * at), dp)
            r.x1 = ctypes.cast(ctypes.c_void_p(x1.data_ptr() + 8 * at1), dp)
            r.on_device = 1
            at, at1 = at + p.n * p.m * p.q, at1 + p.m
        return {"kind": kind, "batch": b, "x": x, "x1": x1, "res": res}
    if kind == "serve":
        P = _many(case, seed)
        s = capi.Server(W.Params(rho2_over_n=True, precision="mixed", adapt_rho=True, adapt_start=1000),
                        store_elements=1 << 23, max_active=256, warps_per_cta=case["warps"])
        return {"kind": kind, "server": s, "problems": P}
    P = _problem(case, seed)
    x = torch.empty((P.m, P.q, P.n), device="cuda", dtype=torch.float64)
    x1 = torch.empty(P.m, device="cuda", dtype=torch.float64)
    if kind == "single":
        return {"kind": kind, "fp64": case["precision"] == "fp64", "solver": capi.Solver(P, _params(case)), "x": x, "x1": x1}
    st = {"x": x, "x1": x1, "rho": [1.0] * 4, "cold": True}
    for k in ("s", "mu"):
        st[k] = torch.empty((P.q, P.n), device="cuda", dtype=torch.float64)
    for k in ("lam", "zeta", "h", "p", "nu"):
        st[k] = torch.empty((P.m, P.q), device="cuda", dtype=torch.float64)
    return {"kind": kind, "problem": P, "params": _params(case), "state": st}


def run(state):
    kind = state["kind"]
    if kind == "quartic":
        c = state["case"]
        return {"x": capi.quartic_min(*state["args"], mode=c["mode"], precision=c["precision"], out=state["out"])}
    if kind == "single":
        s = state["solver"]
        s.reset()
        r = s.solve(x_out=state["x"], x1_out=state["x1"])
        if state["fp64"]:
            return {"x": state["x"], "x1": state["x1"], "objective": r["objective"], "iters": r["iters"]}
        return {"x": state["x"].float(), "x1": state["x1"].float()}
    if kind == "noalloc":
        st = state["state"]
        st["cold"] = True
        r = capi.admm_solve_noalloc(state["problem"], state["params"], st)
        return {"x": st["x"], "s": st["s"], "mu": st["mu"], "x1": st["x1"], "objective": r["objective"], "iters": r["iters"]}
    if kind == "batch":
        b = state["batch"]
        b.reset()
        b.solve()
        rc = ABI.admm_batch_wait(b.h, None, state["res"])
        if rc not in (capi.ADMM_OK, capi.ADMM_ENOTCONVERGED):
            raise RuntimeError(capi.admm_last_error())
        return {"x": state["x"].float(), "x1": state["x1"].float()}
    s = state["server"]
    tickets = [s.submit(p) for p in state["problems"]]
    got = []
    for t in tickets:
        r = None
        while r is None:
            r = s.poll(t, wait_ms=1000, want_x=True)
        got.append(r)
    return {"x": np.concatenate([r["x"].ravel() for r in got]).astype(np.float32),
            "x1": np.concatenate([r["x1"] for r in got]).astype(np.float32)}


# ---------------------------------------------------------------------------
# work: an element update takes about 68 operations (step (a) with Algorithm 1 on the Cardano branch)
# and a column 5.  An instance (or a batch) that fits the caches is read once; a larger one streams
# its arrays in every iteration.
# ---------------------------------------------------------------------------
def _solve_work(sizes, iters, word, state_words, shared=False):
    el = sum(n * m * q for n, m, q in sizes)
    col = sum(n * q for n, m, q in sizes)
    bnd = sum(n * m for n, m, q in sizes)
    coef = bnd if shared else el
    once = word * (4 * coef + 2 * el + 2 * bnd + col + 4 * state_words * col)
    passes = iters if once > 128e6 else 1
    return {"bytes": float(once * passes), "flops": float((68 * el + 5 * col) * iters)}


def work(case):
    kind = case["kind"]
    if kind == "quartic":
        return {"bytes": float(7 * case["count"] * (4 if case["precision"] == "fp32" else 8)), "flops": float(60 * case["count"])}
    if kind in ("batch", "serve"):
        return _solve_work(_shapes(case), min(case.get("iters", 5000), 460), 4, 2)  # about 460 to the stop test
    iters = min(case["iters"], 1400)
    return _solve_work([(case["n"], case["m"], case["q"])], iters, 8 if case["precision"] == "fp64" else 4,
                       1 if case["precision"] == "fp64" else 2, case["recipe"] == "shared")


# ---------------------------------------------------------------------------
# the same numbers in plain torch FP64
# ---------------------------------------------------------------------------
def _polish(A, B, C, D, x, steps=3):
    for _ in range(steps):
        f = ((4 * A * x + 3 * B) * x + 2 * C) * x + D
        d = (12 * A * x + 6 * B) * x + 2 * C
        x = torch.where(d > 0, x - f / torch.where(d > 0, d, 1.0), x)
    return x


def _argmin(A, B, C, D, lo, hi, mode="exact"):
    """Algorithm 1 and the clamp: min of A x^4 + B x^3 + C x^2 + D x over [lo, hi]."""
    quad = A == 0
    a = torch.where(quad, 1.0, A)
    b, c, d = 0.75 * B / a, 0.5 * C / a, 0.25 * D / a
    Q, R = c / 3 - b * b / 9, b * c / 6 - b ** 3 / 27 - d / 2
    disc = Q ** 3 + R * R
    sq = disc.clamp(min=0).sqrt()
    v = torch.where(R >= 0, R + sq, R - sq)
    S = torch.sign(v) * v.abs().pow(1.0 / 3.0)
    one = S + torch.where(S != 0, -Q / torch.where(S != 0, S, 1.0), 0.0) - b / 3
    nq = (-Q).clamp(min=0)
    t = torch.acos((R / torch.where(nq > 0, nq, 1.0).pow(1.5)).clamp(-1, 1)) / 3
    hi3 = _polish(A, B, C, D, 2 * nq.sqrt() * torch.cos(t) - b / 3)
    lo3 = _polish(A, B, C, D, 2 * nq.sqrt() * torch.cos(t + 2 * math.pi / 3) - b / 3)

    def value(x):
        return (((A * x + B) * x + C) * x + D) * x

    def clamp(x):
        return torch.minimum(torch.maximum(x, lo), hi)

    if mode == "exact":
        hi3, lo3 = clamp(hi3), clamp(lo3)
    three = clamp(torch.where(value(lo3) > value(hi3), hi3, lo3))
    best = torch.where(disc > 0, clamp(_polish(A, B, C, D, one)), three)
    return torch.where(quad, clamp(-D / (2 * torch.where(quad, C, 1.0))), best)


def _admm(P, rho, iters, r_tol=1e-6, s_tol=1e-6, s_margin=1.0, adapt=False, tau=1.1, check_every=10):
    """The iteration (a)-(i) of App. A from zeros, Gauss-Seidel over the sources, in FP64."""
    n, m, q = P.n, P.m, P.q
    put = lambda a: torch.as_tensor(a, dtype=torch.float64, device="cuda")  # noqa: E731
    coef = [put(a) for a in (P.f2, P.f1, P.f0, P.g2, P.g1, P.g0)]
    if P.coef_shared:
        coef = [a[:, None, :].expand(m, q, n) for a in coef]
    f2, f1, f0, g2, g1, g0 = coef
    lo, hi, y, c = put(P.lo)[:, None, :], put(P.hi)[:, None, :], put(P.y), put(P.c)[:, None]
    rho = [float(v) for v in rho]
    x = torch.minimum(torch.maximum(torch.zeros((m, q, n), dtype=torch.float64, device="cuda"), lo), hi)
    s, mu = torch.zeros_like(y), torch.zeros_like(y)
    lam, zeta, h, p, nu = (torch.zeros((m, q), dtype=torch.float64, device="cuda") for _ in range(5))
    x1 = torch.zeros(m, dtype=torch.float64, device="cuda")
    sum0, cold, it = g0.sum(-1), True, 0
    for it in range(1, iters + 1):
        old = x.clone()
        for i in range(m):
            xo = old[i]
            phi = s - (x.sum(0) - x[i]) + y + mu
            u = -g0[i] if cold else (g2[i] * xo + g1[i]) * xo + (zeta + lam)[i][:, None]
            A = 0.5 * rho[0] * g2[i] ** 2
            B = rho[0] * g2[i] * g1[i]
            C = f2[i] / q + 0.5 * rho[2] + 0.5 * rho[0] * (g1[i] ** 2 - 2 * g2[i] * u)
            D = f1[i] / q - rho[2] * phi - rho[0] * g1[i] * u
            C[:, 0] += 0.5 * rho[3]
            D[:, 0] -= rho[3] * (x1[i] + nu[i])
            x[i] = _argmin(A, B, C, D, lo[i], hi[i])
        sx, so, muo = x.sum(0), s, mu
        s = (sx - y - mu).clamp(min=0)
        mu = mu + s - sx + y
        gx = (g2 * x + g1) * x
        w = gx.sum(-1) + sum0 - n * lam
        kap = rho[1] / (rho[0] + n * rho[1])
        lamn = kap * (h + p - w)
        z = w + n * lamn
        hn = torch.minimum(z - p, c)
        p = p + hn - z
        x0 = x[:, :, 0]
        x1 = (x0 - nu).mean(1)
        nu = nu + x1[:, None] - x0
        dl = lamn - lam - zeta
        if it % check_every == 0 or it == iters:
            dk = gx + g0 if cold else gx - (g2 * old + g1) * old
            r = max(float(v) for v in ((mu - muo).abs().max(), (lamn - lam).abs().max(), (hn - z).abs().max(),
                                       (x0 - x1[:, None]).abs().max()))
            sg = max(rho[0] * float((dk + dl[:, :, None]).abs().max()), rho[1] * float((hn - h).abs().max()),
                     rho[2] * float((s - so - (x - old).sum(0)).abs().max()))
        zeta, lam, h, cold = lamn - lam, lamn, hn, False
        if it % check_every == 0 or it == iters:
            if r < r_tol and sg < s_margin * s_tol:
                break
            ratio, target = r / sg, r_tol / s_tol
            f = tau if ratio > 1.2 * target else 1 / tau if ratio < 0.8 * target else 1.0
            if adapt and it < iters and f != 1.0:
                lam, p, nu, mu = lam / f, p / f, nu / f, mu / f
                rho = [v * f for v in rho]
    return {"x": x, "s": s, "mu": mu, "x1": x1, "objective": float(((f2 * x + f1) * x + f0).sum() / q), "iters": it}


def exact(case, seed):
    kind = case["kind"]
    if kind == "quartic":
        a = _quartics(case, seed)
        parts = [_argmin(*(v[o:o + (1 << 22)].double() for v in a), mode=case["mode"]) for o in range(0, case["count"], 1 << 22)]
        return {"x": torch.cat(parts)}
    if kind == "serve":
        return None  # thousands of iterations of many instances
    if kind == "batch":
        if case["count"] * case["iters"] > 20000:
            return None
        got = [_admm(p, (1.0, 1.0 / p.n, 1.0, 1.0), case["iters"], s_margin=0.85, adapt=case["adapt"])
               for p in _many(case, seed)]
        return {"x": torch.cat([r["x"].ravel() for r in got]), "x1": torch.cat([r["x1"] for r in got])}
    fp64 = case["precision"] == "fp64"
    r = _admm(_problem(case, seed), (1.0, case["rho2"], 1.0, 1.0), case["iters"], s_margin=1.0 if fp64 else 0.85,
              adapt=case["adapt"])
    keep = ("x", "x1", "objective", "iters") if kind == "single" else ("x", "s", "mu", "x1", "objective", "iters")
    return {k: r[k] for k in keep if fp64 or k in ("x", "x1")}
