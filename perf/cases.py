"""What is measured of this framework: one dict per case, `prepare` makes what a user's program
has in hand, `run` is one pass through the public binding, `work` is what that pass cannot do
without, and `exact` is the same result in plain 64-bit torch.

The kinds follow the calls of the library: the H-matvec, the Nystrom sketch, the preconditioner
applied to a block, a PCG solve, and whole NysADMM solves (lasso, l1-logistic, regularisation
path, batch).  Sizes are those of the repository's workloads and tests.

Results of an FP32-class call (BF16, FP32 or FP8 storage) are returned in FP32, the type such a
call computes in; the library hands some of them out in FP64 containers."""
import math

import torch

from paper_2202_11599_gb300 import nysadmm as nx

_T = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16, "fp8": torch.float8_e4m3fn}
_SIZE = {"f64": 8, "f32": 4, "bf16": 2, "fp8": 1}


def listed():
    return [
        # the smallest call: one H-matvec of the 2,000 x 500 FP64 lasso, all latency and launches
        {"name": "hmatvec_small", "kind": "hmatvec", "dtype": "f64", "n": 2000, "d": 500, "weighted": False},
        # the matvec every PCG step of the large mixed-precision lasso makes
        {"name": "hmatvec_bf16", "kind": "hmatvec", "dtype": "bf16", "n": 100000, "d": 10000, "weighted": False},
        # the plain FP64 form at the size of the stream of lasso instances, odd sizes, with a curvature D
        {"name": "hmatvec_f64", "kind": "hmatvec", "dtype": "f64", "n": 39999, "d": 4001, "weighted": True},
        # P^{-1} on the block of residuals that the 64 columns of a path hold
        {"name": "apply_block", "kind": "apply", "dtype": "f32", "d": 10000, "rank": 200, "k": 64},
        # set-up of the large mixed-precision lasso: the preconditioner of the BF16 copy
        {"name": "sketch_bf16", "kind": "sketch", "dtype": "bf16", "n": 100000, "d": 10000, "rank": 200, "weighted": False},
        # set-up of each instance of the FP64 stream
        {"name": "sketch_f64", "kind": "sketch", "dtype": "f64", "n": 40000, "d": 4000, "rank": 100, "weighted": False},
        # one x-subproblem of the large logistic regression: curvature D, FP32 storage
        {"name": "pcg_f32", "kind": "pcg", "dtype": "f32", "n": 200000, "d": 5000, "rank": 100, "weighted": True,
         "rho": 1.0, "tol": 1e-6},
        # the small FP64 lasso from start to end: latency-bound iterations
        {"name": "lasso_small", "kind": "lasso", "dtype": "f64", "inner": "f64", "n": 2000, "d": 500, "rank": 50,
         "rho": 1.0, "tol": 1e-8, "iters": 200, "steps": 0, "refresh": 0, "mixed": False},
        # the large mixed-precision lasso: FP64 problem matrix, BF16 copy in the loop.  Every other
        # iteration takes a PCG step, as the decaying schedule of the benchmark settles to.
        {"name": "lasso_large", "kind": "lasso", "dtype": "f64", "inner": "bf16", "n": 100000, "d": 10000, "rank": 200,
         "rho": 70.0, "tol": 1e-8, "iters": 60, "steps": 1, "refresh": 100, "mixed": True},
        # 64 points of a regularisation path sharing one FP32 matrix
        {"name": "path", "kind": "path", "dtype": "f32", "n": 50000, "d": 4000, "rank": 50, "rho": 100.0, "k": 64,
         "iters": 12, "steps": 2},
        # uneven independent FP32 instances in one call, d over [500, 4000], n = 10 d
        {"name": "batch", "kind": "batch", "dtype": "f32", "count": 8, "dmin": 500, "dmax": 4000, "rank": 50,
         "rho": 100.0, "iters": 20, "steps": 2},
        # l1-logistic regression: FP64 problem matrix, FP32 copy, curvature and sketch renewed in
        # every outer iteration, adaptive rank
        {"name": "logistic", "kind": "logistic", "dtype": "f64", "inner": "f32", "n": 200000, "d": 5000, "rank": 100,
         "rank_max": 400, "rho": 1.0, "tol": 1e-6, "iters": 6},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the kinds above over their whole range of sizes, odd ones among them."""
    kind = rng.choice(["hmatvec", "hmatvec", "apply", "sketch", "sketch", "pcg", "lasso", "path", "batch", "logistic"])
    if kind == "hmatvec":
        d = _log(rng, 300, 10000)
        return {"kind": kind, "dtype": rng.choice(["f64", "f32", "bf16", "fp8"]), "n": _log(rng, 1000, 100000),
                "d": d, "weighted": rng.random() < 0.4}
    if kind == "apply":
        d = _log(rng, 300, 10000)
        return {"kind": kind, "dtype": rng.choice(["f64", "f32"]), "d": d, "rank": min(d // 3, _log(rng, 20, 300)),
                "k": _log(rng, 1, 64)}
    if kind == "sketch":
        dt = rng.choice(["f64", "f32", "bf16"])
        d = _log(rng, 400, 4000 if dt == "f64" else 10000)
        n = _log(rng, 2000, 40000 if dt == "f64" else 100000)
        return {"kind": kind, "dtype": dt, "n": n, "d": d, "rank": min(d // 4, _log(rng, 20, 300)),
                "weighted": rng.random() < 0.4}
    if kind == "pcg":
        dt = rng.choice(["f32", "f64", "bf16"])
        n, d = _log(rng, 2000, 40000 if dt == "f64" else 150000), _log(rng, 400, 5000)
        return {"kind": kind, "dtype": dt, "n": n, "d": d, "rank": min(d // 4, _log(rng, 20, 150)),
                "weighted": rng.random() < 0.5, "rho": 1.0, "tol": 1e-8 if dt == "f64" else 1e-6}
    if kind == "lasso":
        if rng.random() < 0.5:
            n, d = _log(rng, 1000, 20000), _log(rng, 300, 2500)
            return {"kind": kind, "dtype": "f64", "inner": "f64", "n": n, "d": d, "rank": min(d // 5, 60), "rho": 1.0,
                    "tol": 1e-8, "iters": rng.randint(30, 120), "steps": 0, "refresh": 0, "mixed": False}
        n, d = _log(rng, 5000, 100000), _log(rng, 1000, 10000)
        return {"kind": kind, "dtype": "f64", "inner": rng.choice(["bf16", "f32"]), "n": n, "d": d,
                "rank": min(d // 5, _log(rng, 50, 200)), "rho": 70.0, "tol": 1e-8, "iters": rng.randint(20, 60),
                "steps": 1, "refresh": rng.choice([0, 20, 100]), "mixed": True}
    if kind == "path":
        n, d = _log(rng, 4000, 50000), _log(rng, 500, 4000)
        return {"kind": kind, "dtype": rng.choice(["f32", "bf16"]), "n": n, "d": d, "rank": 50, "rho": 100.0,
                "k": rng.randint(8, 64), "iters": rng.randint(4, 12), "steps": 2}
    if kind == "batch":
        lo = _log(rng, 300, 1000)
        return {"kind": kind, "dtype": rng.choice(["f32", "bf16"]), "count": rng.randint(2, 8), "dmin": lo,
                "dmax": lo + _log(rng, 200, 3000), "rank": 50, "rho": 100.0, "iters": rng.randint(8, 20), "steps": 2}
    n, d = _log(rng, 10000, 150000), _log(rng, 500, 5000)
    return {"kind": kind, "dtype": "f64", "inner": "f32", "n": n, "d": d, "rank": min(100, d // 8),
            "rank_max": min(400, d // 3), "rho": 1.0, "tol": 1e-6, "iters": rng.randint(3, 6)}


# ---------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _chunks(n, d):
    step = max(1, (1 << 27) // d)
    return [(r, min(n, r + step)) for r in range(0, n, step)]


def _values(n, d, g, power, rotate=False, scale=1.0):
    """A = G diag((1 + j)^-power) (times two Householder reflections when `rotate`), FP32."""
    cols = (1.0 + torch.arange(d, device="cuda", dtype=torch.float32)) ** -power * scale
    vs = []
    for _ in range(2 if rotate else 0):
        v = torch.randn(d, generator=g, device="cuda", dtype=torch.float32)
        vs.append(v / v.norm())
    out = torch.empty(n, d, device="cuda", dtype=torch.float32)
    for r0, r1 in _chunks(n, d):
        c = out[r0:r1]
        c.normal_(generator=g).mul_(cols)
        for v in vs:
            c.addr_(c @ v, v, alpha=-2.0)
    return out


def _store(a32, dtype):
    """The framework's matrix of these values; rows on 16-byte boundaries."""
    if dtype == "fp8":
        return nx.Matrix.fp8(a32)
    t = _T[dtype]
    vec = 16 // _SIZE[dtype]
    n, d = a32.shape
    if d % vec == 0:
        return nx.Matrix(a32 if t == torch.float32 else a32.to(t))
    return nx.Matrix.padded(a32, t)


def _omega(d, s, g):
    return torch.randn(d, s, generator=g, device="cuda", dtype=torch.float64)


def _mv(a32, x):
    """A x in FP64, by chunks of rows."""
    return torch.cat([a32[r0:r1].double() @ x for r0, r1 in _chunks(*a32.shape)])


def _mtv(a32, u):
    """A^T u in FP64, by chunks of rows."""
    y = torch.zeros(a32.shape[1], dtype=torch.float64, device="cuda")
    for r0, r1 in _chunks(*a32.shape):
        y += a32[r0:r1].double().T @ u[r0:r1]
    return y


def _planted(d, nnz, g, std=1.0):
    x = torch.zeros(d, dtype=torch.float64, device="cuda")
    at = torch.randperm(d, generator=g, device="cuda")[:nnz]
    x[at] = std * torch.randn(nnz, generator=g, device="cuda", dtype=torch.float64)
    return x


def _weights(n, g):
    """A logistic curvature sigma (1 - sigma), in (0, 1/4]."""
    s = torch.sigmoid(1.5 * torch.randn(n, generator=g, device="cuda", dtype=torch.float64))
    return s * (1.0 - s)


def _dims(case):
    k = max(1, case["count"] - 1)
    # uneven: spread over [dmin, dmax], odd sizes among them
    return [case["dmin"] + (case["dmax"] - case["dmin"]) * i // k + (i % 3 == 1) for i in range(case["count"])]


def _lasso_data(n, d, g, rotate=False, noise=1e-3, frac=0.05):
    a32 = _values(n, d, g, 1.0, rotate)
    b = _mv(a32, _planted(d, max(1, d // 100), g)) + noise * torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
    gamma = frac * float(_mtv(a32, b).abs().max())
    return a32, b, gamma


def _inputs(case, seed):
    """The data of a case before it is handed to the framework: plain tensors and numbers."""
    g = _gen(seed)
    kind = case["kind"]
    if kind in ("hmatvec", "sketch", "pcg"):
        n, d = case["n"], case["d"]
        power, scale = (0.5, 1.0 / math.sqrt(d)) if kind == "pcg" else (1.0, 1.0)
        s = {"a32": _values(n, d, g, power, rotate=kind == "sketch" and case["dtype"] != "f64", scale=scale)}
        s["D"] = _weights(n, g) if case["weighted"] else None
        if kind == "hmatvec":
            s["p"] = torch.randn(d, generator=g, device="cuda", dtype=torch.float64)
        if kind in ("sketch", "pcg"):
            s["Om"] = _omega(d, case["rank"], g)
        if kind == "sketch":
            s["V"] = torch.randn(d, 8, generator=g, device="cuda", dtype=torch.float64)
        if kind == "pcg":
            s["r"] = torch.randn(d, generator=g, device="cuda", dtype=torch.float64)
        if case["dtype"] != "f64":
            for k in ("p", "V", "r"):
                if k in s:
                    s[k] = s[k].float()
        return s
    if kind == "apply":
        d = case["d"]
        s = {"a32": _values(2 * d, d, g, 1.0), "Om": _omega(d, case["rank"], g),
             "V": torch.randn(d, case["k"], generator=g, device="cuda", dtype=torch.float64)}
        if case["dtype"] == "f32":
            s["V"] = s["V"].float()
        return s
    if kind == "lasso":
        noise, frac = (1e-3, 0.05) if case["mixed"] else (0.01, 0.1)
        a32, b, gamma = _lasso_data(case["n"], case["d"], g, rotate=case["mixed"], noise=noise, frac=frac)
        return {"a32": a32, "b": b, "gamma": gamma, "Om": _omega(case["d"], case["rank"], g)}
    if kind == "path":
        a32, b, gmax = _lasso_data(case["n"], case["d"], g, frac=1.0)
        k = case["k"]
        return {"a32": a32, "b": b, "gammas": [gmax * 10.0 ** (-3.0 + 3.0 * i / max(1, k - 1)) for i in range(k)],
                "Om": _omega(case["d"], case["rank"], g)}
    if kind == "batch":
        out = []
        for d in _dims(case):
            a32, b, gamma = _lasso_data(10 * d, d, g)
            out.append({"a32": a32, "b": b, "gamma": gamma, "Om": _omega(d, case["rank"], g)})
        return {"problems": out}
    # logistic: A = N(0, 1/d) diag((1 + j)^-1/2), labels sign(A x* + Logistic(0, 1))
    n, d = case["n"], case["d"]
    a32 = _values(n, d, g, 0.5, scale=1.0 / math.sqrt(d))
    u = torch.rand(n, generator=g, device="cuda", dtype=torch.float64).clamp(1e-12, 1 - 1e-12)
    b = torch.sign(_mv(a32, _planted(d, max(1, d // 50), g, 2.0)) + torch.log(u / (1 - u)))
    b[b == 0] = 1.0
    gamma = 0.05 * float(_mtv(a32, 0.5 - 0.5 * (1.0 + b)).abs().max())
    return {"a32": a32, "b": b, "gamma": gamma, "Om": _omega(d, case["rank_max"], g)}


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    kind = case["kind"]
    if kind == "batch":
        for p in s["problems"]:
            p["A"] = _store(p.pop("a32"), case["dtype"])
            p["rank"], p["Omega"] = case["rank"], p.pop("Om")
        return s
    a32 = s.pop("a32")
    if kind == "apply":
        s["P"] = nx.sketch(_store(a32, "f64"), s.pop("Om"))
        return s
    if case.get("inner", case["dtype"]) != case["dtype"]:
        s["Ain"] = _store(a32, case["inner"])
    s["A"] = _store(a32, case["dtype"])
    if kind == "pcg":
        s["P"] = nx.sketch(s["A"], s.pop("Om"), D=s["D"])
    return s


# ---------------------------------------------------------------- one pass
def _steps(case):
    """PCG steps of each ADMM iteration (None: the tolerance decides)."""
    if not case["steps"]:
        return None
    if case.get("mixed"):
        return [case["steps"] if k % 2 == 0 else 0 for k in range(case["iters"])]
    return [case["steps"]] * case["iters"]


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "hmatvec":
        return nx.hmatvec(state["A"], state["p"], 0.5, state["D"])
    if kind == "apply":
        return state["P"].apply(state["V"], 1.0)
    if kind == "sketch":
        P = nx.sketch(state["A"], state["Om"], D=state["D"])
        return {"lam": P.lam.to(state["A"].compute_dtype), "apply": P.apply(state["V"], 1.0)}
    if kind == "pcg":
        return nx.pcg_solve(state["A"], state["r"], c["rho"], state["P"], tol=c["tol"], D=state["D"], allow_noconv=True)[0]
    if kind == "lasso":
        kw = {"A_inner": state["Ain"], "refine": False} if "Ain" in state else {}
        out = nx.nysadmm_solve("lasso", state["A"], state["b"], state["gamma"], c["rho"], c["rank"], c["tol"], state["Om"],
                               admm_iters=c["iters"], pcg_fixed=_steps(c), hx_refresh=c["refresh"], **kw)
        t = state.get("Ain", state["A"]).compute_dtype
        return {"x": out["x"].to(t), "z": out["z"].to(t)}
    if kind == "path":
        out = nx.nysadmm_solve_path(state["A"], state["b"], state["gammas"], c["rho"], c["rank"], 1e-8, state["Om"],
                                    admm_iters=c["iters"], pcg_fixed=_steps(c))
        t = state["A"].compute_dtype
        return {"X": out["X"].to(t), "Z": out["Z"].to(t)}
    if kind == "batch":
        outs = nx.nysadmm_solve_batch(state["problems"], c["rho"], 1e-10, admm_iters=c["iters"], pcg_maxit=c["steps"],
                                      hx_refresh=10)
        return [{"x": o["x"].float(), "z": o["z"].float()} for o in outs]
    out = nx.nysadmm_solve("logistic", state["A"], state["b"], state["gamma"], c["rho"], c["rank"], c["tol"], state["Om"],
                           admm_iters=c["iters"], A_inner=state["Ain"], rank_max=c["rank_max"], ada_tol=2.0)
    return {"x": out["x"].float(), "z": out["z"].float()}


# ---------------------------------------------------------------- what a pass cannot do without
def _sketch_work(n, d, s, esz):
    # A once, Omega in, U and lam out; two products with A, and about 6 products of d x s panels
    # (orthonormalisation, Gram matrices, B, U) with the s x s eigenproblem
    return {"bytes": n * d * esz + 2 * d * s * 8, "flops": 4.0 * n * d * s + 12.0 * d * s * s + 30.0 * s ** 3}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        w = {"bytes": 0, "flops": 0.0}
        for d in _dims(case):
            n = 10 * d
            sk = _sketch_work(n, d, case["rank"], _SIZE[case["dtype"]])
            passes = 1 + case["iters"] * case["steps"]
            w["bytes"] += sk["bytes"] + passes * n * d * _SIZE[case["dtype"]]
            w["flops"] += sk["flops"] + passes * 4.0 * n * d
        return w
    d = case["d"]
    if kind == "apply":
        e = _SIZE[case["dtype"]]
        return {"bytes": d * case["rank"] * e + 2 * d * case["k"] * e, "flops": 4.0 * d * case["rank"] * case["k"]}
    n, esz = case["n"], _SIZE[case["dtype"]]
    if kind == "hmatvec":
        return {"bytes": n * d * esz + 2 * d * (8 if esz == 8 else 4) + (8 * n if case["weighted"] else 0), "flops": 4.0 * n * d}
    if kind == "sketch":
        return _sketch_work(n, d, case["rank"], esz)
    if kind == "pcg":
        # about six iterations reach the tolerance
        return {"bytes": 6 * n * d * esz, "flops": 6 * 4.0 * n * d}
    inner = _SIZE[case.get("inner", case["dtype"])]
    if kind == "lasso":
        sk = _sketch_work(n, d, case["rank"], inner)
        st = _steps(case)
        passes = sum(st) if st else 4 * case["iters"]
        return {"bytes": sk["bytes"] + n * d * esz + passes * n * d * inner, "flops": sk["flops"] + 2.0 * n * d + passes * 4.0 * n * d}
    if kind == "path":
        sk = _sketch_work(n, d, case["rank"], inner)
        passes = case["iters"] * (case["steps"] + 1) - 1
        return {"bytes": sk["bytes"] + (passes + 1) * n * d * esz, "flops": sk["flops"] + passes * 4.0 * n * d * case["k"]}
    sk = _sketch_work(n, d, case["rank"], inner)
    it = case["iters"]
    return {"bytes": it * (sk["bytes"] + n * d * esz + 5 * n * d * inner), "flops": it * (sk["flops"] + 6 * 4.0 * n * d)}


# ---------------------------------------------------------------- the same in 64 bits
def _stored(a32, dtype):
    """The stored values (by chunks) of a matrix of this type, as FP64."""
    if dtype == "fp8":
        scale = (a32.abs().amax(dim=0) / 448.0).clamp_min(torch.finfo(torch.float32).tiny)
        return lambda r0, r1: (a32[r0:r1] / scale).to(torch.float8_e4m3fn).double() * scale.double()
    t = _T[dtype]
    return lambda r0, r1: a32[r0:r1].to(t).double()


def _h_times(a32, dtype, D, X):
    """A^T D A X in FP64 for the stored values of A."""
    rows = _stored(a32, dtype)
    Y = torch.zeros_like(X)
    for r0, r1 in _chunks(*a32.shape):
        c = rows(r0, r1)
        t = c @ X
        if D is not None:
            t = t * (D[r0:r1] if t.dim() == 1 else D[r0:r1, None])
        Y += c.T @ t
    return Y


def _gram(a32, dtype, D=None):
    d = a32.shape[1]
    H = torch.zeros(d, d, dtype=torch.float64, device="cuda")
    rows = _stored(a32, dtype)
    for r0, r1 in _chunks(*a32.shape):
        c = rows(r0, r1)
        H += c.T @ (c if D is None else c * D[r0:r1, None])
    return H


def _nystrom(a32, dtype, D, Om):
    """(U, lam) of the randomized Nystrom approximation (App. B) from the Gaussian Om, in FP64.
    Matrices below FP64 take the orthonormal test matrix rounded to BF16 values and the shift of
    a 24-bit sketch."""
    d = a32.shape[1]
    Q, R = torch.linalg.qr(Om)
    Q = Q * torch.sign(torch.diagonal(R))
    bits = 52 if dtype == "f64" else 23
    if dtype != "f64":
        Q = Q.float().bfloat16().double()
    Y = _h_times(a32, dtype, D, Q)
    top = math.sqrt(float(torch.linalg.eigvalsh(Y.T @ Y)[-1]))
    nu = math.sqrt(d) * 2.0 ** (math.frexp(top)[1] - 1 - bits)
    Y = Y + nu * Q
    M = Q.T @ Y
    C = torch.linalg.cholesky(0.5 * (M + M.T)).T
    B = torch.linalg.solve_triangular(C, Y, upper=True, left=False)
    sig2, V = torch.linalg.eigh(B.T @ B)
    sig2, V = sig2.flip(0), V.flip(1)
    return B @ V / sig2.sqrt(), (sig2 - nu).clamp_min(0.0)


def _apply(U, lam, rho, V):
    V = V.double()
    return V + U @ (((lam[-1] + rho) / (lam + rho) - 1.0)[:, None] * (U.T @ V))


def _cg(mul, r, x, tol):
    """Conjugate gradients in FP64 from x to a relative residual `tol`."""
    w = r - mul(x)
    p, ww, stop = w.clone(), w @ w, (tol * float(r.norm())) ** 2
    for _ in range(400):
        if float(ww) <= stop:
            break
        v = mul(p)
        a = ww / (p @ v)
        x, w = x + a * p, w - a * v
        ww, old = w @ w, ww
        p = w + (ww / old) * p
    return x


def _soft(v, kappa):
    return torch.sign(v) * (v.abs() - kappa).clamp_min(0.0)


def _lasso_exact(a32, inner, b, gammas, rho, iters):
    """NysADMM's iteration with every x-step solved exactly (FP64 Cholesky)."""
    d, k = a32.shape[1], len(gammas)
    q = _mtv(a32, b)[:, None]
    H = _gram(a32, inner)
    H.diagonal().add_(rho)
    L = torch.linalg.cholesky(H)
    kap = torch.tensor(gammas, dtype=torch.float64, device="cuda")[None, :] / rho
    x = z = u = torch.zeros(d, k, dtype=torch.float64, device="cuda")
    for _ in range(iters):
        x = torch.cholesky_solve(q + rho * (z - u), L)
        z = _soft(x + u, kap)
        u = u + x - z
    return x, z


def exact(case, seed):
    kind = case["kind"]
    if kind == "lasso" and case["n"] * case["d"] ** 2 > 2e12:
        return None  # forming H or solving 60 systems by CG takes minutes in FP64
    s = _inputs(case, seed)
    if kind == "batch":
        out = []
        for p in s["problems"]:
            a32 = p["a32"] if case["dtype"] == "f32" else p["a32"].to(_T[case["dtype"]]).float()
            x, z = _lasso_exact(a32, "f32", p["b"], [p["gamma"]], case["rho"], case["iters"])
            out.append({"x": x[:, 0], "z": z[:, 0]})
        return out
    a32 = s["a32"]
    if kind == "hmatvec":
        p = s["p"].double()
        return _h_times(a32, case["dtype"], s["D"], p) + 0.5 * p
    if kind == "apply":
        return _apply(*_nystrom(a32, "f64", None, s["Om"]), 1.0, s["V"])
    if kind == "sketch":
        U, lam = _nystrom(a32, case["dtype"], s["D"], s["Om"])
        return {"lam": lam.cpu(), "apply": _apply(U, lam, 1.0, s["V"])}
    if kind == "pcg":
        r = s["r"].double()
        mul = lambda v: _h_times(a32, case["dtype"], s["D"], v) + case["rho"] * v  # noqa: E731
        return _cg(mul, r, torch.zeros_like(r), 1e-12)
    if kind == "lasso":
        x, z = _lasso_exact(a32, case["inner"], s["b"], [s["gamma"]], case["rho"], case["iters"])
        return {"x": x[:, 0], "z": z[:, 0]}
    if kind == "path":
        a = a32 if case["dtype"] == "f32" else a32.to(_T[case["dtype"]]).float()
        x, z = _lasso_exact(a, "f32", s["b"], s["gammas"], case["rho"], case["iters"])
        return {"X": x, "Z": z}
    # logistic (Sec. 3.2): every outer iteration's x-step by CG to 1e-10
    b, rho = s["b"], case["rho"]
    x = z = u = torch.zeros(case["d"], dtype=torch.float64, device="cuda")
    for _ in range(case["iters"]):
        t = _mv(a32, x)
        sg = torch.sigmoid(t)
        w = sg * (1.0 - sg)
        q = _mtv(a32, w * t + 0.5 * (1.0 + b) - sg)
        x = _cg(lambda v, w=w: _h_times(a32, "f32", w, v) + rho * v, q + rho * (z - u), x, 1e-10)
        z = _soft(x + u, s["gamma"] / rho)
        u = u + x - z
    return {"x": x, "z": z}
