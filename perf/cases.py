"""What a program that trains and serves SP-SVM models spends its GPU time on,
as cases: whole fits, and the single steps a fit or a prediction is made of,
each through the entry point that a program calls.

The inputs are the repository's workloads: the two-Gaussian problem (n = 2,000,
d = 20, |J| = 100), the MNIST-like sparse features (n = 100,000, d = 784), the
Gaussian mixture (n = 500,000, d = 128, |J| to 4,096), its overlapping form
(component means drawn at 0.3, about 40% of the points active), the subproblems
of the one-vs-rest grid (n 5,000 .. 60,000, |J| 256 .. 2,048) and the serving
stream's requests (1,000 .. 100,000 queries).

Some entry points return FP64 buffers of sums whose terms and partial sums are
FP32 by the library's contract (scores, masked sums, Newton matrix, beta):
those are handed on in FP32, the precision they carry; so is the Newton solve's
direction, which its backward error leaves undetermined below that.
"""
import math

import numpy as np
import torch

import paper_1404_1066_gb300 as sp

DEV = "cuda"


def listed():
    return [
        # a small fit on a fixed random basis in the default form: the Adult-scale
        # two-Gaussian problem, where latency, launches and host reads count
        {"name": "fit_small", "kind": "fit", "data": "two_gaussians", "n": 2000, "d": 20, "m": 100,
         "grow": False, "precision": "fp32", "queries": 1000},
        # a grown fit and the prediction with it: the mixture workload at the
        # serving stream's size, basis appended 64 at a time from 256 candidates
        {"name": "fit_grow", "kind": "fit", "data": "mixture", "n": 100_000, "d": 128, "m": 512,
         "grow": True, "precision": "bf16split", "queries": 20_000},
        # one round's 64 appended kernel rows in each arithmetic form
        {"name": "block_fp32", "kind": "block", "n": 100_000, "d": 784, "m": 64, "precision": "fp32"},
        {"name": "block_split", "kind": "block", "n": 500_000, "d": 128, "m": 64, "precision": "bf16split"},
        # one round's candidate scores
        {"name": "score_split", "kind": "score", "n": 500_000, "d": 128, "m": 256, "precision": "bf16split"},
        # the Newton direction's forward product and line search: a one-vs-rest
        # subproblem, and the full mixture with its whole basis
        {"name": "direction_mid", "kind": "direction", "n": 30_000, "d": 128, "m": 1024},
        {"name": "direction_large", "kind": "direction", "n": 500_000, "d": 128, "m": 4096},
        # the Newton system of the active set (compaction, masked gradient sums,
        # Gram matrix): overlapping mixture in the split form, a one-vs-rest
        # subproblem in the FP32 form
        {"name": "system_split", "kind": "system", "n": 200_000, "d": 128, "m": 2048, "active": 0.43,
         "precision": "bf16split"},
        {"name": "system_fp32", "kind": "system", "n": 60_000, "d": 256, "m": 1024, "active": 0.3,
         "precision": "fp32"},
        # the Newton solve at the largest basis
        {"name": "solve", "kind": "solve", "n": 20_000, "d": 784, "m": 4096},
        # decision values: a small serving request in the default form, and the
        # benchmark's 100,000 queries in the split form
        {"name": "predict_fp32", "kind": "predict", "n": 1000, "d": 784, "m": 512, "precision": "fp32"},
        {"name": "predict_split", "kind": "predict", "n": 100_000, "d": 128, "m": 4096,
         "precision": "bf16split"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fit", "block", "score", "direction", "system", "solve", "predict"])
    d = rng.choice([20, 32, 54, 128, 256, 784, rng.randint(3, 400)])
    precision = rng.choice(["fp32", "bf16split"])
    if kind == "fit":
        n = _log_int(rng, 1000, 60_000)
        m = min(_log_int(rng, 50, 400), n // 8)
        # a fixed basis where the classes overlap: the separated mixture leaves its beta to rounding
        data = rng.choice(["two_gaussians", "mixture", "overlap"])
        return {"kind": kind, "data": data, "n": n, "d": rng.choice([20, 32, 54, 128, 256]), "m": m,
                "grow": data == "mixture" or rng.random() < 0.4, "precision": precision,
                "queries": _log_int(rng, 1000, 20_000)}
    if kind in ("block", "score"):
        n = _log_int(rng, 2000, 500_000)
        hi = 1024 if kind == "block" else 256
        m = max(1, min(_log_int(rng, 16, hi), int(2e10 / (n * d))))
        return {"kind": kind, "n": n, "d": d, "m": m, "precision": precision}
    if kind == "direction":
        n = _log_int(rng, 2000, 500_000)
        return {"kind": kind, "n": n, "d": 128, "m": max(64, min(_log_int(rng, 64, 4096), n // 2))}
    if kind == "system":
        n = _log_int(rng, 2000, 200_000)
        m = min(_log_int(rng, 64, 2048 if precision == "bf16split" else 1024), n // 2)
        return {"kind": kind, "n": n, "d": d, "m": m,
                "active": math.exp(rng.uniform(math.log(0.004), math.log(0.5))), "precision": precision}
    if kind == "solve":
        m = _log_int(rng, 64, 4096)
        return {"kind": kind, "n": 5 * m, "d": 784, "m": m}
    n = _log_int(rng, 1000, 100_000)
    m = max(1, min(_log_int(rng, 64, 4096), int((5e10 if precision == "bf16split" else 1e10) / (n * d))))
    return {"kind": kind, "n": n, "d": d, "m": m, "precision": precision}


# ---- inputs ----------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) + 1)
    return g


def _points(case, g, count):
    """`count` points and their labels (two classes), FP32, and gamma."""
    d = case["d"]
    data = case.get("data") or ("sparse" if d == 784 else "mixture")
    r = lambda *s: torch.randn(*s, generator=g, device=DEV)  # noqa: E731
    u = lambda *s: torch.rand(*s, generator=g, device=DEV)  # noqa: E731
    if data == "sparse":   # MNIST-like: 0 with probability 0.8, else uniform; variance 0.2/3 - 0.01
        X = torch.where(u(count, d) < 0.8, 0.0, 1.0 - u(count, d))
        y = torch.where(u(count) < 0.5, 1.0, -1.0)
        return X, y, 1.0 / (d * (0.2 / 3 - 0.01))
    if data == "two_gaussians":
        comp = u(count) < 0.5
        y = torch.where(comp, 1.0, -1.0)
        X = r(count, d) + 0.5 * y[:, None]
        y = torch.where(u(count) < 0.05, -y, y)
        return X, y, 1.0 / d
    mu = r(10, d) * (0.3 if data == "overlap" else 1.0)
    s = 0.5 + 1.5 * u(10)
    comp = torch.randint(0, 10, (count,), generator=g, device=DEV)
    X = mu[comp] + s[comp, None] * r(count, d)
    return X, torch.where(comp % 2 == 0, 1.0, -1.0), 1.0 / d


def _mid_outputs(y, g):
    """Outputs of a model part of the way through its fit: margins around 1."""
    return y * (1.0 + 0.4 * torch.randn(y.shape[0], generator=g, device=DEV))


def _pick(n, m, g):
    return torch.randperm(n, generator=g, device=DEV)[:m].contiguous()


def _kernel_rows(X, J, gamma, out):
    """out[j] = k(x_J[j], X) in FP32, a few hundred rows at a time."""
    sq = (X * X).sum(1)
    for c in range(0, len(J), 256):
        z = X[J[c:c + 256]]
        d2 = (z * z).sum(1)[:, None] + sq[None, :] - 2.0 * (z @ X.T)
        out[c:c + 256] = torch.exp(-gamma * d2.clamp_min_(0.0))
    return out


def _stored(case, seed):
    """A stored kernel matrix with labels, outputs and the basis."""
    g = _gen(seed)
    n, m = case["n"], case["m"]
    X, y, gamma = _points(case, g, n)
    J = _pick(n, m, g)
    ld = (n + 127) // 128 * 128
    K = torch.zeros((m, ld), dtype=torch.float32, device=DEV)
    _kernel_rows(X, J, gamma, K[:, :n])
    return g, K, y, J, ld


def _kmat(K, n, precision="fp32"):
    m, ld = K.shape
    return sp.KMat(K, sp.SPSVM_FP32, n, m, ld, 0)


def _fit_inputs(case, seed):
    g = _gen(seed)
    n, q = case["n"], case["queries"]
    X, y, gamma = _points(case, g, n + q)
    basis = None if case["grow"] else torch.sort(_pick(n, case["m"], g))[0]
    return X[:n].contiguous(), y[:n].contiguous(), X[n:].contiguous(), gamma, basis


FIT_LAMBDA = {"two_gaussians": 1e-3, "mixture": 1e-4, "overlap": 1e-3}


def _block_inputs(case, seed):
    g = _gen(seed)
    X, y, gamma = _points(case, g, case["n"])
    return X, y, gamma, _pick(case["n"], case["m"], g), g


def _direction_inputs(case, seed):
    """A descent direction scaled to the minimum of the current quadratic
    piece, as a Newton step's is: the search ends near t = 1."""
    g, K, y, J, ld = _stored(case, seed)
    n = case["n"]
    o = _mid_outputs(y, g)
    r = torch.where(y * o < 1.0, o - y, 0.0)
    v = torch.zeros(case["m"], dtype=torch.float64, device=DEV)
    u = torch.zeros(n, dtype=torch.float64, device=DEV)
    for c in range(0, case["m"], 256):
        v[c:c + 256] = -(K[c:c + 256, :n] @ r).double()
    for c in range(0, case["m"], 256):
        u += (v[c:c + 256].float() @ K[c:c + 256, :n]).double()
    act = (y * o < 1.0).double()
    t = -(r.double() * u).sum() / (act * u * u).sum()
    return K, y, J, o, v * t, 1e-4


def _system_inputs(case, seed):
    g, K, y, J, ld = _stored(case, seed)
    o = y * (1.0 + 0.3 * torch.randn(case["n"], generator=g, device=DEV).abs())
    act = torch.rand(case["n"], generator=g, device=DEV) < case["active"]
    o = torch.where(act, 2.0 * y - o, o)   # an active point's margin is below 1
    return K, y, J, o, act.to(torch.uint8), 1e-4


def _solve_inputs(case, seed):
    """The Newton system of the MNIST-like points, 43% of them active, at
    lambda = 1 (C = 1, the paper's setting for two of its datasets): conditioned
    well enough that the solution is determined past FP32."""
    g, K, y, J, ld = _stored(case, seed)
    n = case["n"]
    S = torch.rand(n, generator=g, device=DEV) < 0.43
    Ks = K[:, :n][:, S].double()
    H = K[:, J].double() + Ks @ Ks.T
    return (0.5 * (H + H.T)).contiguous(), Ks @ y[S].double()


def _predict_inputs(case, seed):
    g = _gen(seed)
    X, y, gamma = _points(case, g, case["n"] + case["m"])
    beta = torch.randn(case["m"], generator=g, device=DEV, dtype=torch.float64)
    return X[:case["m"]].contiguous(), beta, X[case["m"]:].contiguous(), gamma


def prepare(case, seed):
    kind, st = case["kind"], {"case": case}
    if kind == "fit":
        X, y, Q, gamma, basis = _fit_inputs(case, seed)
        opts = {"precision": case["precision"], "seed": 7}
        if basis is not None:
            opts |= {"initial_basis": basis.cpu().numpy(), "fixed_basis": True}
        st |= {"X": X, "y": y, "Q": Q, "gamma": gamma, "opts": opts}
    elif kind == "block":
        X, y, gamma, J, g = _block_inputs(case, seed)
        st |= {"P": sp.spsvm_prepare_points(X, case["precision"]), "gamma": gamma, "J": J,
               "out": sp.kmat_empty(case["n"], case["m"])}
    elif kind == "score":
        X, y, gamma, J, g = _block_inputs(case, seed)
        st |= {"P": sp.spsvm_prepare_points(X, case["precision"]), "gamma": gamma, "J": J, "y": y,
               "o": _mid_outputs(y, g)}
    elif kind == "direction":
        K, y, J, o, v, lam = _direction_inputs(case, seed)
        st |= {"K": _kmat(K, case["n"]), "y": y, "J": J, "o": o, "v": v, "lam": lam,
               "u": torch.empty(case["n"], dtype=torch.float32, device=DEV)}
    elif kind == "system":
        K, y, J, o, act, lam = _system_inputs(case, seed)
        n, m = case["n"], case["m"]
        Kc = sp.kmat_empty((n + 127) // 128 * 128, m, case["precision"])
        st |= {"K": _kmat(K, n), "Kc": Kc, "y": y, "J": J, "res": o - y, "act": act, "lam": lam}
    elif kind == "solve":
        st["H"], st["b"] = _solve_inputs(case, seed)
    else:
        st["B"], st["beta"], st["Q"], st["gamma"] = _predict_inputs(case, seed)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "fit":
        model = sp.spsvm_fit(st["X"], st["y"], st["gamma"], FIT_LAMBDA[case["data"]], case["m"], 1e-6,
                             **st["opts"])
        f = sp.spsvm_predict(model, st["Q"])
        out = {"outputs": model.outputs(case["n"]), "decision": f}
        if not case["grow"]:
            out["beta"] = model.basis_and_beta()[1].astype(np.float32)
        return out
    if kind == "block":
        sp.spsvm_kernel_block(st["P"], st["J"], st["gamma"], case["precision"], st["out"])
        return st["out"].buf.view(case["m"], -1)[:, :case["n"]]
    if kind == "score":
        return torch.stack(sp.spsvm_score_candidates(st["P"], st["y"], st["o"], st["J"], st["gamma"],
                                                     1e-4, case["precision"])).float()
    if kind == "direction":
        sp.spsvm_gemv(st["K"], st["v"], st["u"])
        t = sp.spsvm_line_search(st["o"], st["u"], st["y"], st["v"], st["J"], st["lam"])
        return {"u": st["u"], "t": t}
    if kind == "system":
        w1, w2, count, pos = sp.spsvm_compact_active(st["K"], st["act"], st["res"], st["y"], st["Kc"])
        H = sp.spsvm_gram(st["Kc"], count, case["n"], st["K"], st["J"], st["lam"], case["precision"])
        return {"gradient": w1.float(), "rhs": w2.float(), "H": H.float(), "Kc": st["Kc"].buf,
                "count": count, "pos": pos}
    if kind == "solve":
        info, status, x, iters, be = sp.spsvm_solve_mixed(st["H"], st["b"])
        # FP64, determined to cond(H) times the backward error asked for
        return {"x": x.float(), "info": info}
    return sp.spsvm_decision(st["B"], st["beta"], st["Q"], st["gamma"], case["precision"])


def work(case):
    n, d, m, kind = case["n"], case["d"], case["m"], case["kind"]
    if kind == "fit":
        # the kernel rows, and per growth round of 64 two passes over them and a factorisation
        rounds = range(64, m + 64, 64) if case["grow"] else [m]
        f = 2 * n * m * d + sum(4 * n * min(r, m) + min(r, m) ** 3 / 3 for r in rounds)
        return {"bytes": 4 * n * (d + 2) + 4 * case["queries"] * (d + 1),
                "flops": f + 2 * case["queries"] * m * d}
    if kind == "block":
        planes = 6 if case["precision"] == "bf16split" else 4   # bytes of a point's feature
        return {"bytes": n * d * planes + 4 * n + 4 * n * m, "flops": 2 * n * m * d}
    if kind == "score":
        planes = 6 if case["precision"] == "bf16split" else 4
        return {"bytes": n * d * planes + 12 * n + 24 * m, "flops": 2 * n * m * d}
    if kind == "direction":
        return {"bytes": 4 * n * m + 12 * n + 16 * m, "flops": 2 * n * m}
    if kind == "system":
        s = case["active"] * n
        # the active columns read, their copy written (and read by the contraction), H written
        return {"bytes": 12 * s * m + 5 * n + 8 * m * m, "flops": s * m * (m + 1) + 4 * s * m}
    if kind == "solve":
        return {"bytes": 8 * m * m + 16 * m, "flops": m ** 3 / 3 + 4 * m * m}
    return {"bytes": 4 * d * (n + m) + 4 * n + 8 * m, "flops": 2 * n * m * d}


# ---- the same in 64 bits ------------------------------------------------------
def _rbf64(A, B, gamma):
    A, B = A.double(), B.double()
    d2 = (A * A).sum(1)[:, None] + (B * B).sum(1)[None, :] - 2.0 * (A @ B.T)
    return torch.exp(-gamma * d2.clamp_min_(0.0))


def _newton64(K, KJJ, y, lam):
    """The minimiser of lam/2 b'K_JJ b + 1/2 sum max(0, 1 - y o)^2, o = K' b."""
    b = torch.zeros(K.shape[0], dtype=torch.float64, device=DEV)
    f = lambda c: 0.5 * lam * (c @ (KJJ @ c)) + 0.5 * (1.0 - y * (K.T @ c)).clamp_min(0.0).square().sum()  # noqa: E731
    S = None
    for _ in range(100):
        act = y * (K.T @ b) < 1.0
        if S is not None and bool((act == S).all()):
            break
        S = act
        Ks = K[:, S]
        full = torch.linalg.solve(lam * KJJ + Ks @ Ks.T, Ks @ y[S])
        t, f0 = 1.0, f(b)
        while t > 1e-6 and f(b + t * (full - b)) > f0:
            t *= 0.5
        b = b + t * (full - b)
        if t < 1.0:
            S = None
    return b


def exact(case, seed):
    kind, n, m = case["kind"], case["n"], case["m"]
    if kind == "fit":
        if case["grow"]:
            return None   # the basis is the fit's own choice
        X, y, Q, gamma, basis = _fit_inputs(case, seed)
        K = _rbf64(X[basis], X, gamma)
        b = _newton64(K, K[:, basis], y.double(), FIT_LAMBDA[case["data"]])
        return {"outputs": K.T @ b, "decision": _rbf64(Q, X[basis], gamma) @ b, "beta": b}
    if kind == "block":
        X, y, gamma, J, g = _block_inputs(case, seed)
        out = torch.empty((m, n), dtype=torch.float64, device=DEV)
        for c in range(0, m, 64):
            out[c:c + 64] = _rbf64(X[J[c:c + 64]], X, gamma)
        return out
    if kind == "score":
        X, y, gamma, J, g = _block_inputs(case, seed)
        o = _mid_outputs(y, g)
        a = (y * o < 1.0).double()
        r = a * (o.double() - y.double())
        gs, hs = 1e-4 * o[J].double(), torch.full((m,), 1e-4, dtype=torch.float64, device=DEV)
        for c in range(0, m, 64):
            K = _rbf64(X[J[c:c + 64]], X, gamma)
            gs[c:c + 64] += K @ r
            hs[c:c + 64] += (K * K) @ a
        return torch.stack([gs, hs, gs * gs / (2.0 * hs)])
    if kind == "direction":
        K, y, J, o, v, lam = _direction_inputs(case, seed)
        u = torch.zeros(n, dtype=torch.float64, device=DEV)
        for c in range(0, m, 256):
            u += v[c:c + 256] @ K[c:c + 256, :n].double()
        o, y = o.double(), y.double()
        mm, vv = 1.0 - y * o, y * u
        a0, a1 = lam * (v @ o[J]), lam * (v @ u[J])
        lo, hi = 0.0, 64.0
        for _ in range(80):
            t = 0.5 * (lo + hi)
            if float(a0 + a1 * t - (vv * (mm - t * vv).clamp_min(0.0)).sum()) < 0.0:
                lo = t
            else:
                hi = t
        return {"u": u, "t": np.float64(0.5 * (lo + hi))}
    if kind == "system":
        K, y, J, o, act, lam = _system_inputs(case, seed)
        S = act.bool()
        Ks = K[:, :n][:, S].double()
        KJJ = K[:, J].double()
        H = lam * 0.5 * (KJJ + KJJ.T) + Ks @ Ks.T
        return {"gradient": Ks @ (o - y)[S].double(), "rhs": Ks @ y[S].double(), "H": H, "Kc": None,
                "count": None, "pos": None}
    if kind == "solve":
        H, b = _solve_inputs(case, seed)
        x = torch.linalg.solve(H, b)
        for _ in range(2):
            x = x + torch.linalg.solve(H, b - H @ x)
        return {"x": x, "info": None}
    B, beta, Q, gamma = _predict_inputs(case, seed)
    out = torch.empty(n, dtype=torch.float64, device=DEV)
    for c in range(0, n, 8192):
        out[c:c + 8192] = _rbf64(Q[c:c + 8192], B, gamma) @ beta
    return out
