"""The work this library is measured on: calls of its public entry points over the sizes
that its workloads, tests and benchmark use, from the smallest product to the largest.

Inputs come from the seeded generators of ``paper_2510_07929_gb300.workloads`` and are
made before the timed pass, as a program would have them: the problem handle (layouts of
X, RPCholesky factor), device vectors, preallocated results.  Every case works on one
side stream that the handle shares.  Results of the FP32- and TF32-class products are
handed on in 32 bits, the width that carries their accuracy; FP64-class products, solves
and gradients stay in 64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2510_07929_gb300 import kqr
from paper_2510_07929_gb300 import workloads as W

PREC = {"high": kqr.PREC_HIGH, "fp32": kqr.PREC_FP32}
_stream = None


def listed():
    return [
        # The product inside CG on the small RBF workload (n = 2000, p = 10, K stored by default):
        # a few microseconds of work, so latency and launches count.
        {"name": "product_small", "do": "product", "data": "rbf_small", "n": 2000, "p": 10, "m": 1, "prec": "fp32",
         "store": 2},
        # The product inside CG on the mid-size RBF workload (n = 50000, p = 20, entries on the fly).
        {"name": "product_rbf", "do": "product", "data": "rbf_mid", "n": 50000, "p": 20, "m": 1, "prec": "fp32",
         "store": 2},
        # The product inside CG on the benchmark's Laplacian workload, entries on the fly as it states.
        {"name": "product_laplacian", "do": "product", "data": "lap_large", "n": 200000, "p": 50, "m": 1,
         "prec": "fp32", "store": 0},
        # The shared CG product of a (tau, lambda) grid: eight right-hand sides per pass over K.
        {"name": "product_grid", "do": "product", "data": "rbf_small", "n": 19999, "p": 8, "m": 8, "prec": "fp32",
         "store": 2},
        # FP64-class products, which every gradient, Sec. 4 residual and low-rank CG step needs:
        # one vector on the mid-size RBF data, one on Laplacian data, and a grid's eight.
        {"name": "high_rbf", "do": "product", "data": "rbf_mid", "n": 50000, "p": 20, "m": 1, "prec": "high",
         "store": 2},
        {"name": "high_laplacian", "do": "product", "data": "lap_large", "n": 50001, "p": 50, "m": 1, "prec": "high",
         "store": 2},
        {"name": "high_grid", "do": "product", "data": "rbf_small", "n": 10007, "p": 8, "m": 8, "prec": "high",
         "store": 2},
        # The batched workload: 64 RBF problems of 1000 .. 20000 points, 64 right-hand sides each.
        {"name": "batch", "do": "batch", "problems": 64, "nmin": 1000, "nmax": 20000, "p": 8, "m": 64},
        # One linear system of Phase I on the small RBF workload: the first system of a solve, with
        # the Woodbury core built for it and CG of cheap products (latency bound).
        {"name": "system_small", "do": "system", "data": "rbf_small", "n": 2000, "p": 10, "rank0": 0, "phase": 1,
         "rtol": 1e-8},
        # One Newton system of Phase II on the mid-size RBF data at the benchmark's rank (1024): the
        # gradient and its diagonal, the Woodbury core, CG.
        {"name": "system_newton", "do": "system", "data": "rbf_mid", "n": 20011, "p": 20, "rank0": 1024, "phase": 2,
         "rtol": 1e-8},
        # The benchmark's step (set-up on resident data, then a whole solve) on its generator at a
        # size that fits a pass, default options.
        {"name": "solve", "do": "solve", "data": "lap_large", "n": 10000, "p": 50, "rank0": 0, "tau": 0.25,
         "lam": 1e-4, "tol": 1e-9},
        # The backward direction: held-out loss gradient of a solved problem (the gradient workload's
        # generator, tau and lambda, at the gamma of a tuning sweep that the tests also take).
        {"name": "gradient", "do": "gradient", "n": 3000, "nh": 750, "p": 16, "tau": 0.5, "lam": 0.1, "gamma": 1.0},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["product", "product", "product", "high", "high", "batch", "system", "system", "solve",
                     "gradient"])
    if do == "product":
        m = rng.choice([1, 1, 1, 1, 2, 3, 5, 8])
        data = rng.choice(["rbf_small", "rbf_mid", "lap_large"])
        n = _logint(rng, 1000, 120000 if m == 1 else 30000)
        p = rng.randint(2, 50) if data == "lap_large" else rng.randint(2, 32)
        return {"do": do, "data": data, "n": n, "p": p, "m": m, "prec": "fp32", "store": rng.choice([0, 2, 2])}
    if do == "high":
        m = rng.choice([1, 1, 1, 2, 5, 8])
        data = rng.choice(["rbf_small", "rbf_mid", "lap_large"])
        n = _logint(rng, 1000, 50000 if m == 1 else 15000)
        p = rng.randint(2, 50) if data == "lap_large" else rng.randint(2, 32)
        return {"do": "product", "data": data, "n": n, "p": p, "m": m, "prec": "high", "store": 2}
    if do == "batch":
        nmin = _logint(rng, 100, 2000)
        return {"do": do, "problems": rng.randint(8, 64), "nmin": nmin, "nmax": nmin + _logint(rng, 2000, 18000),
                "p": rng.randint(2, 32), "m": rng.randint(1, 64)}
    if do == "system":
        data = rng.choice(["rbf_mid", "lap_large"])
        return {"do": do, "data": data, "n": _logint(rng, 1000, 18000), "p": rng.randint(10, 40),
                "rank0": rng.choice([0, _logint(rng, 64, 1024)]), "phase": rng.choice([1, 2]), "rtol": 1e-8}
    if do == "solve":
        return {"do": do, "data": "lap_large", "n": _logint(rng, 2000, 9000), "p": rng.randint(30, 50), "rank0": 0,
                "tau": rng.choice([0.25, 0.5, 0.75]), "lam": 1e-4, "tol": 1e-9}
    n = _logint(rng, 1000, 2900)
    return {"do": do, "n": n, "nh": rng.randint(n // 8, n // 3), "p": 16, "tau": 0.5, "lam": 0.1, "gamma": 1.0}


# ---- inputs -----------------------------------------------------------------------------
def _work_stream():
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    torch.cuda.set_stream(_stream)
    return _stream


def _data(case, seed):
    gen = W.GENERATORS[case["data"]]
    return gen(n=case["n"], p=case["p"], seed=seed)


def _batch_sizes(case):
    rng = np.random.default_rng(0)   # the sizes belong to the case, not to the seed
    return [int(s) for s in rng.integers(case["nmin"], case["nmax"] + 1, size=case["problems"])]


def _normal(shape, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(shape, dtype=torch.float64, device="cuda", generator=g)


def _batch_inputs(case, seed):
    rng = np.random.default_rng(seed)
    sizes = _batch_sizes(case)
    Xs = [rng.random((n, case["p"])) for n in sizes]
    return Xs, 1.0 / 8.0, _normal((sum(sizes), case["m"]), seed + 1)


def _iterate(case, wl, seed):
    """(alpha, z, Kalpha, beta, sigma, lam, eps) of an iterate in the middle of a solve: about a
    third of the points inside the box, Phase I's sigma = 1 or Phase II's sigma = 1 / lambda."""
    lam = wl.lam
    sigma = 1.0 if case["phase"] == 1 else 1.0 / lam
    w = 0.9 * _normal(case["n"], seed + 2)                      # alpha + z / sigma
    alpha = torch.clamp(w, wl.tau - 1.0, wl.tau)
    y = torch.from_numpy(wl.y).cuda()
    Kalpha = lam * (y + 0.1 * _normal(case["n"], seed + 3))     # fitted values near y
    return alpha, sigma * (w - alpha), Kalpha, 0.1, sigma, lam, 1e-3


def _phase1_rhs(wl, alpha, z, lam):
    y = torch.from_numpy(wl.y).cuda()
    return lam * (y - 0.1 - z + alpha)


def _gradient_inputs(case, seed):
    tr = W.rbf_small(n=case["n"], p=case["p"], seed=seed, tau=case["tau"], lam=case["lam"])
    ho = W.rbf_small(n=case["nh"], p=case["p"], seed=seed + 1000, tau=case["tau"], lam=case["lam"])
    return tr, ho


def prepare(case, seed):
    stream = _work_stream()
    do = case["do"]
    if do == "batch":
        Xs, gamma, V = _batch_inputs(case, seed)
        handle = kqr.Batch(Xs, gamma)
        handle.set_stream(stream)
        return {"case": case, "handle": handle, "V": V, "U": torch.empty_like(V)}
    if do == "gradient":
        tr, ho = _gradient_inputs(case, seed)
        prob = kqr.Problem(tr.X, tr.y, "rbf", case["gamma"], pivot_uniforms=W.pivot_uniforms(1024, seed + 9))
        prob.set_stream(stream)
        prob.solve(case["tau"], case["lam"], 1e-10)
        return {"case": case, "handle": prob, "Xh": ho.X, "yh": ho.y}
    wl = _data(case, seed)
    opts = {"gram_store": case["store"]} if do == "product" else {"rank0": case["rank0"]}
    uniforms = W.pivot_uniforms(1024, seed + 9)
    prob = kqr.Problem(wl.X, wl.y, wl.kind, wl.gamma, pivot_uniforms=uniforms, **opts)
    prob.set_stream(stream)
    state = {"case": case, "handle": prob}
    if do == "product":
        shape = (case["n"], case["m"]) if case["m"] > 1 else (case["n"],)
        state["V"] = _normal(shape, seed + 1)
        state["U"] = torch.empty_like(state["V"])
    elif do == "system":
        state["tau"] = wl.tau
        state["it"] = _iterate(case, wl, seed)
        state["rhs1"] = _phase1_rhs(wl, state["it"][0], state["it"][1], wl.lam)
        state["grad"], state["L"], state["x"] = (torch.empty(case["n"], dtype=torch.float64, device="cuda")
                                                 for _ in range(3))
    else:
        state["uniforms"] = uniforms
    return state


# ---- one pass ---------------------------------------------------------------------------
def run(state):
    case, h = state["case"], state["handle"]
    do = case["do"]
    if do == "product":
        h.kmatvec_dev(state["V"], state["U"], PREC[case["prec"]])
        return state["U"].float() if case["prec"] == "fp32" else state["U"]
    if do == "batch":
        h.kmatmul_dev(state["V"], state["U"])
        return state["U"].float()
    if do == "system":
        alpha, z, Ka, beta, sigma, lam, eps = state["it"]
        grad, L, x = state["grad"], state["L"], state["x"]
        if case["phase"] == 1:       # (2.1): (K + lambda sigma (1 1^T + I)) alpha = b
            L.fill_(lam * sigma)
            b = state["rhs1"]
        else:                        # (3.1): Newton system at the iterate
            h.box_grad_dev(alpha, z, Ka, beta, sigma, state["tau"], lam, eps, grad=grad, Ldiag=L)
            b = -lam * grad
        its = h.pcg_dev(L, lam * sigma, b, x, case["rtol"] * float(b.norm()), 3000)
        return {"x": x, "L": L, "grad": grad if case["phase"] == 2 else b, "solved": its > 0}
    if do == "solve":
        h.refactor(state["uniforms"])
        alpha, beta, kkt, _ = h.solve(case["tau"], case["lam"], case["tol"])
        return {"alpha": alpha, "solved": kkt <= case["tol"]}
    loss, dgamma, dlambda, dX = h.heldout_grad(state["Xh"], state["yh"])
    return {"loss": loss, "d_loggamma": dgamma, "d_loglambda": dlambda, "dX": dX}


# ---- what a pass cannot do without ------------------------------------------------------
def work(case):
    do = case["do"]
    if do == "batch":
        sizes = _batch_sizes(case)
        n, p, m = sum(sizes), case["p"], case["m"]
        entries = float(sum(s * s for s in sizes))
        return {"bytes": 4.0 * n * p + 16.0 * n * m, "flops": entries * (2 * p + 2 * m)}
    n, p = case["n"], case["p"]
    per_entry = 3 * p + 1 if case.get("data") == "lap_large" else 2 * p + 2
    half = n * (n + 1) / 2.0                      # K is symmetric: entries formed once
    if do == "product":
        m = case["m"]
        wide = 4 if case["prec"] == "fp32" else 8
        return {"bytes": wide * n * p + 16.0 * n * m, "flops": half * per_entry + 2.0 * n * n * m}
    if do == "gradient":
        # set-up of the union problem's products: three sets of p + 1 vectors over n + nh points,
        # and two adjoint solves of about 20 products each
        N = n + case["nh"]
        return {"bytes": 8.0 * N * p * 5, "flops": N * (N + 1) / 2.0 * per_entry + 2.0 * N * N * 3 * (p + 1)
                + 40 * 2.0 * n * n}
    r = case["rank0"] or math.ceil(math.sqrt(n))
    core = r * r * n + r ** 3                     # core, factor and inverse
    if do == "system":
        its = 30                                  # products, each with a rank-r preconditioner
        return {"bytes": its * 8.0 * n * 8, "flops": core + half * per_entry + its * (2.0 * n * n + 4.0 * n * r)}
    its = 400
    return {"bytes": its * 8.0 * n * 8, "flops": r * r * n + core + half * per_entry
            + its * (2.0 * n * n + 4.0 * n * r)}


# ---- the same in 64 bits, plain torch ---------------------------------------------------
def _gram_rows(Xr, X, kind, gamma):
    d = torch.zeros(Xr.shape[0], X.shape[0], dtype=torch.float64, device=X.device)
    for k in range(X.shape[1]):
        t = Xr[:, k:k + 1] - X[:, k]
        if kind == "laplacian":
            d += t.abs_()
        else:
            d.addcmul_(t, t)
    return d.mul_(-gamma).exp_()


def _gram_times(X, V, kind, gamma):
    step = max(1, (1 << 27) // X.shape[0])
    return torch.cat([_gram_rows(X[i:i + step], X, kind, gamma) @ V for i in range(0, X.shape[0], step)])


def _optimum(K, y, tau, lam):
    """Exact (alpha, beta, inside) of the dual (1.3): splitting steps for the active set, then
    the equations of that set, repeated until the set stays; None if it never does."""
    n = y.numel()
    eye = torch.eye(n, dtype=torch.float64, device=y.device)
    one = eye.sum(0)
    s = float(K.diagonal().mean()) / lam * 0.3
    inv = torch.cholesky_inverse(torch.linalg.cholesky(K / lam + s * eye))
    inv1 = inv @ one
    v, z = torch.zeros_like(y), torch.zeros_like(y)
    for outer in range(60):
        for _ in range(200):
            a = inv @ (y + s * v - z)
            a = a - (a.sum() / inv1.sum()) * inv1
            v = torch.clamp(a + z / s, tau - 1.0, tau)
            z = z + s * (a - v)
        up, dn = v >= tau, v <= tau - 1.0
        e = (~(up | dn)).nonzero()[:, 0]
        if e.numel() == 0:
            return None
        alpha = torch.where(up, tau * one, torch.where(dn, (tau - 1.0) * one, 0 * one))
        rhs = torch.stack([lam * y[e] - K[e] @ alpha, lam * one[e]], 1)
        sol = torch.linalg.solve(K[e][:, e], rhs)
        beta = (alpha.sum() + sol[:, 0].sum()) / sol[:, 1].sum()
        alpha[e] = sol[:, 0] - beta * sol[:, 1]
        r = y - beta - K @ alpha / lam
        if bool(((alpha[e] > tau - 1.0) & (alpha[e] < tau)).all()) and bool((r[up] >= 0).all()) and bool(
                (r[dn] <= 0).all()):
            return alpha, beta, ~(up | dn)
    return None


def exact(case, seed):
    stream = _work_stream()
    do = case["do"]
    with torch.cuda.stream(stream):
        if do == "batch":
            Xs, gamma, V = _batch_inputs(case, seed)
            at, out = 0, []
            for x in Xs:
                out.append(_gram_times(torch.from_numpy(x).cuda(), V[at:at + len(x)], "rbf", gamma))
                at += len(x)
            return torch.cat(out)
        if do == "gradient":
            return _exact_gradient(case, seed)
        wl = _data(case, seed)
        X, y = torch.from_numpy(wl.X).cuda(), torch.from_numpy(wl.y).cuda()
        n = case["n"]
        if do == "product":
            V = _normal((n, case["m"]), seed + 1)
            U = _gram_times(X, V, wl.kind, wl.gamma)
            return U if case["m"] > 1 else U[:, 0]
        eye = torch.eye(n, dtype=torch.float64, device="cuda")
        K = _gram_times(X, eye, wl.kind, wl.gamma) if n <= 4096 else torch.cat(
            [_gram_rows(X[i:i + 4096], X, wl.kind, wl.gamma) for i in range(0, n, 4096)])
        if do == "system":
            alpha, z, Ka, beta, sigma, lam, eps = _iterate(case, wl, seed)
            if case["phase"] == 1:
                L = torch.full_like(y, lam * sigma)
                b = grad = _phase1_rhs(wl, alpha, z, lam)
            else:
                w = alpha + z / sigma
                v = torch.clamp(w, wl.tau - 1.0, wl.tau)
                grad = Ka / lam - y + beta + sigma * alpha.sum() + sigma * (w - v)
                S = ((w > wl.tau - 1.0) & (w < wl.tau)).double()
                L = lam * sigma * (1.0 - S) + lam * eps
                b = -lam * grad
            A = K + lam * sigma
            A.diagonal().add_(L)
            x = torch.cholesky_solve(b[:, None], torch.linalg.cholesky(A))[:, 0]
            return {"x": x, "L": L, "grad": grad, "solved": None}
        got = _optimum(K, y, case["tau"], case["lam"])
        return None if got is None else {"alpha": got[0], "solved": None}


def _exact_gradient(case, seed):
    tr, ho = _gradient_inputs(case, seed)
    tau, lam, gamma = case["tau"], case["lam"], case["gamma"]
    X, y = torch.from_numpy(tr.X).cuda(), torch.from_numpy(tr.y).cuda()
    Xh, yh = torch.from_numpy(ho.X).cuda(), torch.from_numpy(ho.y).cuda()
    K, Kh = _gram_rows(X, X, "rbf", gamma), _gram_rows(Xh, X, "rbf", gamma)
    got = _optimum(K, y, tau, lam)
    if got is None:
        return None
    alpha, beta, inside = got
    r = yh - beta - Kh @ alpha / lam
    loss = torch.where(r > 0, tau * r, (tau - 1.0) * r).sum()
    g = torch.where(r > 0, -tau * torch.ones_like(r), (1.0 - tau) * torch.ones_like(r))   # d loss / d f_h
    e = inside.nonzero()[:, 0]
    m = e.numel()
    J = torch.zeros(m + 1, m + 1, dtype=torch.float64, device="cuda")
    J[:m, :m] = K[e][:, e] / lam
    J[:m, m] = 1.0
    J[m, :m] = 1.0
    rhs = torch.cat([(Kh[:, e].T @ g) / lam, g.sum()[None]])
    u = torch.zeros_like(y)
    u[e] = torch.linalg.solve(J, rhs)[:m]
    # dl/dtheta = g^T (d f_h) - u^T (d F_E) with f = beta + K alpha / lambda
    dlam = -(g @ (Kh @ alpha)) / lam + (u @ (K @ alpha)) / lam
    D, Dh = -torch.log(K), -torch.log(Kh)                        # gamma ||x - x'||^2
    dgam = -(g @ ((Dh * Kh) @ alpha)) / lam + (u @ ((D * K) @ alpha)) / lam
    dX = torch.empty_like(X)
    for k in range(X.shape[1]):
        dh = Xh[:, k:k + 1] - X[:, k]                            # d k(x_h, x_i) / d x_i = 2 gamma dh k
        dd = X[:, k:k + 1] - X[:, k]
        from_h = 2 * gamma / lam * alpha * ((Kh * dh).T @ g)
        rows = -2 * gamma / lam * u * ((K * dd) @ alpha)         # F_i through its own point
        cols = 2 * gamma / lam * alpha * ((K * dd).T @ u)        # F_i through the other point
        dX[:, k] = from_h - rows - cols
    return {"loss": loss, "d_loggamma": dgam, "d_loglambda": dlam, "dX": dX}
