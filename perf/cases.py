"""What the library is used for, as cases that can be timed and compared.

Each case is one call, or one short sequence of calls, of the public API on
seeded synthetic inputs with the shapes and distributions of inputs/synthetic.py
(generated on the GPU).  The operations:

  product   (A + lambda I) V, krr_kmatvec in one of its three precisions
  batched   the product for several (kernel, sigma) settings, krr_kmatvec_batched
  predict   K(Xtest, Xtrain) alpha, krr_predict
  factor    krr_rpcholesky and one application of the Alg. 1 preconditioner
  solve     krr_rpcholesky and krr_pcg_solve: a whole kernel ridge regression
  krill     krill_build, krill_solve and the predictions at new points
  serve     a closed loop of solve requests through KrrServer

What carries float32 accuracy (the "mixed" products, predictions and
preconditioner, and the solves to a tolerance of 1e-6) is returned as float32,
which is how a program keeps such results; what is computed in float64 or
float-float stays float64.  A solve returns its fitted values y - lambda alpha,
one for each point and right-hand side: two solutions that meet the same
tolerance have the same fitted values to that tolerance, while their
coefficients may differ by the condition number times it.  A restricted model
is solved to 1e-8 and evaluated in float64 for the same reason (its
coefficients are large and cancel); its predictions are kept as float32.
"""
import math

import numpy as np
import torch

import paper_2304_12465_gb300 as K

GAUSSIAN, LAPLACE, MATERN = 0, 1, 2
_DEV = "cuda"


# ------------------------------------------------------------------- cases
def listed():
    return [
        # one small product: a request at the low end of the serving range,
        # and the per-iteration call of a small solve (launches and host work)
        dict(name="product_small", op="product", prec="mixed", N=2000, d=4, m=1, kernel=GAUSSIAN,
             sigma=0.8, mu=1e-5, points="normal"),
        # the product of the ill-conditioned benchmark workload, one call of
        # every inner PCG iteration
        dict(name="product_main", op="product", prec="mixed", N=100_000, d=16, m=4,
             kernel=GAUSSIAN, sigma=0.5, mu=1e-7, points="cube"),
        # the widest request of the serving range: 32 coordinates, 16
        # right-hand sides, Matern, an N that fits no tile
        dict(name="product_wide", op="product", prec="mixed", N=50_021, d=32, m=16, kernel=MATERN,
             sigma=2.0, mu=1e-6, points="normal"),
        # the paper's molecular workload: Laplace with the l1 distance
        dict(name="product_laplace", op="product", prec="mixed", N=60_007, d=8, m=1,
             kernel=LAPLACE, sigma=1.0, mu=1e-6, points="normal"),
        # the float64-accurate product behind every refinement residual
        dict(name="product_ff", op="product", prec="ff", N=40_009, d=16, m=4, kernel=GAUSSIAN,
             sigma=0.5, mu=1e-7, points="cube"),
        # a hyperparameter search step: 4 Matern and 4 Laplace bandwidths, two
        # regularisations each
        dict(name="batched", op="batched", N=40_000, d=8, settings=8, ms=2),
        # predictions of a restricted model (2000 centers) at many new points
        dict(name="predict", op="predict", prec="mixed", N=2000, Nt=200_003, d=20, m=1,
             kernel=GAUSSIAN, sigma=2.0, points="decay"),
        # the preconditioner of the benchmark workload, built and applied once
        dict(name="factor_main", op="factor", prec="mixed", N=100_000, d=16, m=4, kernel=GAUSSIAN,
             sigma=0.5, mu=1e-7, k=1000, points="cube"),
        # the plain float64 configuration, from points to solution
        dict(name="solve_fp64", op="solve", prec="fp64", N=4096, d=8, m=1, kernel=GAUSSIAN,
             sigma=1.5, mu=1e-5, k=200, tol=1e-10, points="normal"),
        # the benchmark workload as a whole
        dict(name="solve_main", op="solve", prec="mixed", N=100_000, d=16, m=4, kernel=GAUSSIAN,
             sigma=0.5, mu=1e-7, k=1000, tol=1e-6, points="cube"),
        # restricted regression at a tenth of the full configuration's points
        dict(name="krill", op="krill", N=200_000, Nt=10_000, d=20, k=1000, kernel=GAUSSIAN,
             sigma=2.0, mu=1e-6, tol=1e-8, points="decay"),
        # a burst of small and medium requests at the server
        dict(name="serve", op="serve", requests=16, n_min=2000, n_max=12_000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _log(rng, lo, hi):
    return float("%.4g" % math.exp(rng.uniform(math.log(lo), math.log(hi))))


def _problem(rng):
    """Kernel, bandwidth and points of a problem as the configurations pair them."""
    points = rng.choice(["normal", "cube", "decay"])
    d = {"normal": rng.choice([1, 3, 4, 5, 8, 13, 16, 24, 32]), "cube": rng.choice([6, 11, 16, 27]),
         "decay": rng.choice([7, 12, 20, 30])}[points]
    sigma = _log(rng, 0.4, 1.0) if points == "cube" else _log(rng, 0.5, 3.0)
    return dict(points=points, d=d, sigma=sigma, kernel=rng.choice([GAUSSIAN, LAPLACE, MATERN]))


def draw(rng):
    op = rng.choice(["product", "product", "product", "batched", "predict", "factor", "solve",
                     "krill", "serve"])
    if op == "product":
        prec = rng.choice(["mixed", "mixed", "ff", "fp64"])
        top = {"mixed": 120_000, "ff": 50_000, "fp64": 12_000}[prec]
        return dict(op=op, prec=prec, N=_log_int(rng, 500, top), m=rng.choice([1, 2, 3, 4, 5, 8, 11, 16]),
                    mu=_log(rng, 1e-8, 1e-4), **_problem(rng))
    if op == "batched":
        return dict(op=op, N=_log_int(rng, 1000, 60_000), d=rng.choice([3, 4, 8, 13, 16]),
                    settings=rng.choice([1, 2, 3, 4, 8]), ms=rng.choice([1, 2]))
    if op == "predict":
        return dict(op=op, prec=rng.choice(["mixed", "mixed", "mixed", "fp64"]),
                    N=_log_int(rng, 500, 10_000), Nt=_log_int(rng, 100, 100_000),
                    m=rng.choice([1, 2, 4, 7, 16]), **_problem(rng))
    if op == "factor":
        N = _log_int(rng, 1000, 100_000)
        return dict(op=op, prec=rng.choice(["mixed", "mixed", "fp64"]), N=N,
                    m=rng.choice([1, 2, 4, 9]), mu=_log(rng, 1e-7, 1e-4),
                    k=_log_int(rng, 40, min(1000, N // 5)), **_problem(rng))
    if op == "solve":
        fp64 = rng.random() < 0.4
        N = _log_int(rng, 1000, 5000 if fp64 else 30_000)
        return dict(op=op, prec="fp64" if fp64 else "mixed", tol=1e-10 if fp64 else 1e-6, N=N,
                    m=rng.choice([1, 2, 4]), mu=_log(rng, 1e-5, 1e-3),
                    k=_log_int(rng, 50, min(500, N // 5)), **_problem(rng))
    if op == "krill":
        return dict(op=op, N=_log_int(rng, 10_000, 300_000), Nt=_log_int(rng, 500, 20_000),
                    d=rng.choice([8, 12, 20]), k=_log_int(rng, 100, 1000), kernel=GAUSSIAN,
                    sigma=2.0, mu=1e-6, tol=1e-8, points="decay")
    return dict(op="serve", requests=rng.randint(3, 16), n_min=_log_int(rng, 1000, 2500),
                n_max=_log_int(rng, 3000, 12_000))


# ------------------------------------------------------------------ inputs
def _points(gen, n, d, kind):
    """normal: x ~ N(0, I).  cube: x uniform on [0, 1]^d with 5% of the rows
    near-duplicates of others.  decay: x ~ N(0, diag(1 / j)).  mixture: eight
    Gaussian clusters of very different widths."""
    if kind == "cube":
        X = torch.rand((n, d), generator=gen, device=_DEV, dtype=torch.float64)
        dup = max(1, n // 20)
        perm = torch.randperm(n, generator=gen, device=_DEV)
        X[perm[:dup]] = X[perm[-dup:]] + 1e-6 * _normal(gen, dup, d)
        return X
    if kind == "mixture":
        means = 3.0 * _normal(gen, 8, d)
        scales = torch.logspace(-1, math.log10(2.0), 8, device=_DEV, dtype=torch.float64)
        comp = torch.randint(0, 8, (n,), generator=gen, device=_DEV)
        return means[comp] + scales[comp, None] * _normal(gen, n, d)
    X = _normal(gen, n, d)
    if kind == "decay":
        X = X / torch.arange(1, d + 1, device=_DEV, dtype=torch.float64).sqrt()
    return X


def _normal(gen, *shape):
    return torch.randn(shape, generator=gen, device=_DEV, dtype=torch.float64)


def _targets(gen, X, m):
    """m smooth functions of the points plus noise, one a row."""
    t = X.sum(1) / math.sqrt(X.shape[1])
    Y = torch.stack([torch.sin((r + 1) * t) for r in range(m)])
    return (Y + 0.01 * _normal(gen, m, X.shape[0])).contiguous()


def _settings(case):
    """Matern bandwidths, then Laplace ones, over the range of a search."""
    S = case["settings"]
    return ([MATERN if q < (S + 1) // 2 else LAPLACE for q in range(S)],
            [0.5 * 2.0 ** (q % 4) for q in range(S)])


def _requests(case, seed):
    rng = np.random.default_rng(seed)
    lo, hi = math.log(case["n_min"]), math.log(case["n_max"])
    out = []
    for i in range(case["requests"]):
        n = int(math.exp(lo + (hi - lo) * (i + 0.5) / case["requests"]))
        d, m = [4, 8, 16, 32][i % 4], 1 + (5 * i) % 8
        X = rng.standard_normal((n, d))
        w = rng.standard_normal(d)
        proj = X @ (w / np.linalg.norm(w))
        Y = np.stack([np.sin((r + 1) * proj) for r in range(m)])
        out.append(dict(X=X, Y=Y + 0.01 * rng.standard_normal((m, n)), kernel=i % 3,
                        sigma=0.5 * 2.0 ** (i % 3), mu=[1e-5, 1e-4][i % 2], k=n // 10,
                        seed=int(rng.integers(1 << 31))))
    return out


def prepare(case, seed):
    """The inputs on the GPU; for the server, the running server and the
    requests as host arrays, as they reach it."""
    op, gen = case["op"], torch.Generator(device=_DEV).manual_seed(seed)
    if op == "serve":
        return dict(case=case, server=K.KrrServer(max_slots=32), requests=_requests(case, seed))
    s = dict(case=case, seed=seed)
    s["X"] = _points(gen, case["N"], case["d"], case.get("points", "mixture"))
    if op == "batched":
        s["V"] = _normal(gen, case["settings"] * case["ms"], case["N"])
    elif op == "krill":
        s["Xt"] = _points(gen, case["Nt"], case["d"], case["points"])
        s["Y"] = _targets(gen, s["X"], 1)
        perm = torch.randperm(case["N"], generator=gen, device=_DEV)[:case["k"]]
        s["centers"] = perm.sort().values
        s["Xc"] = s["X"][s["centers"]].contiguous()
    elif op == "solve":
        s["Y"] = _targets(gen, s["X"], case["m"])
    else:  # a PCG direction, a residual or coefficients
        s["V"] = _normal(gen, case["m"], case["N"])
        if op == "predict":
            s["Xt"] = _points(gen, case["Nt"], case["d"], case["points"])
    return s


def run(s):
    c = s["case"]
    op = c["op"]
    if op == "serve":
        return _serve(s["server"], s["requests"])
    if op == "batched":
        kernels, sigmas = _settings(c)
        lams = [mu * c["N"] for mu in [1e-6, 1e-8][:c["ms"]]] * c["settings"]
        return K.krr_kmatvec_batched(s["X"], kernels, sigmas, lams, s["V"]).float()
    kern, sigma = c["kernel"], c["sigma"]
    if op == "krill":
        P = K.krill_build(s["X"], kern, sigma, s["centers"], c["mu"], seed=s["seed"])
        beta, _ = K.krill_solve(P, s["Y"], tol=c["tol"])
        P.free()
        return K.krr_predict(s["Xc"], kern, sigma, beta, s["Xt"], prec="fp64").float()
    if op == "product":
        out = K.krr_kmatvec(s["X"], kern, sigma, c["mu"] * c["N"], s["V"], prec=c["prec"])
    elif op == "predict":
        out = K.krr_predict(s["X"], kern, sigma, s["V"], s["Xt"], prec=c["prec"])
    else:
        F = K.krr_rpcholesky(s["X"], kern, sigma, c["k"], seed=s["seed"])
        if op == "factor":
            out = K.krr_precond_apply(F, c["mu"], s["V"], prec=c["prec"])
        else:
            alpha, _ = K.krr_pcg_solve(s["X"], kern, sigma, s["Y"], c["mu"], F, tol=c["tol"],
                                       prec=c["prec"])
            out = s["Y"] - c["mu"] * c["N"] * alpha
        F.free()
    return out.float() if c["prec"] == "mixed" else out


def _serve(server, requests):
    ids = [server.submit(r["X"], r["kernel"], r["sigma"], r["Y"], r["mu"], r["k"], tol=1e-6,
                         maxit=3000, seed=r["seed"]) for r in requests]
    done = {d["id"]: d["alpha"] for d in server.drain()}
    return [(r["Y"] - r["mu"] * len(r["X"]) * done[i]).astype(np.float32)
            for i, r in zip(ids, requests)]


# -------------------------------------------------------------------- work
def work(case):
    """Inputs read once and outputs written once; the arithmetic of the method
    as it is defined, with one pass over the kernel matrix for each product it
    needs (a solve: as many as its tolerance takes, about)."""
    op = case["op"]
    if op == "serve":
        n = math.sqrt(case["n_min"] * case["n_max"])
        return {"bytes": case["requests"] * n * (15 + 8) * 8.0,
                "flops": case["requests"] * (60 * n * n * 39 + 3 * n * (n / 10) ** 2)}
    N, d = case["N"], case["d"]
    if op == "batched":
        cols = case["settings"] * case["ms"]
        return {"bytes": 8.0 * N * (d + 2 * cols),
                "flops": float(N) * N * (2 * d + 2 * cols + 8 * case["settings"])}
    if op == "predict":
        m, Nt = case["m"], case["Nt"]
        return {"bytes": 8.0 * (N * (d + m) + Nt * (d + m)), "flops": float(N) * Nt * (2 * d + 2 * m + 1)}
    if op == "krill":
        k, Nt = case["k"], case["Nt"]
        zeta = math.ceil(math.log(k + 1))
        passes = 2 * 45 + 2          # A(:, S) and its transpose in each iteration
        return {"bytes": 8.0 * (N * (d + 1) + k + Nt * (d + 1)),
                "flops": float(N) * k * (2 * d + 3) * (passes + zeta) + 2.0 * k ** 3 + 2.0 * k ** 3 / 3}
    m = case["m"]
    product = float(N) * N * (2 * d + 2 * m + 1)
    if op == "product":
        return {"bytes": 8.0 * N * (d + 2 * m), "flops": product}
    k = case["k"]
    factor = float(N) * k * (2 * d + 1) + 2.0 * N * k * k + k ** 3
    if op == "factor":
        return {"bytes": 8.0 * N * (d + 2 * m), "flops": factor + 4.0 * N * k * m}
    iters = 340 if case["points"] == "cube" else 120
    return {"bytes": 8.0 * N * (d + 2 * m), "flops": factor + iters * (product + 4.0 * N * k * m)}


# ------------------------------------------------------- results in 64 bits
def _kernel(A, B, kern, sigma):
    """Kernel matrix of the rows of A and B from float64 distances."""
    if kern == LAPLACE:
        l1 = torch.zeros((len(A), len(B)), device=_DEV, dtype=torch.float64)
        for a, b in zip(A.T, B.T):
            l1 += (a[:, None] - b).abs_()
        return l1.mul_(-1.0 / sigma).exp_()
    shift = B.mean(0)
    A, B = A - shift, B - shift
    d2 = torch.addmm((A * A).sum(1)[:, None] + (B * B).sum(1), A, B.T, alpha=-2.0).clamp_(min=0.0)
    if kern == GAUSSIAN:
        return d2.mul_(-0.5 / sigma ** 2).exp_()
    q = d2.mul_(5.0).sqrt_().div_(sigma)
    return (1.0 + q + q * q / 3.0) * torch.exp(-q)


def _multiply(A, B, kern, sigma, V):
    """K(A, B) V^T in float64, by blocks of rows; V (m, len(B)) -> (m, len(A))."""
    step = max(1, int(2e8 // len(B)))
    out = [V @ _kernel(A[i:i + step], B, kern, sigma).T for i in range(0, len(A), step)]
    return torch.cat(out, 1)


def _philox(t, j, seed):
    """Word 0 of Philox4x64-10 with counter (t, j, 0, 0) and the pivot key
    (numpy counts up before each block)."""
    ctr = [t, j, 0, 0]
    for i in range(4):
        if ctr[i]:
            ctr[i] -= 1
            break
        ctr[i] = (1 << 64) - 1
    gen = np.random.Philox(counter=np.array(ctr, dtype=np.uint64),
                           key=np.array([seed, 0x5250434850495653], dtype=np.uint64))
    return int(gen.random_raw(1)[0])


def _pivoted_factor(X, kern, sigma, k, seed):
    """Randomly pivoted Cholesky (k x N factor) with the library's documented
    sampling rule: fixed-point weights, draws in order, repeats left out."""
    N = len(X)
    block = min(100, (k + 9) // 10)
    bits = 62 - (N - 1).bit_length()
    floor = N * 2.0 ** -52
    dres = torch.ones(N, device=_DEV, dtype=torch.float64)
    F = torch.zeros((k, N), device=_DEV, dtype=torch.float64)
    rank = t = 0
    while rank < k:
        w = torch.where(dres > floor, (dres.clamp(max=1.0) * 2.0 ** bits).floor(), 0.0 * dres)
        prefix = w.to(torch.int64).cumsum(0).cpu().numpy()
        total = int(prefix[-1])
        if total == 0:
            break
        targets = [(_philox(t, j, seed) * total) >> 64 for j in range(min(block, k - rank))]
        cand = list(dict.fromkeys(int(i) for i in np.searchsorted(prefix, targets, side="right")))
        G = _kernel(X[cand], X, kern, sigma) - F[:rank, cand].T @ F[:rank]
        for row, i in enumerate(cand):
            if G[row, i] > floor:
                f = G[row] / G[row, i].sqrt()
                G[row + 1:] -= f[cand[row + 1:], None] * f
                F[rank] = f
                dres -= f * f
                rank += 1
        dres[cand] = 0.0
        t += 1
    return F[:rank]


def exact(case, seed):
    op = case["op"]
    if op in ("krill", "serve") or (op == "solve" and case["N"] > 12_000):
        return None  # a sketch in float32 and a tolerance decide; too large to solve directly
    s = prepare(case, seed)
    X, N = s["X"], case["N"]
    if op == "batched":
        kernels, sigmas = _settings(case)
        ms, out = case["ms"], []
        for q in range(case["settings"]):
            V = s["V"][q * ms:(q + 1) * ms]
            lam = torch.tensor([mu * N for mu in [1e-6, 1e-8][:ms]], device=_DEV, dtype=torch.float64)
            out.append(_multiply(X, X, kernels[q], sigmas[q], V) + lam[:, None] * V)
        return torch.cat(out)
    kern, sigma = case["kernel"], case["sigma"]
    if op == "predict":
        return _multiply(s["Xt"], X, kern, sigma, s["V"])
    lam = case["mu"] * N
    if op == "product":
        return _multiply(X, X, kern, sigma, s["V"]) + lam * s["V"]
    if op == "factor":
        F, R = _pivoted_factor(X, kern, sigma, case["k"], seed), s["V"]
        core = F @ F.T + lam * torch.eye(len(F), device=_DEV, dtype=torch.float64)
        inner = torch.cholesky_solve(F @ R.T, torch.linalg.cholesky(core))
        return (R - (F.T @ inner).T) / lam
    M = _kernel(X, X, kern, sigma)
    M.diagonal().add_(lam)
    alpha = torch.cholesky_solve(s["Y"].T.contiguous(), torch.linalg.cholesky(M)).T
    return s["Y"] - lam * alpha
