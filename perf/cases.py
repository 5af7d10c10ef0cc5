"""The work a user of this package has it do, as cases that can be timed and checked.

Each case is one call, or one fit, through the public Python API (paper_1905_10587_gb300.api)
on seeded synthetic data of the package's own recipes (the point sets and targets of synth/,
redrawn here on the GPU):

* mixture  10 Gaussian clusters (means U[-5,5]^d, unit variance), sigma = 1, beta = 1e-3;
* cube     U[0,side]^3 at the density of 10^6 points per 10^3 volume, sigma = 0.8, beta = 1e-4;
* normal   N(0, I_d), sigma = sqrt(d), beta = 1e-3;
* unit     U[0,1]^d, sigma = 0.5, beta = 1e-2.

Kinds: kmvm (a kernel product (K + beta I) V), residual (the FP64-accurate residual), apply
(the preconditioner), predict (K(Xtest, X) alpha), fit (build + solve), grad (the held-out loss
and its gradients) and batch (many small problems).  A fit returns what its residual tolerance
determines: on the clusters, where alpha is only fixed to about tol / beta, the predictions on a
test set; on smooth data, where large coefficients cancel in the predictions, the coefficients,
in the single precision that predict takes them in.
"""
import math

import torch

from paper_1905_10587_gb300 import api

DEV = "cuda"


def listed():
    return [
        # the inner loop of every solve with the tensor cores on: the headline product of bench.py
        dict(name="kmvm_tc", kind="kmvm", recipe="mixture", n=100000, d=8, r=1, precision=1),
        # the same call with the default options (FP32 tiles), at an odd size and another dimension
        dict(name="kmvm_fp32", kind="kmvm", recipe="normal", n=30011, d=6, r=1, precision=0),
        # the exact-difference form, which solves fall back to when FP32 expansion is too coarse
        dict(name="kmvm_diff", kind="kmvm", recipe="normal", n=20011, d=12, r=1, precision=2),
        # a block of 16 right-hand sides on 3-D data (the multi-output / batched-solve product)
        dict(name="kmvm_tc_16rhs", kind="kmvm", recipe="cube", n=50021, d=3, r=16, precision=1),
        # the smallest call there is: a handful of query points against a fitted model (serving)
        dict(name="predict_few", kind="predict", recipe="mixture", n=20000, d=8, r=1, m=7, k=200, precision=0),
        # a whole test set at once, several outputs
        dict(name="predict_many", kind="predict", recipe="mixture", n=100000, d=8, r=4, m=20011, k=200,
             precision=0),
        # the verified residual that ends every solve and drives its refinement
        dict(name="residual", kind="residual", recipe="mixture", n=30011, d=8, r=1),
        # one preconditioner application at the headline size (two passes over n x k)
        dict(name="apply", kind="apply", recipe="mixture", n=100000, d=8, r=1, k=1000, precision=1),
        # a small fit with the default options: launches and host reads dominate
        dict(name="fit_small", kind="fit", recipe="unit", n=2000, d=4, r=1, k=100, precision=0),
        # the headline workload: build + solve to 1e-6 on 10^5 points with the tensor cores, and
        # the predictions on a test set
        dict(name="fit_mixture", kind="fit", recipe="mixture", n=100000, d=8, r=1, m=10007, k=1000, precision=1),
        # one hyperparameter step: held-out loss and its gradients (two solves, derivative products)
        dict(name="grad", kind="grad", recipe="mixture", n=4001, d=8, r=1, m=600, k=150, precision=0),
        # many small problems at once, 8 right-hand sides each (batched regression)
        dict(name="batch", kind="batch", recipe="normal", n=3000, d=6, r=8, nprob=8, k=200, precision=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["kmvm"] * 5 + ["predict"] * 2 + ["residual", "apply", "fit", "fit", "grad", "batch"])
    if kind == "kmvm":
        recipe = rng.choice(["mixture", "normal", "normal", "cube"])
        d = 3 if recipe == "cube" else rng.randint(2, 16) if recipe == "normal" else 8
        return dict(kind=kind, recipe=recipe, n=_log(rng, 500, 100000), d=d, r=rng.choice([1, 1, 1, 2, 3, 4, 8, 16]),
                    precision=rng.choice([0, 1, 1, 2]))
    if kind == "predict":
        return dict(kind=kind, recipe="mixture", n=_log(rng, 2000, 100000), d=8, r=rng.choice([1, 1, 4]),
                    m=_log(rng, 1, 20000), k=rng.randint(50, 300), precision=rng.choice([0, 0, 1, 2]))
    if kind == "residual":
        recipe = rng.choice(["mixture", "normal"])
        return dict(kind=kind, recipe=recipe, n=_log(rng, 1000, 40000), d=8 if recipe == "mixture" else rng.randint(2, 16),
                    r=rng.choice([1, 1, 2]))
    if kind == "apply":
        return dict(kind=kind, recipe="mixture", n=_log(rng, 4000, 100000), d=8, r=rng.choice([1, 1, 8]),
                    k=_log(rng, 50, 1000), precision=rng.choice([0, 1]))
    if kind == "fit":
        if rng.random() < 0.5:
            return dict(kind=kind, recipe="unit", n=_log(rng, 500, 8000), d=rng.randint(3, 5), r=1, k=rng.randint(40, 150),
                        precision=rng.choice([0, 1, 2]))
        n = _log(rng, 10000, 40000)
        return dict(kind=kind, recipe="mixture", n=n, d=8, r=1, m=rng.randint(500, 5000), k=rng.randint(100, 500),
                    precision=rng.choice([0, 1]))
    if kind == "grad":
        return dict(kind=kind, recipe="mixture", n=_log(rng, 500, 6000), d=8, r=1, m=rng.randint(100, 900),
                    k=rng.randint(60, 150), precision=0)
    return dict(kind=kind, recipe="normal", n=_log(rng, 1000, 5000), d=rng.randint(3, 12), r=8, nprob=rng.randint(2, 10),
                k=rng.randint(80, 200), precision=1)


# ------------------------------------------------------------------ inputs
def _params(case):
    d = case["d"]
    return {"mixture": (1.0, 1e-3), "cube": (0.8, 1e-4), "normal": (math.sqrt(d), 1e-3), "unit": (0.5, 1e-2)}[case["recipe"]]


def _points(case, g, n, m):
    """n training and m test points of the case's recipe (float32, on the GPU)."""
    d, t = case["d"], n + m
    if case["recipe"] == "mixture":
        mu = torch.rand((10, d), generator=g, device=DEV) * 10 - 5
        lab = torch.randint(0, 10, (t,), generator=g, device=DEV)
        X = mu[lab] + torch.randn((t, d), generator=g, device=DEV)
    elif case["recipe"] == "cube":
        X = torch.rand((t, d), generator=g, device=DEV) * (10.0 * (n / 1e6) ** (1.0 / 3.0))
    elif case["recipe"] == "unit":
        X = torch.rand((t, d), generator=g, device=DEV)
    else:
        X = torch.randn((t, d), generator=g, device=DEV)
    return X[:n].contiguous(), X[n:].contiguous()


def _targets(case, g, X, r):
    n, d = X.shape
    if case["recipe"] == "mixture":
        y = X.norm(dim=1) * torch.cos(X[:, 0]) + 0.05 * torch.randn(n, generator=g, device=DEV)
    elif case["recipe"] == "unit":
        y = torch.sin(2 * math.pi * X.sum(dim=1)) + 0.01 * torch.randn(n, generator=g, device=DEV)
    elif case["recipe"] == "cube":
        y = torch.sin(X).sum(dim=1) + 0.1 * torch.randn(n, generator=g, device=DEV)
    else:
        W = torch.randn((r, d), generator=g, device=DEV)
        return torch.sin(X @ W.t())
    if r == 1:
        return y[:, None].contiguous()
    return torch.cat([y[:, None], torch.randn((n, r - 1), generator=g, device=DEV)], dim=1)


def _inputs(case, seed):
    """Everything drawn for one case, from its seed alone."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    kind, n, r = case["kind"], case["n"], case["r"]
    if kind == "batch":
        probs = []
        for i in range(case["nprob"]):
            ni = max(200, int(n * (0.5 + 1.5 * i / max(1, case["nprob"] - 1))))
            X, _ = _points(case, g, ni, 0)
            probs.append((X, _targets(case, g, X, r)))
        return dict(probs=probs)
    X, Xt = _points(case, g, n, case.get("m", 0))
    out = dict(X=X, Xt=Xt)
    if kind in ("kmvm", "residual", "fit"):
        Y = _targets(case, g, X, r)
        out["Y"] = Y[:, 0].contiguous() if r == 1 else Y
    if kind in ("apply", "predict"):
        out["V"] = torch.randn((n, r) if r > 1 else (n,), generator=g, device=DEV)
    if kind == "residual":
        out["A"] = torch.randn((n, r) if r > 1 else (n,), generator=g, device=DEV, dtype=torch.float64)
    if kind in ("apply", "predict"):
        out["S"] = torch.randperm(n, generator=g, device=DEV)[:case["k"]].to(torch.int32)
    if kind == "grad":
        XX = torch.cat([X, Xt])
        yy = _targets(case, g, XX, 1)[:, 0]
        out["y"], out["yv"] = yy[:n].contiguous(), yy[n:].contiguous()
    return out


def prepare(case, seed):
    st = _inputs(case, seed)
    st["case"] = case
    st["sigma"], st["beta"] = _params(case)
    kind = case["kind"]
    if kind in ("kmvm", "predict", "apply", "fit", "residual"):
        st["ctx"] = api.KRR(precision=case.get("precision", 0))
    if kind in ("apply", "predict"):
        st["ctx"].build(st["X"], st["sigma"], st["beta"], case["k"], anchors=st["S"])
    if kind == "grad":
        st["y"].requires_grad_()
        st["ls"] = torch.tensor(math.log(st["sigma"]), requires_grad=True)
        st["lb"] = torch.tensor(math.log(st["beta"]), requires_grad=True)
    return st


# ------------------------------------------------------------------ one pass
def run(st):
    case, kind, sigma, beta = st["case"], st["case"]["kind"], st["sigma"], st["beta"]
    if kind == "kmvm":
        return st["ctx"].kmvm(st["X"], st["X"], st["Y"], sigma, beta)
    if kind == "predict":
        return st["ctx"].predict(st["Xt"], st["V"])
    if kind == "residual":
        return st["ctx"].residual_hp(st["X"], st["Y"], st["A"], sigma, beta, mode="ff")
    if kind == "apply":
        return st["ctx"].apply_precond(st["V"])
    if kind == "fit":
        ctx = st["ctx"]
        ctx.build(st["X"], sigma, beta, case["k"], seed=1)
        alpha, _ = ctx.solve(st["Y"], tol=1e-6)
        return ctx.predict(st["Xt"], alpha.float()) if case["recipe"] == "mixture" else alpha.float()
    if kind == "grad":
        st["y"].grad = st["ls"].grad = st["lb"].grad = None
        loss = api.validation_loss(st["y"], st["ls"], st["lb"], st["X"], st["Xt"], st["yv"], case["k"],
                                   precision=case["precision"])
        loss.backward()
        return [loss.item(), st["y"].grad, st["ls"].grad, st["lb"].grad]
    probs = [(X, Y, sigma, beta, case["k"]) for X, Y in st["probs"]]
    alphas, _, _ = api.batch_solve(probs, tol=1e-6, precision=case["precision"])
    return [a.float() for a in alphas]


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    kind, n, d, r, m, k = (case["kind"], case["n"], case["d"], case["r"], case.get("m", 0), case.get("k", 0))
    # a kernel value costs its exponent (2d + 2) and an exponential (1); a square product has
    # n^2 / 2 distinct ones; each right-hand side adds a multiply-add per entry
    def square(n):
        return n * n / 2.0 * (2 * d + 3) + 2.0 * r * n * n

    if kind == "kmvm":
        return dict(bytes=4.0 * (n * d + 2 * n * r), flops=square(n))
    if kind == "predict":
        return dict(bytes=4.0 * ((n + m) * d + (n + m) * r), flops=float(n) * m * (2 * d + 3 + 2 * r))
    if kind == "residual":
        return dict(bytes=4.0 * (n * d + n * r) + 16.0 * n * r, flops=square(n))
    if kind == "apply":
        # u = F^T r is complete before F v begins: two reads of F
        return dict(bytes=8.0 * n * k + 8.0 * n * r, flops=4.0 * n * k * r)
    if kind in ("fit", "grad"):
        # sketch, pivoted QR (half its flops at least a read of what is left), factor and Gram
        # matrix, and the products of the solve: about 30 on smooth data, 100 to 800 on the clusters
        its = (2 if kind == "grad" else 1) * (30 if case["recipe"] == "unit" else 100 + n // 150)
        build = 2.0 * n * n * k + 6.0 * n * k * k
        return dict(bytes=4.0 * n * k * (4 + 2 * its) + 4.0 * n * d, flops=build + its * square(n))
    ns = [max(200, int(n * (0.5 + 1.5 * i / max(1, case["nprob"] - 1)))) for i in range(case["nprob"])]
    its = 100
    return dict(bytes=sum(4.0 * q * k * 2 * its for q in ns),
                flops=sum(2.0 * q * q * k + 6.0 * q * k * k + its * square(q) for q in ns))


# ------------------------------------------------------------------ the same in 64 bits
def _kernel(A, B, sigma):
    """exp(-||a - b||^2 / (2 sigma^2)) in float64."""
    A, B = A.double(), B.double()
    c = B.mean(dim=0)
    A, B = A - c, B - c
    D = (A * A).sum(1)[:, None] + (B * B).sum(1)[None, :] - 2.0 * (A @ B.t())
    return torch.exp(D.clamp_(min=0.0) * (-0.5 / (sigma * sigma)))


def _product(A, B, V, sigma):
    V = V.double()
    step = max(1, 200_000_000 // B.shape[0])
    return torch.cat([_kernel(A[i:i + step], B, sigma) @ V for i in range(0, A.shape[0], step)])


def _krr(X, Y, sigma, beta):
    K = _kernel(X, X, sigma)
    K.diagonal().add_(beta)
    Y = Y.double()
    a = torch.cholesky_solve(Y if Y.dim() == 2 else Y[:, None], torch.linalg.cholesky(K))
    return a if Y.dim() == 2 else a[:, 0]


def exact(case, seed):
    kind = case["kind"]
    if kind == "fit" and case["n"] > 20000:
        return None                       # a dense factor of this size takes too long
    st = _inputs(case, seed)
    sigma, beta = _params(case)
    if kind == "kmvm":
        return _product(st["X"], st["X"], st["Y"], sigma) + beta * st["Y"].double()
    if kind == "predict":
        return _product(st["Xt"], st["X"], st["V"], sigma)
    if kind == "residual":
        return st["Y"].double() - _product(st["X"], st["X"], st["A"], sigma) - beta * st["A"]
    if kind == "apply":
        X, S, V = st["X"], st["S"].long(), st["V"].double()
        L = torch.linalg.cholesky(_kernel(X[S], X[S], sigma))
        F = torch.linalg.solve_triangular(L, _kernel(X[S], X, sigma), upper=False).t()
        G = F.t() @ F
        G.diagonal().add_(beta)
        R = V if V.dim() == 2 else V[:, None]
        Z = (R - F @ torch.cholesky_solve(F.t() @ R, torch.linalg.cholesky(G))) / beta
        return Z if V.dim() == 2 else Z[:, 0]
    if kind == "fit":
        a = _krr(st["X"], st["Y"], sigma, beta)
        return _product(st["Xt"], st["X"], a, sigma) if case["recipe"] == "mixture" else a
    if kind == "batch":
        return [_krr(X, Y, sigma, beta) for X, Y in st["probs"]]
    # the gradients of the held-out mean squared error, by autograd through the dense solve
    y = st["y"].double().requires_grad_()
    ls = torch.tensor(float(torch.tensor(math.log(sigma))), dtype=torch.float64, device=DEV, requires_grad=True)
    lb = torch.tensor(float(torch.tensor(math.log(beta))), dtype=torch.float64, device=DEV, requires_grad=True)
    X, Xt = st["X"].double(), st["Xt"].double()

    def kern(A, B):
        D = (A * A).sum(1)[:, None] + (B * B).sum(1)[None, :] - 2.0 * (A @ B.t())
        return torch.exp(D.clamp(min=0.0) * (-0.5 * torch.exp(-2.0 * ls)))

    K = kern(X, X) + torch.exp(lb) * torch.eye(X.shape[0], dtype=torch.float64, device=DEV)
    a = torch.cholesky_solve(y[:, None], torch.linalg.cholesky(K))
    loss = ((kern(Xt, X) @ a)[:, 0] - st["yv"].double()).square().mean()
    loss.backward()
    return [loss.item(), y.grad, ls.grad, lb.grad]
