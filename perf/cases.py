"""Workloads of libkrr that are timed and compared between versions of the library.

Every case goes through the Python binding as a user's program does.  The
sizes are those of the repository's own configurations (the 2,000-point plane,
the 2^20-point cube, the 16-component mixture, the d = 8 batch, the d = 4
gradient, the Matern and high-dimensional tables) and of their neighbourhood.
A case is a dict of plain values whose "kind" is one of

  product   krr_kernel_mvp: Y = (K_hat + gamma I) Q on new points
  prepared  krr_kernel_mvp_points: the same over a prepared point set
  predict   krr_kernel_mvp_rect: Y = K_hat(Xt, X) Q, the regression mean
  fit       krr_fgmres_solve: the weights of a regression
  batch     krr_fgmres_solve_batched: several problems, 16 right-hand sides each
  gradient  autograd.mll_surrogate: gradients of the log marginal likelihood
"""
import math

import numpy as np
import torch

from paper_1408_1237_gb300 import autograd
from paper_1408_1237_gb300 import binding as K


def width(case):
    cloud, d = case["cloud"], case["d"]
    if case.get("family") == "matern":
        return 0.1 if cloud == "cube" else math.sqrt(d)
    if cloud == "mixture":
        return 0.03
    if cloud == "normal":
        return 1.0
    if cloud == "wide":
        return 0.3 * math.sqrt(d)
    return {1: 0.02, 2: 0.1, 3: 0.05}.get(d, 0.2)


def listed():
    return [
        # the smallest call: one weight vector on a few thousand new points,
        # where preparation, launches and waits decide
        dict(name="product_4096", kind="product", cloud="cube", N=4096, d=3, m=1, gamma=1e-3),
        # a serving loop or a caller's own iteration over a fixed point set
        dict(name="prepared_4096", kind="prepared", cloud="cube", N=4096, d=3, m=1, gamma=1e-3),
        # an ordinary kriging-like cloud in the plane, clustered, odd size
        dict(name="product_mixture_50021", kind="product", cloud="mixture", N=50021, d=2, m=1, gamma=1e-3),
        # the headline product of the paper's kind: 2^20 points in the cube
        dict(name="product_cube_1M", kind="product", cloud="cube", N=1 << 20, d=3, m=1, gamma=1e-3),
        # many right-hand sides at once (block iterations, several outputs)
        dict(name="product_cube_16col", kind="product", cloud="cube", N=131072, d=3, m=16, gamma=1e-3),
        # the reduced-precision inner product on normal data in d = 8, where
        # the target blocks are too wide for the expanded form
        dict(name="product_normal_d8_fp16", kind="product", cloud="normal", N=16385, d=8, m=16, gamma=1e-2,
             prec="fp16"),
        # the paper's second kernel function
        dict(name="product_matern_100003", kind="product", cloud="cube", N=100003, d=3, m=1, gamma=1e-2,
             family="matern"),
        # feature vectors of the classification tables (d = 25, padded to 32)
        dict(name="product_d25", kind="product", cloud="wide", N=32768, d=25, m=1, gamma=1e-3),
        # a fitted model of a few outputs evaluated at many test points
        dict(name="predict_4col", kind="predict", cloud="cube", Nt=65541, N=20011, d=3, m=4),
        # the 2,000-point plane (the paper's small study)
        dict(name="fit_2000", kind="fit", cloud="cube", N=2000, d=2, m=1, gamma=1e-2),
        # several Gaussian-process problems of uneven size in one call
        dict(name="batch_6x16", kind="batch", cloud="normal", count=6, n_lo=1024, n_hi=4096, d=8, m=16),
        # one step of a maximum-likelihood fit of width, noise and inputs
        dict(name="gradient_2000", kind="gradient", cloud="cube", N=2000, d=4, probes=32, gamma=1e-2),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["product"] * 5 + ["prepared", "predict", "predict", "fit", "batch", "gradient"])
    if kind == "fit":
        return dict(kind=kind, cloud="cube", N=log_int(500, 4000), d=2, m=rng.choice([1, 1, 2, 5]),
                    gamma=math.exp(rng.uniform(math.log(5e-3), math.log(1e-1))))
    if kind == "batch":
        return dict(kind=kind, cloud="normal", count=rng.randint(2, 6), n_lo=1024, n_hi=log_int(1500, 4096), d=8,
                    m=rng.choice([4, 16]))
    if kind == "gradient":
        return dict(kind=kind, cloud="cube", N=log_int(500, 2000), d=4, probes=rng.choice([8, 16, 32]), gamma=1e-2)
    cloud = rng.choice(["cube", "cube", "mixture", "normal", "wide"])
    d = {"cube": rng.randint(1, 4), "mixture": 2, "normal": rng.randint(5, 8), "wide": rng.randint(9, 64)}[cloud]
    m = rng.choice([1, 1, 1, rng.randint(2, 8), 16])
    case = dict(kind=kind, cloud=cloud, d=d, m=m)
    # a drawn case costs no more than the largest listed product
    most = {"cube": 700000, "mixture": 700000, "normal": 120000, "wide": 60000}[cloud] / (1 if m == 1 else 4)
    if rng.random() < 0.15 and kind == "product" and cloud != "mixture":
        case["family"] = "matern"
        most /= 3
    elif rng.random() < 0.2 and kind != "predict":
        case["prec"] = rng.choice(["fp16", "bf16"])
        most /= 2
    if kind == "predict":
        case.update(Nt=log_int(500, most / 4), N=log_int(500, most / 4))
        return case
    case.update(N=log_int(1000, most / (4 if kind == "prepared" else 1)),
                gamma=math.exp(rng.uniform(math.log(1e-4), math.log(1e-1))))
    return case


# ------------------------------------------------------------------ inputs
def cloud_points(case, n, gen):
    d, dev = case["d"], "cuda"
    if case["cloud"] == "mixture":
        # 16 components of standard deviation 0.02 with means in the unit square
        means = torch.rand(16, 2, device=dev, generator=torch.Generator(dev).manual_seed(gen.initial_seed() + 1))
        label = torch.randint(16, (n,), device=dev, generator=gen)
        return means[label] + 0.02 * torch.randn(n, 2, device=dev, generator=gen)
    if case["cloud"] == "normal":
        return torch.randn(n, d, device=dev, generator=gen)
    return torch.rand(n, d, device=dev, generator=gen)


def columns(m, n, gen):
    q = torch.randn(m, n, device="cuda", generator=gen)
    return q[0].contiguous() if m == 1 else q


def smooth_field(X):
    return torch.sin(2 * math.pi * X[:, 0]) * torch.cos(2 * math.pi * X[:, 1])


def gp_sample(X, sigma, gen, features=1024):
    """A draw from a Gaussian process by random Fourier features, plus noise."""
    omega = torch.randn(X.shape[1], features, device="cuda", generator=gen) / sigma
    phi = 2 * math.pi * torch.rand(features, device="cuda", generator=gen)
    w = torch.randn(features, device="cuda", generator=gen)
    f = math.sqrt(2.0 / features) * (torch.cos(X @ omega + phi) @ w)
    return f + 0.2 * torch.randn(X.shape[0], device="cuda", generator=gen)


def batch_sizes(case):
    """Sizes log-spaced from n_lo to n_hi, made odd."""
    c = case["count"]
    return [int(case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** (k / max(c - 1, 1))) | 1 for k in range(c)]


def batch_gammas(case):
    c = case["count"]
    return [10.0 ** (-3 + 2 * k / max(c - 1, 1)) for k in range(c)]


_matern = []


def matern_handle():
    if not _matern:
        _matern.append(K.Handle())
        K.krr_set_option(K.KRR_OPT_KERNEL, K.KRR_KERNEL_MATERN32, handle=_matern[0])
    return _matern[0]


def prepare(case, seed):
    gen = torch.Generator("cuda").manual_seed(seed)
    kind = case["kind"]
    s = dict(case=case, sigma=width(case), handle=matern_handle() if case.get("family") == "matern" else None)
    if kind in ("product", "prepared"):
        s["X"] = cloud_points(case, case["N"], gen)
        s["Q"] = columns(case["m"], case["N"], gen)
        if kind == "prepared":
            s["points"] = K.Points(s["X"], s["sigma"])
    elif kind == "predict":
        s["X"] = cloud_points(case, case["N"], gen)
        s["Xt"] = cloud_points(case, case["Nt"], gen)
        s["Q"] = columns(case["m"], case["N"], gen)
    elif kind == "fit":
        s["X"] = cloud_points(case, case["N"], gen)
        noise = 0.1 * torch.randn(case["m"], case["N"], device="cuda", generator=gen)
        B = smooth_field(s["X"]) + noise
        s["B"] = B[0].contiguous() if case["m"] == 1 else B
        # weights accurate to float32, the type the prediction product takes
        s["opts"] = K.default_opts(delta=0.1, inner_tol=1e-2, restart=30, tol=1e-8)
    elif kind == "batch":
        s["problems"] = []
        for n, g in zip(batch_sizes(case), batch_gammas(case)):
            B = torch.randn(case["m"], n, device="cuda", generator=gen)
            s["problems"].append(dict(X=cloud_points(case, n, gen), B=B, gamma=g,
                                      Xsol=torch.empty(case["m"], n, device="cuda", dtype=torch.float64)))
        s["opts"] = K.default_opts(inner_tol=1e-2, inner_maxit=400, restart=30, max_cycles=8, tol=1e-8)
    else:
        s["X"] = cloud_points(case, case["N"], gen).requires_grad_()
        s["y"] = gp_sample(s["X"].detach(), 1.5 * s["sigma"], gen)  # the fit starts off its optimum
        s["log_sigma"] = torch.tensor(math.log(s["sigma"]), requires_grad=True)
        s["log_gamma"] = torch.tensor(math.log(case["gamma"]), requires_grad=True)
        s["seed"] = seed
        s["opts"] = K.default_opts(tol=1e-8, max_cycles=20)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "product":
        return K.krr_kernel_mvp(s["X"], s["Q"], s["sigma"], case["gamma"], prec=case.get("prec", "fp32"),
                                handle=s["handle"])
    if kind == "prepared":
        return K.krr_kernel_mvp_points(s["points"], s["Q"], case["gamma"], prec=case.get("prec", "fp32"))
    if kind == "predict":
        return K.krr_kernel_mvp_rect(s["Xt"], s["X"], s["Q"], s["sigma"])
    if kind == "fit":
        x, _ = K.krr_fgmres_solve(s["X"], s["B"], s["sigma"], case["gamma"], opts=s["opts"])
        return x.float()  # weights for the prediction product
    if kind == "batch":
        K.krr_fgmres_solve_batched(s["problems"], case["d"], s["sigma"], case["m"], opts=s["opts"])
        return [p["Xsol"].float() for p in s["problems"]]  # weights for the prediction product
    leaves = (s["X"], s["log_sigma"], s["log_gamma"])
    loss = autograd.mll_surrogate(s["X"], s["log_sigma"], s["log_gamma"], s["y"], n_probes=case["probes"],
                                  seed=s["seed"], opts=s["opts"])
    return dict(zip(("dX", "dlog_sigma", "dlog_gamma"), torch.autograd.grad(loss, leaves)))


def work(case):
    """Inputs and outputs once each; per pair of points the squared distance
    (2 d operations as a dot product), one exponential and 2 m operations of
    the weighted sum.  A solve needs its kernel matrix and one factorisation."""
    kind, d = case["kind"], case["d"]
    if kind in ("product", "prepared"):
        N, m = case["N"], case["m"]
        return dict(bytes=4.0 * N * (d + 2 * m), flops=float(N) * N * (2 * d + 1 + 2 * m))
    if kind == "predict":
        N, Nt, m = case["N"], case["Nt"], case["m"]
        return dict(bytes=4.0 * (N * (d + m) + Nt * (d + m)), flops=float(N) * Nt * (2 * d + 1 + 2 * m))
    if kind == "fit":
        N, m = case["N"], case["m"]
        return dict(bytes=4.0 * N * (d + 2 * m), flops=float(N) * N * (2 * d + 1 + 2 * m) + N ** 3 / 3.0)
    if kind == "batch":
        m, ns = case["m"], batch_sizes(case)
        return dict(bytes=sum(4.0 * n * (d + 2 * m) for n in ns),
                    flops=sum(float(n) * n * (2 * d + 1 + 2 * m) + n ** 3 / 3.0 for n in ns))
    N, m = case["N"], 1 + case["probes"]
    return dict(bytes=4.0 * N * (2 * d + 1), flops=float(N) * N * (2 * d + 1 + 2 * m * (2 + d)) + N ** 3 / 3.0)


# ------------------------------------------------------- 64-bit evaluation
def f32(v):
    return float(np.float32(v))  # sigma and gamma as the C interface receives them


def kernel64(A, B, sigma, family):
    r2 = torch.zeros(A.shape[0], B.shape[0], dtype=torch.float64, device=A.device)
    for k in range(A.shape[1]):
        r2 += (A[:, k, None] - B[None, :, k]) ** 2
    if family == "matern":
        a = math.sqrt(3.0) / sigma * r2.sqrt_()
        return (1.0 + a) * torch.exp(-a)
    return torch.exp_(r2.mul_(-0.5 / sigma ** 2))


def product64(A, B, Q, sigma, family=None):
    """K_hat(A, B) Q^T as rows like Q, in blocks of targets."""
    A, B, Q2 = A.double(), B.double(), Q.double().reshape(-1, B.shape[0])
    step = max(1, (1 << 27) // B.shape[0])
    out = torch.cat([kernel64(A[i:i + step], B, sigma, family) @ Q2.T for i in range(0, A.shape[0], step)])
    return out.T.contiguous() if Q.ndim == 2 else out[:, 0].contiguous()


def solve64(X, B, sigma, gamma):
    k = kernel64(X.double(), X.double(), sigma, None)
    k.diagonal().add_(gamma)
    L = torch.linalg.cholesky(k)
    return torch.cholesky_solve(B.double().reshape(-1, X.shape[0]).T, L).T.reshape(B.shape)


def probes64(seed, N, P):
    """Element (p, i) is -1 where the top bit of SplitMix64 output number
    p N + i + 1 is set (the estimator's documented probes)."""
    mask = (1 << 64) - 1
    c = np.arange(1, N * P + 1, dtype=np.uint64)
    with np.errstate(over="ignore"):
        z = np.uint64(seed & mask) + c * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return torch.from_numpy(np.where(z >> np.uint64(63), -1.0, 1.0).reshape(P, N)).cuda()


def gradient64(X, y, sigma, gamma, seed, P):
    """The Hutchinson estimate of the log-marginal-likelihood gradient with
    dense solves: W = (a a' - U Z' / P) / 2 and w = W + W'."""
    X = X.detach().double()
    N = X.shape[0]
    Z = probes64(seed, N, P)
    sol = solve64(X, torch.cat([y.double()[None], Z]), sigma, gamma)
    a, U = sol[0], sol[1:]
    W = 0.5 * (torch.outer(a, a) - U.T @ Z / P)
    wk = (W + W.T) * kernel64(X, X, sigma, None)
    G = X * wk.sum(1, keepdim=True) - wk @ X
    r2 = torch.zeros_like(wk)
    for k in range(X.shape[1]):
        r2 += (X[:, k, None] - X[None, :, k]) ** 2
    return dict(dX=-G / sigma ** 2, dlog_sigma=(wk * r2).sum() * (0.5 / sigma ** 2), dlog_gamma=gamma * W.trace())


def exact(case, seed):
    kind = case["kind"]
    pairs = float(case.get("Nt", case.get("N", 0))) * case.get("N", 0)
    if pairs > 1.5e11:
        return None  # over 20 seconds in 64 bits
    s = prepare(case, seed)
    sigma, gamma = f32(s["sigma"]), f32(case.get("gamma", 0.0))
    if kind in ("product", "prepared"):
        return product64(s["X"], s["X"], s["Q"], sigma, case.get("family")) + gamma * s["Q"].double()
    if kind == "predict":
        return product64(s["Xt"], s["X"], s["Q"], sigma)
    if kind == "fit":
        return solve64(s["X"], s["B"], sigma, gamma)
    if kind == "batch":
        return [solve64(p["X"], p["B"], sigma, f32(p["gamma"])) for p in s["problems"]]
    # the hyper-parameters as the float32 logarithms give them
    sigma = f32(float(torch.exp(s["log_sigma"].detach())))
    gamma = f32(float(torch.exp(s["log_gamma"].detach())))
    return gradient64(s["X"], s["y"], sigma, gamma, s["seed"], case["probes"])
