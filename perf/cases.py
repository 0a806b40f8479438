"""Performance cases: the calls a program built on this package makes.

Each case is one pass through the public Python entry points on inputs that
are resident on the GPU: Gaussian-process likelihood steps (value, gradient
and everything a sampler keeps), Cholesky factors with their reverse mode,
batches of small GPs, triangular solves, matrix products and GLM likelihoods.
``listed()`` names the representative ones and ``draw`` gives further sizes of
the same ranges.
"""
from __future__ import annotations

import math
import random

import torch

import paper_1907_01063_gb300 as gp

F64 = torch.float64


def listed():
    return [
        # The 256-point GP of the parity configuration, differentiated by autograd as an
        # optimiser or sampler does: the smallest call, launches and latency count.
        dict(name="gp_autograd_256", kind="gp_autograd", n=256, d=2, rho=0.5, sigma=0.1, jitter=1e-8,
             precision="fp64"),
        # One-dimensional GP regression at the size of the paper's Section 4.2 experiments.
        dict(name="gp_fp64_1000", kind="gp", n=1000, d=1, rho=0.3, sigma=0.3, jitter=1e-8, precision="fp64"),
        # An ordinary FP64 GP step (the conditioning tests' size and kernel).
        dict(name="gp_fp64_4096", kind="gp", n=4096, d=16, rho=4.0, sigma=0.256, jitter=0.0, precision="fp64"),
        # An ordinary mixed-precision step at an odd size: ragged tiles everywhere.
        dict(name="gp_mixed_2049", kind="gp", n=2049, d=3, rho=1.0, sigma=0.3, jitter=1e-6, precision="mixed"),
        # The benchmark's GP step.
        dict(name="gp_mixed_16384", kind="gp", n=16384, d=16, rho=4.0, sigma=0.256, jitter=0.0,
             precision="mixed"),
        # Cholesky factor inside a user's own model, forward and backward, odd size.
        dict(name="chol_fp64_6007", kind="chol", n=6007, d=8, rho=2.8, sigma=0.3, precision="fp64"),
        # The benchmark's batch of small GPs in one launch.
        dict(name="batch_fp64_512", kind="batch", batch=512, lo=64, hi=1024, d=4, size_seed=0, precision="fp64"),
        # A smaller batch in mixed precision (a few dozen groups of a hierarchical model).
        dict(name="batch_mixed_96", kind="batch", batch=96, lo=32, hi=512, d=3, size_seed=1, precision="mixed"),
        # Triangular solve with a block of right-hand sides and its reverse mode.
        dict(name="tri_solve_4096", kind="tri", n=4096, m=16),
        # Matrix product and its reverse mode at ragged sizes (Section 3.1 multiplies such shapes).
        dict(name="matmul_2000", kind="matmul", m=2000, k=1537, n=1025),
        # The benchmark's logistic regression: value and gradient over a million rows.
        dict(name="glm_bernoulli_1m", kind="glm", family="bernoulli_logit", n=1 << 20, k=512),
        # A small Poisson regression: a call of some tens of microseconds.
        dict(name="glm_poisson_10k", kind="glm", family="poisson_log", n=10007, k=25),
    ]


def _log_size(rng: random.Random, lo: int, hi: int) -> int:
    """A size spread over the logarithm of [lo, hi]; about half of them odd."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["gp", "gp", "gp", "gp_autograd", "chol", "batch", "tri", "matmul", "gemm", "glm", "glm",
                       "glm_classes", "trsv"])
    if kind in ("gp", "gp_autograd", "chol"):
        precision = rng.choice(["fp64", "mixed"])
        hi = 5200 if precision == "fp64" else 9000
        d = rng.choice([1, 2, 3, 8, 16])
        case = dict(kind=kind, n=_log_size(rng, 200, hi if kind != "gp_autograd" else 3000), d=d,
                    rho=round(rng.uniform(0.5, 1.1) * math.sqrt(d), 3), sigma=round(rng.uniform(0.2, 0.5), 3),
                    precision=precision)
        if kind != "chol":
            case["jitter"] = rng.choice([0.0, 1e-8, 1e-6])
        return case
    if kind == "batch":
        return dict(kind="batch", batch=_log_size(rng, 8, 400), lo=32, hi=rng.choice([128, 300, 512, 800]),
                    d=rng.choice([1, 2, 4, 7]), size_seed=rng.randrange(1 << 20),
                    precision=rng.choice(["fp64", "mixed"]))
    if kind == "tri":
        return dict(kind="tri", n=_log_size(rng, 200, 4500), m=_log_size(rng, 1, 300))
    if kind == "trsv":
        return dict(kind="trsv", n=_log_size(rng, 200, 16384), trans=rng.choice([False, True]))
    if kind == "matmul":
        return dict(kind="matmul", m=_log_size(rng, 64, 3000), k=_log_size(rng, 64, 3000), n=_log_size(rng, 64, 3000))
    if kind == "gemm":  # k far above the output's sizes (the paper's special case)
        return dict(kind="gemm", m=_log_size(rng, 16, 300), k=_log_size(rng, 20000, 500000), n=_log_size(rng, 16, 300))
    if kind == "glm":
        return dict(kind="glm", family=rng.choice(["normal_id", "bernoulli_logit", "poisson_log",
                                                   "neg_binomial_2_log"]),
                    n=_log_size(rng, 500, 500000), k=_log_size(rng, 2, 700))
    return dict(kind="glm_classes", family=rng.choice(["categorical", "ordinal"]), n=_log_size(rng, 500, 200000),
                k=_log_size(rng, 2, 150), classes=rng.randint(3, 10))


# ------------------------------------------------------------------ inputs
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _gen(seed: int, dev):
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    return g


def _gp_data(n, d, rho, sigma, seed, dev):
    """Inputs N(0, 1) and targets: a random-Fourier-feature draw of the SE kernel plus noise."""
    g = _gen(seed, dev)
    X = torch.randn(n, d, generator=g, device=dev, dtype=F64)
    w = torch.randn(d, 256, generator=g, device=dev, dtype=F64) / rho
    b = torch.rand(256, generator=g, device=dev, dtype=F64) * (2.0 * math.pi)
    f = math.sqrt(2.0 / 256) * torch.cos(X @ w + b).sum(1)
    return X, f + sigma * torch.randn(n, generator=g, device=dev, dtype=F64)


def _plain_cov(X, alpha, rho, sigma, jitter):
    n = X.shape[0]
    r2 = torch.zeros(n, n, dtype=F64, device=X.device)
    for t in range(X.shape[1]):
        c = X[:, t]
        diff = c[:, None] - c[None, :]
        r2.addcmul_(diff, diff)
        del diff
    K = r2.mul(-0.5 / (rho * rho)).exp_().mul_(alpha * alpha)
    K.diagonal().add_(sigma * sigma + jitter)
    return K, r2


def _sizes(case):
    rng = random.Random(case["size_seed"])
    return [rng.randint(case["lo"], case["hi"]) for _ in range(case["batch"])]


def _lower_factor(n, g, dev):
    L = torch.randn(n, n, generator=g, device=dev, dtype=F64).tril_(-1).mul_(1.0 / math.sqrt(n))
    L.diagonal().copy_(1.0 + torch.rand(n, generator=g, device=dev, dtype=F64))
    return L


def _inputs(case, seed, dev):
    """The tensors of a case, made from the seed alone."""
    kind = case["kind"]
    g = _gen(seed, dev)

    def randn(*shape):
        return torch.randn(*shape, generator=g, device=dev, dtype=F64)

    if kind in ("gp", "gp_autograd"):
        X, y = _gp_data(case["n"], case["d"], case["rho"], case["sigma"], seed, dev)
        return dict(X=X, y=y)
    if kind == "chol":
        X, _ = _gp_data(case["n"], case["d"], case["rho"], case["sigma"], seed, dev)
        K, _ = _plain_cov(X, 1.0, case["rho"], case["sigma"], 0.0)
        return dict(K=K, Lbar=randn(case["n"], case["n"]).tril_())
    if kind == "batch":
        sizes = _sizes(case)
        rho = 0.2 + 1.8 * torch.rand(case["batch"], generator=g, device=dev, dtype=F64)
        hyp = torch.stack([torch.ones_like(rho), rho, torch.full_like(rho, 0.1)], 1).contiguous()
        rows = sum(sizes)
        X = randn(rows, case["d"])
        scale = torch.repeat_interleave(rho, torch.tensor(sizes, device=dev))
        w = randn(case["d"], 64)
        b = torch.rand(64, generator=g, device=dev, dtype=F64) * (2.0 * math.pi)
        y = math.sqrt(2.0 / 64) * torch.cos((X / scale[:, None]) @ w + b).sum(1) + 0.1 * randn(rows)
        return dict(X=X, y=y, hyp=hyp)
    if kind == "tri":
        return dict(L=_lower_factor(case["n"], g, dev), B=randn(case["n"], case["m"]),
                    Cbar=randn(case["n"], case["m"]))
    if kind == "trsv":
        return dict(L=_lower_factor(case["n"], g, dev), x=randn(case["n"]))
    if kind in ("matmul", "gemm"):
        m, k, n = case["m"], case["k"], case["n"]
        out = dict(A=randn(m, k), B=randn(k, n))
        if kind == "matmul":
            out["Cbar"] = randn(m, n)
        return out
    n, k = case["n"], case["k"]
    X = randn(n, k)
    u = torch.rand(n, generator=g, device=dev, dtype=F64)
    if kind == "glm":
        # the toy data of the paper's Section 4.1: two columns matter, the others are noise
        mu = 3.0 * X[:, 0] - 2.0 * X[:, 1] + 1.0
        beta = randn(k) / math.sqrt(k)
        if case["family"] == "bernoulli_logit":
            y = (u < torch.sigmoid(mu)).to(F64)
        elif case["family"] == "normal_id":
            y = mu + randn(n)
        else:
            y = torch.poisson(torch.exp(mu / 4.0), generator=g)
        return dict(X=X, y=y, beta=beta)
    C = case["classes"]
    y = torch.floor(u * C).clamp_(max=C - 1.0)
    if case["family"] == "categorical":
        return dict(X=X, y=y, alpha=randn(C), beta=randn(k, C) / math.sqrt(k))
    cuts = torch.linspace(-1.5, 1.5, C - 1, device=dev, dtype=F64) + 0.05 * randn(C - 1) / C
    return dict(X=X, y=y, beta=randn(k) / math.sqrt(k), cuts=torch.sort(cuts).values)


_GLM_ALPHA, _GLM_SIGMA = 0.5, 1.3


def prepare(case, seed):
    dev = torch.device("cuda")
    s = dict(case=case, **_inputs(case, seed, dev))
    kind = case["kind"]
    if kind == "gp":  # matrices and workspaces that a sampler's loop keeps
        n = case["n"]
        for name in ("K", "L", "Kbar"):
            s[name] = torch.zeros(n, n, dtype=F64, device=dev)
        s["ws"] = gp.workspace(n, case["precision"])
        s["hyper_ws"] = torch.empty(gp.se_hyper_grad_workspace_size(n), dtype=torch.uint8, device=dev)
        s["info"] = gp.new_info()
    elif kind == "gp_autograd":
        s["hyp"] = torch.tensor([1.0, case["rho"], case["sigma"]], dtype=F64)
    elif kind == "batch":
        s["batch"] = gp.Batch(_sizes(case), precision=case["precision"])
    elif kind == "gemm":
        s["ws"] = gp.gemm_workspace(dev)
    elif kind == "glm" or (kind == "glm_classes" and case["family"] == "ordinal"):
        s["ws"] = gp.glm_workspace(case["k"], dev)
    elif kind == "trsv":
        s["ws"] = gp.workspace(case["n"])
    return s


def run(state):
    s, case = state, state["case"]
    kind = case["kind"]
    if kind == "gp":
        p, rho, sigma = case["precision"], case["rho"], case["sigma"]
        gp.se_cov(s["X"], 1.0, rho, sigma, case["jitter"], out=s["K"], precision=p)
        r = gp.gp_lml(s["K"], s["y"], p, L=s["L"], ws=s["ws"], info=s["info"], check=False)
        Kbar = gp.gp_lml_grad(r["L"], r["alpha"], 1.0, p, out=s["Kbar"], ws=s["ws"])
        grad = gp.se_hyper_grad(s["X"], 1.0, rho, sigma, Kbar, ws=s["hyper_ws"], precision=p)
        return dict(L=r["L"], alpha=r["alpha"], logdet=r["logdet"], value=r["value"], info=r["info"], Kbar=Kbar,
                    grad=grad)
    if kind == "gp_autograd":
        hyp = s["hyp"].detach().requires_grad_()
        value = gp.gp_lml_value(s["X"], s["y"], hyp, case["jitter"], case["precision"])
        value.backward()
        return dict(value=value.detach(), grad=hyp.grad)
    if kind == "chol":
        K = s["K"].detach().requires_grad_()
        L = gp.Chol.apply(K, case["precision"])
        L.backward(s["Lbar"])
        return dict(L=L.detach(), Kbar=K.grad)
    if kind == "batch":
        b = s["batch"]
        value, grad, info = gp.batched_gp_lml_grad(b, s["X"], s["y"], s["hyp"])
        return dict(value=value, grad=grad, info=info, factors=b.K)
    if kind == "tri":
        L, B = s["L"].detach().requires_grad_(), s["B"].detach().requires_grad_()
        C = gp.mdivide_left_tri_low(L, B)
        C.backward(s["Cbar"])
        return dict(C=C.detach(), Lbar=L.grad, Bbar=B.grad)
    if kind == "trsv":
        return gp.trsv(s["L"], s["x"].clone(), trans=case["trans"], ws=s["ws"])
    if kind == "matmul":
        A, B = s["A"].detach().requires_grad_(), s["B"].detach().requires_grad_()
        C = gp.MatMul.apply(A, B)
        C.backward(s["Cbar"])
        return dict(C=C.detach(), Abar=A.grad, Bbar=B.grad)
    if kind == "gemm":
        return gp.gemm(s["A"], s["B"], ws=s["ws"])
    if kind == "glm":
        return gp.glm(case["family"], s["X"], s["y"], _GLM_ALPHA, s["beta"], _GLM_SIGMA, ws=s["ws"])
    if case["family"] == "categorical":
        return gp.glm_categorical(s["X"], s["y"], s["alpha"], s["beta"])
    return gp.glm_ordinal(s["X"], s["y"], s["beta"], s["cuts"], ws=s["ws"])


# ------------------------------------------------------------------ the same results in 64 bits
def _lower_convention(G):
    """Gradient over the entries a Cholesky factorisation reads, from the symmetric gradient."""
    return 2.0 * G.tril(-1) + torch.diag(G.diagonal())


def _plain_gp(X, y, rho, sigma, jitter):
    n = X.shape[0]
    K, r2 = _plain_cov(X, 1.0, rho, sigma, jitter)
    L = torch.linalg.cholesky(K)
    a = torch.cholesky_solve(y[:, None], L)[:, 0]
    logdet = 2.0 * L.diagonal().log().sum()
    value = -0.5 * y.dot(a) - 0.5 * logdet - 0.5 * n * math.log(2.0 * math.pi)
    G = torch.cholesky_inverse(L).neg_()
    G.addr_(a, a).mul_(0.5)
    K.diagonal().sub_(sigma * sigma + jitter)  # the kernel without its noise
    K.mul_(G)
    da = 2.0 * K.sum()
    dr = (K.mul_(r2)).sum() / rho ** 3
    ds = 2.0 * sigma * G.diagonal().sum()
    return dict(L=L, alpha=a, logdet=logdet, value=value, Kbar=_lower_convention(G), grad=torch.stack([da, dr, ds]))


def _plain_glm(case, t):
    X, y = t["X"], t["y"]
    if case["kind"] == "glm":
        eta = X @ t["beta"] + _GLM_ALPHA
        zero = torch.zeros((), dtype=F64, device=X.device)
        s, fam = _GLM_SIGMA, case["family"]
        ds = zero
        if fam == "normal_id":
            z = (y - eta) / s
            lp = (-0.5 * z * z).sum() - X.shape[0] * (math.log(s) + 0.5 * math.log(2.0 * math.pi))
            d, ds = z / s, ((z * z - 1.0) / s).sum()
        elif fam == "bernoulli_logit":
            lp = (y * eta - torch.nn.functional.softplus(eta, threshold=1e6)).sum()
            d = y - torch.sigmoid(eta)
        elif fam == "poisson_log":
            lp = (y * eta - eta.exp() - torch.lgamma(y + 1.0)).sum()
            d = y - eta.exp()
        else:
            phi = torch.tensor(s, dtype=F64, device=X.device)
            mu = eta.exp()
            lp = (torch.lgamma(y + phi) - torch.lgamma(y + 1.0) - torch.lgamma(phi)
                  + phi * (phi.log() - (mu + phi).log()) + y * (eta - (mu + phi).log())).sum()
            d = y - (y + phi) * mu / (mu + phi)
            ds = (torch.digamma(y + phi) - torch.digamma(phi) + phi.log() - (mu + phi).log() + 1.0
                  - (y + phi) / (mu + phi)).sum()
        return dict(lp=lp, dalpha=d.sum(), dbeta=X.T @ d, dsigma=ds)
    idx = y.long()
    rows = torch.arange(X.shape[0], device=X.device)
    if case["family"] == "categorical":
        lsm = torch.log_softmax(X @ t["beta"] + t["alpha"], 1)
        D = -lsm.exp()
        D[rows, idx] += 1.0
        return dict(lp=lsm[rows, idx].sum(), dalpha=D.sum(0), dbeta=X.T @ D)
    eta, cuts = X @ t["beta"], t["cuts"]
    big = torch.full((1,), float("inf"), dtype=F64, device=X.device)
    ext = torch.cat([-big, cuts, big])
    u, v = torch.sigmoid(eta - ext[idx]), torch.sigmoid(eta - ext[idx + 1])
    P = u - v
    du, dv = u * (1.0 - u) / P, -v * (1.0 - v) / P
    dcuts = torch.zeros(ext.numel(), dtype=F64, device=X.device)
    dcuts.index_add_(0, idx, -du)
    dcuts.index_add_(0, idx + 1, -dv)
    return dict(lp=P.log().sum(), dbeta=X.T @ (du + dv), dcuts=dcuts[1:-1].clone())


def exact(case, seed):
    kind = case["kind"]
    t = _inputs(case, seed, _device())
    if kind in ("gp", "gp_autograd"):
        r = _plain_gp(t["X"], t["y"], case["rho"], case["sigma"], case["jitter"])
        if kind == "gp":
            r["info"] = None
            return r
        return dict(value=r["value"], grad=r["grad"].cpu())
    if kind == "chol":
        L = torch.linalg.cholesky(t["K"])
        P = (L.T @ t["Lbar"]).tril_()
        P.diagonal().mul_(0.5)
        S = torch.linalg.solve_triangular(L.T, P, upper=True)
        S = torch.linalg.solve_triangular(L, S, upper=False, left=False)
        return dict(L=L, Kbar=_lower_convention(0.5 * (S + S.T)))
    if kind == "batch":
        value, grad, factors, o = [], [], [], 0
        hyp = t["hyp"].tolist()
        for i, n in enumerate(_sizes(case)):
            r = _plain_gp(t["X"][o:o + n], t["y"][o:o + n], hyp[i][1], hyp[i][2], 0.0)
            value.append(r["value"])
            grad.append(r["grad"])
            factors.append(r["L"].reshape(-1))
            o += n
        return dict(value=torch.stack(value), grad=torch.stack(grad), info=None, factors=torch.cat(factors))
    if kind == "tri":
        C = torch.linalg.solve_triangular(t["L"], t["B"], upper=False)
        Bbar = torch.linalg.solve_triangular(t["L"].T, t["Cbar"], upper=True)
        return dict(C=C, Lbar=-(Bbar @ C.T).tril(), Bbar=Bbar)
    if kind == "trsv":
        A, upper = (t["L"].T, True) if case["trans"] else (t["L"], False)
        return torch.linalg.solve_triangular(A, t["x"][:, None], upper=upper)[:, 0]
    if kind == "matmul":
        return dict(C=t["A"] @ t["B"], Abar=t["Cbar"] @ t["B"].T, Bbar=t["A"].T @ t["Cbar"])
    if kind == "gemm":
        return t["A"] @ t["B"]
    return _plain_glm(case, t)


# ------------------------------------------------------------------ unavoidable work
def work(case):
    """Inputs read once and outputs written once, and the operations of the method's own counts."""
    kind = case["kind"]
    if kind in ("gp", "gp_autograd"):
        n, d = case["n"], case["d"]
        out = n if kind == "gp_autograd" else 2.0 * n * n + 2 * n
        # factor n^3/3, reverse mode 2n^3/3, covariance and its gradient 3d + 20 a lower entry each, solves
        return dict(bytes=8.0 * (n * d + n + out), flops=float(n) ** 3 + n * (n + 1.0) * (3 * d + 20) + 6.0 * n * n)
    if kind == "chol":
        n = case["n"]
        return dict(bytes=8.0 * 3 * n * n, flops=float(n) ** 3)
    if kind == "batch":
        sizes, d = _sizes(case), case["d"]
        return dict(bytes=8.0 * sum(n * n + n * d + n for n in sizes),
                    flops=float(sum(n ** 3 + n * (n + 1) * (3 * d + 20) + 6 * n * n for n in sizes)))
    if kind == "tri":
        n, m = case["n"], case["m"]
        return dict(bytes=8.0 * (n * n + 4.0 * n * m), flops=3.0 * n * n * m)
    if kind == "trsv":
        n = case["n"]
        return dict(bytes=4.0 * n * (n + 1) + 16.0 * n, flops=float(n) * n)
    if kind in ("matmul", "gemm"):
        m, k, n = case["m"], case["k"], case["n"]
        mats = m * k + k * n + m * n
        if kind == "gemm":
            return dict(bytes=8.0 * mats, flops=2.0 * m * n * k)
        return dict(bytes=16.0 * mats, flops=6.0 * m * n * k)
    n, k, C = case["n"], case["k"], case.get("classes", 1) if case.get("family") == "categorical" else 1
    return dict(bytes=8.0 * (n * k + n + 2.0 * k * C), flops=4.0 * n * k * C + 30.0 * n)
