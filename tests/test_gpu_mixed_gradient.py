"""The mixed path's gradient: recorded values, and its error against FP64 over several seeds.

Recorded: the mixed factorisation and adjoint keep 40 bits of their operands, so
another order of FP64 operations anywhere in them rounds later operands anew and
moves the gradient (sums that cancel) by a share of its own error, 1e-12 to 1e-8
of its size.  The order is fixed; what was recorded comes back to the roundoff
of the last sums (1e-13, some hundred FP64 roundoffs).  The inputs are dyadic
numbers, the same on every host.

Error: with dK the measured error of Kbar, the sums of Kbar k, Kbar k r^2 / rho^3
and of the diagonal change by at most |dK|_F |k|_F and so on (Cauchy-Schwarz),
beside the sums' own rounding (2^-40 of the sum of magnitudes is far above it).
Kbar's error itself: 2^-40 = 9e-13 of its rows' scales per product, measured as
2e-11 at n = 16384; 1e-10 leaves a factor of five.
"""
import json
import os

import numpy as np
import pytest
import torch

import paper_1907_01063_gb300 as gp

pytestmark = pytest.mark.gpu

with open(os.path.join(os.path.dirname(__file__), "golden", "mixed_gradient.json")) as f:
    RECORDED = json.load(f)


def inputs(n, d, seed):
    r = np.random.default_rng(seed)
    X = r.integers(-1774, 1775, (n, d)) / 1024.0
    y = X[:, 0] - 0.5 * X[:, -1] + r.integers(-512, 513, n) / 1024.0
    return torch.as_tensor(X, device="cuda"), torch.as_tensor(y, device="cuda")


def mixed_step(X, y, rho, sigma, jitter):
    K = gp.se_cov(X, 1.0, rho, sigma, jitter, precision="mixed")
    r = gp.gp_lml(K, y, "mixed")
    Kbar = gp.gp_lml_grad(r["L"], r["alpha"], 1.0, "mixed")
    return r, Kbar, gp.se_hyper_grad(X, 1.0, rho, sigma, Kbar, precision="mixed").cpu().numpy()


@pytest.mark.parametrize("case", RECORDED, ids=lambda c: f"{c['n']}-{c['seed']}")
def test_recorded_gradients_come_back(case):
    X, y = inputs(case["n"], case["d"], case["seed"])
    r, _, grad = mixed_step(X, y, case["rho"], case["sigma"], case["jitter"])
    assert abs(r["value"].item() - case["value"]) <= 1e-13 * abs(case["value"])
    assert np.linalg.norm(grad - case["grad"]) <= 1e-13 * np.linalg.norm(case["grad"])


@pytest.mark.parametrize("seed", [1, 2, 3, 4])
def test_gradient_error_is_within_the_error_of_kbar(seed):
    n, d, rho, sigma = 8192, 16, 4.0, 0.256
    X, y = inputs(n, d, 100 + seed)
    _, Kbar, grad = mixed_step(X, y, rho, sigma, 0.0)
    r2 = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    for t in range(d):
        r2 += (X[:, t, None] - X[None, :, t]) ** 2
    k = torch.exp(-0.5 / rho ** 2 * r2)
    L = torch.linalg.cholesky(k + sigma ** 2 * torch.eye(n, dtype=torch.float64, device="cuda"))
    a = torch.cholesky_solve(y[:, None], L)[:, 0]
    G = 0.5 * (torch.outer(a, a) - torch.cholesky_inverse(L))
    low = 2.0 * G.tril(-1) + torch.diag(G.diagonal())  # the entries a factorisation reads
    dK = Kbar.tril() - low
    assert dK.norm() <= 1e-10 * low.norm()
    exact = torch.stack([2.0 * (G * k).sum(), (G * k * r2).sum() / rho ** 3, 2.0 * sigma * G.diagonal().sum()])
    kl, e = k.tril(), dK.norm()
    bound = torch.stack([2.0 * e * kl.norm(), e * (kl * r2).norm() / rho ** 3,
                         2.0 * sigma * dK.diagonal().norm() * n ** 0.5])
    size = torch.stack([2.0 * (low.abs() * k).sum(), (low.abs() * k * r2).sum() / rho ** 3,
                        2.0 * sigma * low.diagonal().abs().sum()])
    assert torch.all((torch.as_tensor(grad, device="cuda") - exact).abs() <= bound + 2.0 ** -40 * size)
