"""The GLM kernel for at most 64 covariates at the edges of its row blocks and lane groups, against the oracle."""
import numpy as np
import pytest
import torch

import paper_1907_01063_gb300 as gp
from oracle import oracle as O
from paper_1907_01063_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - b) / max(np.linalg.norm(b), 1e-300))


@pytest.mark.parametrize("k", [1, 2, 3, 8, 9, 16, 17, 31, 32, 33, 63, 64, 65])
@pytest.mark.parametrize("n", [1, 31, 33, 257, 20011, 100003])
def test_value_and_gradient(n, k):
    # sums of n terms, each good to a few units: 1e-12 as for the other sizes
    X, y = W.glm_data(n, max(k, 2), "poisson_log", seed=n + k)
    X = X[:, :k]
    y[0] = 127.0
    if n > 2:
        y[1], y[2] = 128.0, 300.0  # past the table of log y!
    beta = np.random.default_rng(k).standard_normal(k) / np.sqrt(k) / 2
    ref = O.glm("poisson_log", X, y, 0.3, beta)
    Xd = torch.zeros(n, k + 3, dtype=torch.float64, device="cuda")[:, :k]  # a leading dimension of its own
    Xd.copy_(dev(X))
    got = gp.glm("poisson_log", Xd, dev(y), 0.3, dev(beta))
    assert rel(got["lp"].item(), ref["lp"]) <= 1e-12
    scale = np.linalg.norm(np.abs(X).T @ np.abs(y - np.exp(0.3 + X @ beta)))
    assert np.linalg.norm(got["dbeta"].cpu().numpy() - ref["dbeta"]) <= 1e-12 * scale
    again = gp.glm("poisson_log", Xd, dev(y), 0.3, dev(beta))
    assert all(torch.equal(got[q], again[q]) for q in got)
