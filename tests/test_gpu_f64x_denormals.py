"""Factor and adjoint on slices where the inputs are denormal numbers.

2^-1030 K0 has the factor 2^-515 L0, normal numbers, and the adjoint of L0 and
2^-1030 W0 is 2^-1030 Kbar0.  The denormals are whole multiples of 2^-1074, so 2^-44
takes the place of the roundoff; the condition is about 1e4, with a factor of ten
to spare.
"""
import numpy as np
import pytest
import torch

import paper_1907_01063_gb300 as gp
from oracle import oracle as O
from paper_1907_01063_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL = 2.0 ** -44 * 1e5


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("n", [321, 400, 641])
def test_denormal_covariance(n):
    K = O.se_cov(W.gp_inputs(n, 3, n), 1.0, 1.0, 0.3, 1e-6)
    got = gp.chol(dev(np.ldexp(K, -1030))).cpu().numpy()
    assert rel(np.ldexp(got, 515), O.chol(K)) <= TOL


@pytest.mark.parametrize("n", [321, 400, 641])
def test_denormal_upstream_adjoint(n):
    L, Wt = O.chol(O.se_cov(W.gp_inputs(n, 3, n), 1.0, 1.0, 0.3, 1e-6)), W.random_lower(n, n + 1)
    got = gp.chol_adjoint(dev(L), dev(np.ldexp(Wt, -1030))).cpu().numpy()
    assert rel(np.ldexp(got, 1030), O.chol_adjoint(L, Wt)) <= TOL
