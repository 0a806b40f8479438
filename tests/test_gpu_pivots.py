"""Pivots of the FP64 diagonal-block factor over the whole exponent range.

The refined reciprocal: one third-order step from the hardware seed (relative
error 2^-20 or less, cubed far below the roundoff), three roundings: 2 ulp.
Factors of 2^q K0 (q even) are 2^(q/2) L0: near the top of the range the entries
are exact and the error is the FP64 chain's, n 2^-53 times the condition; among
the denormals the entries are whole multiples of 2^-1074, at least 2^40 of them
on the diagonal, so 2^-40 takes the roundoff's place.
"""
import numpy as np
import pytest
import torch

import paper_1907_01063_gb300 as gp
from test_gpu_recip import inputs, ulps

pytestmark = pytest.mark.gpu


def test_pivot_reciprocal_within_two_ulp():
    x = inputs(-1022, 1022, 200000, 2)  # x and 1/x normal
    xd = torch.as_tensor(x, device="cuda")
    out = torch.empty_like(xd)
    st = gp.capi.gpc_test_recip_cubic(x.size, xd.data_ptr(), out.data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert st == gp.GPC_OK
    assert ulps(out.cpu().numpy(), 1.0 / x).max() <= 2


def integer_factor(n):
    """Whole numbers: diagonal in [2^20, 2^21), the rest up to 2^14, so L0 L0^T is exact (below 2^53) and well conditioned."""
    r = np.random.default_rng(n)
    L = np.tril(r.integers(-2 ** 14, 2 ** 14, (n, n)), -1).astype(np.float64)
    L[np.arange(n), np.arange(n)] = r.integers(2 ** 20, 2 ** 21, n)
    return L


def factor(K):
    info = gp.new_info()
    L = gp.chol(torch.as_tensor(K, device="cuda"), info=info, check=False).cpu().numpy()
    assert info.tolist() == [-1, gp.GPC_OK]
    return L


@pytest.mark.parametrize("n", [1, 2, 9, 17, 40, 64, 65, 100, 128])
@pytest.mark.parametrize("q", [0, 980, -1074])
def test_factor_at_the_ends_of_the_range(n, q):
    # pivots of 2^40 to 2^44 times 2^q: on both sides of 2^1022 and up to the largest
    # number, and denormals down to 2^-1034, whose reciprocals overflow
    L0 = integer_factor(n)
    K0 = L0 @ L0.T
    if q > 0:
        K0 *= min(4.0, 0.99 * 2.0 ** 44 / K0.diagonal().max())
        L0 = np.linalg.cholesky(K0)
    K = np.ldexp(K0, q)
    assert np.all(np.isfinite(K)) and np.array_equal(np.ldexp(K, -q), K0)
    err = np.linalg.norm(np.ldexp(factor(K), -q // 2) - L0) / np.linalg.norm(L0)
    assert err <= 8 * n * (2.0 ** -40 if q < 0 else 2.0 ** -52)
