"""Products on BF16 slices at FP64 accuracy (gemm with a workspace) against the oracle.

Bound, per output and derived beforehand: the oracle's triple loop is off by at
most K 2^-53 S (S = sum |a||b|, first order) and so is the product under test
(its own bound is no larger than the FP64 chain's), so they differ by at most
2 (K + 2) 2^-53 S.
"""
import numpy as np
import pytest
import torch

import paper_1907_01063_gb300 as gp
from oracle import oracle as O

pytestmark = pytest.mark.gpu


def check(C, A, B):
    S = np.abs(A) @ np.abs(B)
    K = A.shape[1]
    assert np.all(np.abs(C - O.gemm(A, B)) <= 2 * (K + 2) * 2.0 ** -53 * S + 1e-320)


def run(A, B, ws=None):
    return gp.gemm(torch.as_tensor(A, device="cuda"), torch.as_tensor(B, device="cuda"), ws=ws).cpu().numpy()


@pytest.mark.parametrize("m,n,k", [(640, 640, 129), (257, 513, 511), (513, 300, 1025), (1000, 8, 4099), (130, 70, 9001),
                                   (65, 1000, 640), (900, 900, 128)])
def test_edges_of_tiles_and_chunks(m, n, k):
    r = np.random.default_rng(m + n + k)
    A, B = r.standard_normal((m, k)), r.standard_normal((k, n))
    check(run(A, B), A, B)


@pytest.mark.parametrize("scale", [1.0, 1e-290, 1e140])
def test_wide_rows_fall_back_block_by_block(scale):
    # rows of A and columns of B spread over many binades, some of them: the
    # products there are formed in FP64, the others on slices
    r = np.random.default_rng(3)
    A, B = r.standard_normal((500, 700)), r.standard_normal((700, 400))
    A[40:90] *= np.exp(30.0 * r.standard_normal((50, 700)))
    B[:, 200:220] *= np.exp(30.0 * r.standard_normal((700, 20)))
    A[300, :] = 0.0
    A[301, :350] = 0.0
    B[:350, 7] = 0.0  # with row 301: two half-empty vectors that do not overlap
    A *= scale
    check(run(A, B), A, B)


def test_infinities_nans_and_denormals_match_the_fp64_chain():
    r = np.random.default_rng(4)
    A, B = r.standard_normal((400, 500)), r.standard_normal((500, 300))
    A[5, 7], A[100, 3], B[4, 9] = np.nan, np.inf, -np.inf
    A[250, :] = 1e-310
    C = run(A, B)
    ref = O.gemm(A, B)
    assert np.array_equal(np.isnan(C), np.isnan(ref))
    inf = np.isinf(ref)
    assert np.array_equal(C[inf], ref[inf])
    fine = np.isfinite(ref)
    fine[250] = False
    S = np.abs(np.nan_to_num(A, posinf=0)) @ np.abs(np.nan_to_num(B, neginf=0))
    assert np.all(np.abs(C - ref)[fine] <= (2 * 502 * 2.0 ** -53 * S)[fine])
    assert np.all(np.abs(C[250, 10:] - ref[250, 10:]) <= 1e-322 * 500)


def test_small_workspace_takes_panels():
    r = np.random.default_rng(5)
    A, B = r.standard_normal((1500, 1400)), r.standard_normal((1400, 1300))
    ws = torch.empty(40 << 20, dtype=torch.uint8, device="cuda")
    check(run(A, B, ws), A, B)


def test_exact_products_are_exact():
    r = np.random.default_rng(6)
    A = r.integers(-2 ** 20, 2 ** 20, (300, 600)).astype(np.float64)
    B = r.integers(-2 ** 20, 2 ** 20, (600, 300)).astype(np.float64)
    assert np.array_equal(run(A, B), O.gemm(A, B))


def test_reverse_mode():
    r = np.random.default_rng(7)
    A, B, Cb = r.standard_normal((321, 450)), r.standard_normal((450, 290)), r.standard_normal((321, 290))
    Ab, Bb = gp.gemm_adjoint(*(torch.as_tensor(x, device="cuda") for x in (A, B, Cb)))
    check(Ab.cpu().numpy(), Cb, B.T.copy())
    check(Bb.cpu().numpy(), A.T.copy(), Cb)
