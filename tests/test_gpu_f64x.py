"""Products on BF16 slices at FP64 accuracy (gemm with a workspace) against the oracle.

Bound, per output and derived beforehand: the oracle's triple loop is off by at
most K 2^-53 S (S = sum |a||b|, first order) and so is the product under test
(its own bound is no larger than the FP64 chain's), so they differ by at most
2 (K + 2) 2^-53 S.
"""
import ctypes

import numpy as np
import pytest
import torch

import paper_1907_01063_gb300 as gp
from oracle import oracle as O
from paper_1907_01063_gb300 import workloads as W

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


# ---- the factorisation and its adjoint on slices (orders from 256)
def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def problem(n, seed=0):
    X = W.gp_inputs(n, 3, seed)
    return O.se_cov(X, 1.0, 1.0, 0.3, 1e-6), W.random_lower(n, seed + 1)


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("n", [256, 257, 319, 384, 449, 640, 769, 1025])
def test_factor_and_adjoint_match_the_oracle(n):
    # 1e-12: condition about 1e4 times the unit roundoff, as for the FP64 kernels
    K, Wt = problem(n, n)
    L = O.chol(K)
    assert rel(gp.chol(dev(K)).cpu().numpy(), L) <= 1e-12
    assert rel(gp.chol_adjoint(dev(L), dev(Wt)).cpu().numpy(), O.chol_adjoint(L, Wt)) <= 1e-12


@pytest.mark.parametrize("n", [321, 383, 447, 513])
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("mixed", 1e-8)])
def test_panel_times_inverse_at_ragged_first_blocks(n, precision, tol):
    # top-left blocks of 65, 127, 63 and 1 rows; a row of the upstream gradient far
    # above the others must not cost them digits (each row has its own scale).
    # fp64: as above; mixed: 2^-40 of a row's scale times condition about 1e4
    K, Wt = problem(n, n)
    Wt[n - 3] *= 2.0 ** 20
    Wt[n - 2] *= 2.0 ** -20
    L = O.chol(K)
    assert rel(gp.chol_adjoint(dev(L), dev(Wt), precision).cpu().numpy(), O.chol_adjoint(L, Wt)) <= tol


def test_minimal_workspace_takes_the_fp64_kernels():
    n = 500
    K, Wt = problem(n, 3)
    b = ctypes.c_size_t()
    assert gp.capi.gpc_workspace_min_size(n, gp.GPC_FP64, ctypes.byref(b)) == gp.GPC_OK
    assert b.value < gp.workspace_size(n)
    ws = torch.empty(b.value, dtype=torch.uint8, device="cuda")
    L = O.chol(K)
    assert rel(gp.chol(dev(K), ws=ws).cpu().numpy(), L) <= 1e-12
    assert rel(gp.chol_adjoint(dev(L), dev(Wt), ws=ws).cpu().numpy(), O.chol_adjoint(L, Wt)) <= 1e-12
    y = W.gp_inputs(n, 1, 5)[:, 0]
    assert rel(gp.gp_lml(dev(K), dev(y), ws=ws)["alpha"].cpu().numpy(), O.gp_lml(K, y)["alpha"]) <= 1e-11


def test_a_mixed_workspace_serves_fp64_calls_on_slices():
    n = 500
    K, _ = problem(n, 3)
    assert gp.workspace_size(n, "mixed") >= gp.workspace_size(n, "fp64")
    own = gp.chol(dev(K))
    shared = gp.chol(dev(K), ws=gp.workspace(n, "mixed"))
    assert torch.equal(own, shared)  # the same route, so the same bits


@pytest.mark.parametrize("spread", [0, 12, 40])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -660, 2.0 ** 660])
def test_diagonal_scaling_changes_nothing(spread, scale):
    # K -> D K D with powers of two: L -> D L and Kbar -> D^-1 Kbar D^-1 exactly, so
    # the slices must see the same digits
    n = 450
    K, Wt = problem(n, 7)
    d = 2.0 ** np.round(spread * np.random.default_rng(1).standard_normal(n)) * np.sqrt(scale)
    L = gp.chol(dev(K)).cpu().numpy()
    G = gp.chol_adjoint(dev(L), dev(Wt)).cpu().numpy()
    L2 = gp.chol(dev(d[:, None] * K * d[None, :])).cpu().numpy()
    assert np.abs(L2 / d[:, None] - L).max() <= 1e-13
    G2 = gp.chol_adjoint(dev(d[:, None] * L), dev(Wt / d[:, None])).cpu().numpy()
    assert np.abs(G2 * d[:, None] * d[None, :] - G).max() <= 1e-12 * np.abs(G).max()


def test_adjoint_of_independent_blocks_keeps_the_small_one():
    n, h = 500, 300
    K, Wt = problem(n, 9)
    K[h:, :h] = K[:h, h:] = 0.0
    Wt[h:, :h] = 0.0
    Wt[h:, h:] *= 1e-30
    L = O.chol(K)
    G = gp.chol_adjoint(dev(L), dev(Wt)).cpu().numpy()
    ref = O.chol_adjoint(L, Wt)
    assert rel(G[h:, h:], ref[h:, h:]) <= 1e-12 and rel(G[:h, :h], ref[:h, :h]) <= 1e-12


@pytest.mark.parametrize("bad,value,status", [(300, -1.0, gp.GPC_ERR_NOT_PD), (450, np.nan, gp.GPC_ERR_NAN),
                                              (450, np.inf, gp.GPC_ERR_NAN)])
def test_failing_pivots(bad, value, status):
    K, _ = problem(640, 11)
    K[bad, bad] = value
    info = gp.new_info()
    gp.chol(dev(K), info=info, check=False)
    assert info.tolist() == [bad, status]


@pytest.mark.parametrize("value,status", [(1e9, gp.GPC_ERR_NOT_PD), (1e200, gp.GPC_ERR_NOT_PD), (np.nan, gp.GPC_ERR_NAN)])
def test_row_above_its_diagonal_fails_at_that_row(value, status):
    K, _ = problem(640, 12)
    K[400, 20] = value
    info = gp.new_info()
    gp.chol(dev(K), info=info, check=False)
    assert info.tolist() == [400, status]


def test_nan_in_the_adjoint_spreads():
    n = 400
    K, Wt = problem(n, 13)
    Wt[350, 200] = np.nan
    L = O.chol(K)
    G = gp.chol_adjoint(dev(L), dev(Wt)).cpu().numpy()
    ref = O.chol_adjoint(L, Wt)
    assert np.isnan(G[350, 100]) and np.isnan(ref[350, 100])


@pytest.mark.parametrize("m,n", [(530000, 64), (64, 530000)])
def test_a_large_workspace_does_not_make_panels_too_long(m, n):
    # more operand rows than one launch of the split covers, in a workspace that holds them all
    r = np.random.default_rng(m)
    A, B = r.standard_normal((m, 64)), r.standard_normal((64, n))
    check(run(A, B, torch.empty(3 << 30, dtype=torch.uint8, device="cuda")), A, B)
