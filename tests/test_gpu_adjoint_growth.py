"""Adjoints whose finished diagonal blocks grow far above what they were made from (FP64, orders on slices).

With D' the block whose rows are scaled to their largest entries, the finished
block is D'^-T (..) D'^-1: it grows by up to the square of D'^-1.  Bound: the FP64
sweep's error grows with the inverse, n 2^-53 |D'^-1| relative to the result's
norm, with room for a factor of ten.
"""
import numpy as np
import pytest
import torch

import paper_1907_01063_gb300 as gp
from oracle import oracle as O
from paper_1907_01063_gb300 import workloads as W
from test_gpu_batched import make_batch, run_batch

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def inverse_size(L):
    s = np.abs(L).max(axis=1)
    return np.abs(np.linalg.inv(L / s[:, None])).max()


@pytest.mark.parametrize("n,at", [(400, 399), (400, 300), (500, 130), (641, 513), (1100, 70)])
@pytest.mark.parametrize("bits", [10, 24, 27, 40, 90])
def test_finished_block_above_its_scale(n, at, bits):
    L = W.known_factor(n, seed=n)
    L[at, at] = 2.0 ** -bits
    Wt = W.random_lower(n, seed=n + 1)
    G = gp.chol_adjoint(dev(L), dev(Wt)).cpu().numpy()
    ref = O.chol_adjoint(L, Wt)
    assert np.all(np.isfinite(ref)) and np.all(np.isfinite(G))
    assert np.linalg.norm(G - ref) <= 10 * n * 2.0 ** -53 * inverse_size(L) * np.linalg.norm(ref)


def test_batch_with_a_repeated_input_stays_finite():
    # a repeated input at the smallest noise that leaves a positive pivot: 1 / L_ii up
    # to 2^26, the largest inverse a factorisation in FP64 can end with
    sizes = [200, 260]
    Xs, ys, hyps = make_batch(sizes, seed=5)
    for i, X in enumerate(Xs):
        X *= 100.0
        X[150] = X[7]
        ys[i][150] = ys[i][7] + 1e-9
        hyps[i][1], hyps[i][2] = 0.5, 3e-8
    for precision in ("fp64", "mixed"):
        _, v, g, info = run_batch(sizes, Xs, ys, hyps, precision=precision)
        for i in range(2):
            assert info[i].tolist() in ([-1, gp.GPC_OK], [150, gp.GPC_ERR_NOT_PD])
            if info[i, 1] == gp.GPC_OK:
                assert np.isfinite(v[i]) and np.all(np.isfinite(g[i]))
