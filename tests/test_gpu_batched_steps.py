"""Batches in lockstep (whole 128 blocks, every member a grid entry) against the
CPU oracle, at the edges of blocks and passes."""
import numpy as np
import pytest
import torch

import paper_1907_01063_gb300 as gp
from oracle import oracle as O
from test_gpu_batched import make_batch, run_batch

pytestmark = pytest.mark.gpu

# sigma = 0.1: condition about n / sigma^2 < 1e5, times the unit roundoff and a
# factor of 10 for the value; the gradient's terms cancel by up to 1e2 more
VALUE_TOL, GRAD_TOL = 1e-10, 1e-8


def check(sizes, Xs, ys, hyps, b, v, g, info, members):
    for i in members:
        assert info[i].tolist() == [-1, gp.GPC_OK]
        ref = O.gp_lml_and_grad(Xs[i], ys[i], *hyps[i], 0.0)
        assert abs(v[i] - ref["value"]) <= VALUE_TOL * max(1.0, abs(ref["value"])), (i, sizes[i])
        assert np.linalg.norm(g[i] - ref["grad"]) <= GRAD_TOL * np.linalg.norm(ref["grad"]), (i, sizes[i])
        L = b.factor(i).cpu().numpy()
        K = O.se_cov(Xs[i], *hyps[i], 0.0)
        assert np.all(np.triu(L, 1) == 0.0)
        # backward error of the factorisation: n 2^-53 |K|, with room for the block inverses
        assert np.abs(np.tril(L @ L.T - K)).max() <= 100 * sizes[i] * 2.0 ** -53


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("d", [1, 4])
@pytest.mark.parametrize("sizes", [[97], [128], [129, 1, 127], [255, 256, 257, 8, 120, 136], [520, 40, 384, 385]])
def test_edges_of_blocks(sizes, d, precision):
    Xs, ys, hyps = make_batch(sizes, d=d, seed=3)
    b, v, g, info = run_batch(sizes, Xs, ys, hyps, precision=precision)
    check(sizes, Xs, ys, hyps, b, v, g, info, range(len(sizes)))


def test_passes_and_a_small_workspace():
    # the whole batch at once, in several passes, and (too little for 64 members) one CTA per GP
    sizes = [300 - (7 * i) % 290 for i in range(200)]
    Xs, ys, hyps = make_batch(sizes, seed=4)
    X = torch.as_tensor(np.concatenate(Xs), device="cuda").contiguous()
    y = torch.as_tensor(np.concatenate(ys), device="cuda").contiguous()
    out = []
    for ws in (None, 700 << 20, 300 << 20):
        b = gp.Batch(sizes)
        if ws:
            assert ws < b.ws.numel()
            b.ws = b.ws[:ws]
        before = gp.launch_count()
        v, g, info = gp.batched_gp_lml_grad(b, X, y, torch.as_tensor(hyps))
        launches = gp.launch_count() - before
        out.append((launches, v.cpu().numpy(), g.cpu().numpy()))
        assert np.all(info.cpu().numpy()[:, 1] == gp.GPC_OK)
        check(sizes, Xs, ys, hyps, b, v.cpu().numpy(), g.cpu().numpy(), info.cpu().numpy(), (0, 1, 41, 150, 199))
    assert out[1][0] > out[0][0] > out[2][0] and out[2][0] <= 2
    assert np.array_equal(out[0][1], out[1][1]) and np.array_equal(out[0][2], out[1][2])


def test_failures_and_refused_orders_stay_with_their_member():
    sizes = [260, 200, 150, 130]
    Xs, ys, hyps = make_batch(sizes, seed=5)
    Xs[1][170] = Xs[1][3]  # a repeated input without noise: K is singular at row 170
    hyps[1][2] = 0.0
    hyps[1][1] = 0.02
    Xs[2][140] = np.nan
    b, v, g, info = run_batch(sizes, Xs, ys, hyps)
    assert info[2, 1] == gp.GPC_ERR_NAN and np.isnan(v[2]) and np.all(np.isnan(g[2]))
    assert info[2, 0] == 140
    assert info[1, 1] in (gp.GPC_OK, gp.GPC_ERR_NOT_PD) and (info[1, 1] == gp.GPC_OK or info[1, 0] == 170)
    check(sizes, Xs, ys, hyps, b, v, g, info, (0, 3))
    b = gp.Batch(sizes)
    b.n[1] = 261
    b.n[3] = 0
    X = torch.as_tensor(np.concatenate(Xs), device="cuda").contiguous()
    y = torch.as_tensor(np.concatenate(ys), device="cuda").contiguous()
    _, _, info = gp.batched_gp_lml_grad(b, X, y, torch.as_tensor(hyps))
    assert info.cpu().tolist()[0] == [-1, gp.GPC_OK]
    assert [info.cpu().tolist()[i] for i in (1, 3)] == [[-1, gp.GPC_ERR_INVALID_ARG]] * 2


def test_a_product_that_gives_up_is_reported_per_member():
    sizes = [300, 140, 200]
    Xs, ys, hyps = make_batch(sizes, seed=6)
    Xs[2][150] = np.nan
    gp.get_error(clear=True)
    try:
        gp.set_test_fault(gp.GPC_TEST_WAIT_NS, 1_000_000)
        gp.set_test_fault(gp.GPC_TEST_OZAKI_NO_LOADS, 1)
        _, v, g, info = run_batch(sizes, Xs, ys, hyps)
    finally:
        gp.set_test_fault(gp.GPC_TEST_WAIT_NS, 0)
        gp.set_test_fault(gp.GPC_TEST_OZAKI_NO_LOADS, 0)
    assert gp.get_error(clear=True) == gp.GPC_ERR_TIMEOUT
    assert info[0].tolist() == [-1, gp.GPC_ERR_TIMEOUT] and info[1].tolist() == [-1, gp.GPC_ERR_TIMEOUT]
    assert info[2, 1] in (gp.GPC_ERR_NAN, gp.GPC_ERR_TIMEOUT)  # the product may be what should have met the NaN
    assert np.all(np.isnan(v)) and np.all(np.isnan(g))
    b, v, g, info = run_batch(sizes, Xs, ys, hyps)
    check(sizes, Xs, ys, hyps, b, v, g, info, (0, 1))
    assert info[2].tolist() == [150, gp.GPC_ERR_NAN] and gp.get_error() == gp.GPC_OK
