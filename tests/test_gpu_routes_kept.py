"""Kernels that larger problems no longer reach, at several blocks: the persistent batch launch (more members than
SMs, orders below 256) and the FP64 factorisation and adjoint kernels (orders up to 320, minimal workspaces)."""
import numpy as np
import pytest
import torch

import paper_1907_01063_gb300 as gp
from oracle import oracle as O
from paper_1907_01063_gb300 import workloads as W
from test_gpu_batched import MIXED_GRAD_TOL, MIXED_VALUE_TOL, make_batch, run_batch
from test_gpu_f64_route import kernels
from test_gpu_fp64 import TOL, dev, rel, se_problem

pytestmark = pytest.mark.gpu

ORDERS = [255, 1, 5, 33, 64, 65, 100, 128, 129, 200, 63, 3, 192, 250, 31]


@pytest.mark.parametrize("block", [32, 64])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_persistent_batch_at_several_blocks(block, precision):
    sizes = (ORDERS * 11)[:165]  # more than the SMs, so one CTA per GP
    assert len(sizes) > torch.cuda.get_device_properties(0).multi_processor_count
    Xs, ys, hyps = make_batch(sizes, seed=block)
    run_batch(sizes[:1], Xs[:1], ys[:1], hyps[:1])
    before = gp.launch_count()
    b, v, g, info = run_batch(sizes, Xs, ys, hyps, block, precision)
    assert gp.launch_count() - before <= 2
    assert np.all(info == [-1, gp.GPC_OK])
    vtol, gtol = (1e-10, 1e-8) if precision == "fp64" else (MIXED_VALUE_TOL, MIXED_GRAD_TOL)
    for i in list(range(len(ORDERS))) + [45, 163]:
        ref = O.gp_lml_and_grad(Xs[i], ys[i], *hyps[i], 0.0)
        assert abs(v[i] - ref["value"]) <= vtol * max(1.0, abs(ref["value"])), (i, sizes[i])
        assert np.linalg.norm(g[i] - ref["grad"]) <= gtol * np.linalg.norm(ref["grad"]), (i, sizes[i])
        L = b.factor(i).cpu().numpy()
        assert np.linalg.norm(L - ref["L"]) <= vtol * np.linalg.norm(ref["L"])


@pytest.mark.parametrize("block", [16, 32, 64, 96, 128])
@pytest.mark.parametrize("n", [300, 333, 700])
def test_fp64_kernels_at_block_sizes(n, block):
    old = gp.get_tuning(gp.GPC_TUNE_BLOCK)
    try:
        gp.set_tuning(gp.GPC_TUNE_BLOCK, block)
        ws = torch.empty(gp.workspace_min_size(n, "fp64"), dtype=torch.uint8, device="cuda")
        _, K = se_problem(n, seed=2)
        Lo, Lbar, y = O.chol(K), W.random_lower(n, seed=3), W.gp_inputs(n, 1, seed=4)[:, 0]

        def step():
            return gp.chol(dev(K), ws=ws), gp.chol_adjoint(dev(Lo), dev(Lbar), ws=ws), gp.gp_lml(dev(K), dev(y), ws=ws)

        (L, G, res), names = kernels(step)
        assert not any("f64x" in k for k in names)
        assert sum("potrf" in k for k in names) == 2 * -(-n // block)  # the factor twice
        ref = O.gp_lml(K, y)
        assert rel(L.cpu().numpy(), Lo) <= TOL and rel(G.cpu().numpy(), O.chol_adjoint(Lo, Lbar)) <= TOL
        assert rel(res["alpha"].cpu().numpy(), ref["alpha"]) <= TOL
        assert abs(res["value"].item() - ref["value"]) <= TOL * abs(ref["value"])
    finally:
        gp.set_tuning(gp.GPC_TUNE_BLOCK, old)
