"""Which FP64 factorisations and adjoints run on BF16 slices: one threshold in the order, the same route in any
workspace that is large enough."""
import numpy as np
import pytest
import torch

import paper_1907_01063_gb300 as gp
from oracle import oracle as O
from paper_1907_01063_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def kernels(fn):
    torch.cuda.synchronize()
    gp.trace_enable(True, timeline=True)
    try:
        out = fn()
        torch.cuda.synchronize()
    finally:
        gp.trace_enable(False)
    return out, [s["kernel"] for s in gp.trace_timeline()]


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("n,slices", [(255, False), (256, False), (257, False), (319, False), (320, False), (321, True),
                                      (322, True), (383, True), (384, True)])
def test_one_threshold(n, slices):
    K = O.se_cov(W.gp_inputs(n, 3, n), 1.0, 1.0, 0.3, 1e-6)
    Lo, Wt = O.chol(K), W.random_lower(n, n + 1)
    for ws in (None, gp.workspace(700, "fp64"), gp.workspace(n, "mixed")):
        L, names = kernels(lambda: gp.chol(dev(K), ws=ws))
        assert any("f64x_gemm" in k for k in names) == slices
        G, names = kernels(lambda: gp.chol_adjoint(dev(Lo), dev(Wt), ws=ws))
        assert any("f64x_gemm" in k for k in names) == slices
        # condition about 1e4 times the unit roundoff, as for the FP64 kernels
        assert rel(L.cpu().numpy(), Lo) <= 1e-12 and rel(G.cpu().numpy(), O.chol_adjoint(Lo, Wt)) <= 1e-12
        if ws is None:
            first = L, G
        else:
            assert torch.equal(L, first[0]) and torch.equal(G, first[1])


@pytest.mark.parametrize("depth", [1, 8])
def test_the_mixed_depth_knob_leaves_fp64_calls_alone(depth):
    n = 900
    K = dev(O.se_cov(W.gp_inputs(n, 3, 7), 1.0, 1.0, 0.3, 1e-6))
    ws = gp.workspace(n, "fp64")
    want, _ = kernels(lambda: gp.chol(K, ws=ws))
    old = gp.get_tuning(gp.GPC_TUNE_MIXED_DEFER)
    try:
        gp.set_tuning(gp.GPC_TUNE_MIXED_DEFER, depth)
        L, names = kernels(lambda: gp.chol(K, ws=ws))
    finally:
        gp.set_tuning(gp.GPC_TUNE_MIXED_DEFER, old)
    assert any("f64x_gemm" in k for k in names) and torch.equal(L, want)


@pytest.mark.parametrize("offset", [8, 16, 40, 248])
def test_a_workspace_may_start_at_any_double(offset):
    n = 500
    K = dev(O.se_cov(W.gp_inputs(n, 3, 8), 1.0, 1.0, 0.3, 1e-6))
    Wt, y = dev(W.random_lower(n, 9)), dev(W.gp_inputs(n, 1, 10)[:, 0])
    size = gp.workspace_size(n, "fp64")
    ws = torch.empty(size + offset, dtype=torch.uint8, device="cuda")[offset:]

    def step(ws):
        L = gp.chol(K, ws=ws)
        r = gp.gp_lml(K, y, ws=ws)
        return L, gp.chol_adjoint(L, Wt, ws=ws), r["alpha"], gp.gp_lml_grad(r["L"], r["alpha"], ws=ws)

    got, names = kernels(lambda: step(ws))
    assert any("f64x_gemm" in k for k in names)
    assert all(torch.equal(a, b) for a, b in zip(got, step(None)))


def test_matrices_may_start_at_any_double_with_odd_leading_dimensions():
    n, ld = 450, 463
    Kh, Wt = O.se_cov(W.gp_inputs(n, 3, 8), 1.0, 1.0, 0.3, 1e-6), W.random_lower(n, 9)
    Kp, Wp, Lp, Gp = (torch.zeros(n * ld + 1, dtype=torch.float64, device="cuda")[1:].view(n, ld)[:, :n] for _ in range(4))
    Kp.copy_(dev(Kh))
    Wp.copy_(dev(Wt))
    L = gp.chol(Kp, out=Lp)
    G = gp.chol_adjoint(L, Wp, out=Gp)
    assert torch.equal(L, gp.chol(dev(Kh))) and torch.equal(G, gp.chol_adjoint(L.contiguous(), dev(Wt)))
