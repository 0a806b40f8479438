"""GLM likelihoods called by several host threads whose kernels ask for different amounts of shared memory."""
import numpy as np
import pytest
import torch

import paper_1907_01063_gb300 as gp
from test_gpu_threads import in_threads

pytestmark = pytest.mark.gpu


class GlmCaller:
    def __init__(self, n, k, family):
        g = np.random.default_rng(n + k)
        self.X = torch.as_tensor(g.standard_normal((n, k)), device="cuda")
        self.y = torch.as_tensor(g.integers(0, 3 if family == "ordinal" else 2, n).astype(float), device="cuda")
        self.beta = torch.as_tensor(g.standard_normal(k) / k, device="cuda")
        self.cuts = torch.tensor([-0.5, 0.5], dtype=torch.float64, device="cuda")
        self.family, self.ws, self.stream = family, gp.glm_workspace(k, "cuda"), torch.cuda.Stream()

    def step(self):
        if self.family == "ordinal":
            return gp.glm_ordinal(self.X, self.y, self.beta, self.cuts, ws=self.ws)
        return gp.glm(self.family, self.X, self.y, 0.5, self.beta, 1.0, ws=self.ws)


def test_glm_calls_of_several_shared_memory_sizes():
    # every size above the default limit, so each call needs the limit raised
    callers = [GlmCaller(90000, k, f) for k, f in ((24, "bernoulli_logit"), (31, "bernoulli_logit"), (20, "ordinal"),
                                                   (31, "ordinal"))]
    for c in callers:
        c.ref = c.step()
    torch.cuda.synchronize()

    def work(c):
        # the library's entry point directly: short host work between the calls of the threads
        k = c.X.shape[1]
        out = torch.empty(k + 8, dtype=torch.float64, device="cuda")
        n, x, y, b, o, ws, s = (90000, c.X.data_ptr(), c.y.data_ptr(), c.beta.data_ptr(), out.data_ptr(),
                                c.ws.data_ptr(), c.stream.cuda_stream)
        if c.family == "ordinal":
            args = (n, k, 3, x, k, y, b, c.cuts.data_ptr(), o, o + 64, o + 8, ws, c.ws.numel(), s)
            call = gp.capi.gpc_glm_ordinal
        else:
            args = (gp.GLM_FAMILIES[c.family], n, k, x, k, y, 0.5, b, 1.0, o, o + 8, o + 64, o + 16, ws, c.ws.numel(), s)
            call = gp.capi.gpc_glm
        c.bad = sum(call(*args) != gp.GPC_OK for _ in range(5000))
        c.out = c.step()

    in_threads(callers, work)
    assert [c.bad for c in callers] == [0, 0, 0, 0]
    assert all(torch.equal(c.out[q], c.ref[q]) for c in callers for q in c.ref)
