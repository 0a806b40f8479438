"""Factorisations and adjoints enqueued by several host threads at once, each on its own stream with its own
workspace: the same bits as one thread gives.  And a call beside another thread's graph capture."""
import threading

import numpy as np
import pytest
import torch

import paper_1907_01063_gb300 as gp
from paper_1907_01063_gb300 import workloads as W

pytestmark = pytest.mark.gpu


class Caller:
    """One thread's matrices, workspace and stream."""

    def __init__(self, n, precision, seed):
        X = torch.as_tensor(W.gp_inputs(n, 3, seed), device="cuda")
        self.n, self.precision = n, precision
        self.K = gp.se_cov(X, 1.0, 1.0, 0.3, 1e-6)
        self.W = torch.as_tensor(W.random_lower(n, seed + 1), device="cuda")
        self.ws, self.info = gp.workspace(n, precision), gp.new_info()
        self.L, self.G = torch.zeros_like(self.K), torch.zeros_like(self.K)
        self.stream = torch.cuda.Stream()

    def step(self):
        gp.chol(self.K, self.precision, out=self.L, ws=self.ws, info=self.info, check=False)
        gp.chol_adjoint(self.L, self.W, self.precision, out=self.G, ws=self.ws)

    def reference(self):
        self.step()
        torch.cuda.synchronize()
        self.ref = self.L.clone(), self.G.clone()


def in_threads(callers, work):
    start, errors = threading.Barrier(len(callers)), []

    def body(c):
        try:
            with torch.cuda.stream(c.stream):
                start.wait(60)
                work(c)
        except Exception as e:  # noqa: BLE001 - reported by the test
            errors.append(e)

    threads = [threading.Thread(target=body, args=(c,)) for c in callers]
    for t in threads:
        t.start()
    for t in threads:
        t.join(120)
    assert not any(t.is_alive() for t in threads)
    torch.cuda.synchronize()
    assert not errors, errors


# orders above 896 use the auxiliary stream in the factorisation, two blocks in the adjoint
@pytest.mark.parametrize("specs", [[(1200, "fp64"), (1300, "fp64")], [(1200, "fp64"), (1025, "mixed")],
                                   [(400, "fp64"), (1500, "mixed"), (1100, "fp64"), (600, "mixed")]])
def test_threads_on_their_own_streams_give_one_threads_bits(specs):
    callers = [Caller(n, p, 3 * i) for i, (n, p) in enumerate(specs)]
    for c in callers:
        c.reference()
        c.same = torch.ones((), dtype=torch.bool, device="cuda")

    def work(c):
        for _ in range(25):
            c.L.zero_()
            c.G.zero_()
            c.step()
            c.same &= (c.L == c.ref[0]).all() & (c.G == c.ref[1]).all()

    in_threads(callers, work)
    assert all(bool(c.same) for c in callers)
    assert gp.get_error() == gp.GPC_OK


def test_more_threads_than_auxiliary_streams_are_kept():
    callers = [Caller(300 + 40 * i, "fp64", i) for i in range(11)]
    for c in callers:
        c.reference()

    def work(c):
        for _ in range(10):
            c.step()

    for _ in range(2):
        in_threads(callers, work)
        assert all(torch.equal(c.L, c.ref[0]) and torch.equal(c.G, c.ref[1]) for c in callers)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_calls_beside_another_threads_capture_stay_out_of_it(precision):
    a, b = Caller(1200, precision, 0), Caller(1100, precision, 5)
    a.reference()
    b.reference()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    captured, other_done = threading.Event(), threading.Event()

    def work(c):
        if c is a:
            graph.capture_begin(capture_error_mode="thread_local")
            try:
                c.step()
                captured.set()
                other_done.wait(60)  # the capture stays open while the other thread calls
                c.step()
            finally:
                captured.set()
                graph.capture_end()
        else:
            captured.wait(60)
            for _ in range(3):
                c.step()
            c.stream.synchronize()
            other_done.set()

    b.L.zero_()
    b.G.zero_()
    in_threads([a, b], work)
    assert torch.equal(b.L, b.ref[0]) and torch.equal(b.G, b.ref[1])  # ran at once, not in the graph
    a.L.zero_()
    a.G.zero_()
    b.L.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(a.L, a.ref[0]) and torch.equal(a.G, a.ref[1])
    assert np.all(b.L.cpu().numpy() == 0.0)  # nor is any of it in the graph
