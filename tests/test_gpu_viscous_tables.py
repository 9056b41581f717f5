"""The viscous solve's tables (z pivots, x and y factors) follow beta through any order of
eager calls, captured calls and replays of the captured graphs.

A captured call only records its table kernel, and every replay runs it again, so an eager
call must neither trust tables that were merely recorded nor keep its own where a replay
writes.  The kernels are deterministic: results are those of a plan that has seen one eager
call only, bit for bit."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2609_19130_gb300 import FP64, MIXED, Grid, Plan, synth  # noqa: E402

pytestmark = pytest.mark.gpu

GRIDS = [Grid(24, 18, 12, 2 * math.pi, 1.3, 2.0, beta=1.5), Grid(16, 12, 9, 1.0, 1.0, 1.0)]
A, B = 0.02, 0.01


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_2609_19130_gb300 import build
    build.build()


class Solver:
    def __init__(self, prec):
        self.plan = Plan(GRIDS, precision=prec, refine_steps=0)
        self.prec = prec
        self.ins = [tuple(torch.from_numpy(np.ascontiguousarray(a)).cuda()
                          for a in synth.uniform_velocity_np(60 + i, g.nx, g.ny, g.nz)) for i, g in enumerate(GRIDS)]
        self.out = [tuple(torch.empty_like(t) for t in f) for f in self.ins]
        self.stream = torch.cuda.Stream()
        torch.cuda.synchronize()

    def call(self, beta):
        self.plan.viscous_solve(self.ins, beta, out=self.out, stream=self.stream)

    def eager(self, beta):
        self.call(beta)
        return self.taken()

    def taken(self):
        torch.cuda.synchronize()
        got = [t.clone() for f in self.out for t in f]
        for f in self.out:
            for t in f:
                t.zero_()
        torch.cuda.synchronize()
        return got

    def capture(self, beta):
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=self.stream):
            self.call(beta)
        return graph

    def replay(self, graph):
        with torch.cuda.stream(self.stream):
            graph.replay()
        return self.taken()


@pytest.fixture(scope="module", params=[FP64, MIXED])
def expected(request):
    ref = {}
    for beta in (A, B):
        s = Solver(request.param)
        ref[beta] = s.eager(beta)
        s.plan.close()
    assert not torch.equal(ref[A][0], ref[B][0])
    return request.param, ref


def same(got, ref):
    assert all(torch.equal(a, b) for a, b in zip(got, ref))


@pytest.mark.parametrize("before", [None, A, B])
def test_eager_after_a_capture_that_never_ran(expected, before):
    prec, ref = expected
    s = Solver(prec)
    if before is not None:
        same(s.eager(before), ref[before])
    graph = s.capture(B)
    same(s.eager(B), ref[B])
    same(s.eager(A), ref[A])
    same(s.replay(graph), ref[B])
    s.plan.close()


def test_eager_after_replays(expected):
    prec, ref = expected
    s = Solver(prec)
    ga, gb = s.capture(A), s.capture(B)
    for beta, graph, other in ((A, gb, B), (B, ga, A), (A, ga, A)):
        same(s.eager(beta), ref[beta])
        same(s.replay(graph), ref[other])
        same(s.eager(beta), ref[beta])
    same(s.replay(ga), ref[A])
    same(s.replay(gb), ref[B])
    s.plan.close()
