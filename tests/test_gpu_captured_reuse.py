"""Passes captured into a caller's own graph beside live calls of the same plan: a backward reuses the
state of a forward only while it is in place on the device, whatever order the graph's replays and
the live calls come in. Each backward is a fresh plan's, bit for bit."""
import numpy as np
import pytest
import torch

import workloads as W
from gpu_util import f32, prepared

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2606_01598_gb300 as g
    return g


def _c(x):
    return torch.tensor(np.float32(x), device="cuda")


def _inputs(n, seed):
    th = W.quadrupoles(n, 0.1, seed=seed + 2)
    th6 = np.stack([th[:, 0, 0], th[:, 1, 1], th[:, 2, 2], th[:, 0, 1], th[:, 0, 2], th[:, 1, 2]], 1)
    return [_c(x) for x in prepared(W.molten_nacl(n, seed=seed))], [_c(f32(x)) for x in W.tangent(n, seed=seed + 1)], _c(th6)


# the one-block sort's sizes and the general one's
@pytest.mark.parametrize("n", [302, 700])
@pytest.mark.parametrize("kind", ["backward", "forward + backward", "quad", "quad_backward", "solve"])
def test_live_backward_after_replay(gb, n, kind):
    box = W.molten_nacl(n, seed=5).box
    new = lambda: gb.Plan(box, (24, 25, 27), 5, 0.30, 8.0, max_ions=n, brick=(8, 8, 16))  # noqa: E731
    plan, (A, ca, _), (B, cb, th) = new(), _inputs(n, 100), _inputs(n, 200)
    rho = torch.randn(24, 25, 27, device="cuda")

    def other():
        if kind == "backward":
            plan.backward(*B, None, *cb)
        elif kind == "forward + backward":
            plan.forward(*B)
            plan.backward(*B, None, *cb)
        elif kind == "quad":
            plan.forward_quad(*B, th)
        elif kind == "quad_backward":
            plan.backward_quad(*B, th, None, *cb)
        else:
            plan.solve(rho)

    fresh = new()
    fresh.forward(*A)
    want = fresh.backward(*A, None, *ca)
    other()   # loads the kernels before the capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        other()
    for _ in range(3):
        plan.forward(*A)
        graph.replay()
        got = plan.backward(*A, None, *ca)
        for a, b in zip(got, want):
            assert torch.equal(a, b)
    plan.close()
    fresh.close()


@pytest.mark.parametrize("n", [302, 700])
def test_live_backward_after_a_capture_that_has_not_run(gb, n):
    box = W.molten_nacl(n, seed=5).box
    new = lambda: gb.Plan(box, (24, 25, 27), 5, 0.30, 8.0, max_ions=n, brick=(8, 8, 16))  # noqa: E731
    plan, (A, ca, th), (B, _, _) = new(), _inputs(n, 100), _inputs(n, 200)
    fresh = new()
    fresh.forward(*A)
    want = fresh.backward(*A, None, *ca)
    plan.forward(*A)
    plan.forward_quad(*B, th)   # A's order, Phi and lists are gone, its saved inputs are not
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        plan.forward(*A)
    for a, b in zip(plan.backward(*A, None, *ca), want):
        assert torch.equal(a, b)
    graph.replay()   # and a captured forward that has run serves a live backward
    for a, b in zip(plan.backward(*A, None, *ca), want):
        assert torch.equal(a, b)
    plan.close()
    fresh.close()
