"""Recorded passes take their pointers from each call: calls of one size replay the recorded graph
whatever buffers they bring, and give a fresh plan's direct results bit for bit; a caller that
captures its own graph gets the pass captured with the pointers of that call."""
import numpy as np
import pytest
import torch

import workloads as W
from gpu_util import f32, prepared

pytestmark = pytest.mark.gpu

KINDS = ["forward", "virial", "backward", "quad", "quad_backward", "batch"]


@pytest.fixture(scope="module")
def gb():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2606_01598_gb300 as g
    return g


def _c(x):
    return torch.tensor(np.float32(x), device="cuda")


def _inputs(n, seed):
    fr = W.molten_nacl(n, seed=seed)
    g = W.tangent(n, seed=seed + 1)
    theta = W.quadrupoles(n, 0.1, seed=seed + 2)
    th6 = np.stack([theta[:, 0, 0], theta[:, 1, 1], theta[:, 2, 2], theta[:, 0, 1], theta[:, 0, 2], theta[:, 1, 2]], 1)
    return [_c(x) for x in prepared(fr)], [_c(f32(x)) for x in g], _c(th6), torch.tensor([0.3], dtype=torch.float64,
                                                                                         device="cuda")


def _run(plan, kind, x, nframes=1):
    (pos, q, mu), (gf, gp, gl), th, ge = x
    if kind == "forward":
        out = plan.forward(pos, q, mu, field_grad=True)
    elif kind == "virial":
        out = plan.forward(pos, q, mu, virial=True)
    elif kind == "quad":
        out = plan.forward_quad(pos, q, mu, th)
    elif kind == "quad_backward":
        return list(plan.backward_quad(pos, q, mu, th, ge, gf, gp, gl))
    elif kind == "batch":
        out = plan.forward(pos, q, mu)
        return [out[k] for k in sorted(out)] + list(plan.backward(pos, q, mu, ge.repeat(nframes), gf, gp, gl))
    else:
        out = plan.forward(pos, q, mu)
        return [out[k] for k in sorted(out)] + list(plan.backward(pos, q, mu, ge, gf, None, gl))
    return [out[k] for k in sorted(out)]


def _plan(gb, kind, n):
    box = W.molten_nacl(n, seed=5).box
    if kind == "batch":
        return gb.BatchPlan([box, box], [(24, 24, 25), (24, 30, 27)], [5, 4], [0, n // 2, n], 0.30, 8.0)
    return gb.Plan(box, (24, 25, 27), 5, 0.30, 8.0, max_ions=n)


@pytest.mark.parametrize("kind", KINDS)
def test_other_buffers_replay_bitwise(gb, kind):
    n = 302
    plan = _plan(gb, kind, n)
    kept = []   # every call's buffers stay alive, so each call has its own
    for k in range(5):
        x = _inputs(n, 100 + 10 * k)
        got = _run(plan, kind, x, 2)
        fresh = _plan(gb, kind, n)
        want = _run(fresh, kind, x, 2)
        torch.cuda.synchronize()
        for a, b in zip(got, want):
            assert torch.equal(a, b), (kind, k)
        kept.append((x, got))
        fresh.close()
    plan.close()


def test_caller_capture_after_recording(gb):
    n = 302
    plan = _plan(gb, "forward", n)
    x = _inputs(n, 7)
    for _ in range(3):
        plan.forward(*x[0])
    static = [t.clone() for t in x[0]]
    out = {k: v.clone() for k, v in plan.forward(*static).items()}
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        plan.forward(*static, out=out)
    for k in range(2):
        y = _inputs(n, 50 + k)
        for s, t in zip(static, y[0]):
            s.copy_(t)
        plan.forward(*x[0])   # another call in between
        graph.replay()
        fresh = _plan(gb, "forward", n)
        want = fresh.forward(*y[0])
        torch.cuda.synchronize()
        for key in want:
            assert torch.equal(out[key], want[key]), key
        fresh.close()
    plan.close()
