"""cuFFT plans whose batched transforms would carry two real meshes through one complex transform
(odd last axes such as 39 and 75): a mesh of small values beside one of large ones keeps float32's
digits. The backward with small cotangents (it is linear in them, so the bar is the usual one), force
matching through autograd on a plan that is used again and again, and a batch of frames of very
different charges."""
import numpy as np
import pytest
import torch

import workloads as W
from gpu_util import TOL_HVP, check, f32, prepared, relrmse
from oracle import pme as O2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2606_01598_gb300 as g
    return g


def _c(x):
    return torch.tensor(np.float32(x), device="cuda")


@pytest.mark.parametrize("mesh", [(40, 40, 39), (50, 51, 51), (75, 75, 75), (69, 65, 57), (46, 45, 46)])
def test_backward_of_small_cotangents(gb, mesh):
    fr = W.molten_nacl(512, seed=61)
    pos, q, mu = prepared(fr)
    cot = [f32(1e-6 * f32(x)) for x in W.tangent(fr.n, seed=62)]
    plan = gb.Plan(fr.box, mesh, 5, 0.3, 9.0, max_ions=fr.n, fft="cufft", brick=(8, 8, 16))
    x = [_c(t) for t in (pos, q, mu)]
    hv = O2.PMEOracle(fr.box, mesh, 5, 0.3, 9.0).hvp(pos, q, mu, 0.0, *cot)
    for k in range(2):   # behind a forward on the same inputs, and alone
        if k == 0:
            plan.forward(*x)
        for got, ref in zip(plan.backward(*x, None, *(_c(t) for t in cot)), hv):
            check(f"backward of small cotangents {mesh} (rel RMSE)", relrmse(got.cpu().numpy(), ref), TOL_HVP)
    plan.close()


@pytest.mark.parametrize("mesh,order,tilt", [((75, 75, 75), 5, False), ((75, 74, 75), 4, True), ((72, 81, 90), 6, False),
                                             ((40, 40, 39), 6, True)])
def test_force_matching_step_after_step(gb, mesh, order, tilt):
    n = 2002
    box = W.molten_nacl(n, seed=1).box @ (np.array([[1, 0, 0], [0.15, 1, 0], [-0.1, 0.12, 1]]) if tilt else np.eye(3))
    new = lambda: gb.Plan(box, mesh, order, 0.30, 8.0, max_ions=n, brick=(8, 8, 16))  # noqa: E731
    plan = new()
    for k in range(5):
        fr = W.molten_nacl(n, seed=70 + k)
        x = [_c(t).requires_grad_(True) for t in (fr.pos @ np.linalg.solve(fr.box, box), fr.q, fr.mu)]
        f_ref = _c(0.1 * W.tangent(n, seed=80 + k)[0])
        got = []
        for p in (plan, new()):
            force = -torch.autograd.grad(gb.pme_energy(p, *x), x[0], create_graph=True)[0]
            got.append((force.detach(), *torch.autograd.grad(((force - f_ref) ** 2).mean(), x)))
        for a, b in zip(*got):
            assert torch.equal(a, b), (k, mesh)
        if k == 3:   # a replay of the recorded passes
            pos, q, mu = (t.detach().double().cpu().numpy() for t in x)
            w = (2.0 / (3 * n)) * (got[0][0].double().cpu().numpy() - f_ref.double().cpu().numpy())
            hv = O2.PMEOracle(box, mesh, order, 0.30, 8.0).hvp(pos, q, mu, 0.0, w, 0 * q, 0 * mu)
            for a, r in zip(got[0][1:], hv):
                check(f"force-matching gradient {mesh} (rel RMSE)", relrmse(a.cpu().numpy(), r), TOL_HVP)
    plan.close()


def test_batch_of_large_and_small_charges(gb):
    mesh = (40, 40, 39)
    frs = [W.molten_nacl(n, seed=7 + n) for n in (216, 512, 216)]
    scale = (1.0, 1e-5, 1.0)
    data = [(pos, s * q, s * mu) for s, (pos, q, mu) in zip(scale, (prepared(fr) for fr in frs))]
    off = np.concatenate([[0], np.cumsum([fr.n for fr in frs])]).tolist()
    t = [_c(np.concatenate([d[k] for d in data])) for k in range(3)]
    bp = gb.BatchPlan([fr.box for fr in frs], [mesh] * 3, [4] * 3, off, 0.3, 9.0, fft="cufft")
    got = bp.forward(*t)
    for f, fr in enumerate(frs):
        plan = gb.Plan(fr.box, mesh, 4, 0.3, 9.0, max_ions=fr.n, fft="cufft")
        s = slice(off[f], off[f + 1])
        one = plan.forward(*(x[s].contiguous() for x in t))
        for k in ("force", "phi", "field"):   # the same transforms, a frame at a time
            assert relrmse(got[k][s].cpu().numpy(), one[k].cpu().numpy()) < 2e-6, (f, k)
        plan.close()
    bp.close()
