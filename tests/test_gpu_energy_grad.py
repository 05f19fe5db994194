"""Autograd through the energy: the gradient scaled by the energy's cotangent, the double backward
with some cotangents missing and with one on that factor, and CPU tensors, against the plan's own
forward and backward."""
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


@pytest.mark.parametrize("device", ["cuda", "cpu"])
@pytest.mark.parametrize("which", [(0,), (1, 2), (0, 1, 2)])
def test_scaled_gradient_and_double_backward(gb, device, which):
    n = 258
    fr = W.molten_nacl(n, seed=23)
    x = [torch.tensor(np.float32(t), device=device, requires_grad=True) for t in prepared(fr)]
    cot = [torch.tensor(np.float32(f32(t)), device=device) for t in (W.tangent(n, seed=24)[k] for k in (0, 1, 2))]
    plan = gb.Plan(fr.box, (24, 24, 24), 5, 0.30, 8.0, max_ions=n)
    scale = torch.tensor(0.75, dtype=torch.float64, device=device, requires_grad=True)
    e = gb.pme_energy(plan, *x) * scale
    grads = torch.autograd.grad(e, x, create_graph=True)
    raw = [t.detach() for t in x]
    out = plan.forward(*raw)
    s = torch.tensor(0.75, dtype=torch.float32, device=device)
    expect = (-s * out["force"], s * out["phi"], -s * out["field"])
    for a, b in zip(grads, expect):
        assert torch.equal(a, b)
    loss = sum((grads[k] * cot[k]).sum() for k in which)
    got = torch.autograd.grad(loss, x + [scale])
    v = [cot[k] if k in which else None for k in range(3)]
    hv = plan.backward(*raw, None, None if v[0] is None else -s * v[0], None if v[1] is None else s * v[1],
                       None if v[2] is None else -s * v[2])
    for a, b in zip(got[:3], hv):
        assert torch.equal(a, b)
    # d loss / d scale = gradient (unscaled) . cotangent, a float32 sum of n terms: to 1e-4 of the
    # sum of their magnitudes (n 2^-24 is 2e-5)
    terms = [(expect[k] / s).double() * cot[k].double() for k in which]
    want, size = sum(t.sum() for t in terms), sum(t.abs().sum() for t in terms)
    assert abs(got[3].item() - want.item()) < 1e-4 * size.item()
    plan.close()
