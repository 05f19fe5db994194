"""The energy's gradient under torch's batched cotangents (vmap over the backward), on the CPU over
the stand-in plan: each batch entry is the gradient times its cotangent."""
import torch

import paper_2606_01598_gb300 as gb
from test_energy_grad_cpu import QuarticPlan, inputs


def test_batched_cotangents():
    x, _ = inputs()
    w = torch.tensor([0.5, -2.0, 0.0], dtype=torch.float64)
    got = torch.autograd.grad(gb.pme_energy(QuarticPlan(), *x), x, grad_outputs=w, is_grads_batched=True)
    one = torch.autograd.grad(gb.pme_energy(QuarticPlan(), *x), x)
    for a, b in zip(got, one):
        assert torch.equal(a, w.float().reshape(-1, *[1] * b.dim()) * b)


def test_vectorized_jacobian():
    x, _ = inputs()
    f = lambda *t: gb.pme_energy(QuarticPlan(), *t)  # noqa: E731
    got = torch.autograd.functional.jacobian(f, tuple(x), vectorize=True)
    want = torch.autograd.functional.jacobian(f, tuple(x))
    for a, b in zip(got, want):
        assert torch.equal(a, b)
