"""The energy's autograd functions on the CPU over a stand-in plan: what the energy's cotangent
receives stays differentiable, and a cotangent the caller changes afterwards does not matter."""
import torch

import paper_2606_01598_gb300 as gb


class QuarticPlan:
    """E = sum (q |r|^2 + r . mu + q^3), in torch operations, with the plan's signs of the outputs."""
    device = torch.device("cpu")

    @staticmethod
    def energy(r, q, mu):
        return (q * (r * r).sum(1) + (r * mu).sum(1) + q ** 3).sum()

    def forward(self, r, q, mu, **_):
        with torch.enable_grad():
            x = [t.detach().requires_grad_(True) for t in (r, q, mu)]
            e = self.energy(*x)
            g = torch.autograd.grad(e, x)
        return dict(energy=e.detach().double().reshape(1), force=-g[0], phi=g[1], field=-g[2])

    def backward(self, r, q, mu, g_energy, g_force, g_phi, g_field):
        assert g_energy is None
        with torch.enable_grad():
            x = [t.detach().requires_grad_(True) for t in (r, q, mu)]
            g = torch.autograd.grad(self.energy(*x), x, create_graph=True)
            L = sum((c * s * t).sum() for c, s, t in zip((g_force, g_phi, g_field), (-1.0, 1.0, -1.0), g)
                    if c is not None)
            return torch.autograd.grad(L, x)


def inputs(n=5):
    gen = torch.Generator().manual_seed(3)
    new = lambda *s: torch.randn(*s, generator=gen).requires_grad_(True)  # noqa: E731
    return [new(n, 3), new(n), new(n, 3)], [new(n, 3).detach(), new(n).detach(), new(n, 3).detach()]


def test_directional_derivative_is_differentiable():
    x, v = inputs()
    plan = QuarticPlan()
    _, jvp = torch.autograd.functional.jvp(lambda *t: gb.pme_energy(plan, *t), tuple(x), tuple(v),
                                           create_graph=True)
    got = torch.autograd.grad(jvp, x)
    want = torch.autograd.functional.hvp(QuarticPlan.energy, tuple(x), tuple(v))[1]
    for a, b in zip(got, want):   # float32 products of a few terms of order one
        assert torch.allclose(a, b, rtol=1e-5, atol=1e-5)


def test_cotangent_changed_after_the_gradient():
    x, v = inputs()
    w = torch.tensor(0.5, dtype=torch.float64)
    g = torch.autograd.grad(gb.pme_energy(QuarticPlan(), *x), x, grad_outputs=w, create_graph=True)
    w.fill_(7.0)
    got = torch.autograd.grad(sum((a * b).sum() for a, b in zip(g, v)), x)
    want = torch.autograd.functional.hvp(QuarticPlan.energy, tuple(x), tuple(v))[1]
    for a, b in zip(got, want):
        assert torch.allclose(a, 0.5 * b, rtol=1e-5, atol=1e-5)
