"""Mesh transforms line by line (axes of 64, 128 or 256 points, planes too large for one block)
against cuFFT: the solve (both float32 transforms of one input: the bar the other kernel sets are
held to against each other, 2e-6 of the largest potential) and a forward + backward."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import pme as O2
from gpu_util import TOL_HVP, check, f32, prepared, relmax, relrmse

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2606_01598_gb300 as g
    return g


def _c(x):
    return torch.tensor(np.float32(x), device="cuda")


@pytest.mark.parametrize("mesh", [(64, 128, 256), (64, 256, 128), (64, 256, 256), (256, 256, 256)])
def test_line_solve_matches_cufft(gb, mesh):
    box = np.diag([0.8 * m for m in mesh])
    rho = torch.randn(mesh, generator=torch.Generator().manual_seed(3)).cuda()
    res = {}
    for fft in ("auto", "cufft"):
        plan = gb.Plan(box, mesh, 6, 0.3, 9.0, max_ions=64, fft=fft, brick=(8, 8, 16))
        assert plan.fft_kernels == ("power-of-two" if fft == "auto" else "cufft")
        phi, e = plan.solve(rho)
        res[fft] = (phi.cpu().numpy(), e.item())
        plan.close()
    check(f"line vs cuFFT Phi {mesh} (rel max)", relmax(res["auto"][0], res["cufft"][0]), 2e-6)
    assert abs(res["auto"][1] - res["cufft"][1]) < 1e-6 * abs(res["cufft"][1])


def test_line_forward_backward_no_less_accurate_than_cufft(gb):
    # as the other kernel sets are held: force, phi and field against cuFFT, the backward (third
    # spline derivatives, whose float32 rounding differs more between any two transforms) against
    # the oracle, no less accurate than cuFFT; on the forward's inputs (its Phi kept, only the
    # tangent mesh transformed) and on a fresh plan (both meshes) with the same bits
    fr = W.molten_nacl(2048, seed=31)
    mesh, order = (64, 128, 256), 6
    pos, q, mu = prepared(fr)
    cot = [f32(x) for x in W.tangent(fr.n, seed=32)]
    ge = torch.tensor([0.7], dtype=torch.float64, device="cuda")
    dev = [_c(x) for x in (pos, q, mu)], [_c(x) for x in cot]
    fwd, bwd = {}, {}
    for fft in ("auto", "cufft"):
        plan = gb.Plan(fr.box, mesh, order, 0.3, 9.0, max_ions=fr.n, fft=fft, brick=(8, 8, 16))
        fwd[fft] = plan.forward(*dev[0])
        bwd[fft] = plan.backward(*dev[0], ge, *dev[1])
        fresh = gb.Plan(fr.box, mesh, order, 0.3, 9.0, max_ions=fr.n, fft=fft, brick=(8, 8, 16))
        for x, y in zip(bwd[fft], fresh.backward(*dev[0], ge, *dev[1])):
            assert torch.equal(x, y)
        plan.close()
        fresh.close()
    for k in ("force", "phi", "field"):
        check(f"line vs cuFFT {k} (rel RMSE)", relrmse(fwd["auto"][k].cpu().numpy(), fwd["cufft"][k].cpu().numpy()), 2e-6)
    hv = O2.PMEOracle(fr.box, mesh, order, 0.3, 9.0).hvp(pos, q, mu, 0.7, *cot)
    for x, y, r in zip(bwd["auto"], bwd["cufft"], hv):
        e_line, e_cu = relrmse(x.cpu().numpy(), r), relrmse(y.cpu().numpy(), r)
        check(f"line backward vs oracle (rel RMSE; cuFFT {e_cu:.2e})", e_line, min(TOL_HVP, 1.5 * e_cu + 2e-7))


def test_own_transforms_still_refused_for_large_planes(gb):
    with pytest.raises(gb.PMEError) as e:
        gb.Plan(np.eye(3) * 200.0, (256, 256, 256), 6, 0.3, 9.0, max_ions=64, fft="own")
    assert e.value.status == 5   # PME_ERR_UNSUPPORTED
