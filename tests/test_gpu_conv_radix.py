"""The two-step mesh transforms on both sides of the factor (10) up to which the small set of
DFTs is built: single meshes against the oracle, batches of either kind against single frames."""
import numpy as np
import pytest
import torch

import workloads as W
from gpu_util import TOL_MESH, check_energy, prepared, relmax, relrmse
from oracle import pme as O2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2606_01598_gb300 as g
    return g


@pytest.mark.parametrize("mesh", [(4, 5, 6), (100, 9, 10), (10, 100, 81), (81, 90, 100), (108, 10, 9), (10, 75, 8),
                                  (9, 10, 96)])
def test_solve_matches_oracle(gb, mesh):
    fr = W.molten_nacl(512, seed=41)
    pos, q, mu = prepared(fr)
    o = O2.PMEOracle(fr.box, mesh, 4, 0.3, 9.0)
    rho = np.asarray(np.float32(o.stage_mesh(pos, q, mu)), np.float64)
    Phi_ref, E_ref = o.stage_solve(rho)
    plan = gb.Plan(fr.box, mesh, 4, 0.3, 9.0, max_ions=512, fft="own")
    Phi, E = plan.solve(torch.tensor(np.float32(rho), device="cuda"))
    assert relmax(Phi.cpu().numpy(), Phi_ref) < TOL_MESH
    check_energy(E.item(), E_ref, "E_recip")
    plan.close()


@pytest.mark.parametrize("last", [(100, 90, 81), (16, 96, 45)])
def test_batch_matches_single_frames(gb, last):
    meshes = [(8, 9, 10), (30, 27, 45), last]
    frs = [W.molten_nacl(n, seed=7 + n) for n in (64, 216, 512)]
    data = [prepared(fr) for fr in frs]
    off = np.concatenate([[0], np.cumsum([fr.n for fr in frs])]).tolist()
    t = [torch.tensor(np.float32(np.concatenate([d[k] for d in data])), device="cuda") for k in range(3)]
    bp = gb.BatchPlan([fr.box for fr in frs], meshes, [4, 4, 4], off, 0.3, 9.0)
    got = bp.forward(*t)
    for f, fr in enumerate(frs):
        plan = gb.Plan(fr.box, meshes[f], 4, 0.3, 9.0, max_ions=fr.n, fft="cufft")
        s = slice(off[f], off[f + 1])
        one = plan.forward(*(x[s].contiguous() for x in t))
        for k in ("force", "phi", "field"):   # two float32 transforms
            assert relrmse(got[k][s].cpu().numpy(), one[k].cpu().numpy()) < 2e-6, (f, k)
        plan.close()
    bp.close()
