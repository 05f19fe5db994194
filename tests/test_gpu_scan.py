"""Segment starts of the counting sort over many keys: the pair term of sparse frames whose pair
cells fill one, a few and more than the largest number of scan segments, against the oracle."""
import numpy as np
import pytest
import torch

from gpu_util import TOL_F, check, f32, relrmse, sym6
from oracle import pme as O2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2606_01598_gb300 as g
    return g


@pytest.mark.parametrize("L,rcut", [(24.0, 4.0), (60.0, 6.0), (150.0, 4.5), (150.0, 9.0)])
def test_pair_term_over_many_cells(gb, L, rcut):
    # (12^3, 20^3, 66^3 and 33^3 cells: 1, 2, 36 of double length, and 9 segments); ions in clumps, so that
    # there are partners within the cutoff
    n = 2304
    rng = np.random.default_rng(17)
    centres = rng.uniform(0.0, L, size=(n // 8, 3))
    pos = f32(np.mod(np.repeat(centres, 8, 0) + rng.normal(0.0, 1.2, size=(n, 3)), L))
    q = f32(rng.normal(size=n))
    mu = f32(0.1 * rng.normal(size=(n, 3)))
    plan = gb.Plan(np.eye(3) * L, (16, 16, 16), 4, 0.30, rcut, max_ions=n)
    out, e = plan.pair(*(torch.tensor(np.float32(x), device="cuda") for x in (pos, q, mu)))
    _, phi, g, H = O2.PMEOracle(np.eye(3) * L, (16, 16, 16), 4, 0.30, rcut).stage_pair(pos, q, mu)
    out = out.cpu().numpy()
    check("pair phi (rel RMSE)", relrmse(out[:, 0], phi), TOL_F)
    check("pair grad (rel RMSE)", relrmse(out[:, 1:4], g), TOL_F)
    check("pair hess (rel RMSE)", relrmse(out[:, 4:], sym6(H)), TOL_F)
    plan.close()
