"""The real-space potential of isolated ion pairs, pair by pair, over the arguments of erfc from
near zero to where the cutoff leaves it, against the oracle."""
import numpy as np
import pytest
import torch

from gpu_util import f32
from oracle import pme as O2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2606_01598_gb300 as g
    return g


@pytest.mark.parametrize("alpha,rcut", [(0.05, 6.0), (0.3, 9.0), (0.9, 5.6)])
def test_isolated_pairs(gb, alpha, rcut):
    # 512 pairs on a grid wider than two cutoffs, each of its own separation and direction
    m, L = 8, 8 * (2.2 * rcut)
    rng = np.random.default_rng(23)
    grid = (np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3) + 0.3) * (L / m)
    r = np.linspace(0.02, 0.999, len(grid)) * rcut
    d = rng.normal(size=(len(grid), 3))
    d *= (r / np.linalg.norm(d, axis=1))[:, None]
    pos = f32(np.mod(np.concatenate([grid, grid + d]), L))
    q = f32(rng.uniform(0.5, 1.5, size=len(pos)))
    plan = gb.Plan(np.eye(3) * L, (16, 16, 16), 4, alpha, rcut, max_ions=len(pos))
    out, _ = plan.pair(*(torch.tensor(np.float32(x), device="cuda") for x in (pos, q, 0 * pos)))
    _, phi, _, _ = O2.PMEOracle(np.eye(3) * L, (16, 16, 16), 4, alpha, rcut).stage_pair(pos, q, 0 * pos)
    phi, out = np.asarray(phi), out[:, 0].double().cpu().numpy()
    # float32: erfc itself (3.3e-7), eight roundings, and a separation that is off by up to eight
    # roundings of a cell's edge (at most the cutoff), which erfc(x)/r passes on at most 2 + 2 x^2 times
    x, rr = alpha * np.concatenate([r, r]), np.concatenate([r, r])
    tol = 3.3e-7 + 2.0 ** -24 * (8 + (2 + 2 * x * x) * 8 * (1 + rcut / rr))
    worst = np.max(np.abs(out - phi) / (tol * np.abs(phi)))
    assert worst < 1.0, worst
    plan.close()
