"""The one-block sort of small frames: sizes around its thread counts and its limit, the forward
and the backward (records kept for unchanged inputs, formed again for changed ones), against the
oracle and against a one-frame batch plan, whose sort is always the general one."""
import numpy as np
import pytest
import torch

from gpu_util import TOL_F, check, f32, relrmse
from oracle import pme as O2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2606_01598_gb300 as g
    return g


def _frame(n, seed=5):
    rng = np.random.default_rng(seed + n)
    L = max(12.0, 3.0 * n ** (1 / 3))
    pos = f32(rng.uniform(0.0, L, size=(n, 3)))
    q = f32(rng.normal(size=n))
    mu = f32(0.1 * rng.normal(size=(n, 3)))
    return np.eye(3) * L, pos, q, mu


@pytest.mark.parametrize("mesh", [(16, 16, 16), (30, 27, 45)])
@pytest.mark.parametrize("n", [1, 2, 127, 128, 129, 383, 384, 385])
def test_small_frames(gb, n, mesh):
    box, pos, q, mu = _frame(n)
    t = [torch.tensor(np.float32(x), device="cuda") for x in (pos, q, mu)]
    plan = gb.Plan(box, mesh, 5, 0.35, 5.0, max_ions=n)
    r = plan.forward(*t)
    ref = O2.PMEOracle(box, mesh, 5, 0.35, 5.0).evaluate(pos, q, mu)
    check("phi (rel RMSE)", relrmse(r["phi"].cpu().numpy(), ref["phi"]), TOL_F)
    # a batch of this one frame sorts by the general kernels: the order, so the sums, are the same
    bp = gb.BatchPlan([box], [mesh], [5], [0, n], 0.35, 5.0)
    b = bp.forward(*t)
    for k in ("force", "phi", "field") if n > 2 else ("phi",):   # (one ion's force is rounding alone)
        check(k + " against the general sort", relrmse(r[k].cpu().numpy(), b[k].cpu().numpy()), 1e-6)
    # cotangents: unchanged inputs keep the order, changed ones sort again; both as a new plan's
    rng = np.random.default_rng(1)
    g = [torch.tensor(rng.normal(size=s), dtype=torch.float32, device="cuda") for s in ((n, 3), (n,), (n, 3))]
    moved = [(t[0] + 0.31) % float(box[0, 0]), t[1].flip(0).contiguous(), t[2]]
    for inp in (t, moved, t):
        got = plan.backward(*inp, 1.0, *g)
        new = gb.Plan(box, mesh, 5, 0.35, 5.0, max_ions=n)
        want = new.backward(*inp, 1.0, *g)
        assert all(torch.equal(x, y) for x, y in zip(got, want))
        new.close()
    plan.close()
    bp.close()
