"""The network at ion counts around the 128-row tiles of its channel mixing (scalar rows n, vector
rows 3 n, both products of a stage in one launch): forward and backward against the oracle."""
import numpy as np
import pytest
import torch

import workloads as W
from gpu_util import check, f32, relmax, relrmse
from oracle import net as N
from test_gpu_net import TOL_NET, _params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2606_01598_gb300 as g
    return g


@pytest.mark.parametrize("n", [2, 42, 43, 128, 129])
def test_forward_and_backward(gb, n):
    fr = W.molten_nacl(216, seed=21)
    pos, species = f32(fr.pos)[:n], fr.species[:n]
    params = _params(11)
    net = gb.Net(n, 1)
    net.set_frames(np.array([0, n]), np.stack([fr.box]), species)
    net.set_params(params)
    c = lambda x: torch.tensor(np.float32(x), device="cuda")
    out = net.forward(c(pos))
    rng = np.random.default_rng(n)
    gq, gmu = f32(rng.normal(size=n)), f32(rng.normal(size=(n, 3)))
    gp, gpar = net.backward(c(gq), c(gmu), torch.tensor([0.7], dtype=torch.float64, device="cuda"))
    net.sync_status()
    P = N.to_torch(params, requires_grad=True)
    pos_t = N._t(pos).requires_grad_(True)
    q, mu, e = N.predict(pos_t, species, fr.box, P)
    check("q (rel RMSE)", relrmse(out["q"].cpu().numpy(), q.detach().numpy()), TOL_NET)
    check("mu (rel RMSE)", relrmse(out["mu"].cpu().numpy(), mu.detach().numpy()), TOL_NET)
    check("E_sr (rel max)", relmax(out["e_sr"].cpu().numpy(), np.array([float(e)])), TOL_NET)
    L = (q * N._t(gq)).sum() + (mu * N._t(gmu)).sum() + 0.7 * e
    grads = torch.autograd.grad(L, [pos_t] + list(P.values()))
    check("g_pos (rel RMSE)", relrmse(gp.cpu().numpy(), grads[0].numpy()), TOL_NET)
    got = gb.unpack_params(gpar.cpu().numpy())
    for (name, _), g in zip(P.items(), grads[1:]):
        if name != "bq":      # the neutralisation removes bq
            check(f"g_{name} (rel RMSE)", relrmse(got[name], g.numpy()), TOL_NET)
    net.close()
