"""The network's parameter gradients where a block's partial sum overflows: the sum over the blocks
is that infinity, as in float64 arithmetic, and not the difference of two."""
import numpy as np
import pytest
import torch

import workloads as W
from gpu_util import f32
from test_gpu_net import _params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2606_01598_gb300 as g
    return g


@pytest.mark.parametrize("n", [8, 64, 216])
def test_infinite_partial_stays_infinite(gb, n):
    fr = W.molten_nacl(216, seed=21)
    net = gb.Net(n, 1)
    net.set_frames(np.array([0, n]), np.stack([fr.box]), fr.species[:n])
    net.set_params(_params(11))
    c = lambda x: torch.tensor(np.float32(x), device="cuda")
    net.forward(c(f32(fr.pos)[:n]))
    # dL/dbE is the sum of the ions' cotangents: eight of 1e38 in a block are past float32's range
    _, gpar = net.backward(c(np.zeros(n)), c(np.zeros((n, 3))), torch.tensor([1e38], dtype=torch.float64, device="cuda"))
    assert float(gb.unpack_params(gpar.cpu().numpy())["bE"].reshape(-1)[0]) == np.inf
    net.close()
