"""Which transforms a single frame's plan takes by itself: the two-step kernels, except where planes of
more than half an SM's shared memory are more than the SMs (and cuFFT is not slow) or do not fit."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2606_01598_gb300 as g
    return g


@pytest.mark.parametrize("mesh,kernels", [
    ((100, 100, 100), "general"),
    ((150, 128, 128), "general"),       # one wave of large planes
    ((160, 96, 96), "general"),         # small planes
    ((160, 128, 128), "cufft"),
    ((256, 128, 128), "cufft"),
    ((160, 135, 135), "general"),       # two axes on which cuFFT is slow
    ((16, 192, 144), "cufft"),          # the two-step layout does not fit, the Stockham one does
    ((128, 128, 128), "power-of-two"),
    ((64, 256, 256), "power-of-two"),   # line by line
])
def test_automatic_choice(gb, mesh, kernels):
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the line lies at the number of SMs")
    plan = gb.Plan(np.diag(mesh) * 1.0, mesh, 4, 0.3, 5.0, max_ions=64, brick=(8, 8, 16))
    assert plan.fft_kernels == kernels
    plan.close()
