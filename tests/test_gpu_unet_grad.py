"""Gradients of the network at channel counts whose eight-channel groups do
not repeat over a warp (48) or fill it differently (16, 64), with the
comparison and the tolerances of the test of the default network's gradients
(test_gpu_unet: 5e-2 for the whole gradient, 1e-1 for a layer's block)."""
import pytest

import test_gpu_unet

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ndim,shape,channels", [(2, (32, 64), (48, 16)), (2, (48, 96), (64, 48)),
                                                 (3, (8, 8, 32), (48, 32))])
def test_gradient_at_other_widths(ndim, shape, channels):
    test_gpu_unet.test_gradient_matches_reference(ndim, shape, channels, "mse")
