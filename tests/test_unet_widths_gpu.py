"""The layer-by-layer checks of test_unet_gpu.py at image widths where the kernels split a
row otherwise: one segment of 48, 80, 96 or 112 pixels, three and six segments of 128 (a
middle segment has no wrapped neighbour), and widths that the tcgen05 kernels do not
take (24, 168)."""
import pytest

from test_unet_gpu import (N, run, test_each_backward_tensor, test_each_weight_gradient,  # noqa: F401
                           test_input_and_each_forward_layer, torch)

WIDTHS = [(16, 48, 2), (24, 80, 1), (16, 96, 2), (16, 112, 1), (16, 384, 1), (8, 768, 1), (40, 24, 2), (24, 168, 1)]

# (overrides the shapes of the fixture)
pytestmark = pytest.mark.parametrize("run", WIDTHS, indirect=True, ids=[f"{h}x{w}x{n}" for h, w, n in WIDTHS],
                                     scope="module")
