"""The gradient above 128 rows, where a column of the image takes several tiles
and its last one is ragged: the gated input gradients of k_conv_col clipped at
the image's end (136, 200), the weight gradient's blocks running over several
per column (192, 256), one to several images per tile at the coarser levels.
The bounds of test_gpu_unet.py; at least 500 pixels at the coarsest level."""
import pytest

import test_gpu_unet as T

pytestmark = pytest.mark.gpu

SHAPES = [(136, 128, 2, 3, True), (200, 96, 2, 5, False), (256, 64, 2, 8, True), (192, 64, 3, 3, False)]


@pytest.mark.parametrize("H,W,n,cin,periodic_x", SHAPES)
def test_gradient(H, W, n, cin, periodic_x):
    T.test_gradient_matches_oracle(H, W, n, cin, periodic_x)


@pytest.mark.parametrize("H,W,n,cin,periodic_x", SHAPES)
def test_weight_gradient_kernels(H, W, n, cin, periodic_x):
    T.test_weight_gradient_kernels_agree(H, W, n, cin, periodic_x)
