"""The column convolution (k_conv_col) at the sizes where its tiles are ragged:
heights that do not divide 128 or pass it, batches that do not fill a tile's
images, columns fewer than the SMs, an odd last column of a pair, both
paddings.  Forward against the FP64 reference with BF16 storage emulated, to
the bound of test_gpu_unet.py (1e-2 relative L2: FP32 accumulation order and
the BF16 roundings it flips); a missing row, image, column or tap is above 5e-2."""
import numpy as np
import pytest

from oracle import unet as U
from test_gpu_unet import _dev, _problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,n,cin,periodic_x", [(8, 8, 1, 3, True), (136, 16, 1, 8, True), (40, 24, 5, 8, False),
                                                  (16, 32, 3, 16, True), (256, 8, 2, 4, False), (128, 8, 1, 8, True),
                                                  (64, 72, 3, 8, False)])
def test_forward_at_ragged_tiles(H, W, n, cin, periodic_x):
    import torch
    import paper_2212_07494_gb300 as P
    params, x, t, m = _problem(H, W, n, 3, cin)
    net = P.UNet(H, W, n + 1, cin=cin, periodic_x=periodic_x)
    net.set_params(params)
    xd = _dev(x)
    yd = torch.empty((n, H, W, 3), dtype=torch.float32, device="cuda")
    net.forward(xd.data_ptr(), yd.data_ptr(), n)
    torch.cuda.synchronize()
    y = yd.cpu().numpy().astype(np.float64)
    yb, _ = U.forward(params, x, storage="bf16", periodic_x=periodic_x)
    assert np.linalg.norm(y - yb) < 1e-2 * np.linalg.norm(yb)
    net.close()
