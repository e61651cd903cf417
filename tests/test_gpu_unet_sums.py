"""Which pixels one FP32 sum of a weight or bias gradient adds, in which order.

The additions in a tensor core truncate, and Adam's first steps follow the
sign of a gradient, so the members and the order of these sums are part of
what a training step returns.  A network whose layers copy channel 0 (one
weight of 1 at the centre tap, activations of 1) has the loss weights m, times
4 per level, as every layer's dz, so dW[0][centre][0] is a sum of m over the
layer's pixels.  m is 1 but for two 8 x 8 patches, one above the other, of
+2^60 and -2^60: they cancel exactly, and the ones that a sum holds or adds
between its first and its last large term are lost.  How many are lost shows
where each sum starts and how it runs.  All terms left are integers, so the
expected values are exact: the tolerance is zero.  (The patches end with a
16-pixel slice in either order, so how the unit adds within one does not
matter.)"""
import numpy as np
import pytest

from oracle import unet as U

pytestmark = pytest.mark.gpu

BIG = 2.0 ** 60
LEVEL = {"enc1a": 0, "enc1b": 0, "enc2a": 1, "enc2b": 1, "enc3a": 2, "enc3b": 2, "bota": 3, "botb": 3, "up3": 2, "dec3a": 2,
         "dec3b": 2, "up2": 1, "dec2a": 1, "dec2b": 1, "up1": 0, "dec1a": 0, "dec1b": 0, "head": 0}


def _sums(n, H, W, cin, cout, sms):
    """The pixels (image, y, x) of each sum, in order: an index array [pixels, 3] per sum."""
    img, y, x = np.meshgrid(np.arange(n), np.arange(H), np.arange(W), indexing="ij")
    pix = np.stack([img, y, x], -1)
    HB = min(H, 64)
    NB = 64 // HB
    if 64 % HB or H % HB or n % NB:
        flat = pix.reshape(-1, 3)   # mma.sync: 2048 pixels of the images read line by line
        return [flat[k:k + 2048] for k in range(0, len(flat), 2048)]
    # tcgen05: blocks of HB rows of NB images at one x, x running first
    blocks = pix.reshape(n // NB, NB, H // HB, HB, W, 3).transpose(0, 2, 4, 1, 3, 5).reshape(-1, 64, 3)
    CA = min(cin, 64)
    tiles = -(-(9 * cin // CA) // (128 // CA))
    splits = min(-(-2 * sms // tiles), max(len(blocks) // 8, 1))
    per = -(-len(blocks) // splits)
    return [blocks[k:k + per].reshape(-1, 3) for k in range(0, len(blocks), per)]


def _kept(m, sums):
    """The ones of m that its sums keep."""
    kept = 0
    for s in sums:
        v = m[s[:, 0], s[:, 1], s[:, 2]].reshape(-1, 16)
        big, acc = 0.0, 0
        for r in v:
            large = np.abs(r) > 1
            if big or large.any():
                big += r[large].sum()
                acc = 0
            else:
                acc += len(r)
        assert big == 0.0
        kept += acc
    return kept


def _copy_net(P, H, W, n):
    net = P.UNet(H, W, n, cin=3, periodic_x=True)
    p = np.zeros(net.n)
    sl, _ = U.layer_slices(3)
    for name, ci, co, relu, wo, bo in sl:
        if name == "enc1a":
            p[bo] = 1.0
        else:
            p[wo + 4 * ci] = 1.0
    net.set_params(p)
    return net, sl


def _grad(net, m):
    import torch
    n, H, W = m.shape
    x = torch.ones((n, H, W, 3), device="cuda")
    t = torch.zeros((n, H, W, 3), device="cuda")
    md = torch.tensor(m, dtype=torch.float32, device="cuda")
    _, g = net.grad(x.data_ptr(), t.data_ptr(), md.data_ptr(), n, 0.5)
    return g.astype(np.float64)


# 128 x 256 and 64 x 128: blocks of one and of several images; batch 3: the levels
# with several images per block go to mma.sync; 192: three blocks per column;
# W = 120 and 136: an odd number of columns at the coarser levels
@pytest.mark.parametrize("H,W,n,image,x0", [(128, 256, 8, 1, 120), (128, 256, 8, 7, 248), (64, 128, 8, 3, 120), (64, 128, 3, 1, 120),
                                            (192, 128, 2, 1, 120), (128, 136, 8, 5, 0), (128, 120, 4, 3, 112)])
def test_weight_gradient_sums(H, W, n, image, x0):
    import torch
    import paper_2212_07494_gb300 as P
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    net, sl = _copy_net(P, H, W, n)
    m = np.ones((n, H, W))
    m[image, H - 16:H - 8, x0:x0 + 8] = BIG
    m[image, H - 8:, x0:x0 + 8] = -BIG
    g = _grad(net, m)
    net.close()
    bad = {}
    for name, ci, co, relu, wo, bo in sl:
        q = 1 << LEVEL[name]
        sums = _sums(n, H // q, W // q, -(-ci // 16) * 16, -(-co // 32) * 32, sms)
        want = q * q * _kept(m[:, ::q, ::q], sums)
        if g[wo + 4 * ci] != want:
            bad[name] = (g[wo + 4 * ci], want)
    assert not bad, bad


def test_bias_gradient_sums():
    """The head's bias: a thread adds 16 pixels 256 apart, in FP32."""
    import paper_2212_07494_gb300 as P
    net, sl = _copy_net(P, 128, 256, 1)
    bo = sl[-1][5]
    for first, thread in ((0, 0), (4096, 77), (28672, 255)):
        m = np.ones(128 * 256)
        m[first + thread] = BIG
        m[first + thread + 15 * 256] = -BIG
        assert _grad(net, m.reshape(1, 128, 256))[bo] == 128 * 256 - 16, (first, thread)
    net.close()


def test_adam_rounding():
    """Four Adam steps from the library's own gradients and parameters: both moments add a rounded product of the old
    moment to an exact one of the gradient (one fused multiply-add), every other operation is rounded on its own.
    Emulated in extended precision with a rounding to FP32 after each operation: equal bit for bit (products of two
    FP32 values and their sum with a third round the same from 64 bits of mantissa but for ties of one in 2^40)."""
    import torch
    import paper_2212_07494_gb300 as P
    f, L = np.float32, np.longdouble
    if np.finfo(L).nmant < 63:
        pytest.skip("no extended precision")
    H, W, n = 32, 64, 2
    rng = np.random.default_rng(1)
    net = P.UNet(H, W, n, cin=3)
    net.set_params(0.05 * rng.normal(size=net.n))
    x, t = (torch.tensor(rng.normal(size=(n, H, W, 3)), dtype=torch.float32, device="cuda") for _ in range(2))
    w = torch.ones((n, H, W), device="cuda")
    b1, b2, lr, eps = f(0.9), f(0.999), f(1e-3), f(1e-8)
    o1, o2 = f(1) - b1, f(1) - b2
    m, v = np.zeros(net.n, f), np.zeros(net.n, f)
    for k in range(1, 5):
        p = net.params().copy()
        g = np.asarray(net.grad(x.data_ptr(), t.data_ptr(), w.data_ptr(), n, 1 / (3.0 * n * H * W))[1], f)
        net.adam(float(lr))
        m = (L(o1) * g + L(1) * (b1 * m)).astype(f)
        v = ((o2 * g).astype(L) * g + L(1) * (b2 * v)).astype(f)
        c1, c2 = f(1) - f(float(b1) ** k), f(1) - f(float(b2) ** k)
        want = p - (lr * (m / c1)) / (np.sqrt(v / c2) + eps)
        assert np.array_equal(net.params(), want), (k, np.mean(net.params() != want))
    net.close()
