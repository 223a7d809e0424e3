"""The convolutions' tile edges: grids that are no multiple of the 8 x 16 x (1, 2, 3) voxel tiles (or of the 8 x 8 x 4 tiles
of the weight gradient), channel counts that are no multiple of 16, more than one block of 64 output channels,
and the decoder's concatenation with a boundary inside a group of eight channels; against the numpy oracle.

Tolerances as in the other U-Net tests (FP32 accumulation of up to 27 x 96 products and sums over the voxels:
about 1e-5 relative forward and 1e-4 in the gradients, with a factor 10).  Weights and biases keep the ReLUs'
inputs away from 0, where a rounding would switch a gradient on or off.
"""
import numpy as np
import pytest

from oracle import unet_oracle as U

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _rel(a, b):
    return float(np.abs(a - b).max() / max(np.abs(b).max(), 1e-30))


def _weights(ref, seed):
    """Small weights (biases stay the parameters' last entries per layer) and biases of about +-1."""
    rng = np.random.default_rng(seed)
    w = []
    for ci, co in ref:
        w += [rng.uniform(-1, 1, co * ci * 27) * 0.1 * np.sqrt(6.0 / (27 * ci)),
              rng.uniform(0.8, 1.2, co) * np.where(np.arange(co) % 4 == 3, -1, 1)]
    return np.concatenate(w).astype(np.float32)


def _layers(base, levels):
    ch = [min(base << l, 4 * base) for l in range(levels)]
    conv = []
    for l in range(levels):
        conv += [(4 if l == 0 else ch[l - 1], ch[l]), (ch[l], ch[l])]
    for l in range(levels - 2, -1, -1):
        conv += [(ch[l + 1] + ch[l], ch[l]), (ch[l], ch[l])]
    return conv + [(ch[0], 3)]


# (levels, base, (z, y, x), batch); the fifth runs the two-plane tiles, the sixth the three-plane ones (288 blocks each)
@pytest.mark.parametrize("levels,base,shape,batch", [(1, 5, (3, 17, 9), 2), (2, 12, (6, 18, 10), 1), (1, 70, (2, 5, 3), 1),
                                                     (3, 17, (4, 8, 12), 3), (1, 20, (31, 34, 41), 1),
                                                     (1, 12, (47, 34, 41), 1)])
def test_unet_tile_edges(levels, base, shape, batch):
    from paper_1809_00828_gb300 import fcm
    net = fcm.UNet(in_ch=4, out_ch=3, base=base, levels=levels, seed=1)
    net.set(_weights(_layers(base, levels), 5))
    rng = np.random.default_rng(3)
    x = (0.2 * rng.standard_normal((batch, 4) + shape)).astype(np.float32)
    xd = torch.from_numpy(x).cuda()  # backward reads it again
    out = net.forward(xd).cpu().numpy()
    ref = U.UNetOracle(net.get(), 4, 3, base, levels)
    out_ref = ref.forward(x.astype(np.float64))
    assert _rel(out, out_ref) < 1e-4
    gout = rng.standard_normal(out.shape).astype(np.float32)
    net.zero_grad()
    din = net.backward(torch.from_numpy(gout).cuda(), want_din=True).cpu().numpy()
    _, g = net.get(with_grad=True)
    din_ref, g_ref = ref.backward(gout.astype(np.float64))
    assert _rel(din, din_ref) < 1e-3
    assert _rel(g, g_ref) < 1e-3
    # a second backward accumulates, and the same inputs give the same bits
    out2 = net.forward(xd).cpu().numpy()
    net.backward(torch.from_numpy(gout).cuda())
    _, g2 = net.get(with_grad=True)
    assert np.array_equal(out, out2) and np.array_equal(g2, g + g)
    net.close()


def test_infinities_and_nan_pass_through():
    from paper_1809_00828_gb300 import fcm
    net = fcm.UNet(in_ch=1, out_ch=1, base=1, levels=1, seed=1)
    w = np.zeros(net.nparam, np.float32)
    w[13] = w[28 + 13] = w[56 + 13] = 1.0  # identity taps
    net.set(w)
    x = torch.ones((1, 1, 4, 4, 8), device="cuda")
    x[0, 0, 1, 1, 2] = float("inf")
    x[0, 0, 3, 3, 7] = 3.0e38
    y = net.forward(x)
    # 0 * inf = NaN in the neighbours, as for FP32 products; ReLU maps NaN to 0
    assert torch.isinf(y[0, 0, 1, 1, 2]) or torch.isnan(y[0, 0, 1, 1, 2])
    assert float(y[0, 0, 3, 3, 7]) == float(np.float32(3.0e38)) and float(y[0, 0, 3, 0, 0]) == 1.0
    net.close()


def test_where_infinities_go():
    """Identity taps: an infinite voxel stays itself; 0 * inf makes its neighbours NaN, which a ReLU maps to 0 and the
    output layer (no ReLU) passes on.  -inf and NaN are 0 after the first ReLU, and so are their neighbours."""
    from paper_1809_00828_gb300 import fcm
    net = fcm.UNet(in_ch=1, out_ch=1, base=1, levels=1, seed=1)
    w = np.zeros(net.nparam, np.float32)
    w[13] = w[28 + 13] = w[56 + 13] = 1.0
    net.set(w)
    x = np.ones((4, 4, 16), np.float32)
    want = x.copy()
    x[1, 1, 2], x[3, 1, 6], x[3, 1, 10], x[3, 3, 15] = np.inf, -np.inf, np.nan, 3.0e38
    want[0:3, 0:3, 1:4] = np.nan
    want[1, 1, 2] = np.inf
    want[2:4, 0:3, 5:8] = want[2:4, 0:3, 9:12] = 0.0
    want[3, 3, 15] = 3.0e38
    y = net.forward(torch.from_numpy(x).cuda().view(1, 1, 4, 4, 16)).cpu().numpy().reshape(4, 4, 16)
    assert np.array_equal(y, want, equal_nan=True)
    net.close()


def test_an_infinite_gradient_stays_infinite():
    """The bias gradient (a plain sum) of a layer whose CTAs add several tiles to running sums."""
    from paper_1809_00828_gb300 import fcm
    net = fcm.UNet(in_ch=4, out_ch=3, base=100, levels=1, seed=1)
    net.forward(torch.ones((1, 4, 20, 20, 20), device="cuda"))
    g = torch.zeros((1, 3, 20, 20, 20), device="cuda")
    g[0, 0, 9, 9, 9] = float("inf")
    g[0, 1] = 1.0
    net.zero_grad()
    net.backward(g)
    _, grad = net.get(with_grad=True)
    assert np.array_equal(grad[-3:], [np.inf, 8000.0, 0.0])
    net.close()
