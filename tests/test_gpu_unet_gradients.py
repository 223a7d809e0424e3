"""Weight gradients of wide layers, where few CTAs share the voxels of a channel pair, against 64 bits.

Bound (relative, 2-norm): the layer's input and the gradient of its output are FP32 results, each within about
2^-23, and the sum over N voxels is made of FP32 chains of at most N / 256 additions, whose rounding errors of at
most 2^-24 of the running sum add up as a random walk to sqrt(N / 512) 2^-25 of the whole.  Weights and biases keep
the ReLUs' inputs away from 0, where a rounding would switch a gradient on or off.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("base,shape,batch", [(100, (25, 31, 17), 2), (256, (32, 32, 32), 1)])
def test_weight_gradients_of_wide_layers(base, shape, batch):
    from paper_1809_00828_gb300 import fcm
    F = torch.nn.functional
    chan = [(4, base), (base, base), (base, 3)]
    rng = np.random.default_rng(5)
    w = [np.concatenate([rng.uniform(-1, 1, co * ci * 27) * 0.1 * np.sqrt(6.0 / (27 * ci)),
                         rng.uniform(0.8, 1.2, co) * np.where(np.arange(co) % 4 == 3, -1, 1)]).astype(np.float32)
         for ci, co in chan]
    net = fcm.UNet(in_ch=4, out_ch=3, base=base, levels=1, seed=1)
    net.set(np.concatenate(w))
    x = 0.2 * torch.from_numpy(rng.standard_normal((batch, 4) + shape).astype(np.float32)).cuda()
    gout = torch.from_numpy(rng.standard_normal((batch, 3) + shape).astype(np.float32)).cuda()
    net.forward(x)
    net.zero_grad()
    net.backward(gout)
    _, grad = net.get(with_grad=True)
    par = []
    for (ci, co), v in zip(chan, w):
        t = torch.from_numpy(v).cuda()
        par.append((t[:-co].bfloat16().double().view(co, ci, 3, 3, 3).requires_grad_(), t[-co:].double()))
    v = x.double()
    with torch.backends.cudnn.flags(enabled=False):
        for k, (a, b) in enumerate(par):
            v = F.conv3d(v, a, b, padding=1)
            v = F.relu(v) if k < 2 else v
        v.backward(gout.double())
    at = 0
    n = batch * int(np.prod(shape))
    for (ci, co), (a, _) in zip(chan, par):
        g = torch.from_numpy(grad[at:at + 27 * ci * co]).cuda().double()
        at += 27 * ci * co + co
        err = float((g - a.grad.flatten()).norm() / a.grad.norm())
        assert err < 2 * 2.0 ** -23 + (n / 512) ** 0.5 * 2.0 ** -25, (ci, co, err)
    net.close()
