"""The bounded wait of the U-Net's convolutions for the tensor core: with a limit of 0 every convolution gives up (its
products land, the kernel returns), the caller learns of it, no parameter is updated from what it left, and with the
default limit everything is as before.
"""
import numpy as np
import pytest

from paper_1809_00828_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _net(base=20):
    from paper_1809_00828_gb300 import fcm
    return fcm.UNet(in_ch=4, out_ch=3, base=base, levels=2, seed=1)


def test_a_forward_pass_that_timed_out_is_reported_once():
    from paper_1809_00828_gb300 import fcm
    net = _net()
    x = torch.randn((2, 4, 8, 8, 16), device="cuda")
    ref = net.forward(x)
    net.check()
    net.set_wait_limit(0)
    net.forward(x)
    with pytest.raises(fcm.FcmError) as e:
        net.check()
    assert e.value.status == fcm.FCM_ETIMEOUT
    net.check()
    net.forward(x)
    torch.cuda.synchronize()
    with pytest.raises(fcm.FcmError) as e:  # the next call reports it and does nothing else
        net.forward(x)
    assert e.value.status == fcm.FCM_ETIMEOUT
    net.check()
    net.set_wait_limit(-1)
    assert torch.equal(net.forward(x), ref)
    net.check()
    net.close()


def test_no_update_from_gradients_that_timed_out():
    from paper_1809_00828_gb300 import fcm
    net = _net()
    x, g = torch.randn((1, 4, 8, 8, 8), device="cuda"), torch.randn((1, 3, 8, 8, 8), device="cuda")
    w = net.get()
    net.forward(x)  # the buffers of this shape
    net.set_wait_limit(0)
    torch.cuda.synchronize()
    torch.cuda._sleep(200_000_000)  # the calls below are queued before any of them runs
    net.zero_grad()
    net.forward(x)
    net.backward(g)
    net.adam(1e-2, 1)
    with pytest.raises(fcm.FcmError) as e:
        net.get()
    assert e.value.status == fcm.FCM_ETIMEOUT
    assert np.array_equal(net.get(), w)
    net.set_wait_limit(-1)
    net.zero_grad()
    net.forward(x)
    net.backward(g)
    net.adam(1e-2, 1)
    assert not np.array_equal(net.get(), w)
    net.close()


def test_a_flexible_solve_with_a_network_that_timed_out():
    from paper_1809_00828_gb300 import fcm
    s = fcm.Solver(I.workload_porous(5, 8, 2, 6, 1e-8, 3, 1e-9))
    s.precond_build()
    net, b = _net(4), s.rhs()
    u, its, _, st = s.fpcg_solve(net, 0.1, b, 1e-6, 500, coarse_iters=2)
    assert st == fcm.FCM_OK
    net.set_wait_limit(0)
    with pytest.raises(fcm.FcmError, match="convolution") as e:
        s.fpcg_solve(net, 0.1, b, 1e-6, 500, coarse_iters=2)
    assert e.value.status == fcm.FCM_ETIMEOUT and s.last_solve()["status"] == fcm.FCM_ETIMEOUT
    assert s.get_info()["device_error"] == 0
    net.check()  # the solve's failure is not the network's own
    net.set_wait_limit(-1)
    u2, its2, _, _ = s.fpcg_solve(net, 0.1, b, 1e-6, 500, coarse_iters=2)
    assert its2 == its and torch.equal(u2, u)
    net.close()
    s.close()
