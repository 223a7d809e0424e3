"""Threads that read one network while another sets it: every read is one set's parameters, whole."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_readers_get_whole_parameters():
    from paper_1809_00828_gb300 import fcm
    net = fcm.UNet(in_ch=4, out_ch=3, base=24, levels=3, seed=1)
    net.set(np.full(net.nparam, 1.0, np.float32))
    start, stop, torn, errors = threading.Barrier(5), threading.Event(), [], []

    def read():
        try:
            start.wait()
            while not stop.is_set():
                w = net.get()
                if w.min() != w.max():
                    torn.append((float(w.min()), float(w.max())))
        except Exception as e:  # noqa: BLE001 (reported below)
            errors.append(e)

    readers = [threading.Thread(target=read) for _ in range(4)]
    for t in readers:
        t.start()
    start.wait()
    for k in range(300):
        net.set(np.full(net.nparam, float(k % 7), np.float32))
    stop.set()
    for t in readers:
        t.join()
    assert not errors and not torn
    net.close()
