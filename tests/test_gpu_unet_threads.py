"""Networks of different widths run side by side in host threads.

Their convolutions share kernels whose shared-memory need differs from launch to launch; a launch must not
depend on the size another thread asked for last.
"""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_two_networks_in_two_threads():
    import torch
    from paper_1808_07150_gb300 import learned
    shape = (8, 16, 8)
    x = torch.rand(int(np.prod(shape)), device="cuda")
    errors = []

    def work(channels):
        try:
            stream = torch.cuda.Stream()
            with learned.UNet(shape, channels) as net:
                net.init(3)
                pred = torch.zeros_like(x)
                for _ in range(400):
                    net.forward(x, 1.0, pred, stream=stream)
                    net.backward(target=x, want_loss=False, stream=stream)
                stream.synchronize()
        except Exception as e:
            errors.append(e)

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(c,)) for c in ((16, 16), (32, 16), (16, 128), (64, 32))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    assert learned.device_error() == 0
