"""Networks used by several threads at once: every thread has its own network,
grid and buffers, and gets the gradients that it gets alone."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def NN():
    from paper_2401_17183_gb300 import build as B
    B.build()
    from paper_2401_17183_gb300 import nn
    nn.load()
    return nn


# (H, W): one kernel instance, launched with the shared memory of each row width
@pytest.mark.parametrize("grids", [[(32, 64), (16, 128), (64, 32)], [(32, 64), (32, 64)]])
def test_backward_in_threads(NN, grids):
    torch = pytest.importorskip("torch")
    B, co, work = 1, 3, []
    for k, (H, W) in enumerate(grids):
        net = NN.Net(8, co, 64, H, W, B, storage=NN.VLB_NN_BF16, seed=k)
        g = torch.Generator().manual_seed(k)
        x, dy = (torch.rand((B, c, H, W), generator=g).cuda() for c in (8, co))
        work.append((net, x, dy, torch.zeros_like(dy)))
    torch.cuda.synchronize()

    def one(w):
        net, x, dy, y = w
        net.forward(x.data_ptr(), y.data_ptr(), B)
        net.backward(dy.data_ptr(), B)
        return net.grads()

    alone = [one(w) for w in work]
    wrong = []

    def loop(w, want):
        for _ in range(150):
            try:
                if not np.array_equal(one(w), want):
                    wrong.append("other gradients")
            except Exception as e:
                wrong.append(str(e))

    threads = [threading.Thread(target=loop, args=a) for a in zip(work, alone)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, (len(wrong), wrong[0])
