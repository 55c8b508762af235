"""The tensor-core kernels of the warm-start network against its CUDA-core
form, at the sizes where their dispatch and tiles can go wrong: levels that
fit and levels that do not, row widths that are not whole pixel groups or are
odd, a single sample, output channels beyond the fused head."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# width, H, W, batch, output channels
CASES = [(16, 32, 64, 2, 3), (64, 32, 64, 1, 3), (32, 32, 96, 3, 1), (16, 64, 40, 2, 3), (16, 512, 12, 1, 2),
         (32, 16, 32, 2, 5), (16, 32, 256, 1, 4)]


@pytest.fixture(scope="module")
def NN():
    from paper_2401_17183_gb300 import build as B
    B.build()
    from paper_2401_17183_gb300 import nn
    nn.load()
    return nn


@pytest.mark.parametrize("width,H,W,B,co", CASES)
def test_tensor_core_forward_and_gradients(NN, width, H, W, B, co):
    torch = pytest.importorskip("torch")
    net = NN.Net(8, co, width, H, W, B, storage=NN.VLB_NN_BF16, seed=5)
    rng = np.random.default_rng(9)
    p = net.params()
    o = 0
    for cout, cin, k in NN.layer_shapes(8, co, width):
        o += cout * cin * k * k
        p[o:o + cout] = rng.uniform(-0.1, 0.1, cout)
        o += cout
    net.set_params(p)
    x = torch.from_numpy(rng.uniform(-1, 1, (B, 8, H, W)).astype(np.float32)).cuda()
    dy = torch.from_numpy(rng.uniform(-1, 1, (B, co, H, W)).astype(np.float32)).cuda()
    y = torch.zeros_like(dy)
    net.set_tensor_cores(False)
    net.forward(x.data_ptr(), y.data_ptr(), B)
    y_fma = y.cpu().numpy().copy()
    net.set_tensor_cores(True)
    net.forward(x.data_ptr(), y.data_ptr(), B)
    y_tc = y.cpu().numpy()
    # the two differ by bfloat16 roundings of activations that fall the other way
    assert np.linalg.norm(y_tc - y_fma) < 1e-2 * np.linalg.norm(y_fma)
    # gradients through the same stored activations: FP32 products and sums both
    # ways. A sum of n products is off by about sqrt(n) 2^-24 of its terms' norm; the
    # longest chains (4096 pixels, 11 layers deep) give about 1e-5 / 2
    net.backward(dy.data_ptr(), B)
    g_tc = net.grads()
    net.set_tensor_cores(False)
    net.backward(dy.data_ptr(), B)
    g = net.grads()
    o = 0
    for cout, cin, k in NN.layer_shapes(8, co, width):
        for n in (cout * cin * k * k, cout):
            assert np.linalg.norm(g_tc[o:o + n] - g[o:o + n]) <= 1e-5 * np.linalg.norm(g[o:o + n])
            o += n


def test_tensor_core_gradient_not_finite(NN):
    """An infinite and a NaN output gradient reach the parameters as such."""
    torch = pytest.importorskip("torch")
    net = NN.Net(8, 3, 16, 32, 64, 1, storage=NN.VLB_NN_BF16, seed=5)
    x = torch.rand((1, 8, 32, 64), device="cuda")
    y = torch.zeros((1, 3, 32, 64), device="cuda")
    net.forward(x.data_ptr(), y.data_ptr(), 1)
    for bad in (float("inf"), float("nan")):
        dy = torch.zeros_like(y)
        dy[0, 1, 7, 9] = bad
        net.backward(dy.data_ptr(), 1)
        assert not np.isfinite(net.grads()).all()
