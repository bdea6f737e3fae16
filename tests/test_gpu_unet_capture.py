"""U-Net calls inside a CUDA graph capture: the first call of any size on a new
network can be captured (it neither allocates nor waits), and a graph's replays
stay right when later calls need more room than the captured one had.

Predictions of the same samples have the same bits however many go through the
network at once, so replays are compared exactly."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
Q = pytest.importorskip("paper_1512_02796_gb300")

pytestmark = pytest.mark.gpu

N = 32


@pytest.fixture(params=[0, 1], ids=["tcgen05", "mma.sync"])
def engine(request):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    Q.qpat_conv3d_set_engine(request.param)
    yield request.param
    Q.qpat_conv3d_set_engine(0)


def samples(B, seed=0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return (torch.randn((B, N ** 3, 3), generator=g, device="cuda"), torch.rand((B, N ** 3), generator=g, device="cuda"))


def predict(net, x):
    y = torch.empty(x.shape[:2], device="cuda")
    net.predict(x, y)
    return y


def train(net, x, t):
    """An Adam step that reads no loss back."""
    lib = Q.load()
    p = lambda a: ctypes.c_void_p(a.data_ptr())  # noqa: E731
    rc = lib.qpat_unet_train_dev(net.handle, p(x), p(t), x.shape[0], ctypes.c_float(1e-3), None,
                                 ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0, lib.qpat_last_error()


@pytest.mark.parametrize("B", [1, 3])
def test_first_predict_in_a_capture(engine, B):
    x, _ = samples(8)
    want = predict(Q.UNet(N, 1), x)
    net, y = Q.UNet(N, 1), torch.zeros((B, N ** 3), device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        net.predict(x[:B], y)
    g.replay()
    assert torch.equal(y, want[:B])
    assert torch.equal(predict(net, x), want)  # more samples at once: the room grows
    y.zero_()
    filler = [torch.full((1 << 24,), float("nan"), device="cuda") for _ in range(8)]  # whoever gets freed memory writes it
    g.replay()
    assert torch.equal(y, want[:B])
    del filler


@pytest.mark.parametrize("B", [1, 3])
def test_first_training_step_in_a_capture(engine, B):
    x, t = samples(8)
    ref, net = Q.UNet(N, 1), Q.UNet(N, 1)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        train(net, x[:B], t[:B])
    g.replay()
    train(ref, x[:B], t[:B])
    a, b = net.get_params(), ref.get_params()
    before = Q.UNet(N, 1).get_params()
    # one Adam step of rate 1e-3 moves a parameter by at most 1e-3, in the direction of its gradient's sign
    assert np.abs(a - before).max() <= 1.001e-3 and np.abs(a - before).max() > 0.5e-3
    assert np.mean(np.sign(a - before) == np.sign(b - before)) > 0.99
    train(net, x, t)  # more room
    g.replay()
    assert np.isfinite(net.get_params()).all()
