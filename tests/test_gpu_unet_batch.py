"""The U-Net on several samples at once, and the tcgen05 convolution's boxes.

* Convolution: ragged grids (sides that no box divides, sides below a tile)
  and channel counts on both sides of the resident / streamed weights, against
  the mma.sync engine: the same exact BF16 products in FP32 sums of another
  order, at most 27 Cin terms: 1e-5 of the result's scale, as the layer tests.
* Prediction: rows of an MMA do not mix, so a sample's prediction does not
  depend on the samples beside it: the same bits one by one and together.
* Gradient of 4 samples: the mean-squared error of the batch scales every
  gradient by 1/4, exactly in BF16; the sums over samples then differ from the
  four single gradients' sum by FP32 summation order only (1e-5 of the norm).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
Q = pytest.importorskip("paper_1512_02796_gb300")

pytestmark = pytest.mark.gpu


def _need():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("n,cin,cout", [(2, 16, 16), (6, 32, 16), (10, 16, 64), (18, 96, 32), (34, 48, 16), (34, 64, 128),
                                        (66, 16, 32), (130, 16, 16), (12, 192, 64), (20, 128, 128)])
def test_convolution_boxes(n, cin, cout):
    _need()
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    x = torch.randn((n ** 3, cin), generator=g, device="cuda").bfloat16()
    w = (torch.randn((27, cout, cin), generator=g, device="cuda") / np.sqrt(27 * cin)).bfloat16()
    b = torch.randn(cout, generator=g, device="cuda")
    got = []
    for engine in (0, 1):
        Q.qpat_conv3d_set_engine(engine)
        try:
            o = torch.empty((n ** 3, cout), dtype=torch.bfloat16, device="cuda")
            o32 = torch.empty((n ** 3, cout), device="cuda")
            Q.qpat_conv3d_bf16_dev(x, w, b, cout, True, n, o, o32)
            assert torch.equal(o, o32.bfloat16())
            got.append(o32)
        finally:
            Q.qpat_conv3d_set_engine(0)
    assert float((got[0] - got[1]).abs().max()) < 1e-5 * float(got[1].abs().max())
    assert Q.qpat_conv3d_tc_timeouts() == 0


@pytest.mark.parametrize("n,B", [(32, 3), (48, 2)])
@pytest.mark.parametrize("floor", [0.0, 1e-6])
def test_prediction_of_a_batch_equals_the_samples(n, B, floor):
    _need()
    net = Q.UNet(n, seed=3)
    net.set_log_output(floor)
    try:
        x = torch.randn((B, n ** 3, 3), device="cuda")
        both = net.predict(x, torch.empty((B, n ** 3), device="cuda"))
        for b in range(B):
            one = net.predict(x[b:b + 1].contiguous(), torch.empty((1, n ** 3), device="cuda"))
            assert torch.equal(one[0], both[b])
        Q.qpat_conv3d_set_engine(1)
        try:
            other = net.predict(x, torch.empty((B, n ** 3), device="cuda"))
        finally:
            Q.qpat_conv3d_set_engine(0)
        assert float((other - both).norm() / other.norm()) < 2e-2
    finally:
        net.close()


def test_gradient_of_a_batch_is_the_mean_of_the_samples():
    _need()
    n, B = 32, 4
    net = Q.UNet(n, seed=5)
    try:
        x = torch.randn((B, n ** 3, 3), device="cuda")
        t = torch.rand((B, n ** 3), device="cuda")
        loss, g = net.grad(x, t)
        parts = [net.grad(x[b:b + 1].contiguous(), t[b:b + 1].contiguous()) for b in range(B)]
        ref = sum(p[1].astype(np.float64) for p in parts) / B
        assert abs(loss - sum(p[0] for p in parts) / B) < 1e-5 * loss
        assert np.linalg.norm(g - ref) < 1e-5 * np.linalg.norm(ref)
    finally:
        net.close()
