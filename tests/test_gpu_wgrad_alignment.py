"""The weight gradient of the BF16 convolution takes tensors on any boundary of a
BF16 number (slices of larger buffers), with the bits of the aligned ones."""
import pytest

torch = pytest.importorskip("torch")
Q = pytest.importorskip("paper_1512_02796_gb300")

pytestmark = pytest.mark.gpu


def shifted(a, by):
    """The same values, starting `by` elements behind a 256-byte boundary."""
    room = torch.zeros(a.numel() + by, dtype=a.dtype, device=a.device)
    room[by:] = a.reshape(-1)
    return room[by:].view(a.shape)


@pytest.mark.parametrize("n,cin,cout", [(4, 16, 16), (8, 48, 16), (8, 192, 64), (12, 128, 128)])
@pytest.mark.parametrize("ix,iy", [(1, 0), (0, 1), (3, 5), (8, 8)])
def test_wgrad(n, cin, cout, ix, iy):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.randn((n ** 3, cin), generator=g, device="cuda").bfloat16()
    dy = torch.randn((n ** 3, cout), generator=g, device="cuda").bfloat16()
    out = []
    for a, b in ((x, dy), (shifted(x, ix), shifted(dy, iy))):
        dw, db = torch.empty((27, cout, cin), device="cuda"), torch.empty(cout, device="cuda")
        partial = torch.empty(Q.qpat_conv3d_bf16_wgrad_scratch(n, cin, cout), device="cuda")
        Q.qpat_conv3d_bf16_wgrad_dev(a, b, n, dw, db, partial)
        torch.cuda.synchronize()
        out.append((dw, db))
    assert torch.equal(out[0][0], out[1][0])
    assert torch.equal(out[0][1], out[1][1])
