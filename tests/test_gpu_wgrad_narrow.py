"""Weight gradient of layers with 3 or 4 input channels, or one output channel, at widths and
heights that are not multiples of its 64 x 8 tiles (and smaller than one), against the
oracle; and the general kernel, which takes the same layer from an unaligned input.

Tolerance: FP32 sums of at most 64 pixels a row and tile, a few tiles per warp, eight warps
and 608 partial sums, so fewer than 1000 additions in a chain: 1000 x 2^-24 = 6e-5 of the
sum of magnitudes."""
import numpy as np
import pytest

from test_gpu_cnn import G, bf16, pad_ch  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("cin,cin_p,cout,cout_p", [(3, 4, 32, 32), (4, 4, 5, 8), (32, 32, 1, 4), (20, 32, 1, 8), (4, 8, 1, 4),
                                                   (2, 4, 32, 32)])
@pytest.mark.parametrize("B,H,W", [(1, 3, 5), (2, 37, 70), (1, 8, 64), (3, 65, 130)])
@pytest.mark.parametrize("shift", [0, 1])
def test_narrow_weight_gradient(G, cin, cin_p, cout, cout_p, B, H, W, shift):  # noqa: F811
    from oracle import cnn
    lib = G._lib()
    rng = np.random.default_rng(B * H * W + cin)
    xr, xd = bf16(pad_ch(rng.normal(size=(B, H, W, cin)), cin_p))
    # shift: the input starts two bytes past an aligned address
    buf = torch.zeros(xd.numel() + 8, dtype=torch.bfloat16, device="cuda")
    xs = buf[shift:shift + xd.numel()]
    xs.copy_(xd.reshape(-1))
    dz = pad_ch(rng.normal(size=(B, H, W, cout)), cout_p).astype(np.float32)
    dzd = torch.from_numpy(dz).cuda()
    dw = torch.empty(9 * cin * cout, dtype=torch.float32, device="cuda")
    db = torch.empty(cout, dtype=torch.float32, device="cuda")
    scratch = torch.empty(int(lib.mpfc_cnn_wgrad_scratch_bytes(B, H, W)), dtype=torch.uint8, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    assert lib.mpfc_cnn_conv_backward_weight(xs.data_ptr(), B, H, W, cin, cin_p, dzd.data_ptr(), cout, cout_p,
                                             dw.data_ptr(), db.data_ptr(), scratch.data_ptr(), s) == 0
    torch.cuda.synchronize()
    d64 = dz[..., :cout].astype(np.float64)
    gw, gb = cnn.conv3x3_grad_weight(xr[..., :cin], d64)
    aw, ab = cnn.conv3x3_grad_weight(np.abs(xr[..., :cin]), np.abs(d64))
    assert np.all(np.abs(dw.cpu().numpy().reshape(9, cin, cout) - gw) <= 6e-5 * aw)
    assert np.all(np.abs(db.cpu().numpy() - gb) <= 6e-5 * ab)
