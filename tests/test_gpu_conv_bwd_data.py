"""The convolutions at the edges of a CTA's share: one item each, grids of two to six rows (every item an edge row),
one-segment grids, uneven shares; and the backward-data entry against the forward on flipped weights, bit for bit."""
import numpy as np
import pytest

from oracle import conv_oracle as CO
from paper_1904_10070_gb300 import vlb
from tests.test_gpu_conv import SHAPES, _dev, _host, _rand, _stream

pytestmark = pytest.mark.gpu

GRIDS = [(2, 128), (2, 256), (2, 25600), (4, 12800), (6, 7808), (152, 128), (154, 256), (304, 384), (1100, 128)]


@pytest.mark.parametrize("H,W", GRIDS)
@pytest.mark.parametrize("cin,cout", SHAPES)
def test_forward_and_backward_data(cin, cout, H, W):
    import torch
    rng = np.random.default_rng(13 * H + W + 7 * cin + cout)
    x, w = _rand(rng, (H, W, cin)), _rand(rng, (cout, 3, 3, cin), 0.1)
    b = rng.normal(size=cout).astype(np.float32).astype(np.float64)
    yf = torch.full((H, W, cout), float("nan"), dtype=torch.float32, device="cuda")
    yb = torch.full((H, W, cout), float("nan"), dtype=torch.bfloat16, device="cuda")
    dw = _dev(w, torch.bfloat16)
    vlb.vlb_conv3x3_fwd(H, W, cin, cout, _dev(x, torch.bfloat16), dw, _dev(b, torch.float32), None, 1, yb, yf, _stream())
    vlb.vlb_conv_status(_stream(), clear=False)
    ref = CO.conv3x3(x, w, b, relu=True)
    bound = 2 * 9 * cin * 2.0 ** -24 * CO.conv3x3(np.abs(x), np.abs(w)) + 2.0 ** -24 * np.abs(b)
    assert np.all(np.abs(_host(yf) - ref) <= bound + 1e-30)
    np.testing.assert_array_equal(_host(yb), CO.bf16_round(_host(yf)))

    dy, act = _dev(_rand(rng, (H, W, cout)), torch.bfloat16), _dev(_rand(rng, (H, W, cin)), torch.bfloat16)
    wf = torch.empty((cin, 3, 3, cout), dtype=torch.bfloat16, device="cuda")
    vlb.vlb_conv3x3_flip(cin, cout, dw, wf, _stream())
    for mask in (None, act):
        dx = torch.full((H, W, cin), float("nan"), dtype=torch.bfloat16, device="cuda")
        want = torch.empty_like(dx)
        vlb.vlb_conv3x3_fwd(H, W, cout, cin, dy, wf, None, mask, 0, want, None, _stream())
        vlb.vlb_conv3x3_bwd_data(H, W, cin, cout, dy, dw, mask, dx, _stream())
        vlb.vlb_conv_status(_stream(), clear=False)
        assert torch.equal(dx, want)


def test_backward_data_refuses_bad_arguments():
    import torch
    t = torch.zeros(64, dtype=torch.bfloat16, device="cuda")
    for H, W, cin, cout in ((3, 128, 64, 64), (2, 100, 64, 64), (2, 128, 32, 64)):
        with pytest.raises(vlb.VlbError):
            vlb.vlb_conv3x3_bwd_data(H, W, cin, cout, t, t, None, t, _stream())
    with pytest.raises(vlb.VlbError):
        vlb.vlb_conv3x3_bwd_data(2, 128, 64, 64, None, t, None, t, _stream())
