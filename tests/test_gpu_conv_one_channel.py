"""3x3 convolutions of one channel onto more than 32, and the input gradient of the
transposed layer, take the general form: the same bits as the tiled one, which a second
channel of zeros selects (both add the same products in the same order)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("many", [32, 33, 64])
@pytest.mark.parametrize("n,h,w", [(1, 1, 1), (2, 9, 65), (3, 30, 34)])
def test_one_channel_equals_one_and_a_zero_channel(many, n, h, w):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_03617_gb300 import native as N
    rng = np.random.default_rng(7)
    x = torch.from_numpy(rng.standard_normal((n, 1, h, w)).astype(np.float32)).cuda()
    wt = torch.from_numpy((rng.standard_normal((many, 1, 3, 3)) / 3).astype(np.float32)).to(torch.bfloat16).cuda()
    bias = torch.from_numpy(rng.standard_normal(many).astype(np.float32)).cuda()
    zx, zw = torch.cat([x, torch.zeros_like(x)], 1).contiguous(), torch.cat([wt, torch.zeros_like(wt)], 1).contiguous()
    assert torch.equal(N.conv3x3(0, x, wt, bias=bias, relu=True), N.conv3x3(0, zx, zw, bias=bias, relu=True))
    v = wt.transpose(0, 1).contiguous()                      # many input channels, one output
    zv = torch.cat([v, torch.zeros_like(v)], 0).contiguous()
    assert torch.equal(N.conv3x3(1, x, v), N.conv3x3(1, zx, zv))
