"""The tiled tensor-core convolutions (at most 64 channels on both sides) at the
edges of their tiles: widths around the 32- and 64-pixel tiles, odd heights and
widths (scalar loads, ragged last tiles), channel counts around the 16-channel
stages and the N tiles of 16, 32 and 64, more tiles than SMs, and the general form
(more than 64 input channels).

Against the fp64 oracle with the same bfloat16 operands the only difference is
float32 accumulation (1e-5 of max|ref|).  Against the general form, reached with a
65th channel of zeros, the forward pass and the input gradient are equal to
the last bit: both accumulate the same products in the same order."""
import numpy as np
import pytest

from oracle import cnn as C

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-5


@pytest.fixture(scope="module")
def native():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_03617_gb300 import native as N
    N.load()
    return N


def _maxrel(a, b):
    return float(np.max(np.abs(a - b)) / np.max(np.abs(b)))


# (Cin, Cout, stride, upsample, N, H, W)
EDGES = [(1, 1, 1, 0, 1, 1, 1), (16, 16, 1, 0, 1, 3, 31), (17, 33, 1, 0, 1, 5, 64), (64, 64, 1, 0, 1, 9, 65),
         (63, 2, 1, 0, 2, 4, 96), (64, 64, 1, 0, 2, 6, 130), (15, 48, 2, 0, 1, 8, 66), (33, 64, 2, 0, 2, 6, 128),
         (64, 17, 2, 0, 1, 14, 126), (20, 32, 1, 1, 1, 3, 17), (64, 32, 1, 1, 2, 5, 32), (48, 64, 1, 1, 1, 2, 65),
         (4, 8, 1, 0, 40, 18, 64), (80, 24, 1, 0, 1, 6, 20), (70, 64, 2, 0, 1, 6, 20), (65, 5, 1, 1, 1, 4, 10)]


def _data(Cin, Cout, N, H, W, seed):
    rng = np.random.default_rng(seed)
    x = rng.standard_normal((N, Cin, H, W)).astype(np.float32)
    wb = torch.from_numpy((rng.standard_normal((Cout, Cin, 3, 3)) / np.sqrt(9 * Cin)).astype(np.float32)).to(
        torch.bfloat16)
    return x, wb, rng.standard_normal(Cout).astype(np.float32), rng


@pytest.mark.parametrize("shape", EDGES, ids=[str(s) for s in EDGES])
def test_against_the_oracle(native, shape):
    Cin, Cout, S, U, N, H, W = shape
    x, wb, bias, rng = _data(Cin, Cout, N, H, W, 11)
    W64 = wb.to(torch.float64).numpy()
    xd = torch.from_numpy(x).cuda()
    y = native.conv3x3(0, xd, wb.cuda(), bias=torch.from_numpy(bias).cuda(), stride=S, upsample=U).cpu().numpy()
    xin = C.up2(x.astype(np.float64)) if U else x.astype(np.float64)
    ref = C.conv(C.round_bf16(xin), W64, bias.astype(np.float64), stride=S)
    assert _maxrel(y, ref) < TOL
    g = rng.standard_normal(ref.shape).astype(np.float32)
    gd = torch.from_numpy(g).cuda()
    gref, wref, _ = C.conv_backward(xin, W64, g.astype(np.float64), stride=S, round_operands=True)
    gw = native.conv3x3(2, xd, b=gd, stride=S, upsample=U, cout=Cout).cpu().numpy()
    assert _maxrel(gw, wref.reshape(Cout, Cin * 9)) < TOL
    if not U and Cin <= 64:
        gin = native.conv3x3(1, gd, wb.cuda(), stride=S, in_hw=(H, W)).cpu().numpy()
        assert _maxrel(gin, gref) < TOL


@pytest.mark.parametrize("S,U,H,W", [(1, 0, 6, 70), (2, 0, 9, 70), (1, 1, 4, 33), (1, 0, 8, 32)])
def test_equal_to_the_general_form(native, S, U, H, W):
    x, wb, bias, rng = _data(64, 48, 2, H, W, 12)
    xd, wd, bd = torch.from_numpy(x).cuda(), wb.cuda(), torch.from_numpy(bias).cuda()
    pad = lambda t, dim: torch.cat([t, torch.zeros_like(t.narrow(dim, 0, 1))], dim).contiguous()  # noqa: E731
    y = native.conv3x3(0, xd, wd, bias=bd, stride=S, upsample=U, relu=True)
    y65 = native.conv3x3(0, pad(xd, 1), pad(wd, 1), bias=bd, stride=S, upsample=U, relu=True)
    assert torch.equal(y, y65)
    if not U:
        wg = torch.from_numpy((rng.standard_normal((64, 48, 3, 3)) / 20).astype(np.float32)).to(torch.bfloat16).cuda()
        g = torch.from_numpy(rng.standard_normal((2, 64, -(-H // S), -(-W // S))).astype(np.float32)).cuda()
        a = native.conv3x3(1, g, wg, stride=S, in_hw=(H, W))
        b = native.conv3x3(1, pad(g, 1), pad(wg, 0), stride=S, in_hw=(H, W))
        assert torch.equal(a, b)
