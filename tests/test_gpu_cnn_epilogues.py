"""The steps fused into the network's convolutions (skip sum, masks, 2 x 2 pooling of the
upsampled layer's gradient, the skip's gradient, bias gradients) against the same network
put together from the plain convolutions and elementwise operations: forward pass to
the last bit, gradients to the rounding of float32 sums in another order (1e-5 of the
largest entry, as for the plain convolutions).

Shapes: one tile of either width, full-resolution tiles of 32 pixels (32 x 32, 90 x 20)
and of 64, ragged ones, more tiles than SMs, and the smallest grid."""
import numpy as np
import pytest

from paper_2506_03617_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [(1, 2, 2), (2, 32, 32), (1, 90, 20), (3, 30, 34), (2, 16, 64), (40, 18, 96), (9, 66, 70)]


def _layers(theta):
    out, off = [], 0
    for ci, co, *_ in I.CNN_LAYERS:
        w = theta[off:off + ci * co * 9].to(torch.bfloat16).reshape(co, ci, 3, 3).contiguous()
        off += ci * co * 9
        out.append((w, theta[off:off + co].contiguous()))
        off += co
    return out


@pytest.mark.parametrize("shape", SHAPES, ids=[str(s) for s in SHAPES])
def test_network_equals_its_plain_parts(shape):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_03617_gb300 import native as N
    n, h, w = shape
    rng = np.random.default_rng(4)
    theta = I.cnn_initial_params(9).astype(np.float32)
    theta += (0.02 * rng.standard_normal(theta.size)).astype(np.float32)          # biases too
    net = N.Cnn(n, h, w)
    net.set_params(theta)
    x = torch.from_numpy(rng.standard_normal((n, 3, h, w)).astype(np.float32)).cuda()
    gy = torch.from_numpy(rng.standard_normal((n, 2, h, w)).astype(np.float32)).cuda()
    L = _layers(torch.from_numpy(theta).cuda())

    def fwd(l, v, stride=1, up=False, relu=True):
        return N.conv3x3(0, v, L[l][0], bias=L[l][1], stride=stride, upsample=up, relu=relu)

    a1 = fwd(0, x)
    a2 = fwd(1, a1, stride=2)
    a3 = fwd(2, a2)
    a4 = fwd(3, a3)
    r5 = fwd(4, a4, up=True)
    a5 = r5 + a1
    assert torch.equal(net.forward(x), fwd(5, a5, relu=False))

    def bwd(l, g, stride=1, hw=None):
        return N.conv3x3(1, g.contiguous(), L[l][0], stride=stride, in_hw=hw)

    def masked(g, a):
        return torch.where(a > 0, g, torch.zeros_like(g))

    g1 = bwd(5, gy)
    g5 = masked(g1, r5)
    up = bwd(4, g5)
    pooled = ((up[..., 0::2, 0::2] + up[..., 0::2, 1::2]) + up[..., 1::2, 0::2]) + up[..., 1::2, 1::2]
    g4 = masked(pooled, a4)
    g3 = masked(bwd(3, g4), a3)
    g2 = masked(bwd(2, g3), a2)
    g0 = masked(bwd(1, g2, stride=2, hw=(h, w)) + g1, a1)
    parts = [(x, g0, 1, False), (a1, g2, 2, False), (a2, g3, 1, False), (a3, g4, 1, False), (a4, g5, 1, True),
             (a5, gy, 1, False)]
    grad, off = net.backward(x, gy), 0
    for (ci, co, *_), (inp, g, stride, ups) in zip(I.CNN_LAYERS, parts):
        gw = N.conv3x3(2, inp.contiguous(), b=g.contiguous(), stride=stride, upsample=ups, cout=co).reshape(-1)
        got = grad[off:off + gw.numel()]
        assert float((got - gw).abs().max()) <= 1e-5 * float(gw.abs().max())
        off += gw.numel()
        ref = g.double().sum(dim=(0, 2, 3))
        scale = float(g.double().abs().sum(dim=(0, 2, 3)).max())
        assert float((grad[off:off + co].double() - ref).abs().max()) <= 1e-6 * scale
        off += co
    assert off == grad.numel()
