"""The bias gradients of the learned stage are summed in a fixed order: the same inputs
give the same bits, on a grid of many tiles per CTA and on one with fewer tiles than
SMs.  (The weight gradients are added by atomics and agree to float32 rounding.)"""
import numpy as np
import pytest

from paper_2506_03617_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(8, 64, 96), (1, 16, 32), (3, 30, 34)])
def test_bias_gradients_repeat_bit_for_bit(shape):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_03617_gb300 import native as N
    n, h, w = shape
    net = N.Cnn(n, h, w)
    net.set_params(I.cnn_initial_params(5))
    rng = np.random.default_rng(2)
    x = torch.from_numpy(rng.standard_normal((n, 3, h, w)).astype(np.float32)).cuda()
    gy = torch.from_numpy(rng.standard_normal((n, 2, h, w)).astype(np.float32)).cuda()
    net.forward(x)
    grads = [net.backward(x, gy) for _ in range(8)]
    off = 0
    for ci, co, *_ in I.CNN_LAYERS:
        wslice, bslice = slice(off, off + ci * co * 9), slice(off + ci * co * 9, off + ci * co * 9 + co)
        off = bslice.stop
        for g in grads[1:]:
            assert torch.equal(g[bslice], grads[0][bslice])
            assert float((g[wslice] - grads[0][wslice]).abs().max()) < 1e-5 * float(grads[0][wslice].abs().max())
    assert off == net.num_params
    # the last layer's bias gradient is the sum of gy: no convolution in between
    ref = gy.double().sum(dim=(0, 2, 3))
    assert float((grads[0][-2:].double() - ref).abs().max()) < 1e-6 * float(gy.double().abs().sum())
