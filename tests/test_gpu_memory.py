"""A call that runs out of device memory reports it and leaves nothing behind: the next
call does not find the CUDA runtime's last error and take it for its own."""
import numpy as np
import pytest

from paper_2506_03617_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 1024 * 1024
VEC = N * 16                                 # one complex128 vector, eight 2 MB pages


@pytest.fixture(scope="module")
def native():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_03617_gb300 import native as M
    M.load()
    return M


def _problem(native):
    g = I.Grid(2, (992, 992), 16)
    p = I.paper_params(g, I.homogeneous(g), ppw=10.0)
    P = native.Problem.from_grid(g, I.homogeneous(g), p)
    P.set_params(prec="c128", exp_tol=1e-3, theta_max=6.0, t=0.05 * p.t)
    return P


def _free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def test_out_of_memory_is_reported_once(native):
    x = torch.from_numpy(I.random_complex(N, 1)).cuda()
    y = torch.empty_like(x)
    ref = _problem(native).apply_phi(0, x)[0].clone()
    P = _problem(native)
    op = P.apply_operator(x)
    filler = torch.empty(_free() - 3 * VEC, dtype=torch.uint8, device="cuda")
    with pytest.raises(native.MxpError) as e:
        P.apply_phi(0, x, out=y)             # seven vectors
    assert e.value.status == 2               # MXP_ENOMEM
    P.apply_operator(x, out=y)
    with pytest.raises(native.MxpError) as e:
        native.Cnn(64, 256, 256)
    assert e.value.status == 2
    P.apply_operator(x, out=y)
    torch.cuda.synchronize()
    del filler
    torch.cuda.empty_cache()
    assert torch.equal(y, op)
    assert float((P.apply_phi(0, x, out=y)[0] - ref).abs().max()) <= 1e-13 * float(ref.abs().max())
    assert native.Cnn(1, 16, 16).num_params > 0
    torch.cuda.synchronize()
