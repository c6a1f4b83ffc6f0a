"""Chained complex128 sweeps: their time grows with the grid.  A sweep that lets the
next ones start before it waits for the one before it fills the SMs with waiting
blocks, and later blocks crowd onto a few of them: 6.3 us a sweep on 224^2 against 3.1
on 144^2, 5.5 on 24^3 against 2.6 on 16^3.  Work grows by 2.5 and 3.4, but at these
sizes a sweep is its launch and one point's latency: evenly placed, the ratios are
1.25 and 1.1.  Bound 1.6: half way to the crowded ones, times of one process."""
import numpy as np
import pytest

from paper_2506_03617_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def native():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_03617_gb300 import native as N
    N.load()
    return N


def _sweep_us(native, n, npml):
    g = I.Grid(len(n), tuple(v - 2 * npml for v in n), npml)
    c = 1.0 + np.random.default_rng(3).random(g.shape)
    P = native.Problem.from_grid(g, c, I.paper_params(g, c, ppw=10.0))
    P.set_params(prec="c128", exp_tol=1e-3, theta_max=6.0)
    x = torch.from_numpy(I.random_complex(g.n_total, 1)).cuda()
    y = P.empty()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = 1e30
    for rep in range(6):
        a.record(P.stream)
        sweeps = P.apply_phi(0, x, out=y)[1]
        b.record(P.stream)
        b.synchronize()
        if rep:
            best = min(best, a.elapsed_time(b) * 1e3 / sweeps)
    return best


@pytest.mark.parametrize("small,large,npml", [((144, 144), (224, 224), 16), ((16, 16, 16), (24, 24, 24), 3)])
def test_sweep_time_grows_with_the_grid(native, small, large, npml):
    t0, t1 = _sweep_us(native, small, npml), _sweep_us(native, large, npml)
    assert t1 < 1.6 * t0, (t0, t1)
