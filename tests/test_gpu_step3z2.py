"""Two Taylor steps per launch in 3D (complex64, bfloat16 storage): the same values
as single-step launches to the last bit, on grids at the edges of its tiles (28 and
60 columns, 14 rows), of its z segments and of the grid itself, with rows that are no
multiple of 4 (padded buffers), for even and odd Taylor degrees, exp, psi_1 and psi_2.
The single-step sweeps (fuse_k = 1) are checked against the oracle elsewhere."""
import numpy as np
import pytest

from paper_2506_03617_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GRIDS = [((2, 3, 1), 0), ((3, 1, 2), 0), ((4, 14, 5), 0), ((28, 15, 7), 0), ((29, 13, 33), 0), ((20, 6, 4), 4),
         ((49, 10, 9), 4), ((60, 28, 3), 0), ((61, 29, 40), 0), ((1, 4, 5), 1), ((90, 20, 21), 3), ((117, 5, 70), 2)]


@pytest.fixture(scope="module")
def native():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_03617_gb300 import native as N
    N.load()
    return N


@pytest.mark.parametrize("ni,npml", GRIDS, ids=[f"{n}-{p}" for n, p in GRIDS])
@pytest.mark.parametrize("prec", ["c64", "bf16s"])
def test_equal_to_single_steps(native, ni, npml, prec):
    g = I.Grid(3, ni, npml)
    c = 1.0 + np.random.default_rng(5).random(g.shape)
    p = I.paper_params(g, c, ppw=10.0)
    x = torch.from_numpy(I.random_complex(g.n_total, 3)).cuda()
    G = native.Problem.from_grid(g, c, p)
    degrees = set()
    for tol in (1e-2, 1e-3):
        for which in (0, 1, 2):
            out = []
            for fuse in (1, 0):
                # no fused z-marching configuration: the tuner would time it
                G.set_params(prec=prec, exp_tol=tol, theta_max=4.0, fuse_k=fuse, t=p.t * 0.2)
                if G.sweep_kernel() == "fused_3d":
                    pytest.skip("the tuner chose the fused kernel")
                out.append(G.apply_phi(which, x)[0])
                degrees.add(G.plan(which)[2] % 2)
            assert torch.equal(out[0], out[1]), (tol, which, float((out[0] - out[1]).abs().max()))
    assert degrees == {0, 1}
