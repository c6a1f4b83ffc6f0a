"""Tables that only save time (the scaled diagonal of the complex128 actions, 16 bytes an
unknown) against the problems' vectors: given back where a vector no longer fits, also to
another problem of the same batch, tried again when the parameters change, and not kept
by a problem whose actions don't use them.  The device's memory is filled by an ordinary
allocation that leaves a stated number of vectors free."""
import numpy as np
import pytest

from paper_2506_03617_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NI, NPML = (2016, 2016), 16
VEC = 2048 * 2048 * 16                       # one complex128 vector, 32 2 MB pages


@pytest.fixture(scope="module")
def native():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_03617_gb300 import native as N
    N.load()
    return N


def _problem(native, seed, **kw):
    g = I.Grid(2, NI, NPML)
    c = 1.0 + np.random.default_rng(seed).random(g.shape)
    p = I.paper_params(g, c, ppw=10.0)
    P = native.Problem.from_grid(g, c, p)
    P.set_params(prec="c128", exp_tol=1e-3, theta_max=6.0, t=0.05 * p.t, **kw)
    return P


def _free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def _launches(native, P, x, y):
    n0 = native.kernel_launch_count()
    P.apply_phi(0, x, out=y)
    return native.kernel_launch_count() - n0


class _Filled:
    """Leaves about `vectors` vectors of device memory."""

    def __init__(self, vectors):
        self.left = int(vectors * VEC)

    def __enter__(self):
        self.block = torch.empty(_free() - self.left, dtype=torch.uint8, device="cuda")
        assert abs(_free() - self.left) <= VEC // 4

    def __exit__(self, *exc):
        del self.block
        torch.cuda.empty_cache()


def test_vectors_take_the_tables_memory_and_the_table_comes_back(native):
    x = torch.from_numpy(I.random_complex(VEC // 16, 1)).cuda()
    full = _problem(native, 1)
    ref = full.apply_phi(0, x)[0]
    P, y = _problem(native, 1), torch.empty_like(x)
    plain = _launches(native, full, x, y)    # its table is made: conversions and sweeps
    del full
    with _Filled(7.5):                       # seven vectors, not the diagonal too
        P.apply_phi(0, x, out=y)
        assert torch.cuda.mem_get_info()[0] < VEC
    assert float((y - ref).abs().max()) <= 1e-13 * float(ref.abs().max())
    assert _launches(native, P, x, y) == plain
    P.set_params(exp_tol=1e-3)
    assert _launches(native, P, x, y) == plain + 1           # the table is made again
    assert torch.equal(y, ref)


def test_other_precision_gives_the_table_back(native):
    P = _problem(native, 2)
    x = torch.from_numpy(I.random_complex(VEC // 16, 1)).cuda()
    y = P.apply_phi(0, x)[0]
    before = _free()
    P.set_params(prec="c64", persist_cfg=-2, fuse_k=1)
    assert _free() - before >= 0.9 * VEC
    P.set_params(prec="c128", persist_cfg=-1, fuse_k=0)
    assert torch.equal(P.apply_phi(0, x)[0], y)


def test_a_batch_uses_its_other_problems_tables(native):
    """Vectors of a batch with restart 2 and one source: 4 slots, 3 + 2 + 3 Krylov vectors
    and 2 more, 14 a problem; 7 base vectors.  A has base and table, B nothing yet: 35
    vectors are wanted, 34.5 are free, so B fits only when A's table goes too."""
    # kernels and graphs are loaded before the memory is filled: that takes some too
    g = I.Grid(2, (40, 36), 6)
    w = [native.Problem.from_grid(g, I.homogeneous(g), I.paper_params(g, I.homogeneous(g), ppw=10.0)) for _ in range(2)]
    for P in w:
        P.set_params(prec="c128", exp_tol=1e-3, theta_max=6.0, inner_restart=2, inner_fixed=1)
    s = torch.from_numpy(I.random_complex(g.n_total, 1)).cuda()
    native.solve_batch(w, [0, 1], [s, s.clone()], [torch.zeros_like(s) for _ in range(2)], restart=2, maxit=2)
    A = _problem(native, 3, inner_restart=2, inner_fixed=1)
    x = torch.from_numpy(I.random_complex(VEC // 16, 1)).cuda()
    ref = A.apply_phi(0, x)[0]
    B = _problem(native, 4, inner_restart=2, inner_fixed=1)
    bs = [x.clone(), x.clone()]
    xs = [torch.zeros_like(x) for _ in bs]
    with _Filled(34.5):
        st = native.solve_batch([A, B], [0, 1], bs, xs, restart=2, maxit=1)
    assert all(s["outer_iters"] == 1 for s in st)
    assert all(bool(torch.isfinite(torch.view_as_real(v)).all()) and float(v.abs().max()) > 0 for v in xs)
    y = A.apply_phi(0, x)[0]                 # without its table
    assert float((y - ref).abs().max()) <= 1e-13 * float(ref.abs().max())
