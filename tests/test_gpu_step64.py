"""The complex128 sweep at the edges of its warps and bodies: widths around 32,
single rows and planes, no PML and a PML wider than a warp, 3D, faces, and both
scalar forms (sigma imaginary with rho = 1, and general sigma, rho), through
mxp_horner_step against the oracle's operator; and a slab inside the grid, whose
interior starts at a negative local row.

out = rho (y + sigma (A_s - mu) p + gamma v): every value is a sum of at most 20
products of rounding error 1.1e-16 each, with terms at most a few times max|out|,
hence the operator parity bound 1e-13 of max|out|."""
import numpy as np
import pytest

import oracle
from paper_2506_03617_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [((1, 1), 0, None), ((1, 5), 3, None), ((31, 3), 0, None), ((32, 9), 2, None), ((33, 17), 16, None),
         ((20, 40), 33, None), ((95, 6), 0, I.MARMOUSI_BC), ((5, 4, 3), 0, None), ((33, 7, 9), 3, None),
         ((12, 2, 20), 5, None)]


@pytest.fixture(scope="module")
def native():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_03617_gb300 import native as N
    N.load()
    return N


def _setup(ni, npml, bc):
    g = I.Grid(len(ni), ni, npml)
    rng = np.random.default_rng(7)
    c = 1.0 + rng.random(g.shape)
    p = I.paper_params(g, c, ppw=10.0)
    codes = None if bc is None else [I.BC_CODES[b] for b in bc]
    vecs = [I.random_complex(g.n_total, s) for s in (1, 2, 3)]
    return g, c, p, codes, vecs


@pytest.mark.parametrize("ni,npml,bc", CASES, ids=[f"{c[0]}-{c[1]}" for c in CASES])
@pytest.mark.parametrize("prec", ["c128", "c64"])
def test_horner_step(native, ni, npml, bc, prec):
    g, c, p, codes, (x, y, v) = _setup(ni, npml, bc)
    O = oracle.Problem.from_grid(g, c, p, bc=codes)
    G = native.Problem.from_grid(g, c, p)
    if bc:
        G.set_boundary(bc)
    G.set_params(prec=prec)                 # c64: the sweep forms its diagonal per point
    mu = G.plan(0)[0]
    ax = O.apply(x, shifted=True) - mu * x
    xd, yd, vd = (torch.from_numpy(t).cuda() for t in (x, y, v))
    if prec == "c128":
        G.apply_phi(0, xd)                  # makes the scaled diagonal
    h2 = g.h * g.h
    for sigma, gamma, rho, yy, vv in [(0.3j * h2, 0j, 1 + 0j, yd, None), (0.3j * h2, 0.2 - 0.1j, 1 + 0j, yd, vd),
                                      ((0.2 + 0.1j) * h2, 0.4j, 0.6 - 0.8j, yd, vd), (0.5j * h2, 0j, 1 + 0j, None, None),
                                      (0.5j * h2, 1j, 0.8 + 0.6j, None, vd)]:
        out = G.horner_step(sigma, xd, y=yy, v=vv, gamma=gamma, rho=rho).cpu().numpy()
        ref = rho * ((y if yy is not None else 0) + sigma * ax + (gamma * v if vv is not None else 0))
        assert np.max(np.abs(out - ref)) <= 1e-13 * np.max(np.abs(ref))


@pytest.mark.parametrize("ni,npml,bc", CASES, ids=[f"{c[0]}-{c[1]}" for c in CASES])
def test_operator_forms(native, ni, npml, bc):
    """The operator of a complex128 problem and the one beside low-precision actions."""
    g, c, p, codes, (x, _, _) = _setup(ni, npml, bc)
    O = oracle.Problem.from_grid(g, c, p, bc=codes)
    G = native.Problem.from_grid(g, c, p)
    if bc:
        G.set_boundary(bc)
    xd = torch.from_numpy(x).cuda()
    for prec in ("c128", "c64", "bf16s"):
        G.set_params(prec=prec)
        for shifted in (False, True):
            out, ref = G.apply_operator(xd, shifted=shifted).cpu().numpy(), O.apply(x, shifted=shifted)
            assert np.max(np.abs(out - ref)) <= 1e-13 * np.max(np.abs(ref))


@pytest.mark.parametrize("dim", [2, 3])
def test_slab_rows(native, dim):
    ni = (37, 30) if dim == 2 else (9, 8, 26)
    g, c, p, _, (x, y, _) = _setup(ni, 6, None)
    rows, row = g.n[-1], g.n_total // g.n[-1]
    G = native.Problem.from_grid(g, c, p)
    ref = G.horner_step(0.1j * g.h * g.h, torch.from_numpy(x).cuda(), y=torch.from_numpy(y).cuda()).cpu().numpy()
    for r0, r1 in [(0, 9), (3, 20), (14, 25), (20, rows)]:
        S = native.Problem.slab(g, r0, r1 - r0, np.asarray(c).reshape(-1)[r0 * row:r1 * row],
                                (float(c.min()), float(c.max())), p)
        cut = slice(r0 * row, r1 * row)
        out = S.horner_step(0.1j * g.h * g.h, torch.from_numpy(x[cut].copy()).cuda(),
                            y=torch.from_numpy(y[cut].copy()).cuda()).cpu().numpy()
        lo, hi = (0 if r0 == 0 else row), (None if r1 == rows else -row)     # rows whose neighbours the slab holds
        a, b = out[lo:hi], ref[cut][lo:hi]
        assert np.max(np.abs(a - b)) <= 1e-13 * np.max(np.abs(ref))
