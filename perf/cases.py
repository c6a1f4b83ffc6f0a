"""The calls that a user of this library times: sizes, inputs, one pass, its work
and its result in 64 bits.

``listed()`` holds the named cases, ``draw()`` more of the same ranges.  A case
is a dict of plain values; ``prepare`` builds the problem (or the network) and
its inputs on the GPU, ``run`` makes one pass through the public entry points
and ``exact`` computes the same outputs with plain torch in 64 bits.

Low-precision 2D problems name the kernel configuration (``persist_cfg`` or
``tile_cfg``): the autotuner times its candidates, so two processes may settle
on configurations with another Taylor degree, whose results differ by more than
rounding.  The configurations named here are the ones it settles on.
"""
import math

import numpy as np
import torch

from paper_2506_03617_gb300 import inputs as I
from paper_2506_03617_gb300 import native as N

DEV = "cuda:0"


# ------------------------------------------------------------------ the cases

def _case(kind, **kw):
    c = dict(kind=kind, dim=2, nx=128, ny=128, nz=1, npml=16, medium="layered", ppw=8.0, prec="c64",
             exp_tol=1e-6, theta=0.0, which=0, inner_fixed=0, persist_cfg=-1, tile_cfg=-1, batch=1, faces=False)
    c.update(kw)
    return c


def listed():
    return [
        # the residual check of a small problem: one operator apply, launch latency only
        _case("operator", name="operator_c128_160", medium="homogeneous", ppw=10.0, prec="c128"),
        # the FP64 action in parity mode on the smallest configuration (128^2 + 16 PML)
        _case("phi", name="exp_c128_160", medium="homogeneous", ppw=10.0, prec="c128", exp_tol=1e-12),
        # the FP64 action on the 1024^2 layered medium, the plain path every faster one is judged by
        _case("phi", name="exp_c128_1088", nx=1024, ny=1024, npml=32, prec="c128", exp_tol=1e-3, theta=6.0),
        # psi_1 in FP64 on a 3D lens
        _case("phi", name="psi1_c128_3d_128", dim=3, nx=96, ny=96, nz=96, medium="lens", ppw=10.0, prec="c128",
              exp_tol=1e-3, theta=6.0, which=1),
        # the preconditioner of the headline solve: Algorithm 1 in complex64 on the 1024^2 layered medium
        _case("matexpre", name="matexpre_c64_1088", nx=1024, ny=1024, npml=32, exp_tol=1e-3, theta=6.0,
              persist_cfg=10),
        # mixed boundary conditions, no PML, a ragged wide grid (the Marmousi-shaped case)
        _case("phi", name="exp_c64_faces_1700x350", nx=1700, ny=350, npml=0, medium="marmousi", ppw=10.0,
              faces=True, persist_cfg=8),
        # psi_1 with bfloat16 storage on a medium-sized grid
        _case("phi", name="psi1_bf16s_544", nx=512, ny=512, prec="bf16s", exp_tol=1e-3, theta=4.0, which=1,
              persist_cfg=10),
        # the 3D action of the 256^3 configuration, larger than the L2 cache
        _case("phi", name="exp_c64_3d_288", dim=3, nx=256, ny=256, nz=256, medium="homogeneous", ppw=10.0,
              exp_tol=1e-3, theta=6.0),
        # Algorithm 1 on a 3D grid whose sides are no multiples of anything
        _case("matexpre", name="matexpre_c64_3d_odd", dim=3, nx=97, ny=70, nz=83, medium="lens", ppw=10.0,
              inner_fixed=3),
        # several sources on media of two sizes, solved in one call
        _case("batch", name="batch_c64_288_544", nx=256, ny=512, batch=3, tile_cfg=7),
        # the learned stage's training: forward and parameter gradient of a batch of crops
        _case("cnn_train", name="cnn_train_32x64", nx=64, ny=64, batch=32),
        # the learned stage inside a solve: one forward pass over the whole 1088^2 grid
        _case("cnn_forward", name="cnn_forward_1088", nx=1088, ny=1088),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["operator", "phi2", "phi2", "phi3", "phi3", "matexpre2", "matexpre3", "cnn_train",
                       "cnn_forward"])
    if kind == "operator":
        if rng.random() < 0.5:
            return _case("operator", nx=_log_int(rng, 64, 2048), ny=_log_int(rng, 64, 2048), prec="c128",
                         npml=rng.choice([0, 16, 32]))
        return _case("operator", dim=3, nx=_log_int(rng, 32, 256), ny=_log_int(rng, 32, 256),
                     nz=_log_int(rng, 32, 256), medium="lens", ppw=10.0, prec="c128")
    if kind == "phi2":
        prec = rng.choice(["c128", "c64", "bf16s"])
        hi = 512 if prec == "c128" else 960
        which = rng.choice([0, 0, 1] if prec != "c128" else [0, 1, 2])
        return _case("phi", nx=_log_int(rng, 64, hi), ny=_log_int(rng, 64, hi), prec=prec, which=which,
                     npml=rng.choice([16, 17, 32]), exp_tol=1e-12 if prec == "c128" else 1e-6,
                     persist_cfg=-1 if prec == "c128" else 10)
    if kind == "phi3":
        prec = rng.choice(["c128", "c64", "c64", "bf16s"])
        hi = 80 if prec == "c128" else 160
        return _case("phi", dim=3, nx=_log_int(rng, 24, hi), ny=_log_int(rng, 24, hi), nz=_log_int(rng, 24, hi),
                     medium=rng.choice(["homogeneous", "lens"]), ppw=10.0, prec=prec,
                     which=rng.choice([0, 0, 1, 2]), npml=rng.choice([12, 16]), exp_tol=1e-3, theta=4.0)
    if kind == "matexpre2":
        return _case("matexpre", nx=_log_int(rng, 96, 640), ny=_log_int(rng, 96, 640), exp_tol=1e-6,
                     npml=rng.choice([16, 32]), persist_cfg=10, inner_fixed=rng.randint(2, 8))
    if kind == "matexpre3":
        return _case("matexpre", dim=3, nx=_log_int(rng, 24, 112), ny=_log_int(rng, 24, 112),
                     nz=_log_int(rng, 24, 112), medium="lens", ppw=10.0, inner_fixed=rng.randint(1, 4))
    if kind == "cnn_train":
        return _case("cnn_train", nx=2 * _log_int(rng, 8, 64), ny=2 * _log_int(rng, 8, 64),
                     batch=_log_int(rng, 1, 32))
    return _case("cnn_forward", nx=2 * _log_int(rng, 16, 544), ny=2 * _log_int(rng, 16, 544))


# ------------------------------------------------------------------ inputs

def _grid(case, n=None):
    ni = (case["nx"], case["ny"], case["nz"])[:case["dim"]] if n is None else (n, n)
    return I.Grid(case["dim"], tuple(int(v) for v in ni), int(case["npml"]))


def _medium(case, grid, seed):
    if case["medium"] == "homogeneous":
        return I.homogeneous(grid)
    if case["medium"] == "lens":
        u = np.random.default_rng(seed).uniform(0.35, 0.65, 3)
        return I.lens(grid, center=tuple(u[d] * grid.ni[d] * grid.h for d in range(grid.dim)))
    if case["medium"] == "marmousi":
        return I.marmousi_like(grid, seed)
    return I.layered_grf(grid, seed)


def _medium_and_params(case, seed, n=None):
    grid = _grid(case, n)
    c = _medium(case, grid, seed)
    return grid, c, I.paper_params(grid, c, ppw=case["ppw"])


def _problem(case, grid, c, p):
    prob = N.Problem(grid.dim, grid.ni, grid.npml, c, grid.h)
    prob.set_params(omega=p.omega, shift_s=p.shift, t=p.t, c_pml=p.cpml, fprtol=p.fprtol, prec=case["prec"],
                    exp_tol=case["exp_tol"], theta_max=case["theta"], persist_cfg=case["persist_cfg"],
                    tile_cfg=case["tile_cfg"], inner_fixed=case["inner_fixed"])
    if case["faces"]:
        prob.set_boundary(I.MARMOUSI_BC)
    return prob


def _wave(grid, p, seed):
    """A unit-norm wave field: a few plane waves at the slowest wavenumber times a
    smooth amplitude, plus a little noise, as the Krylov vectors look."""
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    rng = np.random.default_rng(seed)
    ax = [torch.from_numpy(grid.node_coords(d)).to(DEV) for d in range(grid.dim)]
    view = [x.reshape([-1 if d == a else 1 for a in reversed(range(grid.dim))]) for d, x in enumerate(ax)]
    v = 0.05 * torch.randn(grid.shape, dtype=torch.complex128, device=DEV, generator=gen)
    k = p.omega
    for _ in range(3):
        u = rng.standard_normal(grid.dim)
        u *= k / np.linalg.norm(u)
        phase = sum(float(u[d]) * view[d] for d in range(grid.dim)) + float(rng.uniform(0, 2 * math.pi))
        v += torch.polar(torch.ones_like(phase), phase)
    ctr = rng.uniform(0.2, 0.8, grid.dim)
    r2 = sum((view[d] - float(ctr[d]) * grid.ni[d] * grid.h) ** 2 for d in range(grid.dim))
    v *= torch.exp(-2.0 * r2)
    v = v.reshape(-1)
    return v / torch.linalg.vector_norm(v)


def _source(grid, seed):
    ctr = I.random_centers(grid, 1, seed=seed)[0]
    return torch.from_numpy(I.rhs_from_source(I.gaussian_source(grid, center=ctr)).ravel()).to(DEV)


def _crops(case, seed):
    """Network input (Re r, Im r, c / c_max) and target with r, z of unit mean square."""
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    b, h, w = case["batch"], case["ny"], case["nx"]
    g = I.Grid(2, (w, h), 0)
    c = I.layered_grf(g, seed)
    x = torch.randn((b, 3, h, w), device=DEV, generator=gen)
    s = torch.nn.functional.avg_pool2d(x[:, :2], 3, 1, 1)      # correlated over a few cells, as residuals are
    x[:, :2] = s / s.square().mean().sqrt()
    x[:, 2] = torch.from_numpy((c / c.max()).astype(np.float32)).to(DEV)
    t = torch.nn.functional.avg_pool2d(x[:, :2], 5, 1, 2)
    return x.contiguous(), (t / t.square().mean().sqrt()).contiguous()


def _theta(case, seed):
    theta = I.cnn_initial_params(I.SEED_BASE + 7000 + int(seed) % 1000)
    off = 0                                        # small biases, as after some training
    rng = np.random.default_rng(seed)
    for ci, co, *_ in I.CNN_LAYERS:
        off += ci * co * 9
        theta[off:off + co] = 0.05 * rng.standard_normal(co)
        off += co
    return theta


BATCH_TARGET = 1e-6


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("cnn_train", "cnn_forward"):
        x, t = _crops(case, seed)
        net = N.Cnn(case["batch"], case["ny"], case["nx"])
        net.set_params(_theta(case, seed))
        return dict(kind=kind, net=net, x=x, t=t)
    if kind == "batch":
        probs, bs, of = [], [], []
        for q, n in enumerate((case["nx"], case["ny"])):
            grid, c, p = _medium_and_params(case, seed + 17 * q, n)
            probs.append(_problem(case, grid, c, p))
            for s in range(case["batch"]):
                bs.append(_source(grid, 1000 * seed + 10 * q + s))
                of.append(q)
        return dict(kind=kind, probs=probs, bs=bs, of=of)
    grid, c, p = _medium_and_params(case, seed)
    prob = _problem(case, grid, c, p)
    x = _source(grid, seed) if kind == "matexpre" else _wave(grid, p, seed)
    return dict(kind=kind, prob=prob, x=x, which=case["which"])


def run(state):
    kind = state["kind"]
    if kind == "operator":
        return state["prob"].apply_operator(state["x"])
    if kind == "phi":
        return state["prob"].apply_phi(state["which"], state["x"])[0]
    if kind == "matexpre":
        return state["prob"].apply_matexpre(state["x"])[0]
    if kind == "batch":
        xs = [torch.empty_like(b) for b in state["bs"]]
        N.solve_batch(state["probs"], state["of"], state["bs"], xs, rtol=BATCH_TARGET)
        return xs
    net, x, t = state["net"], state["x"], state["t"]
    y = net.forward(x)
    if kind == "cnn_forward":
        return y
    gy = (y - t) * (2.0 / y.numel())               # mean squared error
    return dict(y=y, grad=net.backward(x, gy))


# ------------------------------------------------------------------ work

# sweeps of one action: sub-steps times degree of the Taylor plan for the row-sum
# norm of t (A_s - mu), t = 40 h^2 (2D: about 236 with a PML, 167 without; 3D: 340)
_NORM = {2: 236.0, 3: 340.0}


def _sweeps(case, which):
    theta = case["theta"] or (6.0 if case["prec"] == "c128" else 4.0)
    nu = 167.0 if case["npml"] == 0 else _NORM[case["dim"]]
    S, m = N.taylor_plan(nu, case["exp_tol"] * (0.1 if which else 1.0), theta, 1)
    return S * m


def _unknowns(case, n=None):
    return int(np.prod(_grid(case, n).n))


_INNER = 29        # inner GMRES iterations of an apply at 1088^2 (tolerance 0.08)
_BATCH_ACTIONS = {256: 9 * 9, 512: 11 * 15}        # outer times inner iterations of a source


def work(case):
    kind, dim = case["kind"], case["dim"]
    if kind.startswith("cnn"):
        px = case["batch"] * case["nx"] * case["ny"]
        flops = 0.0
        for l, (ci, co, *_) in enumerate(I.CNN_LAYERS):
            flops += 2.0 * 9 * ci * co * px / (4 if l in (1, 2, 3) else 1)
        if kind == "cnn_forward":
            return dict(bytes=4.0 * 5 * px, flops=flops)
        first = 2.0 * 9 * 3 * 32 * px              # no input gradient of the first layer
        return dict(bytes=4.0 * 9 * px, flops=3.0 * flops - first)
    per = 24.0 if dim == 2 else 32.0               # flops of one interior point update
    if kind == "batch":
        flops = byt = 0.0
        for n in (case["nx"], case["ny"]):
            flops += case["batch"] * _BATCH_ACTIONS.get(n, 120) * _sweeps(case, 0) * _unknowns(case, n) * per
            byt += (case["batch"] * 32.0 + 8.0) * _unknowns(case, n)
        return dict(bytes=byt, flops=flops)
    n = _unknowns(case)
    byt = 40.0 * n                                  # input, output and medium
    if kind == "operator":
        return dict(bytes=byt, flops=per * n)
    if kind == "phi":
        return dict(bytes=byt, flops=per * n * _sweeps(case, case["which"]))
    inner = case["inner_fixed"] or _INNER
    flops = per * n * (_sweeps(case, 1) + inner * _sweeps(case, 0))
    flops += 8.0 * n * inner * (inner + 3)          # Gram-Schmidt: dots and updates
    return dict(bytes=byt, flops=flops)


# ------------------------------------------------------------------ exact values

class _Op:
    """The operator of Eq. helmholtz with the PML of Eq. pml-1d-s in 64 bits."""

    def __init__(self, case, grid, c, p, shifted=True):
        self.grid, dim, h = grid, grid.dim, grid.h
        self.shape = grid.shape
        self.wp, self.wm = [], []
        diag = torch.from_numpy(p.omega ** 2 / c ** 2).to(DEV).to(torch.complex128)
        if shifted:
            diag = diag * complex(1.0, p.shift)
        for d in range(dim):
            x = grid.node_coords(d)
            L, delta = grid.ni[d] * h, grid.npml * h

            def inv(z):
                if grid.npml == 0:
                    return np.ones(len(z), dtype=np.complex128)
                r = (np.maximum(-z, 0.0) + np.maximum(z - L, 0.0)) / delta
                return 1.0 / (1.0 + 1j * p.cpml / (delta * p.omega) * r * r)

            wp = inv(x) * inv(x + 0.5 * h) / h ** 2
            wm = inv(x) * inv(x - 0.5 * h) / h ** 2
            view = [-1 if a == d else 1 for a in reversed(range(dim))]
            wp, wm = (torch.from_numpy(w).to(DEV).reshape(view) for w in (wp, wm))
            diag = diag - (wp + wm)
            self.wp.append(wp)
            self.wm.append(wm)
        if case["faces"]:
            kh = 0.5 * p.omega * h / torch.from_numpy(c).to(DEV)
            ghost = torch.complex(torch.ones_like(kh), kh) / torch.complex(torch.ones_like(kh), -kh)
            for f, bc in enumerate(I.MARMOUSI_BC):
                d, ax = f // 2, dim - 1 - f // 2
                at = 0 if f % 2 == 0 else self.shape[ax] - 1
                w = (self.wm if f % 2 == 0 else self.wp)[d].select(ax, at)
                g = ghost.select(ax, at) if bc == "absorbing" else 1.0
                diag.select(ax, at).add_(w * g)
        self.diag = diag.contiguous()
        self.norm = float((diag.abs() + sum((a.abs() + b.abs()) for a, b in zip(self.wp, self.wm))).max())

    def __call__(self, p):
        out = self.diag * p
        for d in range(self.grid.dim):
            ax = self.grid.dim - 1 - d
            n = self.shape[ax]
            lo, hi = slice(0, n - 1), slice(1, n)

            def cut(t, s):
                return t.narrow(ax, s.start, s.stop - s.start) if t.shape[ax] > 1 else t

            cut(out, lo).addcmul_(cut(self.wp[d], lo), cut(p, hi))
            cut(out, hi).addcmul_(cut(self.wm[d], hi), cut(p, lo))
        return out


def _taylor_action(op, t, which, x):
    """exp(M) x, psi_1(M) x or psi_2(M) x, M = i t A, by Taylor sums over sub-steps
    of norm <= 8 of the matrix augmented by the scalar rows of psi."""
    steps = max(1, math.ceil(t * op.norm / 8.0))
    v = x.reshape(op.shape)
    u = v.clone() if which == 0 else torch.zeros_like(v)
    z = (0.0, 1.0, 0.0)[which]                      # scalar that feeds v into the grid block
    for _ in range(steps):
        term, acc, feed = u, u.clone(), z
        for k in range(1, 200):
            term = op(term).mul_(1j * t / (steps * k))
            if feed:
                term.add_(v, alpha=feed / (steps * k))
            feed = 1.0 / steps if which == 2 and k == 1 else 0.0
            acc.add_(term)
            if k % 8 == 0 and float(term.abs().max()) < 1e-18 * float(acc.abs().max()):
                break
        if which == 2:
            z += 1.0 / steps
        u = acc
    return u.reshape(-1)


def _gmres(apply, rhs, tol, fixed, restart=30, maxit=1000):
    x = torch.zeros_like(rhs)
    beta0 = float(torch.linalg.vector_norm(rhs))
    r, total = rhs, 0
    target = fixed or maxit
    while total < target:
        beta = float(torch.linalg.vector_norm(r))
        V = [r / beta]
        H = np.zeros((restart + 1, restart), dtype=np.complex128)
        est = beta
        for j in range(min(restart, target - total)):
            w = apply(V[j])
            for _ in range(2):
                for i in range(j + 1):
                    h = complex(torch.vdot(V[i], w))
                    H[i, j] += h
                    w = w - h * V[i]
            hn = float(torch.linalg.vector_norm(w))
            H[j + 1, j] = hn
            V.append(w / hn)
            total += 1
            e = np.zeros(j + 2, dtype=np.complex128)
            e[0] = beta
            y = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)[0]
            est = float(np.linalg.norm(e - H[:j + 2, :j + 1] @ y))
            if not fixed and est <= tol * beta0:
                break
        for i, yi in enumerate(y):
            x = x + complex(yi) * V[i]
        if (not fixed and est <= tol * beta0) or total >= target:
            break
        r = rhs - apply(x)
    return x


def _direct(op, b):
    """The solution of the 2D system by block elimination along y."""
    ny, nx = op.shape
    b = b.reshape(ny, nx)
    wpx, wmx = op.wp[0].reshape(-1), op.wm[0].reshape(-1)
    wpy, wmy = op.wp[1].reshape(-1), op.wm[1].reshape(-1)
    line = torch.diag(wpx[:-1], 1) + torch.diag(wmx[1:], -1)
    inv, rhs = [], []
    for j in range(ny):
        a, f = line + torch.diag(op.diag[j]), b[j]
        if j:
            a = a - (wmy[j] * wpy[j - 1]) * inv[-1]
            f = f - wmy[j] * (inv[-1] @ rhs[-1])
        inv.append(torch.linalg.inv(a))
        rhs.append(f)
    x = [None] * ny
    for j in reversed(range(ny)):
        x[j] = inv[j] @ (rhs[j] if j == ny - 1 else rhs[j] - wpy[j] * x[j + 1])
    return torch.stack(x).reshape(-1)


def _net64(case, seed, x):
    """Parameters (weights as the bfloat16 values the network holds) and output in 64 bits."""
    F = torch.nn.functional
    theta = torch.from_numpy(_theta(case, seed)).to(DEV)
    ws, bs, off = [], [], 0
    for ci, co, *_ in I.CNN_LAYERS:
        ws.append(theta[off:off + ci * co * 9].to(torch.bfloat16).double().reshape(co, ci, 3, 3).requires_grad_())
        off += ci * co * 9
        bs.append(theta[off:off + co].double().requires_grad_())
        off += co
    conv = lambda l, v, s=1: F.conv2d(v, ws[l], bs[l], stride=s, padding=1)  # noqa: E731
    a1 = F.relu(conv(0, x.double()))
    a = F.relu(conv(1, a1, 2))
    a = F.relu(conv(3, F.relu(conv(2, a))))
    a = F.relu(conv(4, F.interpolate(a, scale_factor=2, mode="nearest"))) + a1
    return ws, bs, conv(5, a)


def exact(case, seed):
    kind = case["kind"]
    if kind.startswith("cnn"):
        x, t = _crops(case, seed)
        with torch.set_grad_enabled(kind == "cnn_train"):
            ws, bs, y = _net64(case, seed, x)
            if kind == "cnn_forward":
                return y
            loss = (y - t.double()).square().mean()
            grads = torch.autograd.grad(loss, [v for wb in zip(ws, bs) for v in wb])
        return dict(y=y.detach(), grad=torch.cat([g.reshape(-1) for g in grads]))
    if kind == "batch":
        out = []
        for q, n in enumerate((case["nx"], case["ny"])):
            grid, c, p = _medium_and_params(case, seed + 17 * q, n)
            op = _Op(case, grid, c, p, shifted=False)
            out += [_direct(op, _source(grid, 1000 * seed + 10 * q + s)) for s in range(case["batch"])]
        return out
    grid, c, p = _medium_and_params(case, seed)
    if kind == "operator":
        return _Op(case, grid, c, p, shifted=False)(_wave(grid, p, seed).reshape(grid.shape)).reshape(-1)
    op = _Op(case, grid, c, p)
    if kind == "phi":
        return _taylor_action(op, p.t, case["which"], _wave(grid, p, seed))
    rt = _taylor_action(op, p.t, 1, _source(grid, seed))
    return _gmres(lambda v: v - _taylor_action(op, p.t, 0, v), rt, p.fprtol, case["inner_fixed"])
