"""The solver's workloads as callable cases: time steps, the preconditioner, the explicit loads, set-up,
the warm-start network and the morphology projection, each through the calls a program makes.

``listed()`` names the cases, ``draw(rng)`` makes one more of the same ranges, ``prepare`` builds what a
program holds before the call (mesh, system, preconditioner, state, network, inputs), ``run`` is one pass
and returns its outputs, ``work`` its unavoidable bytes and flops, and ``exact`` the same outputs in 64
bits from plain torch / numpy where that is affordable.

Inputs.  A time step is called in earnest on a state that earlier steps have smoothed, with chemical
potentials that belong to it.  ``_evolve`` makes such states without the library: the same model
(polynomial potential, Section 4's parameters) advanced from seeded noise by a cosine-spectral
semi-implicit scheme on the nodes of the same box.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2204_03575_gb300 import ch, inputs, warmstart

TAU, EPS, K_EVAP, G_SUB = 1e-4, 1e-3, 5e-3, 0.01  # the paper's values (the library's defaults)
CHI, FH_N, FH_DELTA = (1.0, 0.3, 0.3), (20.0, 20.0, 1.0), 1e-10
SPECTRAL_STEPS = 16
GEOMETRY = ("dim", "nx", "ny", "nz", "Lx", "Ly", "Lz")


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # one time step of the plain FP64 form on the smallest configuration (1089 nodes): latency and launches
        dict(name="step_2d_32_fp64", kind="step", dim=2, nx=32, ny=32, Lx=1.0, Ly=1.0, base=0.33, precision=0, krylov=0),
        # the headline workload, FP64 throughout and with FP32 V-cycles
        dict(name="step_2d_512_fp64", kind="step", dim=2, nx=512, ny=512, Lx=1.0, Ly=1.0, base=0.33, precision=0,
             krylov=0),
        dict(name="step_2d_512_mixed", kind="step", dim=2, nx=512, ny=512, Lx=1.0, Ly=1.0, base=0.33, precision=1,
             krylov=0),
        # the 3D film: Kuhn tetrahedra, FP32 V-cycles
        dict(name="step_3d_128x128x32_mixed", kind="step", dim=3, nx=128, ny=128, nz=32, Lx=1.0, Ly=1.0, Lz=0.25,
             base=0.30, precision=1, krylov=0),
        # the paper's 800 x 400 point grid on its 10 x 2.5 box with its Krylov method
        dict(name="step_2d_799x399_minres", kind="step", dim=2, nx=799, ny=399, Lx=10.0, Ly=2.5, base=0.35, precision=0,
             krylov=1),
        # 64 independent runs of uneven sizes advanced together
        dict(name="batch_64_mixed", kind="batch", runs=64, spec=0, precision=1),
        # a step from the warm-start network's prediction
        dict(name="guess_2d_256_mixed", kind="guess", nx=256, ny=256, precision=1),
        # loss and gradients of the warm-start network on one training batch
        dict(name="train_256_batch8", kind="train", nx=256, ny=256, batch=8),
        # Algorithm 1 alone (one application), FP64, on a 3D box of odd sizes
        dict(name="apply_3d_63x47x41_fp64", kind="apply", dim=3, nx=63, ny=47, nz=41, Lx=1.0, Ly=1.0, Lz=0.5, base=0.30),
        # right-hand sides with the Flory-Huggins potential, 3D
        dict(name="rhs_3d_128x128x32_fh", kind="rhs", dim=3, nx=128, ny=128, nz=32, Lx=1.0, Ly=1.0, Lz=0.25, base=0.30,
             potential=3),
        # mesh, system and preconditioner of a new parameter set (sweeps over tau and eps rebuild them), and the
        # preconditioner's first application
        dict(name="setup_2d_256_fp64", kind="setup", dim=2, nx=256, ny=256, Lx=1.0, Ly=1.0),
        # a morphology handed to a finite-difference device grid
        dict(name="project_512_to_1024", kind="project", nx=512, ny=512, gx=1024, gy=1024),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _box(rng, dim, lo, hi, nodes):
    """Cells of a box whose node count stays within `nodes`, sides spread over [lo, hi] by logarithm."""
    while True:
        n = [_log_int(rng, lo, hi) for _ in range(dim)]
        if math.prod(c + 1 for c in n) <= nodes:
            break
    if dim == 2:
        lx, ly = rng.choice([(1.0, 1.0), (10.0, 2.5)])
        return dict(dim=2, nx=n[0], ny=n[1], Lx=lx, Ly=ly)
    return dict(dim=3, nx=n[0], ny=n[1], nz=n[2], Lx=1.0, Ly=1.0, Lz=rng.choice([0.25, 0.5]))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "batch", "guess", "train", "apply", "rhs", "setup", "project"])
    base = round(rng.uniform(0.28, 0.36), 3)
    if kind == "step":
        dim = rng.choice([2, 2, 3])
        box = _box(rng, 2, 24, 800, 270_000) if dim == 2 else _box(rng, 3, 8, 128, 300_000)
        return dict(kind=kind, **box, base=base, precision=rng.choice([0, 1]), krylov=rng.choice([0, 0, 0, 1]))
    if kind == "batch":
        return dict(kind=kind, runs=_log_int(rng, 3, 64), spec=rng.randrange(1, 1 << 20), precision=rng.choice([0, 1, 1]))
    if kind == "guess":
        return dict(kind=kind, nx=_log_int(rng, 48, 256), ny=_log_int(rng, 48, 256), precision=rng.choice([0, 1]))
    if kind == "train":
        return dict(kind=kind, nx=_log_int(rng, 48, 256), ny=_log_int(rng, 48, 256), batch=rng.randint(1, 8))
    if kind == "apply":
        dim = rng.choice([2, 3])
        box = _box(rng, 2, 48, 800, 270_000) if dim == 2 else _box(rng, 3, 12, 80, 200_000)
        return dict(kind=kind, **box, base=base)
    if kind == "rhs":
        dim = rng.choice([2, 3])
        box = _box(rng, 2, 24, 800, 270_000) if dim == 2 else _box(rng, 3, 8, 128, 540_000)
        return dict(kind=kind, **box, base=base, potential=rng.choice([0, 3]))
    if kind == "setup":
        dim = rng.choice([2, 3])
        box = _box(rng, 2, 32, 400, 66_000) if dim == 2 else _box(rng, 3, 8, 48, 40_000)
        return dict(kind=kind, **box)
    return dict(kind=kind, nx=_log_int(rng, 32, 512), ny=_log_int(rng, 32, 512), gx=_log_int(rng, 32, 1024),
                gy=_log_int(rng, 32, 1024))


# ---------------------------------------------------------------- inputs
def _uniform(seed, stream, shape):
    g = torch.Generator(device="cuda").manual_seed((int(seed) * 64 + stream) & 0x7FFFFFFF)
    return torch.rand(shape, dtype=torch.float64, device="cuda", generator=g)


def _mirror(u):
    """The even extension of a nodal field along every axis (n + 1 points -> 2 n)."""
    for ax in range(u.dim()):
        n = u.shape[ax] - 1
        u = torch.cat([u, u.narrow(ax, 1, n - 1).flip(ax)], ax)
    return u


def _evolve(cells, lengths, base_p, base_n, seed, stream=0, keep=1):
    """The last `keep` states (N x 4: phi_p, phi_nfa, mu_p, mu_nfa, x fastest) of SPECTRAL_STEPS
    semi-implicit steps from base +/- 0.01 noise, zero flux."""
    cells, lengths = list(reversed(cells)), list(reversed(lengths))
    shape = [c + 1 for c in cells]
    k2 = 0.0
    for ax, (c, length) in enumerate(zip(cells, lengths)):
        f = torch.fft.rfftfreq(2 * c, 1.0 / (2 * c)) if ax == len(cells) - 1 else torch.fft.fftfreq(2 * c, 1.0 / (2 * c))
        k = (f.to(device="cuda", dtype=torch.float64) * (math.pi / length)) ** 2
        k2 = k2 + k.reshape([-1 if a == ax else 1 for a in range(len(cells))])
    full = [2 * c for c in cells]
    inner = tuple(slice(0, s) for s in shape)
    p = base_p + 0.01 * (2 * _uniform(seed, 2 * stream, shape) - 1)
    n = base_n + 0.01 * (2 * _uniform(seed, 2 * stream + 1, shape) - 1)
    out = []
    for step in range(SPECTRAL_STEPS):
        s = 1.0 - p - n
        fields, mus = [], []
        for u, f in ((p, 7 * p * n * n - 0.2 * s), (n, 7 * n * p * p - 0.2 * s)):
            fh = torch.fft.rfftn(_mirror(f))
            uh = (torch.fft.rfftn(_mirror(u)) - TAU * k2 * fh) / (1 + TAU * EPS * k2 * k2)
            fields.append(torch.fft.irfftn(uh, s=full)[inner])
            mus.append(torch.fft.irfftn(fh + EPS * k2 * uh, s=full)[inner])
        p, n = fields
        if step >= SPECTRAL_STEPS - keep:
            out.append(torch.stack([t.reshape(-1) for t in (p, n, *mus)], 1).contiguous())
    return out


def _columns(state):
    return [state[:, c].contiguous() for c in range(4)]


def _params(case, **kw):
    geo = {k: case[k] for k in GEOMETRY if k in case}
    return ch.Params(**geo, **kw)


def _cells(case):
    d = case.get("dim", 2)
    return [case[k] for k in ("nx", "ny", "nz")[:d]], [case.get(k, 1.0) for k in ("Lx", "Ly", "Lz")[:d]]


def prepare(case, seed):
    kind = case["kind"]
    cells, lengths = _cells(case) if kind != "batch" else (None, None)
    if kind == "step":
        kw = dict(precision=case["precision"], krylov=case["krylov"])
        if case["krylov"]:
            kw["rtol"] = 1e-7  # the paper's tolerance for its method
        p = _params(case, **kw)
        system = ch.System(ch.Mesh(p), p)
        state = ch.State(system, ch.Precond(system))
        (x,) = _evolve(cells, lengths, case["base"], case["base"], seed)
        return dict(case=case, state=state, x=_columns(x))
    if kind == "batch":
        spec = inputs.batch_runs(case["runs"], seed=case["spec"])
        p = ch.Params(precision=case["precision"])
        system = ch.System(ch.Mesh(p, runs=[ch.Params(nx=nx, ny=ny) for nx, ny, _, _ in spec]), p)
        state = ch.State(system, ch.Precond(system))
        x = torch.cat([_evolve((nx, ny), (1.0, 1.0), bp, bn, seed, stream=r)[0]
                       for r, (nx, ny, bp, bn) in enumerate(spec)])
        return dict(case=case, state=state, x=_columns(x))
    if kind in ("guess", "train"):
        nx, ny = case["nx"], case["ny"]
        if kind == "guess":
            state = warmstart.make_state(nx, ny, case["precision"])
            q2, q, s = _evolve(cells, lengths, 0.33, 0.31, seed, keep=3)
            net = ch.WarmStartNet(ny + 1, nx + 1, 1)
            net.fit_norm(s.unsqueeze(0))
            net.set_params(warmstart.init_params(net.nparams, seed & 0xFFFF))
            return dict(case=case, state=state, net=net, s=s, q=q, q2=q2, x=_columns(s))
        system = warmstart.make_system(nx, ny)
        hist = [_evolve(cells, lengths, 0.25 + 0.02 * b, 0.40 - 0.015 * b, seed, stream=b, keep=3)
                for b in range(case["batch"])]
        q2, q, s = (torch.stack(t).contiguous() for t in zip(*hist))
        net = ch.WarmStartNet(ny + 1, nx + 1, case["batch"])
        net.fit_norm(s)
        net.set_params(warmstart.init_params(net.nparams, seed & 0xFFFF))
        return dict(case=case, system=system, net=net, s=s, q=q, q2=q2)
    if kind == "apply":
        p = _params(case)
        system = ch.System(ch.Mesh(p), p)
        # what the Krylov method hands the preconditioner: a residual-like vector, rough and zero-mean
        (x,) = _evolve(cells, lengths, case["base"], case["base"], seed)
        v = (x - x.mean(0)) / x.std(0) + 0.3 * (2 * _uniform(seed, 9, tuple(x.shape)) - 1)
        return dict(case=case, pc=ch.Precond(system), v=(v / v.norm()).contiguous())
    if kind == "rhs":
        p = _params(case, potential=case["potential"])
        (x,) = _evolve(cells, lengths, case["base"], case["base"], seed)
        return dict(case=case, system=ch.System(ch.Mesh(p), p), x=_columns(x)[:2])
    if kind == "setup":
        # a sweep's parameter set: tau and eps around the paper's values
        u = _uniform(seed, 0, (2,)).tolist()
        n = math.prod(c + 1 for c in cells)
        return dict(case=case, tau=TAU * 10 ** (u[0] - 0.5), eps=EPS * 10 ** (u[1] - 0.5),
                    v=2 * _uniform(seed, 1, (n, 4)) - 1)
    if kind == "project":
        (x,) = _evolve(cells, lengths, 0.33, 0.33, seed)
        return dict(case=case, x=_columns(x)[:2])
    raise ValueError(kind)


# ---------------------------------------------------------------- one pass
def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind in ("step", "batch"):
        st["state"].set(*st["x"])
        st["state"].step()
        return st["state"].get()
    if kind == "guess":
        pred = st["net"].predict(st["s"], st["q"], st["q2"])
        st["state"].set(*st["x"])
        st["state"].step_guess(pred)
        return dict(st["state"].get(), pred=pred)
    if kind == "train":
        # lr = 0: loss and gradients without the parameter update (the call held-out losses make)
        loss = st["net"].train_residual(st["system"], st["s"], st["q"], st["q2"], 0.0)
        return dict(loss=loss, grads=st["net"].get_params()[1])
    if kind == "apply":
        return st["pc"].apply(st["v"])
    if kind == "rhs":
        return st["system"].rhs(*st["x"])
    if kind == "setup":
        p = _params(case, tau=st["tau"], eps=st["eps"])
        system = ch.System(ch.Mesh(p), p)
        return dict(system=system.csr(), w=ch.Precond(system).apply(st["v"]))
    if kind == "project":
        return ch.morphology_project(*st["x"], case["nx"], case["ny"], 1.0, 1.0, case["gx"], case["gy"])
    raise ValueError(kind)


# ---------------------------------------------------------------- unavoidable work of one pass
def _sizes(dim, cells):
    n = math.prod(c + 1 for c in cells)
    return n, (7 if dim == 2 else 15) * n, (2 if dim == 2 else 6) * math.prod(cells)


def _apply_flops(nnz):
    """Algorithm 1 on both species: four H V-cycles and one M V-cycle with nine and five fine-level
    operator products each (coarser levels add about a fifth), 4 flops per entry."""
    return 1.2 * (4 * 11 + 7) * 4.0 * nnz


def work(case):
    kind = case["kind"]
    if kind == "batch":
        spec = inputs.batch_runs(case["runs"], seed=case["spec"])
        n = sum((nx + 1) * (ny + 1) for nx, ny, _, _ in spec)
        nnz = 7 * n
    else:
        cells, _ = _cells(case)
        n, nnz, elems = _sizes(case.get("dim", 2), cells)
    if kind in ("step", "batch", "guess"):
        its = 10 if kind != "guess" else 7
        net = 9 * 2.0 * (16 * 32 + 32 * 32 + 32 * 8) * n if kind == "guess" else 0.0
        # the state in, the fields out; per iteration Algorithm 1, the block operator and Gram-Schmidt
        return dict(bytes=(32.0 + 40.0 + (128.0 if kind == "guess" else 0.0)) * n,
                    flops=net + its * (_apply_flops(nnz) + 16.0 * nnz + 16.0 * its * n))
    if kind == "train":
        b = case["batch"]
        return dict(bytes=96.0 * n * b, flops=3 * 9 * 2.0 * (16 * 32 + 32 * 32 + 32 * 8) * n * b + 48.0 * nnz * b)
    if kind == "apply":
        return dict(bytes=64.0 * n, flops=_apply_flops(nnz))
    if kind == "rhs":
        pts = (27 if case["dim"] == 3 else 9) if case["potential"] == 3 else 4
        return dict(bytes=48.0 * n, flops=elems * pts * 2.0 * (4 * (case["dim"] + 1) + 10) + 4.0 * nnz)
    if kind == "setup":
        # the system's pattern and three value arrays written, both hierarchies' levels about as much again
        return dict(bytes=2.0 * 28.0 * nnz + 64.0 * n, flops=_apply_flops(nnz))
    g = float(case["gx"]) * case["gy"]
    return dict(bytes=16.0 * n + 17.0 * g, flops=0.0)


# ---------------------------------------------------------------- the same outputs in 64 bits
def _mesh64(cells, lengths):
    """Coordinates, simplices and the facets of y = 0 and y = Ly of the uniform mesh."""
    d = len(cells)
    ax = [torch.arange(c + 1, dtype=torch.float64, device="cuda") * (length / c) for c, length in zip(cells, lengths)]
    grid = torch.meshgrid(*reversed(ax), indexing="ij")
    X = torch.stack([g.reshape(-1) for g in reversed(grid)], 1)
    strides = [1, cells[0] + 1, (cells[0] + 1) * (cells[1] + 1)][:d]
    idx = torch.meshgrid(*[torch.arange(c, device="cuda") for c in reversed(cells)], indexing="ij")
    corner = sum(i.reshape(-1) * s for i, s in zip(idx, reversed(strides)))
    perms = [(0, 1), (1, 0)] if d == 2 else [(0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)]
    tets = []
    for perm in perms:
        v = [corner]
        for a in perm:
            v.append(v[-1] + strides[a])
        tets.append(torch.stack(v, 1))
    el = torch.cat(tets)
    if d == 2:
        i = torch.arange(cells[0], device="cuda")
        bot = torch.stack([i, i + 1], 1)
    else:
        k, i = torch.meshgrid(torch.arange(cells[2], device="cuda"), torch.arange(cells[0], device="cuda"), indexing="ij")
        b = (i + strides[2] * k).reshape(-1)
        bot = torch.cat([torch.stack([b, b + 1, b + 1 + strides[2]], 1), torch.stack([b, b + strides[2], b + 1 + strides[2]], 1)])
    return X, el, bot, bot + strides[1] * cells[1]


def _measure(X, s):
    """Measures and barycentric gradients (E x (k + 1) x D) of k-simplices."""
    J = X[s[:, 1:]] - X[s[:, :1]]
    k = J.shape[1]
    gram = J @ J.transpose(1, 2)
    vol = torch.sqrt(torch.linalg.det(gram)) / math.factorial(k)
    g = torch.linalg.solve(gram, J)
    return vol, torch.cat([-g.sum(1, keepdim=True), g], 1)


def _collapsed(k, pts):
    """Product Gauss-Legendre rule collapsed onto the k-simplex: barycentric points and weights (sum 1)."""
    x, w = np.polynomial.legendre.leggauss(pts)
    x, w = 0.5 * (x + 1), 0.5 * w
    lam, wt = [], []
    for ids in np.ndindex(*([pts] * k)):
        u = [x[i] for i in ids]
        xi, left, ww = [], 1.0, 1.0
        for a, i in enumerate(ids):
            xi.append(u[a] * left)
            ww *= w[i] * (1 - u[a]) ** (k - 1 - a)
            left *= 1 - u[a]
        lam.append([1 - sum(xi)] + xi)
        wt.append(ww * math.factorial(k))
    return lam, wt


def _load(X, s, p, n, pts, f):
    """(int f_p lambda_i, int f_n lambda_i) over the simplices s for f(phi_p, phi_n) by quadrature."""
    vol, _ = _measure(X, s)
    out = torch.zeros(2, X.shape[0], dtype=torch.float64, device="cuda")
    P, N = p[s], n[s]
    for lam, w in zip(*_collapsed(s.shape[1] - 1, pts)):
        bary = torch.tensor(lam, dtype=torch.float64, device="cuda")
        for row, val in zip(out, f(P @ bary, N @ bary)):
            for a in range(s.shape[1]):
                row.index_add_(0, s[:, a], vol * w * lam[a] * val)
    return out


def _fh(a, b):
    s = 1 - a - b
    la, lb, ls = (torch.log(t.clamp_min(FH_DELTA)) + 1 for t in (a, b, s))
    pn, ps, ns = CHI
    return (la / FH_N[0] - ls / FH_N[2] + pn * b + ps * (s - a) - ns * b,
            lb / FH_N[1] - ls / FH_N[2] + (pn - ps) * a + ns * (s - b))


def _poly(a, b):
    s = 1 - a - b
    return 7 * a * b * b - 0.2 * s, 7 * b * a * a - 0.2 * s


class _Fem64:
    """M, K, the loads and the block operator of one box, element by element in 64 bits."""

    def __init__(self, cells, lengths):
        self.X, self.el, self.bot, self.top = _mesh64(cells, lengths)
        vol, g = _measure(self.X, self.el)
        d = len(cells)
        self.Ke = vol[:, None, None] * (g @ g.transpose(1, 2))
        eye = torch.ones(d + 1, d + 1, dtype=torch.float64, device="cuda") + torch.eye(d + 1, dtype=torch.float64, device="cuda")
        self.Me = vol[:, None, None] * eye / ((d + 1) * (d + 2))
        self.n = self.X.shape[0]
        self.a, self.c = TAU, TAU / EPS

    def mul(self, Ae, x):
        y = torch.einsum("eij,ejc->eic", Ae, x[self.el])
        return torch.zeros_like(x).index_add(0, self.el.reshape(-1), y.reshape(-1, x.shape[1]))

    def apply(self, x):
        m, k = self.mul(self.Me, x), self.mul(self.Ke, x)
        return torch.cat([m[:, :2] + self.a * k[:, 2:], self.a * k[:, :2] - self.c * m[:, 2:]], 1)

    def rhs(self, p, n, potential=0):
        F = _load(self.X, self.el, p, n, 3, _fh) if potential == 3 else _load(self.X, self.el, p, n, 4, _poly)
        sub = torch.full_like(p[:1], G_SUB)
        g = _load(self.X, self.bot, p, n, 4, lambda a, b: (sub, sub))
        g = g + _load(self.X, self.top, p, n, 4, lambda a, b: (K_EVAP * a * (1 - a - b), K_EVAP * b * (1 - a - b)))
        m = self.mul(self.Me, torch.stack([p, n], 1))
        return torch.cat([m + TAU * g.T, -self.c * F.T], 1)

    def dense(self):
        M = torch.zeros(self.n * self.n, dtype=torch.float64, device="cuda")
        K = torch.zeros_like(M)
        at = (self.el[:, :, None] * self.n + self.el[:, None, :]).reshape(-1)
        M.index_add_(0, at, self.Me.reshape(-1))
        K.index_add_(0, at, self.Ke.reshape(-1))
        return M.reshape(self.n, self.n), K.reshape(self.n, self.n)


def _exact_step(case, seed):
    cells, lengths = _cells(case)
    if math.prod(c + 1 for c in cells) > 2500:
        return None  # a dense solve of the step's system is affordable on small meshes only
    fem = _Fem64(cells, lengths)
    (x,) = _evolve(cells, lengths, case["base"], case["base"], seed)
    b = fem.rhs(x[:, 0], x[:, 1])
    M, K = fem.dense()
    A = torch.cat([torch.cat([M, fem.a * K], 1), torch.cat([fem.a * K, -fem.c * M], 1)])
    sol = torch.linalg.solve(A, torch.cat([b[:, :2], b[:, 2:]]))
    p, n = sol[:fem.n, 0], sol[:fem.n, 1]
    return dict(phi_p=p, phi_nfa=n, phi_s=1 - p - n, mu_p=sol[fem.n:, 0], mu_nfa=sol[fem.n:, 1])


def _exact_train(case, seed):
    cells, lengths = _cells(case)
    nx, ny, B = case["nx"], case["ny"], case["batch"]
    hist = [_evolve(cells, lengths, 0.25 + 0.02 * b, 0.40 - 0.015 * b, seed, stream=b, keep=3) for b in range(B)]
    q2, q, s = (torch.stack(t) for t in zip(*hist))
    d, D = s - q, s - 2 * q + q2
    r1, r2 = (t.square().mean(1, keepdim=True).sqrt().clamp_min(1e-30) for t in (d, D))
    flat = s.reshape(-1, 4)
    x = torch.cat([(s - flat.mean(0)) / flat.std(0), d / r1, D / r2], 2)
    x = x.reshape(B, ny + 1, nx + 1, 12).permute(0, 3, 1, 2)
    rng = np.random.default_rng(seed & 0xFFFF)  # the seeded He-uniform start, output bias 1
    vals = []
    for i, (size, fan, nb) in enumerate([(9 * 16 * 32, 9 * 12, 32), (9 * 32 * 32, 9 * 32, 32), (9 * 32 * 8, 9 * 32, 8)]):
        lim = np.sqrt(6.0 / fan) * (0.1 if i == 2 else 1.0)
        vals += [rng.uniform(-lim, lim, size), np.zeros(nb)]
    vals[-1][:4] = 1.0
    theta = torch.from_numpy(np.concatenate(vals).astype(np.float32)).double().cuda().requires_grad_(True)
    at = 0

    def take(*shape):
        nonlocal at
        v = theta[at:at + math.prod(shape)].reshape(shape)
        at += math.prod(shape)
        return v

    for cin, used, cout, outs in ((16, 12, 32, 32), (32, 32, 32, 32), (32, 32, 8, 4)):
        w, bias = take(3, 3, cin, cout), take(cout)
        cols = torch.nn.functional.unfold(x, 3, padding=1)  # B x (channels x 9) x pixels
        y = torch.einsum("bkp,ko->bop", cols, w[:, :, :used, :outs].permute(2, 0, 1, 3).reshape(used * 9, outs))
        y = (y + bias[:outs, None]).reshape(B, outs, ny + 1, nx + 1)
        x = y.relu() if outs == 32 else y
    out = x.permute(0, 2, 3, 1).reshape(B, -1, 4)
    fem = _Fem64(cells, lengths)
    loss = 0.0
    for b in range(B):
        rex = fem.rhs(s[b, :, 0], s[b, :, 1]) - fem.apply(2 * s[b] - q[b])
        r = rex - fem.apply(out[b] * D[b])
        for sp in (0, 1):
            loss = loss + torch.log(r[:, sp::2].square().sum() / rex[:, sp::2].square().sum()) / (2 * B)
    (grad,) = torch.autograd.grad(loss, theta)
    return dict(loss=float(loss), grads=grad.cpu().numpy())


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        return _exact_step(case, seed)
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "rhs":
        cells, lengths = _cells(case)
        (x,) = _evolve(cells, lengths, case["base"], case["base"], seed)
        return _Fem64(cells, lengths).rhs(x[:, 0], x[:, 1], case["potential"])
    if kind == "setup":
        cells, lengths = _cells(case)
        u = _uniform(seed, 0, (2,)).tolist()
        tau, eps = TAU * 10 ** (u[0] - 0.5), EPS * 10 ** (u[1] - 0.5)
        fem = _Fem64(cells, lengths)
        at = (fem.el[:, :, None] * fem.n + fem.el[:, None, :]).reshape(-1)
        keys, inv = torch.unique(at, return_inverse=True)  # sorted: the rows in order, columns ascending
        M, K = (torch.zeros(len(keys), dtype=torch.float64, device="cuda").index_add_(0, inv, v.reshape(-1))
                for v in (fem.Me, fem.Ke))
        rowptr = torch.zeros(fem.n + 1, dtype=torch.int64, device="cuda")
        rowptr[1:] = torch.bincount(keys // fem.n, minlength=fem.n).cumsum(0)
        return dict(system=(rowptr.int(), (keys % fem.n).int(), M, K, tau * K + math.sqrt(tau / eps) * M), w=None)
    if kind == "project":
        (x,) = _evolve(*_cells(case), 0.33, 0.33, seed)
        pix = []
        for g, n in ((case["gx"], case["nx"]), (case["gy"], case["ny"])):
            pts = (np.arange(g) + 0.5) * (1.0 / g)
            pix.append(np.clip(np.floor(pts / (1.0 / n) + 0.5).astype(np.int64), 0, n))
        img = (x[:, 0] > x[:, 1]).cpu().numpy().reshape(case["ny"] + 1, case["nx"] + 1)
        inside = img[np.ix_(pix[1], pix[0])]
        return inside.astype(np.uint8), np.where(inside, 1e-10, 0.1), np.where(inside, 0.1, 1e-10)
    return None  # a preconditioner is an approximation, a batch or a guessed step too large for a dense solve
