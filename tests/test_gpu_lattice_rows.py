"""The lattice form of the operator and of FP64 smoothing against the assembled rows, at cell counts whose
coordinates i (L / n) are not exact: the cells of an axis then have several widths a few ulp of the coordinate
apart (relative to the cell, 1.4e-13 on 799 cells of [0, 10], 1e-11 on 50000 of [0, 1]), the assembled entries
differ as much, and every row has to be its own.

Tolerances.  y_i = (A x)_i has at most 30 products: with k terms summed in any order the error is at most
(k + 2) u sum |a||x|, u = 2^-53: 32 u per node.  A smoothing pass against the same recurrence in extended
precision: per step three or four roundings of values of the iterate's size, damped by the next steps (the
smoother is a contraction on the modes it targets and adds nothing on the others): 16 u of the largest value.
"""
import numpy as np
import pytest
import scipy.sparse as sp

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
BOXES = [dict(nx=33, ny=31), dict(nx=799, ny=399, Lx=10.0, Ly=2.5), dict(nx=50000, ny=3), dict(nx=400000, ny=1),
         dict(nx=1, ny=57, Ly=0.9), dict(dim=3, nx=33, ny=21, nz=17, Lz=0.5), dict(dim=3, nx=1, ny=2, nz=41, Lz=0.7),
         "batch"]


def _system(lib, kw, **more):
    if kw == "batch":
        runs = [lib.Params(nx=57, ny=33, Lx=0.9, **more), lib.Params(nx=1, ny=9, Lx=3.0, **more),
                lib.Params(nx=41, ny=29, **more), lib.Params(nx=57, ny=33, **more)]
        return lib.System(lib.Mesh(runs[0], runs=runs), runs[0]), runs[0]
    p = lib.Params(**kw, **more)
    return lib.System(lib.Mesh(p), p), p


def _csr(rowptr, col, val, n):
    return sp.csr_matrix((val.cpu().numpy(), col.cpu().numpy(), rowptr.cpu().numpy()), shape=(n, n))


def _mul(A, x):
    """A x in extended precision (every row of A has entries)."""
    return np.add.reduceat(A.data.astype(np.longdouble)[:, None] * x[A.indices], A.indptr[:-1], axis=0)


@pytest.mark.parametrize("kw", BOXES, ids=str)
def test_operator_has_the_assembled_rows(lib, kw):
    import torch
    system, p = _system(lib, kw)
    rowptr, col, m, k, _ = system.csr()
    M, K = _csr(rowptr, col, m, system.n), _csr(rowptr, col, k, system.n)
    a, c = np.longdouble(p.tau * p.mobility), np.longdouble(p.tau * p.mobility / p.eps)
    rng = np.random.default_rng(2)
    x = rng.standard_normal((system.n, 4))
    lib.profile_read(reset=True)
    y = system.apply_A(torch.from_numpy(x).cuda()).cpu().numpy()
    # which form ran: the lattice form counts 66 bytes per node, the CSR form 20 per stored entry and more
    assert lib.profile_read(reset=True)["apply_A_f64"]["bytes"] == 66.0 * system.n

    def blocks(M, K, c, x):
        mx, kx = _mul(M, x), _mul(K, x)
        return np.concatenate([mx[:, :2] + a * kx[:, 2:], a * kx[:, :2] + c * mx[:, 2:]], 1)

    want, size = blocks(M, K, -c, x.astype(np.longdouble)), blocks(abs(M), abs(K), c, abs(x).astype(np.longdouble))
    assert float((abs(y - want) / size).max()) <= 32 * U
    # the right-hand side's mass product (tau g is zero inside the box)
    phi = 0.3 + 0.05 * rng.standard_normal((system.n, 2))
    dev = [torch.from_numpy(t).cuda() for t in phi.T.copy()]
    b = system.rhs(*dev).cpu().numpy()
    g = np.stack([t.cpu().numpy() for t in system.loads(*dev)[2:]], 1)
    want, size = _mul(M, phi.astype(np.longdouble)) + np.longdouble(p.tau) * g, _mul(M, abs(phi).astype(np.longdouble))
    assert float((abs(b[:, :2] - want) / (size + p.tau * abs(g))).max()) <= 32 * U


def _smooth(L, b, x):
    """One pass of the level's Chebyshev smoother on x."""
    lo, hi = (np.longdouble(t) for t in L["bounds"])
    theta, delta = (hi + lo) / 2, (hi - lo) / 2
    rho, d = delta / theta, np.longdouble(0)
    for s in range(L["degree"]):
        r = L["dinv"] * (b - _mul(L["A"], x))
        if s == 0:
            d = r / theta
        else:
            new = 1 / (2 * theta / delta - rho)
            d, rho = new * rho * d + 2 * new / delta * r, new
        x = x + d
    return x


def _vcycle(levels, b, x, l=0):
    L = levels[l]
    if l + 1 == len(levels):
        A = L["A"].toarray()
        for _ in range(5):  # refined to extended precision
            x = x + np.linalg.solve(A, (b - _mul(L["A"], x)).astype(np.float64))
        return x
    x = _smooth(L, b, x)
    r = _mul(L["R"], b - _mul(L["A"], x))
    x = x + _mul(L["P"], _vcycle(levels, r, np.zeros(r.shape, np.longdouble), l + 1))
    return _smooth(L, b, x)


def _levels(pc, which):
    exported = [pc.level(which, l) for l in range(len(pc.levels(which)))]
    out = []
    for l, e in enumerate(exported):
        A = _csr(*e["A"], e["rows"])
        L = dict(A=A, bounds=e["bounds"], degree=e["degree"], dinv=(1 / A.diagonal().astype(np.longdouble))[:, None])
        if l + 1 < len(exported):
            rowptr, col, val = (t.cpu().numpy() for t in e["P"])
            L["P"] = sp.csr_matrix((val, col, rowptr), shape=(e["rows"], exported[l + 1]["rows"]))
            L["R"] = L["P"].T.tocsr()
        out.append(L)
    return out


@pytest.mark.parametrize("kw", [dict(nx=399, ny=200, Lx=10.0, Ly=2.5), dict(nx=33, ny=31), dict(nx=64, ny=3, Lx=0.9),
                                dict(dim=3, nx=33, ny=21, nz=17, Lz=0.5), "batch"], ids=str)
@pytest.mark.parametrize("which", [0, 1])
def test_fp64_smoothing_has_the_assembled_rows(lib, kw, which):
    """One launch per step (ch_smooth, and the V-cycles of the larger meshes) and one per pass (small 2D meshes)."""
    import torch
    system, _ = _system(lib, kw, coarse_max=64)
    pc = lib.Precond(system)
    levels = _levels(pc, which)
    assert len(levels) >= 2
    b, x0 = np.random.default_rng(4).standard_normal((2, system.n, 2))
    bl, bd = b.astype(np.longdouble), torch.from_numpy(b).cuda()
    for degree in (1, 5):
        want = _smooth(dict(levels[0], degree=degree), bl, x0.astype(np.longdouble))
        got = torch.from_numpy(x0.copy()).cuda()
        pc.smooth(which, bd, got, degree)
        assert float(abs(got.cpu().numpy() - want).max()) <= 16 * U * float(abs(want).max())
    want = _vcycle(levels, bl, np.zeros(b.shape, np.longdouble))
    got = pc.vcycle(which, bd).cpu().numpy()
    assert float(abs(got - want).max()) <= 16 * U * float(abs(want).max())


def test_fp32_cycles_of_a_long_thin_grid(lib):
    """400000 x 1 cells: the rows of one position differ by more than 2^-36 of the diagonal, and FP32 V-cycles take the
    classes by cell widths, a launch per step (the lattice form counts 2 bytes of class id per node and its vectors).  Against
    the oracle to the bound of the other FP32 V-cycle tests."""
    import torch
    from oracle import ch_oracle as o
    from test_zy_vcycle_oracle import TOL, _exported, _oracle_levels
    system, _ = _system(lib, dict(nx=400000, ny=1), precision=1)
    pc = lib.Precond(system)
    levels = _oracle_levels(_exported(pc, 0))
    degree, n = levels[0]["degree"], system.n
    b = np.random.default_rng(4).standard_normal((n, 2))
    bd = torch.from_numpy(b).cuda()
    lib.profile_read(reset=True)
    got = pc.vcycle(0, bd).cpu().numpy()
    step = lib.profile_read(reset=True)["cheb_step_f32"]
    assert step["launches"] == 2 * degree - 1
    assert step["bytes"] <= (2.0 + 4.0 * 10) * n * step["launches"]
    for k in range(2):
        want = o.vcycle(levels, b[:, k])
        assert np.abs(got[:, k] - want).max() / np.abs(want).max() <= TOL[1]
