"""The block operator, the right-hand sides and the steps in lattice form (one table row per position class)
against the assembled CSR matrices, on boxes of every rim shape (one cell thick, odd, batched), on a grid
too long and thin for the classes (coordinate rounding: the CSR form), and with a non-finite entry, which
must reach its neighbours only.  y = A x is a sum of at most 30 products, so the two forms differ by a few
ulp of sum |a||x|: 1e-13 of the largest entry, the tolerance of the other operator tests."""
import numpy as np
import pytest
import scipy.sparse as sp

pytestmark = pytest.mark.gpu

BOXES = [dict(nx=1, ny=1), dict(nx=2, ny=5), dict(nx=1, ny=40), dict(nx=37, ny=23, Lx=10.0, Ly=2.5),
         dict(dim=3, nx=1, ny=1, nz=1), dict(dim=3, nx=1, ny=6, nz=2, Lz=0.3), dict(dim=3, nx=7, ny=5, nz=9, Lx=2.0),
         dict(nx=400000, ny=1)]


def _matrices(system):
    rowptr, col, m, k, _ = (t.cpu().numpy() for t in system.csr())
    shape = (system.n, system.n)
    return sp.csr_matrix((m, col, rowptr), shape=shape), sp.csr_matrix((k, col, rowptr), shape=shape)


def _system(lib, kw, runs=None):
    p = lib.Params(**kw)
    mesh = lib.Mesh(p, runs=runs)
    return lib.System(mesh, p), p


@pytest.mark.parametrize("kw", BOXES + ["batch"])
def test_operator_and_rhs_match_the_assembled_matrices(lib, kw):
    import torch
    if kw == "batch":
        runs = [lib.Params(nx=5, ny=3), lib.Params(nx=1, ny=9, Lx=3.0), lib.Params(nx=16, ny=2, Ly=0.5)]
        system, p = _system(lib, dict(nx=5, ny=3), runs)
    else:
        system, p = _system(lib, kw)
    M, K = _matrices(system)
    a, c = p.tau * p.mobility, p.tau * p.mobility / p.eps
    rng = np.random.default_rng(1)
    x = rng.standard_normal((system.n, 4))
    y = system.apply_A(torch.from_numpy(x).cuda()).cpu().numpy()
    ref = np.hstack([M @ x[:, :2] + a * (K @ x[:, 2:]), a * (K @ x[:, :2]) - c * (M @ x[:, 2:])])
    for col in range(4):
        assert np.abs(y[:, col] - ref[:, col]).max() <= 1e-13 * np.abs(ref[:, col]).max()
    phi = 0.3 + 0.05 * rng.standard_normal((2, system.n))
    dev = [torch.from_numpy(t).cuda() for t in phi]
    b = system.rhs(*dev).cpu().numpy()
    Fp, Fn, gp, gn = (t.cpu().numpy() for t in system.loads(*dev))
    want = np.stack([M @ phi[0] + p.tau * gp, M @ phi[1] + p.tau * gn, -c * Fp, -c * Fn], 1)
    assert np.abs(b - want).max() <= 1e-13 * np.abs(want).max()


def test_a_non_finite_entry_reaches_its_neighbours_only(lib):
    import torch
    runs = [lib.Params(nx=4, ny=3), lib.Params(nx=3, ny=5)]
    system, _ = _system(lib, dict(nx=4, ny=3), runs)
    M, _ = _matrices(system)
    for bad in (0, 4, 5, 19, 20, 23, system.n - 1):  # corners and row ends of both runs
        x = np.ones((system.n, 4))
        x[bad] = np.nan
        y = system.apply_A(torch.from_numpy(x).cuda()).cpu().numpy()
        assert set(np.flatnonzero(np.isnan(y).any(1))) == set(M[:, [bad]].nonzero()[0])
