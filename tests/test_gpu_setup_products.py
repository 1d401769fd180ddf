"""The set-up's sparse products and coarse inverse at their edges, through the exported hierarchies: rows
past each table size of the hashed product (and the heap merge beyond the largest), rows past the
in-register sort, coarsest levels around the 32-pivot blocks of the inverse.  A_{l+1} = P^T A P to 1e-13
of the largest entry (sums of at most a few thousand terms of one sign pattern, rounding below 1e-13),
and Algorithm 1 with a one-level hierarchy is its exact form: 1e-11 as in the parity tests."""
import numpy as np
import pytest
import scipy.sparse as sp

pytestmark = pytest.mark.gpu


def _csr(t, shape):
    return sp.csr_matrix((t[2].cpu().numpy(), t[1].cpu().numpy(), t[0].cpu().numpy()), shape=shape)


@pytest.mark.parametrize("kw", [dict(nx=33, ny=31, coarse_max=64), dict(nx=200, ny=7, coarse_max=20),
                                dict(dim=3, nx=20, ny=18, nz=16, Lz=0.5, coarse_max=40),
                                # strong coupling only along x: long aggregates, wide coarse rows
                                dict(dim=3, nx=40, ny=36, nz=34, Lx=1.0, Ly=3.0, Lz=0.3, amg_theta=0.2, coarse_max=60)])
def test_galerkin_products(lib, kw):
    p = lib.Params(**kw)
    pc = lib.Precond(lib.System(lib.Mesh(p), p))
    for which in (0, 1):
        n = len(pc.levels(which))
        lv = [pc.level(which, l) for l in range(n)]
        for l in range(n - 1):
            rows, nxt = lv[l]["rows"], lv[l + 1]["rows"]
            A, P = _csr(lv[l]["A"], (rows, rows)), _csr(lv[l]["P"], (rows, nxt))
            C = _csr(lv[l + 1]["A"], (nxt, nxt))
            for M in (A, P, C):  # sorted rows without duplicates
                d = np.diff(M.indices.astype(np.int64))
                d[np.diff(M.indptr).cumsum()[:-1] - 1] = 1
                assert (d > 0).all()
            D = (P.T @ A @ P - C).tocsr()
            assert abs(D).max() <= 1e-13 * abs(C).max()


@pytest.mark.parametrize("nx,ny", [(3, 7), (4, 6), (7, 7), (30, 32), (31, 31), (63, 64)])
def test_coarse_inverse_sizes(lib, nx, ny):
    """One-level hierarchies of 32, 35, 64, 1023, 1024 and 4160 > 4096 (two levels) rows."""
    import torch
    p = lib.Params(nx=nx, ny=ny, coarse_max=4096)
    system = lib.System(lib.Mesh(p), p)
    pc = lib.Precond(system)
    rowptr, col, m, _, h = system.csr()
    rng = np.random.default_rng(0)
    b = rng.standard_normal((system.n, 2))
    for which, val in ((0, m), (1, h)):
        if len(pc.levels(which)) > 1:
            continue
        A = _csr((rowptr, col, val), (system.n, system.n))
        x = pc.vcycle(which, torch.from_numpy(b).cuda()).cpu().numpy()
        assert np.linalg.norm(A @ x - b) <= 1e-11 * np.linalg.norm(b)
