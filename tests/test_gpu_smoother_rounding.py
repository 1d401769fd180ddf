"""The Chebyshev smoother's rounding error.  ch_smooth against the same recurrence in extended precision, beside
the error of that recurrence evaluated on the host in the working precision with fused multiply-adds and the
direction kept: x' = x - beta e', e' = carry e + D^-1 (A x - b).  The two do the same operations, so their errors
agree to a few percent of the root mean square (allowed: 5 %; about a thousand nodes and more, the largest
difference between two orders of the same sums is 2 %).  Forms that are not as accurate lie outside: the
momentum term from x - x_prev is 13 to 27 % further off at these degrees, tables with the diagonal folded in
30 % and more.  Input and operator are rounded to the working precision first."""
import numpy as np
import pytest
import scipy.sparse as sp

pytestmark = pytest.mark.gpu

LD = np.longdouble


def _recurrence(A, dinv, b, x, degree, bounds, T):
    """The smoother with every operation rounded to T (rows of A in column order, fused multiply-adds)."""
    W = np.float64 if T is np.float32 else LD
    rowptr, width = A.indptr, int(np.diff(A.indptr).max())
    col, val = np.zeros((A.shape[0], width), int), np.zeros((A.shape[0], width), T)
    at = np.arange(A.nnz) - np.repeat(rowptr[:-1], np.diff(rowptr))
    row = np.repeat(np.arange(A.shape[0]), np.diff(rowptr))
    col[row, at], val[row, at] = A.indices, A.data

    def fma(a, u, v):
        return (np.asarray(a).astype(W) * u.astype(W) + v.astype(W)).astype(T)

    lo, hi = bounds
    theta, delta = (hi + lo) / 2, (hi - lo) / 2
    sigma = theta / delta  # (the coefficients' roundings are common to all nodes: the library's order)
    rho, beta = 1 / sigma, 1 / theta
    b, x, dinv = b.astype(T), x.astype(T), dinv.astype(T)[:, None]
    for s in range(degree):
        r = -b
        for d in range(width):
            r = fma(val[:, d:d + 1], x[col[:, d]], r)
        r = (dinv * r).astype(T)
        if s == 0:
            e = r
        else:
            new = 1 / (2 * sigma - rho)
            after = 2 * new / delta
            e = fma(T(new * rho * beta / after), e, r)
            rho, beta = new, after
        x = fma(T(-beta), e, x)
    return x


@pytest.mark.parametrize("kw", [dict(nx=33, ny=31), dict(nx=64, ny=40), dict(dim=3, nx=16, ny=12, nz=10, Lz=0.5)], ids=str)
@pytest.mark.parametrize("which", [0, 1])
@pytest.mark.parametrize("precision", [0, 1])
def test_rounding_is_that_of_the_kept_direction(lib, kw, which, precision):
    import torch
    T = np.float32 if precision else np.float64
    p = lib.Params(precision=precision, coarse_max=64, **kw)
    system = lib.System(lib.Mesh(p), p)
    pc = lib.Precond(system)
    level = pc.level(which, 0)
    rowptr, col, val = (t.cpu().numpy() for t in level["A"])
    dinv = (1 / sp.csr_matrix((val, col, rowptr), shape=(system.n, system.n)).diagonal()).astype(T)
    A = sp.csr_matrix((val.astype(T).astype(np.float64), col, rowptr), shape=(system.n, system.n))
    b, x0 = np.random.default_rng(6).standard_normal((2, system.n, 2)).astype(T).astype(np.float64)
    for degree in (3, 5):
        exact = _recurrence(A, dinv, b, x0, degree, [LD(t) for t in level["bounds"]], LD)
        same = _recurrence(A, dinv, b, x0, degree, level["bounds"], T)
        x = torch.from_numpy(x0.copy()).cuda()
        pc.smooth(which, torch.from_numpy(b).cuda(), x, degree)
        rms = [float(np.sqrt(np.mean((t - exact) ** 2))) for t in (x.cpu().numpy(), same)]
        assert rms[0] <= 1.05 * rms[1], (degree, rms)
