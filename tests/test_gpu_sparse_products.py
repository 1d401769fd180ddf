"""The set-up's sparse product and transposition on matrices made for their branches: products whose longest row has a
given number of columns on either side of every table size (64 slots hold 48 columns, then 192, 768, 3072; longer rows take
the merge), rows of many terms on few columns, empty rows, one long row among short ones; transposed rows on either side
of the 256 entries that are ranked in shared memory.

The pattern has to be exact.  A value is the sum of its terms in a fixed order: at most (terms + 1) u sum |a||b| off,
u = 2^-53, and the same from run to run."""
import ctypes

import numpy as np
import pytest
import scipy.sparse as sp

import probes

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module")
def probe(lib, tmp_path_factory):
    dll = probes.load(lib, "products_probe.cu", tmp_path_factory.mktemp("probe"))
    vp, i = ctypes.c_void_p, ctypes.c_int
    dll.product_probe.restype = dll.transpose_probe.restype = ctypes.c_int64
    dll.product_probe.argtypes = [i] * 3 + [vp] * 6 + [ctypes.c_int64] + [vp] * 3
    dll.transpose_probe.argtypes = [i] * 2 + [vp] * 3 + [ctypes.c_int64] + [vp] * 3
    return dll


def _csr(rows, ncols, rng):
    """Rows of sorted distinct columns with values of both signs."""
    rowptr = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    col = np.concatenate([np.sort(r) for r in rows]).astype(np.int32) if rowptr[-1] else np.zeros(0, np.int32)
    return sp.csr_matrix((rng.standard_normal(rowptr[-1]), col, rowptr), shape=(len(rows), ncols))


def _arrays(M):
    return [a.ctypes.data for a in (M.indptr, M.indices, M.data)]


def _result(call, rows, ncols, room):
    rowptr, col, val = np.zeros(rows + 1, np.int32), np.zeros(room, np.int32), np.zeros(room)
    nnz = call(room, rowptr.ctypes.data, col.ctypes.data, val.ctypes.data)
    assert 0 <= nnz <= room, nnz
    return sp.csr_matrix((val[:nnz], col[:nnz], rowptr), shape=(rows, ncols))


# columns of the longest row of the product; terms per column there; columns of B
CASES = [(20, 1, 40), (48, 1, 48), (48, 3, 10000), (49, 1, 10000), (192, 2, 10000), (193, 1, 10000), (768, 1, 10000),
         (769, 2, 10000), (3072, 1, 10000), (3073, 1, 10000), (5000, 2, 10000), (60, 40, 60), (60, 40, 10000)]


@pytest.mark.parametrize("columns,terms,m", CASES)
def test_products(probe, columns, terms, m):
    rng = np.random.default_rng(columns + terms)
    # B: `terms` groups of rows that share `columns` columns between them, 50 columns a row, then short rows
    per = 50
    wide = rng.permutation(m)[:columns]
    b_rows = [wide[k:k + per] for _ in range(terms) for k in range(0, columns, per)]
    groups = len(b_rows)
    b_rows += [rng.permutation(m)[:rng.integers(0, 4)] for _ in range(200)]
    B = _csr(b_rows, m, rng)
    # A: one row that takes all the groups, empty rows, short rows (of short rows of B)
    short = [groups + rng.permutation(200)[:rng.integers(0, 6)] for _ in range(150)]
    A = _csr(short[:70] + [np.arange(groups)] + short[70:], len(b_rows), rng)
    ones = [sp.csr_matrix((np.ones(M.nnz), M.indices, M.indptr), shape=M.shape) for M in (A, B)]
    pattern = (ones[0] @ ones[1]).tocsr()  # the terms of each entry
    pattern.sort_indices()
    assert np.diff(pattern.indptr).max() == columns
    room = pattern.nnz + 10

    def product():
        return _result(lambda *out: probe.product_probe(A.shape[0], A.shape[1], m, *_arrays(A), *_arrays(B), *out),
                       A.shape[0], m, room)

    C = product()
    assert np.array_equal(C.indptr, pattern.indptr) and np.array_equal(C.indices, pattern.indices)
    want = (A.toarray().astype(np.longdouble) @ B.toarray().astype(np.longdouble)) if m <= 100 else None
    size = (abs(A) @ abs(B)).tocsr()
    size.sort_indices()
    if want is None:  # extended precision row by row
        vals = np.zeros(C.nnz, np.longdouble)
        for i in range(A.shape[0]):
            acc = np.zeros(m, np.longdouble)
            for q in range(A.indptr[i], A.indptr[i + 1]):
                r = slice(B.indptr[A.indices[q]], B.indptr[A.indices[q] + 1])
                acc[B.indices[r]] += np.longdouble(A.data[q]) * B.data[r].astype(np.longdouble)
            c = slice(C.indptr[i], C.indptr[i + 1])
            vals[c] = acc[C.indices[c]]
    else:
        vals = want[np.repeat(np.arange(C.shape[0]), np.diff(C.indptr)), C.indices]
    assert (abs(C.data - vals) <= (pattern.data + 1) * U * size.data).all()
    assert np.array_equal(product().data, C.data)


@pytest.mark.parametrize("longest", [1, 31, 255, 256, 257, 900])
def test_transposes(probe, longest):
    rng = np.random.default_rng(longest)
    n, m = max(longest, 40), 70
    cols = [[] for _ in range(n)]
    for r in rng.permutation(n)[:longest]:  # column 7 has `longest` entries, column 8 none
        cols[r].append(7)
    for r in range(n):
        cols[r] += [c for c in rng.permutation(m)[:2] if c not in (7, 8)]
    A = _csr([np.array(c, dtype=np.int64) for c in cols], m, rng)
    C = _result(lambda *out: probe.transpose_probe(n, m, *_arrays(A), *out), m, n, A.nnz)
    want = A.T.tocsr()
    want.sort_indices()
    assert np.diff(want.indptr).max() >= longest
    assert np.array_equal(C.indptr, want.indptr) and np.array_equal(C.indices, want.indices)
    assert np.array_equal(C.data, want.data)


@pytest.mark.parametrize("nx,ny,precision", [(63, 63, 0), (62, 63, 0), (61, 61, 1), (8, 8, 0)])
def test_one_level_hierarchies_solve_exactly(lib, nx, ny, precision):
    """The largest dense inverse (4096 rows) and sizes beside the 32-pivot blocks; a V-cycle is then the solve itself.  FP64
    1e-11 as in the parity tests; FP32 2e-6 as in the V-cycle tests (inverse and vectors rounded to FP32, cond <= 20 on M)."""
    import torch
    p = lib.Params(nx=nx, ny=ny, coarse_max=4096, precision=precision)
    system = lib.System(lib.Mesh(p), p)
    pc = lib.Precond(system)
    rowptr, col, m, _, _ = (t.cpu().numpy() for t in system.csr())
    assert len(pc.levels(0)) == 1
    M = sp.csr_matrix((m, col, rowptr), shape=(system.n, system.n))
    b = np.random.default_rng(0).standard_normal((system.n, 2))
    x = pc.vcycle(0, torch.from_numpy(b).cuda()).cpu().numpy()
    assert np.linalg.norm(M @ x - b) <= (2e-6 if precision else 1e-11) * np.linalg.norm(b)
