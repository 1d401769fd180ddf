"""Restrictions at every width the set-up may choose, 256 (a block per row) included, with and without the coarse level's
first step fused, in both precisions: the set-up picks a width by timing, so a V-cycle alone may run any of them.  Rows
of 0, 1, 63, 64, 255, 256, 257 and 1500 entries.  A row sum of k terms in any order is at most (k + 1) u sum |r||x| off, and the
fused step two roundings more."""
import ctypes

import numpy as np
import pytest

import probes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def probe(lib, tmp_path_factory):
    f = probes.load(lib, "restrict_probe.cu", tmp_path_factory.mktemp("probe")).restrict_probe
    vp, i = ctypes.c_void_p, ctypes.c_int
    f.argtypes = [i] * 3 + [vp] * 4 + [i, vp, ctypes.c_double, vp, vp]
    return f


@pytest.mark.parametrize("first", [False, True])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("width", [1, 2, 4, 8, 16, 32, 256])
def test_row_sums(probe, width, precision, first):
    import torch
    T, u = (np.float32, 2.0 ** -24) if precision else (np.float64, 2.0 ** -53)
    rng = np.random.default_rng(3)
    counts = [0, 1, 63, 64, 255, 256, 257, 1500, 5, 700]
    cols = 2000
    rowptr = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    col = np.concatenate([np.sort(rng.permutation(cols)[:k]) for k in counts]).astype(np.int32)
    val, x = rng.standard_normal(rowptr[-1]).astype(T), rng.standard_normal((cols, 2)).astype(T)
    dinv, invtheta = rng.uniform(0.5, 2.0, len(counts)).astype(T), 0.7
    dev = [torch.from_numpy(a).cuda() for a in (rowptr, col, val, x, dinv)]
    bc = torch.full((len(counts), 2), float("nan"), dtype=dev[3].dtype, device="cuda")
    xc = torch.full_like(bc, float("nan"))
    torch.cuda.synchronize()
    assert probe(precision, len(counts), cols, *(t.data_ptr() for t in dev[:4]), width, dev[4].data_ptr() if first else None,
                 invtheta, bc.data_ptr(), xc.data_ptr() if first else None) == 0
    bc, xc = bc.cpu().numpy(), xc.cpu().numpy()
    for i, k in enumerate(counts):
        q = slice(rowptr[i], rowptr[i + 1])
        terms = val[q, None].astype(np.longdouble) * x[col[q]].astype(np.longdouble)
        want, size = terms.sum(0), abs(terms).sum(0)
        assert (abs(bc[i] - want) <= (k + 1) * u * size).all(), (i, k)
        if first:
            f = np.longdouble(T(invtheta)) * np.longdouble(dinv[i])
            assert (abs(xc[i] - f * bc[i]) <= 2.5 * u * abs(f * bc[i])).all(), (i, k)
    assert first or np.isnan(xc).all()
