"""The end of the Gram-Schmidt passes on given vectors (krylov_probe.cu, compiled here against the library's own
kernels): V_{j+1} = (W - V h2) / h_{j+1,j} in FP64, node by node, however small the vector's entry or large h2.

Tolerance: the sum over nv terms runs in two halves of fused multiply-adds, then one addition, one subtraction
and the scaling: (nv / 2 + 4) u sum |h2_k V_k| + 3 u |W - V h2| per entry, u = 2^-53, all divided by h_{j+1,j}."""
import ctypes

import numpy as np
import pytest

import probes

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
MAXM = 64


@pytest.fixture(scope="module")
def probe(lib, tmp_path_factory):
    f = probes.load(lib, "krylov_probe.cu", tmp_path_factory.mktemp("probe")).orth_probe
    f.argtypes = [ctypes.c_int] * 3 + [ctypes.c_void_p] * 4
    return f


def _species(x, s):  # the components of species s as one vector: (phi, mu) per node
    return x[..., s::2].reshape(*x.shape[:-2], -1)


def _vectors(n, nv, kind, seed):
    """Per species an orthonormal basis of nv vectors and W: random, or nearly in the basis's span."""
    rng = np.random.default_rng(seed)
    V, W = np.zeros((nv, n, 4)), np.zeros((n, 4))
    for s in (0, 1):
        q = np.linalg.qr(rng.standard_normal((2 * n, min(nv + 1, 2 * n))))[0].T
        V[:, :, s::2] = q[:nv].reshape(nv, n, 2)
        c = rng.standard_normal(nv)
        w = rng.standard_normal(2 * n) if kind == "random" else c @ q[:nv]
        if kind.startswith("lean"):  # what the first projection leaves is that part of W
            w = w + float(kind[5:]) * rng.standard_normal(2 * n) / np.sqrt(2 * n)
        W[:, s::2] = w.reshape(n, 2)
    W[n // 2] *= 1e-9  # (a node where the vector is small)
    return V, W


def _run(probe, n, nv, blocks, V, W):
    import torch
    Vd, Wd = torch.from_numpy(V).cuda(), torch.from_numpy(W).cuda()
    nxt = torch.full((n, 4), np.nan, dtype=torch.float64, device="cuda")
    nh = 2 * (MAXM + 1)
    out = np.zeros(2 * nh + 2 + 2 * MAXM)
    torch.cuda.synchronize()
    assert probe(n, nv, blocks, Vd.data_ptr(), Wd.data_ptr(), nxt.data_ptr(), out.ctypes.data) == 0
    h1, h2 = out[:nh].reshape(2, -1)[:, :nv], out[nh:2 * nh].reshape(2, -1)[:, :nv]
    R = out[2 * nh + 2:].reshape(2, MAXM)[:, :nv]
    return Wd.cpu().numpy(), nxt.cpu().numpy(), h1, h2, out[2 * nh:2 * nh + 2], R


@pytest.mark.parametrize("n,nv,blocks,kind", [(3000, 30, 20, "random"), (3000, 30, 20, "lean 1e-6"), (700, 64, 5, "lean 1e-6"),
                                              (700, 33, 40, "lean 1e-4"), (257, 1, 1, "lean 1e-6"), (3000, 16, 33, "lean 1e-9")])
def test_correction_is_fp64(probe, n, nv, blocks, kind):
    V, W = _vectors(n, nv, kind, seed=nv)
    W1, got, _, h2, hinv, _ = _run(probe, n, nv, blocks, V, W)
    for s in (0, 1):
        v, w = _species(V, s).astype(np.longdouble), _species(W1, s).astype(np.longdouble)
        corr, size = h2[s] @ v, abs(h2[s]) @ abs(v)
        bound = U * ((nv / 2 + 4) * size + 3 * abs(w - corr)) * hinv[s]
        assert (abs(_species(got, s) - (w - corr) * np.longdouble(hinv[s])) <= bound).all()


@pytest.mark.parametrize("n,nv,blocks,kind", [(4, 8, 1, "random"), (4, 7, 1, "random"), (40, 64, 3, "lean 1e-15"), (32, 64, 20, "random"),
                                              (3000, 30, 20, "lean 0"), (3000, 30, 20, "lean 1e-12"), (3000, 30, 20, "random")])
def test_the_next_vector_has_unit_length(probe, n, nv, blocks, kind):
    """Also where the basis spans the space, or W to rounding, and the second projection takes most of what the
    first left.  The norm is a sum of 2 n squares, its rounding below 1e-13.  h_{j+1,j} belongs to the column: with
    earlier rotations that are identities the new entry of R is the hypotenuse of h_{j,j} and h_{j+1,j}."""
    V, W = _vectors(n, nv, kind, seed=nv)
    _, got, h1, h2, hinv, R = _run(probe, n, nv, blocks, V, W)
    for s in (0, 1):
        assert hinv[s] > 0.0
        assert abs(np.linalg.norm(_species(got, s)) - 1.0) <= 1e-13
        assert abs(R[s, nv - 1] / np.hypot(h1[s, nv - 1] + h2[s, nv - 1], 1.0 / hinv[s]) - 1.0) <= 1e-13
