"""Rounding error of the Flory-Huggins loads: the product rule in extended precision against the device's loads
and against the same rule evaluated point by point in numpy's doubles.  Both sum f' over the rule's points, whose
large terms (the logarithms, 1 and the interaction terms) cancel before they are weighted, so their errors are
alike: at most 1.25 times the plain evaluation's in the root mean square over all nodes (a few percent by the
order of the sums; logarithms off by an ulp, or integrals combined after the sums, give 1.4 to 6).  Smooth fields,
concentrations over nine decades, and constant fields of powers of two, whose logarithms are table entries."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LD = np.longdouble


def _rule(dim, T):
    root = np.sqrt(T(15)) / 10
    x, w = [T(1) / 2 - root, T(1) / 2, T(1) / 2 + root], [T(5) / 18, T(4) / 9, T(5) / 18]
    for i in range(3):
        for j in range(3):
            for k in range(3 if dim == 3 else 1):
                u, v = x[i], x[j]
                if dim == 2:
                    yield [1 - u - v * (1 - u), u, v * (1 - u)], 2 * w[i] * w[j] * (1 - u)
                else:
                    xi = [u, v * (1 - u), x[k] * (1 - u) * (1 - v)]
                    yield [1 - sum(xi)] + xi, 6 * w[i] * w[j] * w[k] * (1 - u) ** 2 * (1 - v)


def _loads(p, X, el, phi, T):
    X, P, N = X.astype(T), phi[0].astype(T)[el], phi[1].astype(T)[el]
    J = X[el[:, 1:]] - X[el[:, :1]]
    if J.shape[1] == 2:
        vol = abs(J[:, 0, 0] * J[:, 1, 1] - J[:, 0, 1] * J[:, 1, 0]) / 2
    else:
        vol = abs((J[:, 0] * np.cross(J[:, 1], J[:, 2])).sum(1)) / 6
    cpn, cps, cns = T(p.chi_pn), T(p.chi_ps), T(p.chi_ns)
    ip, inn, ins = (T(1.0 / t) for t in (p.N_p, p.N_nfa, p.N_s))
    out = np.zeros((2, len(X)), T)
    F = np.zeros((2,) + el.shape, T)
    for lam, w in _rule(J.shape[1], T):
        a = sum(lam[k] * P[:, k] for k in range(el.shape[1]))
        b = sum(lam[k] * N[:, k] for k in range(el.shape[1]))
        s = 1 - a - b
        la, lb, ls = (np.log(np.maximum(t, T(p.fh_delta))) + 1 for t in (a, b, s))
        fa = la * ip - ls * ins + cpn * b + cps * (s - a) - cns * b
        fb = lb * inn - ls * ins + (cpn - cps) * a + cns * (s - b)
        for k in range(el.shape[1]):
            F[0, :, k] += w * lam[k] * fa
            F[1, :, k] += w * lam[k] * fb
    for q in range(2):
        np.add.at(out[q], el, F[q] * vol[:, None])
    return out


@pytest.mark.parametrize("fields", ["smooth", "dense", "decades", "powers of two"])
@pytest.mark.parametrize("kw", [dict(nx=40, ny=24), dict(nx=25, ny=33, Lx=10.0, Ly=2.5),
                                dict(dim=3, nx=8, ny=7, nz=9, Lz=0.5)], ids=str)
def test_error_is_that_of_the_plain_evaluation(lib, kw, fields):
    import torch
    p = lib.Params(potential=3, **kw)
    system = lib.System(lib.Mesh(p), p)
    X, el = (t.cpu().numpy() for t in system.mesh.copy()[:2])
    rng = np.random.default_rng(3)
    if fields in ("smooth", "dense"):
        base = 0.3 if fields == "smooth" else 0.42
        phi = [base + 0.05 * np.cos(3 * X @ rng.standard_normal(X.shape[1])) + 1e-3 * rng.random(system.n) for _ in range(2)]
    elif fields == "decades":
        phi = list(0.45 * 10 ** (-9 * rng.random((2, system.n))))
    else:
        phi = [np.full(system.n, 0.25), np.full(system.n, 0.5)]
    got = np.stack([t.cpu().numpy() for t in system.loads(*(torch.from_numpy(f).cuda() for f in phi))[:2]])
    want, plain = _loads(p, X, el, phi, LD), _loads(p, X, el, phi, np.float64)
    rms = [float(np.sqrt(np.mean((t - want) ** 2))) for t in (got, plain)]
    print(kw, fields, rms)
    if fields == "powers of two":  # (no average over many roundings: three of the load's size)
        assert float(abs(got - want).max()) <= 3 * 2.0 ** -53 * float(abs(want).max()) + 3 * rms[1]
    else:
        assert rms[0] <= 1.25 * rms[1], rms
