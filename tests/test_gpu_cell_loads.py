"""The explicit loads formed per grid cell, at cell counts around the kernels' blocks (32 cells, 128 threads) and
on boxes one cell thick, against the oracle: 1e-12 (Flory-Huggins) and 1e-13 of the largest entry, the
tolerances of the load parity tests."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("potential", [0, 3])
@pytest.mark.parametrize("kw", [dict(nx=1, ny=1), dict(nx=33, ny=2), dict(dim=3, nx=1, ny=2, nz=33), dict(dim=3, nx=5, ny=4, nz=3)])
def test_loads_match_the_oracle_on_thin_boxes(lib, kw, potential):
    import torch
    from oracle import ch_oracle as o
    p = lib.Params(potential=potential, **kw)
    system = lib.System(lib.Mesh(p), p)
    op = o.Params(**kw)
    rng = np.random.default_rng(2)
    phi = rng.uniform(0.05, 0.6, (2, system.n))
    F = [t.cpu().numpy() for t in system.loads(*(torch.from_numpy(t).cuda() for t in phi))[:2]]
    om = o.mesh(op)
    ref = o.load_vector_fh(om, phi[0], phi[1], op) if potential == 3 else o.load_vector(om, phi[0], phi[1])
    for g, r in zip(F, ref):
        assert np.abs(g - r).max() <= (1e-12 if potential == 3 else 1e-13) * np.abs(r).max()


@pytest.mark.parametrize("beyond", [[], [2.0 ** 64, 1e20]])
@pytest.mark.parametrize("kw", [dict(nx=20, ny=11), dict(dim=3, nx=6, ny=5, nz=4)])
def test_flory_huggins_logarithms_over_their_range(lib, kw, beyond):
    """Concentrations from denormal to 3, then to 1e20 (the logarithm tables' end and beyond it), some below the
    guard: 1e-12 of the largest entry as above (each logarithm is good to 2^-53 (1 + |log x|)).
    No pair of values sums to nearly 1: 1 - phi_p - phi_n would cancel, in the oracle as here."""
    import torch
    from oracle import ch_oracle as o
    p = lib.Params(potential=3, **kw)
    system = lib.System(lib.Mesh(p), p)
    rng = np.random.default_rng(3)
    phi = rng.choice([1e-310, 1e-12, 1e-9, 1e-3, 0.25, 0.375, 0.0625, 3.0, -0.1] + beyond, (2, system.n))
    F = [t.cpu().numpy() for t in system.loads(*(torch.from_numpy(t).cuda() for t in phi))[:2]]
    op = o.Params(**kw)
    for g, r in zip(F, o.load_vector_fh(o.mesh(op), phi[0], phi[1], op)):
        assert np.isfinite(g).all()
        assert np.abs(g - r).max() <= 1e-12 * np.abs(r).max()
