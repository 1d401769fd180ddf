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
