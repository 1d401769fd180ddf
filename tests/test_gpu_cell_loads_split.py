"""The polynomial loads of 3D meshes of few cells (a thread per simplex) and of many (a thread per cell): the same sums in
the same order.  A run's loads do not depend on what is batched with it, so a small box alone and the same box in a
batch beyond the line (152 x 64 cells) have to agree bit for bit, and the small box with the oracle as in the parity
tests."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("box", [dict(nx=1, ny=1, nz=1), dict(nx=5, ny=4, nz=3, Lx=1.3), dict(nx=21, ny=20, nz=23, Lz=0.5)], ids=str)
@pytest.mark.parametrize("potential", [0, 1, 2])
def test_alone_and_in_a_large_batch(lib, box, potential):
    import torch
    p = lib.Params(dim=3, potential=potential, **box)
    other = lib.Params(dim=3, potential=potential, nx=24, ny=22, nz=20)
    alone, batch = lib.System(lib.Mesh(p), p), lib.System(lib.Mesh(p, runs=[p, other]), p)
    gen = torch.Generator().manual_seed(2)
    phi = [0.4 * torch.rand(batch.n, dtype=torch.float64, generator=gen).cuda() for _ in range(2)]
    a = alone.loads(*(t[:alone.n].contiguous() for t in phi))
    b = batch.loads(*phi)
    for x, y in zip(a, b):
        assert torch.equal(x, y[:alone.n])
