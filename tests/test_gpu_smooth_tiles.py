"""The tile form of the finest level's smoothing passes (2D, one launch per pass) against the oracle's
V-cycle, at sizes around the tiles' edges: 64-column regions in FP32 (52 to 62 output columns at halos 6 to
1), 16-column ones in FP64, meshes of one row of cells, meshes smaller than a tile, several runs of unlike
size in one batch, a mesh large enough for two blocks per SM, and FP64 meshes on both sides of the line where
the single steps take over.

The hierarchy is the device's (coarsest level capped at 32 rows, or one level's direct solve would answer);
bounds as in the other V-cycle tests: FP64 1e-12 relative (sums of at most 9 terms over a handful of
passes), FP32 2e-6 (unit roundoff 6e-8 through the same passes)."""
import numpy as np
import pytest
import torch

from oracle import ch_oracle as o
from test_zy_vcycle_oracle import TOL, _exported, _oracle_levels

pytestmark = pytest.mark.gpu

SIZES = [dict(nx=53, ny=3), dict(nx=54, ny=58), dict(nx=57, ny=1), dict(nx=1, ny=130), dict(nx=109, ny=53),
         dict(nx=12, ny=11), dict(nx=66, ny=127), dict(nx=54, ny=54, cheb_degree=1), dict(nx=107, ny=9, cheb_degree=5),
         dict(nx=64, ny=64), dict(nx=640, ny=640), "batch"]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("which", [0, 1])
@pytest.mark.parametrize("kw", SIZES, ids=str)
def test_tiled_passes_equal_the_oracle_vcycle(lib, kw, which, precision):
    if kw == "batch":
        runs = [lib.Params(precision=precision, coarse_max=32, nx=a, ny=b) for a, b in ((61, 5), (17, 64), (3, 3))]
        p = runs[0]
    else:
        runs, p = None, lib.Params(precision=precision, coarse_max=32, **kw)
    system = lib.System(lib.Mesh(p, runs=runs), p)
    pc = lib.Precond(system)
    levels = _oracle_levels(_exported(pc, which))
    assert len(levels) >= 2
    b = np.random.default_rng(5 + which).standard_normal((system.n, 2))
    for cycles in (1, 2):
        got = pc.vcycle(which, torch.from_numpy(b).cuda(), cycles).cpu().numpy()
        for k in range(2):
            want = None
            for _ in range(cycles):
                want = o.vcycle(levels, b[:, k]) if want is None else o.vcycle(levels, b[:, k], x0=want.copy())
            err = np.abs(got[:, k] - want).max() / np.abs(want).max()
            assert err <= TOL[precision], (kw, which, k, cycles, err)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("kw", [dict(nx=57, ny=1), dict(nx=66, ny=53), dict(nx=20, ny=20, vcycles_M=2)], ids=str)
def test_last_pass_stores_the_application(lib, kw, precision):
    """Algorithm 1's first half is M's V-cycles alone: the tile pass that stores its result in FP64 and the cycle
    that a conversion follows are the same arithmetic, bit for bit."""
    p = lib.Params(precision=precision, coarse_max=32, **kw)
    system = lib.System(lib.Mesh(p), p)
    pc = lib.Precond(system)
    v = torch.from_numpy(np.random.default_rng(8).standard_normal((system.n, 4))).cuda()
    w = pc.apply(v)
    assert torch.equal(w[:, :2], pc.vcycle(0, v[:, :2].contiguous(), kw.get("vcycles_M", 1)))
    assert torch.isfinite(w).all()
