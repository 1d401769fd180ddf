"""V-cycles whose coarse levels have long rows: row sums over every width the set-up may choose, one block per
row for restrictions of 64 entries a row and more, and the dense solve.  Against the oracle's V-cycle on the
device's own hierarchy; bounds as in the other V-cycle tests."""
import numpy as np
import pytest
import torch

from oracle import ch_oracle as o
from test_zy_vcycle_oracle import TOL, _exported, _oracle_levels

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("autotune", [0, 1])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("kw", [dict(nx=31, ny=33, nz=29, coarse_max=40), dict(nx=40, ny=40, nz=20, coarse_max=8),
                                dict(nx=25, ny=17, nz=9, coarse_max=300)], ids=str)
def test_long_rows(lib, kw, precision, autotune):
    p = lib.Params(precision=precision, dim=3, Lz=0.5, autotune=autotune, **kw)
    system = lib.System(lib.Mesh(p), p)
    pc = lib.Precond(system)
    exported = _exported(pc, 1)
    levels = _oracle_levels(exported)
    for l, (_, r, _) in enumerate(pc.tiles(1)[:-1]):
        long_rows = exported[l]["P"].nnz >= 64 * exported[l + 1]["A"].shape[0]
        print(f"{kw} precision={precision} level {l}: restriction width {r}")
        assert r in (1, 2, 4, 8, 16, 32) or (r == 256 and long_rows and autotune), (l, r)
    b = np.random.default_rng(3).standard_normal((system.n, 2))
    got = pc.vcycle(1, torch.from_numpy(b).cuda(), 1).cpu().numpy()
    for k in range(2):
        want = o.vcycle(levels, b[:, k])
        err = np.abs(got[:, k] - want).max() / np.abs(want).max()
        assert err <= TOL[precision], (kw, k, err)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("kw", [dict(nx=150, ny=121, coarse_max=8), dict(nx=400, ny=40, Lx=10.0, coarse_max=8), "batch"], ids=str)
def test_restriction_without_a_residual(lib, kw, precision):
    """FP32 levels below the finest of a 2D mesh restrict by R b - (R A) x where the product has no more entries
    than A: no residual is formed there (the launch counters say so) and the cycle is the oracle's; FP64
    levels keep the residual."""
    if kw == "batch":
        runs = [lib.Params(precision=precision, coarse_max=8, nx=a, ny=b) for a, b in ((133, 80), (97, 141), (60, 61))]
        p = runs[0]
    else:
        runs, p = None, lib.Params(precision=precision, **kw)
    system = lib.System(lib.Mesh(p, runs=runs), p)
    pc = lib.Precond(system)
    levels = _oracle_levels(_exported(pc, 1))
    assert len(levels) >= 3
    b = np.random.default_rng(11).standard_normal((system.n, 2))
    torch.cuda.synchronize()
    lib.profile_read(reset=True)
    got = pc.vcycle(1, torch.from_numpy(b).cuda(), 2).cpu().numpy()
    launches = {k: v["launches"] for k, v in lib.profile_read(reset=True).items()}
    residuals = sum(v for k, v in launches.items() if k.startswith("vresidual_coarse"))
    restrictions = sum(v for k, v in launches.items() if k.startswith("restrict_coarse"))
    assert restrictions == 2 * (len(levels) - 2)
    assert residuals < restrictions if precision == 1 else residuals == restrictions
    for k in range(2):
        want = o.vcycle(levels, b[:, k], x0=o.vcycle(levels, b[:, k]))
        err = np.abs(got[:, k] - want).max() / np.abs(want).max()
        assert err <= TOL[precision], (kw, k, err)
