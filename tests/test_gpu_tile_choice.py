"""High smoothing degrees in FP32: a tile recomputes a halo as deep as the degree, so from some degree on a launch per
step is faster on meshes of many tiles (ch_params.cheb_degree goes to 16).  The launch counters say which form
ran: one launch per pass by tiles, one per step otherwise.  Both are the oracle's V-cycle to the bound of the
other FP32 V-cycle tests."""
import numpy as np
import pytest
import torch

from oracle import ch_oracle as o
from test_zy_vcycle_oracle import TOL, _exported, _oracle_levels

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw,degree,tiled", [(dict(nx=256, ny=256), 15, True), (dict(nx=300, ny=97), 16, True),
                                             (dict(nx=512, ny=512), 8, True), (dict(nx=700, ny=700), 16, False),
                                             (dict(nx=700, ny=700), 5, True), ("batch", 16, False), ("batch", 5, True)], ids=str)
def test_tiles_where_they_are_faster(lib, kw, degree, tiled):
    p = lib.Params(precision=1, cheb_degree=degree, **({} if kw == "batch" else kw))
    runs = None
    if kw == "batch":
        runs = [lib.Params(precision=1, cheb_degree=degree, nx=150 + 7 * r, ny=200 - 9 * r) for r in range(16)]
    system = lib.System(lib.Mesh(p, runs=runs), p)
    pc = lib.Precond(system)
    levels = _oracle_levels(_exported(pc, 1))
    b = np.random.default_rng(2).standard_normal((system.n, 2))
    bd = torch.from_numpy(b).cuda()
    lib.profile_read(reset=True)
    got = pc.vcycle(1, bd).cpu().numpy()
    steps = lib.profile_read(reset=True)["cheb_step_f32"]["launches"]
    assert steps == (2 if tiled else 2 * degree - 1)
    for k in range(2):
        want = o.vcycle(levels, b[:, k])
        assert np.abs(got[:, k] - want).max() / np.abs(want).max() <= TOL[1]
