"""The Krylov basis at its edges: nearly exhausted Krylov spaces (the second Gram-Schmidt correction is then
not small and is formed in FP64), bases past the 16-vector chunks of the dot products, runs of one block
and of several.  Steps solved to rtol 1e-13 equal the oracle's; the fields' error is below
cond(A) * rtol * |x| / |field| <= 1.5e2 * 1e-13 * 10 = 1.5e-10 on these meshes (cond(A) <= 143)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [dict(nx=1, ny=1, restart=12), dict(nx=2, ny=1, restart=20), dict(nx=3, ny=2, restart=30),
                                dict(nx=17, ny=15, restart=16), dict(nx=17, ny=16, restart=17),
                                dict(nx=48, ny=40, restart=64), dict(dim=3, nx=2, ny=2, nz=2, restart=40)])
@pytest.mark.parametrize("precision", [0, 1])
def test_step_matches_the_oracle_for_exhausted_and_long_bases(lib, kw, precision):
    import torch
    from oracle import ch_oracle as o
    from paper_2204_03575_gb300 import inputs
    geo = {k: v for k, v in kw.items() if k != "restart"}
    p = lib.Params(rtol=1e-13, max_iter=1000, precision=precision, **kw)
    system = lib.System(lib.Mesh(p), p)
    state = lib.State(system, lib.Precond(system))
    pp, pn = inputs.initial_state(system.n, 0.33, 0.33, 0.01, seed=3)
    state.set(torch.from_numpy(pp).cuda(), torch.from_numpy(pn).cuda())
    state.step()
    got = {k: v.cpu().numpy() for k, v in state.get().items()}
    ref = o.Solver(o.Params(**geo))
    nxt = ref.step(o.initial(ref.N, pp, pn))
    for name in ("phi_p", "phi_nfa", "mu_p", "mu_nfa"):
        r = getattr(nxt, name)
        err = np.abs(got[name] - r).max() / np.abs(r).max()
        assert err <= 1.5e-10, f"{name}: relative error {err:.3e}"
