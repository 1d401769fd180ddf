"""A training call that runs out of device memory fails with CH_ERR_OOM and leaves the network usable: the next call
allocates what is missing and returns the same loss and gradients as a network that never failed.  The failure is made on
the host (warmstart_probe.cu compiles the library's own source with a counted allocator), one allocation after another."""
import ctypes

import numpy as np
import pytest

import probes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def probe(lib, tmp_path_factory):
    f = probes.load(lib, "warmstart_probe.cu", tmp_path_factory.mktemp("probe")).train_probe
    f.argtypes = [ctypes.c_void_p] * 2 + [ctypes.c_int] * 3 + [ctypes.c_void_p] * 5 + [ctypes.c_int] + [ctypes.c_void_p] * 2
    return f


@pytest.mark.parametrize("preconditioned", [False, True])
def test_the_next_call_after_a_failed_allocation(lib, probe, preconditioned):
    import torch
    from paper_2204_03575_gb300 import warmstart
    nx, ny, B = 24, 18, 3
    system = warmstart.make_system(nx, ny)
    pc = lib.Precond(system)
    gen = torch.Generator().manual_seed(5)
    q2 = 0.3 + 0.05 * torch.rand(B, system.n, 4, dtype=torch.float64, generator=gen)
    q = q2 + 1e-3 * torch.rand(B, system.n, 4, dtype=torch.float64, generator=gen)
    x = q + 1e-3 * torch.rand(B, system.n, 4, dtype=torch.float64, generator=gen)
    x, q, q2 = (t.cuda() for t in (x, q, q2))
    params = warmstart.init_params(lib.lib().ch_ws_nparams(), 1).astype(np.float32)
    norm = np.concatenate([np.full(8, 0.1), np.full(8, 2.0), np.ones(4)]).astype(np.float32)
    torch.cuda.synchronize()

    def run(fail_at):
        loss, grads = ctypes.c_float(), np.zeros(len(params), np.float32)
        status = probe(system._h, pc._h if preconditioned else None, ny + 1, nx + 1, B, params.ctypes.data, norm.ctypes.data,
                       x.data_ptr(), q.data_ptr(), q2.data_ptr(), fail_at, ctypes.addressof(loss), grads.ctypes.data)
        return status, loss.value, grads

    status, loss, grads = run(0)
    assert status == lib.OK and np.isfinite(loss) and np.abs(grads).max() > 0
    failed = 0
    for fail_at in range(1, 20):
        status, again, g = run(fail_at)
        assert again == loss and np.array_equal(g, grads), fail_at
        if status == lib.OK:  # past the call's last allocation
            break
        assert status == lib.ERR_OOM
        failed += 1
    assert failed == (7 if preconditioned else 5)
