"""A learned step that runs out of device memory for its history fails with CH_ERR_OOM; called again, it and the steps after
it are those of a state that never failed, bit for bit.  The failure is made on the host (learned_probe.cu compiles the
library's own source with a counted allocator), one allocation after another."""
import ctypes

import numpy as np
import pytest

import probes

pytestmark = pytest.mark.gpu


def test_the_next_call_after_a_failed_allocation(lib, tmp_path):
    import torch
    from paper_2204_03575_gb300 import warmstart
    probe = probes.load(lib, "learned_probe.cu", tmp_path).learned_probe
    probe.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int] * 2 + [ctypes.c_void_p]
    nx, ny = 20, 17
    system = warmstart.make_system(nx, ny)
    pc, net = lib.Precond(system), warmstart.zero_net(nx, ny)
    torch.cuda.synchronize()

    def run(fail_at):
        x = np.zeros((system.n, 4))
        return probe(system._h, pc._h, net._h, 5, fail_at, x.ctypes.data), x

    status, want = run(0)
    assert status == lib.OK and np.isfinite(want).all()
    for fail_at in (1, 2, 3):
        status, x = run(fail_at)
        assert status == lib.ERR_OOM and np.array_equal(x, want), fail_at
