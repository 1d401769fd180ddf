"""The weight-gradient kernels at the edges of their tiles (segments of at most 160 pixels, strips of image
rows) against the CPU oracle's gradients.  Both sides round activations and output gradients to BF16 at
the same places, so they differ where FP32 accumulation moves a value across a rounding boundary:
2e-2 per layer in the L2 norm, as in the other gradient tests."""
import numpy as np
import pytest

from oracle import warmstart_oracle as wo

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,B", [(1, 1, 1), (1, 16, 2), (2, 160, 1), (3, 161, 2), (5, 321, 1), (40, 17, 3), (97, 33, 1)])
def test_gradients_at_tile_edges(lib, H, W, B):
    import torch
    rng = np.random.default_rng(5)
    net = lib.WarmStartNet(H, W, max_batch=max(B, 2))
    theta = (rng.standard_normal(net.nparams) * 0.2).astype(np.float32)
    # padded entries (input channels 12-15, output channels 4-7) are ignored by the network
    theta[:9 * 16 * 32].reshape(9, 16, 32)[:, 12:] = 0
    theta[-(9 * 32 * 8 + 8):-8].reshape(9, 32, 8)[:, :, 4:] = 0
    theta[-4:] = 0
    net.set_params(theta)
    norm = (rng.standard_normal(8) * 0.05, rng.uniform(0.5, 2.0, 8), np.array([0.7, 1.2, 0.5, 0.9]))
    net.set_norm(*norm)
    x = rng.standard_normal((B, H * W, 4)).astype(np.float32)
    q = (x - 0.1 * rng.standard_normal(x.shape)).astype(np.float32)
    q2 = (q - 0.1 * rng.standard_normal(x.shape)).astype(np.float32)
    n = (x + 0.1 * rng.standard_normal(x.shape)).astype(np.float32)
    net.train_step(*(torch.from_numpy(a).cuda() for a in (x, q, q2, n)), 0.0)
    g = net.get_params()[1]
    img = lambda a: a.astype(np.float64).reshape(B, H, W, 4)
    _, ref = wo.loss_and_grads(theta.astype(np.float64), img(x), img(q), img(q2), img(n), norm, bf=True, lap=0.0)
    k = 0
    for m in (9 * 16 * 32, 32, 9 * 32 * 32, 32, 9 * 32 * 8, 8):
        a, b = g[k:k + m], ref[k:k + m]
        assert np.linalg.norm(a - b) <= 2e-2 * max(np.linalg.norm(b), 1e-12), (k, m)
        k += m


def test_inputs_off_the_vector_alignment_give_the_same_results(lib):
    """The states are read four channels at a time where they are aligned for it; a contiguous view that
    starts 8 bytes off gives the same prediction and gradients, bit for bit."""
    import torch
    H, W, B = 9, 21, 2
    rng = np.random.default_rng(6)
    net = lib.WarmStartNet(H, W, max_batch=B)
    net.set_params((rng.standard_normal(net.nparams) * 0.2).astype(np.float32))
    hist = [torch.from_numpy(rng.standard_normal((B, H * W, 4))).cuda() for _ in range(3)]

    def off(t):
        buf = torch.empty(t.numel() + 1, dtype=t.dtype, device="cuda")[1:].view(t.shape)
        buf.copy_(t)
        assert buf.data_ptr() % 32 == 8
        return buf

    a = net.predict(*(t[0].contiguous() for t in hist))
    b = net.predict(*(off(t[0].contiguous()) for t in hist))
    assert torch.equal(a, b)
    p = lib.Params(nx=W - 1, ny=H - 1)
    system = lib.System(lib.Mesh(p), p)
    la = net.train_residual(system, *hist, 0.0)
    ga = net.get_params()[1]
    lb = net.train_residual(system, *(off(t) for t in hist), 0.0)
    assert la == lb
    np.testing.assert_array_equal(ga, net.get_params()[1])
