"""The denoiser's parameter vectors: copies in and out, the update of every layer, and the packed
weights after an update."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(4, 4, 4), (8, 12, 20), (16, 32, 128)])
def test_update_reaches_every_layer_and_its_packed_weights(sde_gpu, shape):
    """Adam's first step from zero moments moves a parameter by -lr g / (|g| + 1e-8).  Rounding: the
    moments and their corrections cancel to 1e-5 (1 - 0.999 in FP32 is off by 2e-5 of itself, half
    of that under the root), the subtraction to half an ulp of the parameter on each side of the
    difference.  Gradients below 1e-3 of their layer's largest are left out: their sums over
    unordered atomics may change sign from one call to the next."""
    import torch
    S = sde_gpu
    rng = np.random.default_rng(3)
    net, fresh = S.Denoiser(*shape, batch_max=1, seed=1), S.Denoiser(*shape, batch_max=1, seed=2)
    p0 = net.get_params()
    p0 = (p0 + 0.02 * rng.standard_normal(p0.shape)).astype(np.float32)
    net.set_params(p0)
    assert np.array_equal(net.get_params(), p0)
    gen = torch.Generator(device="cuda").manual_seed(9)
    low = torch.rand(shape, device="cuda", generator=gen)
    rho = 0.5 + torch.rand(shape, device="cuda", generator=gen)
    high = 0.8 * low
    g, _ = net.gradients(low, rho, high)
    lr = 1e-2
    net.train_step(low, rho, high, lr=lr)
    S.denoise_status()
    p1 = net.get_params()
    step = p1.astype(np.float64) - p0
    want = -lr * g.astype(np.float64) / (np.abs(g.astype(np.float64)) + 1e-8)
    tol = 1e-4 * lr + 2.0 ** -22 * np.maximum(np.abs(p0), np.abs(p1))
    for i, parts in enumerate(zip(net.split(step), net.split(want), net.split(tol), net.split(g))):
        for s_, w_, t_, g_ in zip(*parts):
            big = np.abs(g_) > 1e-3 * np.abs(g_).max()
            assert big.any(), i
            assert (np.abs(s_ - w_) <= t_)[big].all(), i
    # a second network that is given the same parameters computes the same doses, bit for bit:
    # the packed weights after an update are those after a copy
    fresh.set_params(p1)
    a, b = net.infer(low, rho), fresh.infer(low, rho)
    S.denoise_status()
    assert torch.equal(a, b)
    assert not torch.equal(a, low)
    net.close()
    fresh.close()
