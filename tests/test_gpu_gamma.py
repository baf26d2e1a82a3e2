"""The gamma index on the GPU against the oracle's over the forms its search takes: grids one
voxel thin, anisotropic voxels, distances below and above a voxel, coarse and fine search steps."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,voxel,dta,steps", [
    ((5, 7, 130), (1.0, 1.0, 1.0), 0.5, 10), ((1, 40, 33), (1.0, 1.0, 1.0), 0.5, 10),
    ((9, 3, 1), (1.0, 0.5, 2.0), 1.3, 7), ((12, 20, 24), (1.0, 0.5, 2.0), 3.0, 5),
    ((16, 17, 19), (0.5, 0.5, 0.5), 2.0, 1), ((3, 4, 5), (1.0, 1.0, 1.0), 1.0, 50), ((1, 1, 1), (1.0, 1.0, 1.0), 1.0, 3)])
@pytest.mark.parametrize("noise", [0.02, 0.2])
def test_gamma_equals_the_oracle_gamma(sde_gpu, oracle_lib, shape, voxel, dta, steps, noise):
    """FP32 against FP64: a voxel's decision differs only where its smallest gamma is within
    FP32 rounding of 1 (about 1e-5 of them), so at most one voxel of these grids."""
    import torch
    from oracle import analysis as A
    g = torch.Generator().manual_seed(sum(shape) + steps)
    ref = (1.0 + torch.sin(torch.arange(int(np.prod(shape))) * 0.37)).reshape(shape).float()
    ref = ref * (1 + 0.02 * torch.randn(shape, generator=g))
    ev = ref * (1 + noise * torch.randn(shape, generator=g))
    got = sde_gpu.gamma3d(ref.cuda(), ev.cuda(), voxel, dta_mm=dta, steps=steps)
    want, passed, mask = A.gamma_pass_rate(ref.double().numpy(), ev.double().numpy(), voxel, dta_mm=dta,
                                           step_frac=steps, return_map=True)
    assert abs(got - want) <= 1.01 / mask.sum(), (got, want)


def test_gamma_of_doses_that_are_not_finite(sde_gpu):
    """A NaN or infinite evaluated dose fails at its voxel and spoils no other one; a NaN reference
    voxel is not evaluated."""
    import torch
    ref = torch.ones(6, 8, 40)
    ev = torch.ones(6, 8, 40)
    ev[2, 3, 10] = float("nan")
    ev[4, 5, 30] = float("inf")
    got = sde_gpu.gamma3d(ref.cuda(), ev.cuda(), (1.0, 1.0, 1.0))
    assert abs(got - (1 - 2 / ref.numel())) < 1e-9
    ref[0, 0, 0] = float("nan")
    got = sde_gpu.gamma3d(ref.cuda(), ev.cuda(), (1.0, 1.0, 1.0))
    assert abs(got - (1 - 2 / (ref.numel() - 1))) < 1e-9
