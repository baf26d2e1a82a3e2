"""The convolution's epilogue groups and the phases of the tensor-memory accumulators.  A group waits
for an accumulator by the parity of how often it was filled, so it must not be two fillings
behind: on the CPU, for the plans of a sweep of shapes; on the GPU, the results of layers whose items
are a single block of sixteen columns, many per multiprocessor."""
import itertools

import pytest

import paper_2511_03115_gb300 as S


def test_no_group_is_two_fillings_of_an_accumulator_behind():
    """The groups' walk of kernel k_conv3d_brick: blocks of sixteen columns of all tiles of a CTA's items,
    in turn; item i is in accumulator i % nacc.  Every item has been waited for from its
    accumulator's previous one on, and each block is one group's."""
    walks = set()
    for D, H, W in itertools.product((1, 12, 700), (1, 2, 3, 5, 8, 16, 31, 128), (1, 2, 8, 15, 30, 62, 63, 126, 128, 129, 256)):
        for Cin, Cout in itertools.product((16, 32, 96, 192), (16, 32, 48, 80, 96, 128, 256)):
            try:
                b = S.conv3d_plan(5000 // D, D, H, W, Cin, Cout)
            except S.SdeError:
                continue
            walks.add((b["tiles"] * (b["Cp"] // 16), b["nacc"], b["groups"]))
    assert any(blocks == 1 for blocks, _, _ in walks)
    for blocks, nacc, groups in walks:
        taken = []
        for g in range(groups):
            waited = -1
            for at in range(g, 40 * blocks, groups):
                item = at // blocks
                assert item < nacc or waited >= item - nacc, (blocks, nacc, groups, g, item)
                waited = item
                taken.append(at)
        assert sorted(taken) == list(range(40 * blocks))


@pytest.mark.gpu
@pytest.mark.parametrize("n,shape,Cin,Cout", [(64, (16, 8, 8), 16, 16), (1, (700, 8, 8), 32, 16), (1, (700, 1, 128), 32, 16),
                                              (1, (1250, 1, 256), 16, 16), (3, (400, 3, 29), 16, 48)])
def test_single_block_items_match_float64(sde_gpu, n, shape, Cin, Cout):
    """Items of one, two and three blocks.  FP32 accumulation of at most 864 products, as for the other
    convolution tests: 1e-5 of the largest value."""
    import torch
    g = torch.Generator().manual_seed(Cin + Cout + n)
    x = torch.randn(n, *shape, Cin, generator=g).to(torch.bfloat16)
    w = (0.2 * torch.randn(Cout, 27, Cin, generator=g)).to(torch.bfloat16)
    y = S.conv3d(S.to_pcg(x.cuda()), w.cuda(), fp32=True)
    S.denoise_status()
    wt = w.double().reshape(Cout, 3, 3, 3, Cin).permute(0, 4, 1, 2, 3)
    ref = torch.nn.functional.conv3d(x.double().permute(0, 4, 1, 2, 3), wt, padding=1).permute(0, 2, 3, 4, 1)
    assert (y.cpu().double() - ref).abs().max().item() <= 1e-5 * ref.abs().max().item() + 1e-5


@pytest.mark.gpu
def test_a_batch_of_small_volumes_is_denoised_as_each_alone(sde_gpu):
    import torch
    n, shape = 32, (24, 8, 8)
    many, one = S.Denoiser(*shape, batch_max=n, seed=4), S.Denoiser(*shape, batch_max=1, seed=4)
    p = many.get_params()
    many.split(p)[10][0][:] = 0.02  # the untrained output layer is zero
    many.set_params(p)
    one.set_params(p)
    g = torch.Generator(device="cuda").manual_seed(8)
    low = torch.rand(n, *shape, device="cuda", generator=g)
    rho = 0.5 + torch.rand(*shape, device="cuda", generator=g)  # a batch has one density map
    out = many.infer(low, rho)
    S.denoise_status()
    assert not torch.equal(out, low)
    for i in range(n):
        assert torch.equal(out[i], one.infer(low[i].contiguous(), rho)), i
    S.denoise_status()
    many.close()
    one.close()
