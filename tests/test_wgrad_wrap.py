"""The weight gradient where its ring of planes wraps: on the CPU, that every MMA of a cut window has a
width the tensor core takes; on the GPU, wide rows against float64 over more planes than the
ring holds."""
import itertools

import pytest

import paper_2511_03115_gb300 as S

WIDTHS = [1, 7, 8, 15, 16, 17, 31, 33, 63, 64, 75, 100, 127, 128, 129, 160, 200, 224, 239, 240, 241, *range(244, 257)]


def wgrad64(x, dy):
    """dw [Cout, 27, Cin] in float64 of channels-last x and dy."""
    import torch
    n, D, H, W, Cin = x.shape
    Cout = dy.shape[-1]
    ref = torch.zeros(Cout, 27, Cin, dtype=torch.float64, device=x.device)
    xp = torch.nn.functional.pad(x.double(), (0, 0, 1, 1, 1, 1, 1, 1))
    for t in range(27):
        w = xp[:, t // 9:t // 9 + D, t // 3 % 3:t // 3 % 3 + H, t % 3:t % 3 + W]
        ref[:, t] = dy.double().reshape(-1, Cout).T @ w.reshape(-1, Cin)
    return ref


@pytest.mark.parametrize("W", WIDTHS)
def test_every_mma_has_a_width_of_sixteen_columns_multiples(W):
    """An MMA of M = 128 takes N in multiples of 16 up to 256.  The short order's ring moves on by a plane
    an item, so a window of three planes is cut after one and after two of them."""
    for n, D, H in ((1, 24, 24), (1, 64, 64), (1, 192, 128), (2, 5, 7)):
        for Cin, Cout in itertools.product((16, 32, 96, 144, 192), range(16, 129, 16)):
            try:
                S.conv3d_wgrad_plan(n, D, H, W, Cin, Cout)
            except S.SdeError:
                continue
            b = S.conv3d_wgrad_ring(n, D, H, W, Cin, Cout)
            columns, plane = 8 * b["ngr"], 8 * b["gpp"] * (b["Ty"] + 2)
            widths = [columns]
            if not b["order"]:
                widths += [plane, columns - plane, 2 * plane, columns - 2 * plane]
            assert all(16 <= w <= 256 and w % 16 == 0 for w in widths), (n, D, H, Cin, Cout, b, widths)


@pytest.mark.gpu
@pytest.mark.parametrize("Cin,Cout,shape", [(96, 64, (24, 24, 248)), (96, 64, (24, 24, 253)), (96, 64, (24, 24, 256)),
                                            (96, 48, (24, 24, 256)), (96, 128, (24, 24, 206)), (32, 64, (24, 40, 250))])
def test_wide_rows_match_float64(sde_gpu, Cin, Cout, shape):
    """FP32 accumulation over at most 2e4 positions per sum: 1e-4 of the largest gradient, as for the
    other weight-gradient tests."""
    import torch
    b = S.conv3d_wgrad_ring(1, *shape, Cin, Cout)
    assert b["order"] == 0 and b["items"] // b["G"] + 2 > b["XS"]
    g = torch.Generator(device="cuda").manual_seed(Cin + Cout)
    x = (0.5 * torch.randn(1, *shape, Cin, device="cuda", generator=g)).to(torch.bfloat16)
    dy = (0.5 * torch.randn(1, *shape, Cout, device="cuda", generator=g)).to(torch.bfloat16)
    dw = torch.zeros(Cout, 27, Cin, device="cuda")
    S.conv3d_wgrad(S.to_pcg(x), S.to_pcg(dy), dw)
    S.denoise_status()
    ref = wgrad64(x, dy)
    assert (dw.double() - ref).abs().max().item() <= 1e-4 * ref.abs().max().item() + 1e-4
