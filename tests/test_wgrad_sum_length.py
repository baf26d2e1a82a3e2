"""How many K steps a CTA of the weight gradient adds up in one FP32 sum: never more than the row-block
plan, whose errors are the measure (an accumulator drops up to 2^-23 of itself a step)."""
import itertools

import pytest

import paper_2511_03115_gb300 as S


def steps(b):
    return -(-b["items"] // b["G"]) * b["kst"]


@pytest.mark.parametrize("W", [1, 2, 5, 8, 12, 15, 16, 17, 18, 20, 24, 30, 33, 40, 48, 50, 64, 75, 100, 127, 128, 200, 250, 256])
def test_sums_are_no_longer_than_the_row_block_plans(W):
    for n, D, H in ((1, 24, 24), (1, 64, 63), (1, 192, 128), (2, 5, 7), (1, 45, 61)):
        for Cin, Cout, sms in itertools.product(range(16, 193, 16), (16, 32, 48, 64, 80, 128), (152, 132)):
            try:
                p = S.conv3d_wgrad_plan(n, D, H, W, Cin, Cout, sms=sms)
            except S.SdeError:
                continue
            b = S.conv3d_wgrad_ring(n, D, H, W, Cin, Cout, sms=sms)
            assert steps(b) <= steps(p) and b["G"] <= b["items"], (n, D, H, Cin, Cout, sms)
            # no wave of CTAs more than that takes
            one = max(1, sms // (Cin // (8 * b["load"])))
            if not b["order"] and b["G"] > one:
                assert steps(dict(b, G=one * ((b["G"] - 1) // one))) > steps(p)


@pytest.mark.gpu
@pytest.mark.parametrize("Cin,Cout,shape", [(192, 32, (192, 128, 16)), (192, 32, (192, 128, 24)), (192, 48, (100, 64, 8)),
                                            (64, 32, (60, 61, 20))])
def test_long_sums_of_narrow_rows_match_float64(sde_gpu, Cin, Cout, shape):
    import torch
    b = S.conv3d_wgrad_ring(1, *shape, Cin, Cout)
    assert b["order"] == 0
    g = torch.Generator(device="cuda").manual_seed(Cin + Cout + shape[2])
    x = (0.5 * torch.randn(1, *shape, Cin, device="cuda", generator=g)).to(torch.bfloat16)
    dy = (0.5 * torch.randn(1, *shape, Cout, device="cuda", generator=g)).to(torch.bfloat16)
    dw = torch.zeros(Cout, 27, Cin, device="cuda")
    S.conv3d_wgrad(S.to_pcg(x), S.to_pcg(dy), dw)
    S.denoise_status()
    ref = torch.zeros(Cout, 27, Cin, dtype=torch.float64, device="cuda")
    D, H, W = shape
    xp = torch.nn.functional.pad(x.double(), (0, 0, 1, 1, 1, 1, 1, 1))
    for t in range(27):
        w = xp[:, t // 9:t // 9 + D, t // 3 % 3:t // 3 % 3 + H, t % 3:t % 3 + W]
        ref[:, t] = dy.double().reshape(-1, Cout).T @ w.reshape(-1, Cin)
    err, top = (dw.double() - ref).abs().max().item(), ref.abs().max().item()
    assert err <= steps(b) * 2.0 ** -23 * top + 1e-4
