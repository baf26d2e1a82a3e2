"""A value that is not finite in one input channel reaches the weight gradients of that channel alone: on
the CPU, that no window of the weight gradient reads another channel's values; on the GPU,
infinities at the rows' ends in one channel against float64 in the others."""
import itertools

import pytest

import paper_2511_03115_gb300 as S

WIDTHS = [1, 2, 3, 5, 8, 13, 14, 15, 16, 17, 18, 30, 31, 32, 33, 48, 63, 75, 100, 126, 127, 128, 129, 143, 200, 240, 254, 256]


@pytest.mark.parametrize("W", WIDTHS)
def test_windows_stay_in_their_channels(W):
    """Position f of the plane slots holds group f / (Yb P) mod gpp (those from `load` on are never
    written) and column f mod P, of which the first and the last are zero padding."""
    seen = set()
    for n, D, H in ((1, 24, 24), (1, 192, 128), (1, 700, 60), (2, 5, 7)):
        for Cin, Cout in itertools.product((16, 32, 96, 192), (16, 32, 48, 64, 80, 128)):
            try:
                b = S.conv3d_wgrad_ring(n, D, H, W, Cin, Cout)
            except S.SdeError:
                continue
            P, Yb, gpp, kst, back, load = b["P"], b["Ty"] + 2, b["gpp"], b["kst"], b["back"], b["load"]
            key = (b["order"], b["Ty"], gpp, kst, back, load, b["nt"], b["xoff"], b["drun"])
            if key in seen:
                continue
            seen.add(key)
            used = b["drun"] // 16
            assert Cin % (8 * load) == 0 and 0 <= back < 16 and (back == 0 or kst > 1) and load in (1, gpp)
            assert used + back <= 16 * kst
            for g, r, t, j in itertools.product(range(load), range(3), range(b["nt"]), range(kst)):
                first = (g * Yb + r) * P + b["xoff"] + t + 16 * j - (back if j == kst - 1 else 0)
                for f in range(first, first + 16):
                    group, x = f // (Yb * P) % gpp, f % P
                    assert group == g or group >= load or x in (0, P - 1), (b, g, r, t, j)
            # each position of dy once, the last step's at its end: it meets the x of its own place
            for k in range(used):
                j = min(k // 16, kst - 1)
                at = k + (back if j == kst - 1 else 0)
                assert at // 16 == j and k == at - (back if j == kst - 1 else 0)


@pytest.mark.gpu
@pytest.mark.parametrize("Cin,Cout,shape,order", [(32, 32, (3, 5, 17), 0), (48, 48, (4, 9, 33), 0), (32, 80, (3, 4, 75), 0),
                                                  (32, 16, (5, 6, 8), 0), (48, 64, (6, 5, 3), 0), (16, 96, (4, 6, 1), 0),
                                                  (176, 32, (40, 50, 128), 1), (192, 32, (28, 61, 128), 1)])
@pytest.mark.parametrize("bad", [8, 7])
def test_other_channels_gradients_stay_finite(sde_gpu, Cin, Cout, shape, order, bad):
    """1e-4 of the largest gradient, as for the other weight-gradient tests."""
    import torch
    b = S.conv3d_wgrad_ring(1, *shape, Cin, Cout)
    assert b["order"] == order
    g = torch.Generator(device="cuda").manual_seed(Cin + 3 * Cout)
    x = (0.5 * torch.randn(1, *shape, Cin, device="cuda", generator=g)).to(torch.bfloat16)
    dy = (0.5 * torch.randn(1, *shape, Cout, device="cuda", generator=g)).to(torch.bfloat16)
    x[:, :, :, :16, bad] = float("inf")
    x[:, :, :, -16:, bad] = float("nan")
    dw = torch.zeros(Cout, 27, Cin, device="cuda")
    S.conv3d_wgrad(S.to_pcg(x), S.to_pcg(dy), dw)
    S.denoise_status()
    fine = [c for c in range(Cin) if c != bad]
    ref = torch.zeros(Cout, 27, len(fine), dtype=torch.float64, device="cuda")
    D, H, W = shape
    xp = torch.nn.functional.pad(x[..., fine].double(), (0, 0, 1, 1, 1, 1, 1, 1))
    for t in range(27):
        w = xp[:, t // 9:t // 9 + D, t // 3 % 3:t // 3 % 3 + H, t % 3:t % 3 + W]
        ref[:, t] = dy.double().reshape(-1, Cout).T @ w.reshape(-1, len(fine))
    got = dw[:, :, fine].double()
    assert torch.isfinite(got).all()
    assert (got - ref).abs().max().item() <= 1e-4 * ref.abs().max().item() + 1e-4
    assert not torch.isfinite(dw[:, :, bad]).all()
