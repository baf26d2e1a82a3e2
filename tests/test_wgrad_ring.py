"""The weight gradient's rings: on the CPU, that every copy, operand window and accumulator of the
layout stays inside its buffer and that the taps it forms are each tap once, over every
position; on the GPU, the gradient against float64 at the edges of the layout's choices."""
import itertools

import pytest

import paper_2511_03115_gb300 as S

HEADER, CAP = 1024, 227 * 1024
WIDTHS = [1, 2, 8, 14, 15, 16, 17, 30, 32, 33, 64, 75, 112, 127, 128, 129, 130, 192, 255, 256]


@pytest.mark.parametrize("W", WIDTHS)
@pytest.mark.parametrize("n,D,H", [(2, 5, 6), (1, 700, 120), (1, 150, 64)])
def test_rings_stay_inside_their_buffers(W, n, D, H):
    for Cin, Cout in itertools.product(range(16, 193, 16), range(16, 129, 16)):
        try:
            p = S.conv3d_wgrad_plan(n, D, H, W, Cin, Cout)
        except S.SdeError:  # a refused shape stays refused
            with pytest.raises(S.SdeError):
                S.conv3d_wgrad_ring(n, D, H, W, Cin, Cout)
            continue
        b = S.conv3d_wgrad_ring(n, D, H, W, Cin, Cout)
        ns, nt, kst, ra, P, Ty, gpp, ngr = (b[k] for k in ("ns", "nt", "kst", "ra", "P", "Ty", "gpp", "ngr"))
        Yb = Ty + 2
        assert P == W + 2 and H % Ty == 0 and b["items"] == n * (H // Ty) * D and ra == 256 * kst
        assert b["drun"] <= ra and b["drun"] % 16 == 0 and Cin % (8 * gpp) == 0
        assert ns * Cout <= 128  # at most sixteen copies, two per copying warp
        assert ngr % 2 == 0 and 8 * ngr <= 256 and nt * 8 * ngr <= 512
        assert (3 * gpp - 1) * Yb + 3 <= ngr <= (3 * gpp - 1) * Yb + 4
        # dy slots: ns x Cout/8 runs; M = 128 reads sixteen runs from a slot's start
        assert b["dslot"] == ns * (Cout // 8) * ra
        assert HEADER + (b["DS"] - 1) * b["dslot"] + 16 * ra <= b["smem"] <= CAP
        assert b["x_off"] == HEADER + b["DS"] * b["dslot"]
        # plane slots at one stride over groups, rows and planes
        assert b["xslot"] == gpp * Yb * P * 16
        # the first window starts one position before a slot at most, the last one ends inside
        assert b["xoff"] >= -1
        top = (ngr - 1) * P + b["xoff"] + nt - 1 + 16 * kst - 1  # from the first of three planes
        assert b["x_off"] + (b["XS"] - 3) * b["xslot"] + 16 * (top + 1) <= b["smem"]
        assert 2 <= b["DS"] <= 4 and b["XS"] <= 12 and max(ra, P * 16) < 1 << 18
        assert b["XS"] == 3 * b["DS"] if b["order"] else b["XS"] >= b["DS"] + 2
        if b["order"]:  # the row-block plan's items and K steps
            assert (Ty, kst, b["items"], b["G"]) == (p["Ty"], p["kst"], p["items"], p["G"])
        assert 1 <= b["G"] <= b["items"]


@pytest.mark.parametrize("Cin,Cout,n,D,H,W", [(16, 32, 1, 4, 4, 16), (16, 48, 1, 4, 4, 33), (16, 128, 1, 4, 4, 17),
                                              (96, 32, 1, 192, 128, 128), (32, 16, 1, 192, 128, 128),
                                              (192, 64, 1, 96, 64, 64)])
def test_every_tap_is_formed_once_from_every_position(Cin, Cout, n, D, H, W):
    """The kernel's sums restated on one item: every (row group, offset, copy) that is stored is one
    tap, and its positions are the item's voxels, each once, against the shifted x."""
    b = S.conv3d_wgrad_ring(n, D, H, W, Cin, Cout)
    P, Ty, Yb, K = b["P"], b["Ty"], b["Ty"] + 2, 16 * b["kst"]
    taps = {}
    for t, q, i in itertools.product(range(b["nt"]), range(b["ngr"]), range(b["ns"])):
        r, pg = q % Yb, q // Yb
        dz, g, dx = pg // b["gpp"], pg % b["gpp"], t + i - 1
        if r > 2 or dz > 2 or (b["ns"] == 2 and i == 1 and t == 0):
            continue
        assert (g, dz, r, dx) not in taps
        pairs = {}
        for k in range(K):
            if 16 * k >= b["drun"]:
                continue  # zeros
            f = k + b["dyx"] - i + 1  # dy position in the padded rows from (y0, x = -1)
            yv, xv = divmod(f, P)
            if not (0 <= yv < Ty and 1 <= xv <= W):
                continue  # padding: zero
            at = r * P + k + b["xoff"] + t  # x position in the plane's rows from (y0 - 1, x = -1)
            pairs[(yv, xv - 1)] = divmod(at, P)
        for v in itertools.product(range(Ty), range(W)):
            want = (v[0] + r, v[1] + dx + 1)
            if v in pairs:
                assert pairs[v] == want
            else:
                assert not 1 <= want[1] <= W  # only products with the zero border are left out
        taps[(g, dz, r, dx)] = True
    assert len(taps) == 27 * b["gpp"]


@pytest.mark.gpu
@pytest.mark.parametrize("Cin,Cout,n,shape", [
    (16, 16, 1, (1, 1, 16)), (32, 32, 2, (3, 5, 17)), (48, 48, 1, (2, 9, 33)), (96, 64, 1, (7, 3, 64)),
    (192, 80, 1, (2, 2, 31)), (16, 128, 2, (4, 3, 130)), (64, 112, 1, (5, 4, 15)), (144, 32, 1, (40, 2, 128)),
    (32, 16, 1, (2, 37, 256)), (80, 96, 1, (3, 6, 1)), (48, 32, 1, (1, 200, 128)),
    # sums long enough for the row-block order, with one and several rows an item
    (176, 32, 1, (40, 50, 128)), (192, 64, 1, (66, 36, 64)), (192, 16, 1, (30, 60, 128))])
def test_wgrad_matches_float64(sde_gpu, Cin, Cout, n, shape):
    """FP32 accumulation over at most 2e4 positions per sum: 1e-4 of the largest gradient, as for the
    other weight-gradient tests; the call adds to what dw holds."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(Cin * 7 + Cout)
    D, H, W = shape
    x = (0.5 * torch.randn(n, D, H, W, Cin, device="cuda", generator=g)).to(torch.bfloat16)
    dy = (0.5 * torch.randn(n, D, H, W, Cout, device="cuda", generator=g)).to(torch.bfloat16)
    buf = torch.full((Cout * 27 * Cin + 1,), 2.0, device="cuda")
    dw = buf[1:].view(Cout, 27, Cin)  # 4-byte aligned only
    sde_gpu.conv3d_wgrad(sde_gpu.to_pcg(x), sde_gpu.to_pcg(dy), dw)
    sde_gpu.denoise_status()
    ref = torch.zeros(Cout, 27, Cin, dtype=torch.float64, device="cuda")
    xp = torch.nn.functional.pad(x.double(), (0, 0, 1, 1, 1, 1, 1, 1))
    for t in range(27):
        w = xp[:, t // 9:t // 9 + D, t // 3 % 3:t // 3 % 3 + H, t % 3:t % 3 + W]
        ref[:, t] = dy.double().reshape(-1, Cout).T @ w.reshape(-1, Cin)
    assert float(buf[0]) == 2.0
    assert (dw.double() - 2.0 - ref).abs().max().item() <= 1e-4 * ref.abs().max().item() + 1e-4
