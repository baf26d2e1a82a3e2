"""The weight gradient's copying warps and the fillings of its slots (CPU).  A warp waits for a slot by
the parity of how often it was released, so no filling of a slot may complete without the warp:
otherwise a warp that is held up finds the slot released twice, waits for a third time that does
not come, and the call ends in a timeout although its sums were right."""
import itertools

import pytest

import paper_2511_03115_gb300 as S

WARPS = 8


@pytest.mark.parametrize("n,D,H,W", [(1, 192, 128, 128), (1, 96, 64, 64), (1, 300, 64, 128), (2, 5, 6, 33), (1, 40, 50, 256),
                                     (1, 200, 60, 14), (1, 200, 60, 40)])
def test_no_filling_completes_without_a_copying_warp(n, D, H, W):
    """The copies of kernel k_wgrad_ring: dy copy i is warp i % 8's; in the long order warp w brings group
    w % gpp of plane w / gpp, in the short order the planes' copies go round the warps."""
    for Cin, Cout in itertools.product((16, 32, 64, 96, 192), range(16, 129, 16)):
        try:
            b = S.conv3d_wgrad_ring(n, D, H, W, Cin, Cout)
        except S.SdeError:
            continue
        nd, gpp, part = b["ns"] * Cout // 8, b["gpp"], set(range(b["copiers"]))
        assert b["copiers"] <= WARPS and b["arrivals"] in (1, b["copiers"])
        arrive = part if b["arrivals"] > 1 else {0}
        dy = {i % WARPS for i in range(nd)}
        if b["order"]:  # dy rows and planes fill one slot
            planes = set(range(3 * gpp))
            assert dy | planes <= part  # every copy is made
            assert dy | planes | arrive == part, b
        else:
            assert dy <= part
            assert dy | arrive == part, b
            for turn in range(nd, nd + 8 * gpp, gpp):
                brings = {(turn + q) % WARPS for q in range(gpp)}
                assert brings <= part and brings | arrive == part, b
