"""Runs too small to fill the GPU share their histories among fewer warps and lanes: the tally and the
balance stay those of any other split of the same histories."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 33, 607, 609, 9_729, 19_455, 19_457, 38_913, 60_001])
@pytest.mark.parametrize("params", [{}, {"theta_cut_sigmas": 2.5}, {"theta_cut_sigmas": 2.5, "secondary_fraction": 0.6}])
def test_any_split_of_a_small_run_gives_the_same_tally(sde_gpu, n, params):
    """The whole run, its two uneven parts, and other launch shapes (one warp a block, refills of
    single lanes): whole numbers, so equal."""
    from sde_workloads import water100
    wl = water100(n)
    with sde_gpu.SdeDose(wl, **params) as d:
        d.run(wl.spots, seed=5)
        _, ref, bal = d.fetch(dose=False)
        assert bal["histories"] == n and bal["incident"] == bal["deposited"] + bal["escaped"] + bal["removed"]
        cut = n // 3
        d.reset()
        d.run(wl.spots, seed=5, first=0, count=cut)
        d.run(wl.spots, seed=5, first=cut)
        _, parts, bal2 = d.fetch(dose=False)
        assert np.array_equal(ref, parts) and bal == bal2
        for tuning in ({"warps_per_block": 1, "blocks_per_sm": 2}, {"refill_min": 4, "batch": 64}):
            d.set_tuning(**tuning)
            d.reset()
            d.run(wl.spots, seed=5)
            _, other, bal3 = d.fetch(dose=False)
            assert np.array_equal(ref, other) and bal == bal3
