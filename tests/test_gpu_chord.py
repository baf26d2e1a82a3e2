"""The chord tally's voxel traversal against the oracle's chord splitter on tracks that no random
number bends: along and across faces, steps shorter and longer than a voxel, leaving the grid."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("h", [(1.0, 1.0, 1.0), (0.5, 0.5, 0.5), (0.2, 0.35, 0.15), (2.0, 1.0, 0.5)])
@pytest.mark.parametrize("u", [(0.0, 0.0, 1.0), (0.0, 0.0, -1.0), (1.0, 0.0, 0.0), (-0.6, 0.0, 0.8), (0.5, -0.7, 0.4),
                               (-1.0, -1.0, -1.0)])
def test_straight_tracks_match_the_oracle(sde_gpu, oracle_lib, h, u):
    """One history without straggling, scattering or events: the tally differs from the oracle's
    FP64 split by FP32 positions only.  Along a track of 200 steps of 0.5 mm in a 24 mm box a
    position is off by at most 200 roundings of half an ulp of 24 (2e-4 mm), so a face moves
    that much of a step's deposit (4e-4 of it per crossed face, FP32 energies 1e-4 more)."""
    from sde_workloads import WATER, Workload, pencil
    n = [int(round(24.0 / v)) for v in h]
    wl = Workload("box", tuple(n), h, (0.0, 0.0, 0.0), np.ones((n[2], n[1], n[0]), np.float32),
                  np.zeros((n[2], n[1], n[0]), np.uint8), [WATER], pencil(90.0, 1, 12.03, 11.98, 12.01, u=u))
    _, eg, bg = sde_gpu.run_workload(wl, seed=3, tally_mode=1, physics_mask=0)
    _, eo, bo = oracle_lib.run_workload(wl, seed=3, tally_mode=1, physics_mask=0)
    assert bg["incident"] == bg["deposited"] + bg["escaped"] + bg["removed"] and bg["steps"] == bo["steps"]
    step = bo["deposited"] / bo["steps"]
    assert np.abs(eg.astype(np.float64) - eo.astype(np.float64)).max() <= 4e-3 * step, step
