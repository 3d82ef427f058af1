"""loc_estimate against the oracle at the edges of its kernels: bins that leave a quarter empty or end a
batch of eight early, rows that end within a 16-byte group, cells of a tile outside the grid, the sizes
on either side of the grouped second pass (32768 groups), disks that hold one cell, a part and all of
the map.  Tolerances as in test_gpu_estimate.py: states exact, sums to 1e-6, values to 1e-6."""
import numpy as np
import pytest

import paper_1910_00572_gb300 as loc
from oracle import readout as R

pytestmark = pytest.mark.gpu

SIZES = [(1, 1, 1), (3, 5, 2), (16, 16, 3), (17, 15, 5), (64, 64, 32), (101, 99, 36), (40, 25, 256),
         (364, 362, 33), (364, 360, 7), (520, 509, 9), (511, 513, 24), (520, 504, 6)]


@pytest.mark.parametrize("storage", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("H,W,K", SIZES, ids=str)
def test_estimate_matches_oracle(H, W, K, storage):
    rng = np.random.default_rng(H * W + K)
    occ = (rng.random((H, W)) < 0.1).astype(np.uint8)
    occ[H // 2, W // 2] = 0
    b = rng.random((K, H, W)).astype(np.float32) * (occ == 0)
    cell = 0.1
    h = loc.loc_create(occ, loc.loc_params_default(H=H, W=W, K=K, cell_m=cell, storage=storage))
    try:
        for uniform in (True, False):                   # the restart state reads the map
            if not uniform:
                loc.loc_set_belief(h, b)
            ref = loc.loc_belief(h).astype(np.float64)
            for radius, dk in ((0.0, 0), (0.12 * min(H, W) * cell, 2), (10.0 * (H + W), K)):
                got, want = loc.loc_estimate(h, radius, dk), R.estimate(ref, cell, 0.0, radius, dk)
                for key in ("k", "j", "i", "second_j", "second_i"):
                    assert got[key] == want[key], (key, got, want)
                assert abs(got["mass_near"] - want["mass_near"]) <= 1e-6 * want["mass_near"]
                assert abs(got["p"] - want["p"]) <= 1e-6 * want["p"]
                assert abs(got["second_p"] - want["second_p"]) <= 1e-6 * want["second_p"]
    finally:
        loc.loc_destroy(h)
