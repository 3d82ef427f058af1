"""The dense scan update at every number of bins that picks another form of its scorer (a thread owns
every 16th bin: 1 to 6, 8 or 16 of them, all in use or not), on grids whose cells come in fours and whose
last block is full or not.  Bounds as in test_gpu_dense.py: each state within (n_used + 8) 2^-23 (|log L|
+ |max log L| + 2) + 2^-20 relative, and 1e-6."""
import math

import numpy as np
import pytest

import paper_1910_00572_gb300 as loc
from oracle import dense as D

pytestmark = pytest.mark.gpu

BINS = [1, 15, 16, 17, 32, 33, 48, 49, 64, 65, 80, 81, 96, 97, 112, 128, 129, 250, 256]


@pytest.mark.parametrize("H,W", [(16, 16), (13, 17)], ids=str)
@pytest.mark.parametrize("K", BINS)
def test_update_matches_oracle(H, W, K):
    rng = np.random.default_rng(K)
    occ = (rng.random((H, W)) < 0.15).astype(np.uint8)
    occ[H // 2, W // 2] = 0
    cell, r_max, sig, A = 0.1, 1.5, 0.4, K * max(1, 72 // K)
    b = (rng.random((K, H, W)) * (occ == 0)).astype(np.float32)
    n = 24
    z = rng.uniform(0.1, 1.6, n).astype(np.float32)
    h = loc.loc_create(occ, loc.loc_params_default(H=H, W=W, K=K, cell_m=cell))
    try:
        loc.loc_set_belief(h, b)
        loc.loc_range_table(h, A, r_max)
        loc.loc_lidar_update_dense(h, z, -math.pi, 2 * math.pi / n, 1, sig)
        got = loc.loc_belief(h).astype(np.float64)
    finally:
        loc.loc_destroy(h)
    prior = b.astype(np.float64) / b.astype(np.float64).sum()
    table = D.range_table(occ, A, r_max, cell)
    ref, logL, mx, _ = D.dense_update(prior, occ, table, 0.0, z, -math.pi, 2 * math.pi / n, r_max, 1, sig)
    n_used = int((z < r_max).sum())
    rel = (n_used + 8) * 2.0 ** -23 * (np.abs(logL) + abs(mx) + 2.0) + 2.0 ** -20
    err = np.abs(got - ref)
    assert err.max() <= 1e-6
    assert (err <= np.where(np.isfinite(rel), rel, 0.0) * ref + 1e-12).all()
    assert (got[:, occ != 0] == 0).all()
