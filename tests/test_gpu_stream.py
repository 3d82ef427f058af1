"""The streaming propagation kernel (tile configurations 3, 16 and 17) at the edges of its tiles:
rows around the 28-row tile, widths around the 64-cell tile, bin counts around the 7-deep theta
ring and the 8 planes in flight, and more tiles than SMs (several tiles per persistent CTA).

It performs the passes of the synchronous configurations on every cell, so its stored values equal
those of configuration 2 bit for bit; the normalisers are the same sums in another order, within a
few FP64 roundings and the FP32 rounding of 2 against 4 values summed before each compensated
addition (relative 2^-23 at most), which the readback multiplies in as one FP32 factor."""
import numpy as np
import pytest

import paper_1910_00572_gb300 as loc
from synth import fields

pytestmark = pytest.mark.gpu

SHAPES = [(1, 8, 8), (27, 64, 9), (28, 72, 14), (29, 56, 15), (57, 136, 16), (84, 128, 22), (565, 576, 8)]


@pytest.mark.parametrize("storage", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("H,W,K", SHAPES, ids=lambda v: str(v))
def test_streaming_tiles_equal_the_synchronous_ones(H, W, K, storage):
    rng = np.random.default_rng(H + W + K)
    occ = (rng.random((H, W)) < 0.15).astype(np.uint8)
    occ[H // 2, W // 2] = 0
    b = fields.belief_like(occ, K, seed=H, dtype=np.float32)
    tiles = (2, 3, 16, 17)
    hs = [loc.loc_create(occ, loc.loc_params_default(H=H, W=W, K=K, cell_m=0.05, storage=storage, tile=t,
                                                     kernel=loc.LOC_KERNEL_TILED)) for t in tiles]
    try:
        for first in (True, False):                     # the uniform start read from the map, a belief
            for h in hs:
                if not first:
                    loc.loc_set_belief(h, b)
                loc.loc_step(h, 0.031, -0.044, 0.05)
            want, z = loc.loc_belief(hs[0]), loc.loc_stats(hs[0])["last_Z"]
            for h in hs[1:]:
                assert abs(loc.loc_stats(h)["last_Z"] - z) <= 2.0 ** -23 * z
                np.testing.assert_allclose(loc.loc_belief(h), want, rtol=2.0 ** -21, atol=0)
            am = [loc.loc_argmax(h) for h in hs]
            assert all(a[:3] == am[0][:3] for a in am)
    finally:
        for h in hs:
            loc.loc_destroy(h)


RAGGED = [(1, 1, 8), (29, 61, 9), (31, 66, 11), (57, 133, 16), (40, 250, 22), (565, 577, 8)]


@pytest.mark.parametrize("storage", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("H,W,K", RAGGED, ids=lambda v: str(v))
def test_streaming_ragged_rows_equal_the_generic_kernel(H, W, K, storage):
    """Rows of any width (odd, even, a multiple of 4 but not of 16 bytes), shifts within a cell and
    beyond a tile: the generic kernel's operations in its order, so its stored values; normalisers as
    above."""
    rng = np.random.default_rng(H + W + K)
    occ = (rng.random((H, W)) < 0.15).astype(np.uint8)
    occ[H // 2, W // 2] = 0
    b = fields.belief_like(occ, K, seed=H, dtype=np.float32)
    if not b.any():
        b = np.repeat((occ == 0)[None].astype(np.float32), K, 0)
    hs = [loc.loc_create(occ, loc.loc_params_default(H=H, W=W, K=K, cell_m=0.05, storage=storage, kernel=k))
          for k in (loc.LOC_KERNEL_GENERIC, loc.LOC_KERNEL_AUTO)]
    try:
        for u, first in ((0.031, True), (0.031, False), (0.9, False), (0.0, False)):
            for h in hs:
                if not first:
                    loc.loc_set_belief(h, b)
                loc.loc_step(h, u, -0.044 if u else 0.0, 0.05)
            want, z = loc.loc_belief(hs[0]), loc.loc_stats(hs[0])["last_Z"]
            assert abs(loc.loc_stats(hs[1])["last_Z"] - z) <= 2.0 ** -23 * z
            np.testing.assert_allclose(loc.loc_belief(hs[1]), want, rtol=2.0 ** -21, atol=0)
    finally:
        for h in hs:
            loc.loc_destroy(h)
