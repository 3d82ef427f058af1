"""Floyd-Steinberg selection on both forms of the block hand-off, bit-exact against the oracle's FP32 C
code: inboxes in shared memory, up to 6848 columns where each warp has one 32-row block and up to 3392
where it has several (above 2048 rows), and global memory beyond."""
import numpy as np
import pytest

import paper_1910_00572_gb300 as loc
from oracle import lidar as OL
from synth import fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W", [(70, 6848), (70, 6849), (33, 9000), (2049, 3392), (2049, 3393), (4129, 257)], ids=str)
def test_selection_is_bit_exact(H, W):
    m = fields.map_like(H, W, seed=H + W)
    fs = float(OL.fs_factor(m, H * W // 50))
    h = loc.loc_create(np.zeros((H, W), np.uint8), loc.loc_params_default(H=H, W=W, K=1, cell_m=0.05))
    try:
        for _ in range(2):                       # the second time over the first one's scratch
            sel, count = loc.loc_dither(h, m, fs)
            want = OL.fs_select(m, fs)
            assert count == int(want.sum())
            assert np.array_equal(sel, want)
    finally:
        loc.loc_destroy(h)
