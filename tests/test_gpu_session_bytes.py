"""What a session holds on the device after a scan update and every readout is at most what
loc_session_bytes says, the figure that sessions are admitted by."""
import math

import numpy as np
import pytest

import paper_1910_00572_gb300 as loc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,K,storage,beams", [(16, 16, 8, "f32", 36), (512, 512, 8, "f32", 360), (200, 304, 16, "bf16", 1080),
                                                 (311, 205, 9, "f16", 1080), (1024, 1024, 8, "bf16", 360)], ids=str)
def test_a_session_holds_what_it_is_admitted_for(H, W, K, storage, beams):
    import torch
    held = {}

    def alloc(n, stream):
        t = torch.empty(max(n, 1), dtype=torch.uint8, device="cuda")
        held[t.data_ptr()] = (t, (n + 511) // 512 * 512)
        return t.data_ptr()
    occ = (np.random.default_rng(H).random((H, W)) < 0.1).astype(np.uint8)
    occ[H // 2, W // 2] = 0
    p = loc.loc_params_default(H=H, W=W, K=K, cell_m=0.05, storage=storage, stream=loc.torch_stream(), n_samples=256)
    z = np.full(beams, 1.0, np.float32)
    loc.loc_set_allocator(alloc, lambda ptr, stream: held.pop(ptr))
    try:
        h = loc.loc_create(occ, p)
        for _ in range(2):
            loc.loc_step(h, 0.03, 0.01, 0.0)
            loc.loc_estimate(h, 0.5, 1)
            loc.loc_marginal(h)
            loc.loc_lidar_update(h, z, 0.0, 2 * math.pi / beams, 10.0, 1, 0.5)
            loc.loc_argmax(h)
            loc.loc_sync(h)
        total = sum(n for _, n in held.values())
        loc.loc_destroy(h)
    finally:
        loc.loc_set_allocator(None, None)
    assert not held
    assert total <= loc.loc_session_bytes(p), (total, loc.loc_session_bytes(p))
