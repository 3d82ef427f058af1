"""A registered allocator may hand out any address: the kernels' wide loads (of the map, of the belief
and of the scans' tables) see aligned memory, every result is that of a session on cudaMalloc's memory,
and what was handed out comes back."""
import math

import numpy as np
import pytest

import paper_1910_00572_gb300 as loc

pytestmark = pytest.mark.gpu


def use(H, W, K, storage, occ, z):
    """Every kind of call once; the results."""
    h = loc.loc_create(occ, loc.loc_params_default(H=H, W=W, K=K, cell_m=0.05, storage=storage, n_samples=64,
                                                   stream=loc.torch_stream()))
    try:
        out = []
        for _ in range(2):
            loc.loc_step(h, 0.03, 0.01, 0.0)
            out += [loc.loc_belief(h), loc.loc_marginal(h), *loc.loc_argmax(h), *loc.loc_estimate(h, 0.2, 1).values()]
        loc.loc_lidar_update(h, z, 0.0, 2 * math.pi / z.size, 10.0, 2, 0.5)
        out += [loc.loc_belief(h), loc.loc_samples(h)]
        loc.loc_range_table(h, 2 * K, 10.0)
        loc.loc_lidar_update_dense(h, z, 0.0, 2 * math.pi / z.size, 2, 0.5)
        return out + [loc.loc_belief(h)]
    finally:
        loc.loc_destroy(h)


@pytest.mark.parametrize("offset", ["map by 1", 1, 4, 8], ids=str)
@pytest.mark.parametrize("H,W,K,storage", [(40, 72, 8, "f32"), (37, 53, 9, "f32"), (40, 72, 8, "bf16")], ids=str)
def test_addresses_of_any_alignment(H, W, K, storage, offset):
    import torch
    rng = np.random.default_rng(H + W)
    occ = (rng.random((H, W)) < 0.1).astype(np.uint8)
    occ[H // 2, W // 2] = 0
    z = rng.uniform(0.3, 1.5, 36).astype(np.float32)
    want = use(H, W, K, storage, occ, z)
    held = {}

    def alloc(n, stream):
        t = torch.empty(n + 64, dtype=torch.uint8, device="cuda")
        p = t.data_ptr() + (offset if offset != "map by 1" else int(n == H * W))
        held[p] = t
        return p
    loc.loc_set_allocator(alloc, lambda p, stream: held.pop(p))
    try:
        got = use(H, W, K, storage, occ, z)
    finally:
        loc.loc_set_allocator(None, None)
    assert not held
    assert len(got) == len(want) and all(np.array_equal(a, b) for a, b in zip(got, want))
