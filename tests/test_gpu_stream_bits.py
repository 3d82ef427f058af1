"""The streaming propagation stores the values of the kernels whose place it takes, bit for bit: those of
the synchronous tiles where TMA applies (configuration 2 against 3, 16 and 17, alone and in a batch), those
of the generic kernel on other widths.  Compared on the stored tensors themselves, which a session takes
from a registered allocator (its first two allocations)."""
import numpy as np
import pytest

import paper_1910_00572_gb300 as loc

pytestmark = pytest.mark.gpu


@pytest.fixture()
def memory():
    """Device memory from torch while the test's sessions live: the tensors in the order of their requests."""
    import torch
    order = []

    def alloc(n, stream):
        order.append(torch.empty(n, dtype=torch.uint8, device="cuda"))
        return order[-1].data_ptr()
    loc.loc_set_allocator(alloc, lambda p, stream: None)
    yield order
    loc.loc_set_allocator(None, None)


class Session:
    def __init__(self, memory, occ, K, storage, **kw):
        H, W = occ.shape
        first = len(memory)
        self.h = loc.loc_create(occ, loc.loc_params_default(H=H, W=W, K=K, cell_m=0.05, storage=storage, **kw))
        self.both, self.cur = memory[first:first + 2], 0
        self.nbytes = K * H * W * (4 if storage == "f32" else 2)

    def stored(self):
        """The tensor after one more step."""
        self.cur ^= 1
        loc.loc_sync(self.h)
        return self.both[self.cur][:self.nbytes].cpu().numpy()


def case(H, W, K):
    rng = np.random.default_rng(H * W + K)
    occ = (rng.random((H, W)) < 0.15).astype(np.uint8)
    occ[H // 2, W // 2] = 0
    # a belief over many orders of magnitude: each rounding shows in some state
    b = np.exp(rng.uniform(-25.0, 0.0, (K, H, W))).astype(np.float32) * (occ == 0)
    return occ, b


MOVES = [(0.031, -0.044, 0.05), (0.9, 0.37, -0.3), (0.0, 0.0, 0.0), (-0.05, 0.1, 2.0)]


def close(sessions):
    for s in sessions:
        loc.loc_destroy(s.h)


@pytest.mark.parametrize("storage", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("H,W,K", [(1, 8, 8), (29, 72, 14), (57, 136, 16), (113, 200, 21), (565, 576, 9)], ids=str)
def test_aligned_rows(memory, H, W, K, storage):
    occ, b = case(H, W, K)
    ss = [Session(memory, occ, K, storage, tile=t, kernel=loc.LOC_KERNEL_TILED) for t in (2, 3, 16, 17)]
    batch = None
    try:
        for s in ss:
            loc.loc_set_belief(s.h, b)
        for n, m in enumerate(MOVES):
            for s in ss:                        # the first move reads the same belief in every session
                loc.loc_set_belief(s.h, b)
                loc.loc_step(s.h, *m)
            want = ss[0].stored()
            for s in ss[1:]:
                assert np.array_equal(s.stored(), want), n
        batch = loc.loc_batch_create([ss[1].h], tile=3)
        for s in ss[:2]:
            loc.loc_set_belief(s.h, b)
        loc.loc_step(ss[0].h, *MOVES[0])
        loc.loc_batch_step(batch, *([x] for x in MOVES[0]))
        loc.loc_batch_sync(batch)
        want = ss[0].stored()
        assert np.array_equal(ss[1].stored(), want)
    finally:
        if batch is not None:
            loc.loc_batch_destroy(batch)
        close(ss)


@pytest.mark.parametrize("storage", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("H,W,K", [(1, 1, 8), (29, 61, 9), (57, 134, 16), (40, 250, 22), (565, 577, 9)], ids=str)
def test_other_widths(memory, H, W, K, storage):
    occ, b = case(H, W, K)
    if not b.any():
        b = np.repeat((occ == 0)[None].astype(np.float32), K, 0)
    ss = [Session(memory, occ, K, storage, kernel=k) for k in (loc.LOC_KERNEL_GENERIC, loc.LOC_KERNEL_AUTO)]
    try:
        for m in MOVES:
            for s in ss:
                loc.loc_set_belief(s.h, b)
                loc.loc_step(s.h, *m)
            want = ss[0].stored()
            assert np.array_equal(ss[1].stored(), want), m
    finally:
        close(ss)
