"""A restart's step (the first one, or after all mass was lost: the input is the map) of the streaming
kernel: the stored values of the synchronous tiles bit for bit, whatever the shift; in a batch, where a
stage that held the map takes another session's planes next, those of the sessions alone; and at most
three times an ordinary step's time (1.3 to 2.0 measured; with one warp reading the map it was 6 to 8)."""
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


def session(memory, H, W, K, storage, seed=0, **kw):
    """A new session, and its two belief buffers as bytes (the step writes the second one first)."""
    rng = np.random.default_rng(seed + H * W)
    occ = (rng.random((H, W)) < 0.15).astype(np.uint8)
    occ[H // 2, W // 2] = 0
    first = len(memory)
    h = loc.loc_create(occ, loc.loc_params_default(H=H, W=W, K=K, cell_m=0.05, storage=storage, **kw))
    n = K * H * W * (4 if storage == "f32" else 2)
    return h, [m[:n] for m in memory[first:first + 2]], occ


MOVES = [(0.0, 0.0), (0.031, -0.044), (0.9, 0.37), (-2.3, 4.1)]


@pytest.mark.parametrize("storage", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("H,W,K", [(1, 8, 8), (29, 72, 9), (57, 136, 16), (90, 64, 21), (565, 576, 8)], ids=str)
def test_first_step_equals_the_synchronous_one(memory, H, W, K, storage):
    for u, v in MOVES:
        ss = [session(memory, H, W, K, storage, tile=t, kernel=loc.LOC_KERNEL_TILED) for t in (2, 3, 16)]
        for h, _, _ in ss:
            loc.loc_step(h, u, v, 0.1)
            loc.loc_sync(h)
        want = ss[0][1][1].cpu().numpy()
        for _, both, _ in ss[1:]:
            assert np.array_equal(both[1].cpu().numpy(), want), (u, v)
        for h, _, _ in ss:
            loc.loc_destroy(h)


@pytest.mark.parametrize("storage", ["f32", "bf16"])
def test_batch_of_restarted_and_other_sessions(memory, storage):
    shapes = [(224, 256, 12), (300, 320, 11), (224, 256, 10), (400, 264, 9), (500, 512, 8)]
    ss = [session(memory, *s, storage, seed=n) for n, s in enumerate(shapes)]
    alone = [session(memory, *s, storage, seed=n, tile=3, kernel=loc.LOC_KERNEL_TILED) for n, s in enumerate(shapes)]
    batch = loc.loc_batch_create([h for h, _, _ in ss], tile=3)
    try:
        for n, (H, W, K) in enumerate(shapes):
            if n % 2:                                   # every second session holds a belief
                b = np.random.default_rng(n).random((K, H, W)).astype(np.float32) * (ss[n][2] == 0)
                for q in (ss, alone):
                    loc.loc_set_belief(q[n][0], b)
        for tick in range(2):
            loc.loc_batch_step(batch, 0.05, -0.03, 0.02)
            loc.loc_batch_sync(batch)
            for (h, both, _), (_, mine, _) in zip(alone, ss):
                loc.loc_step(h, 0.05, -0.03, 0.02)
                loc.loc_sync(h)
                assert np.array_equal(mine[1 - tick].cpu().numpy(), both[1 - tick].cpu().numpy())
    finally:
        loc.loc_batch_destroy(batch)
        for h, _, _ in ss + alone:
            loc.loc_destroy(h)


@pytest.mark.parametrize("H,W,K,storage", [(1024, 1024, 36, "f32"), (1024, 1024, 36, "bf16")], ids=str)
def test_restart_takes_about_a_step(memory, H, W, K, storage):
    import torch
    first, later = [], []
    for _ in range(7):
        h, _, _ = session(memory, H, W, K, storage, stream=loc.torch_stream())
        memory[0].zero_()                               # the stream is busy when the timed work is enqueued
        for times in (first, later):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            loc.loc_step(h, 0.04, 0.01, 0.0)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        loc.loc_destroy(h)
    assert np.median(first) <= 3.0 * np.median(later), (first, later)
