"""The streaming propagation's bounded waits, without a GPU fault: loc_debug_step_stall withholds a
tile from the warps that wait for it, the waits give up after 0.2 s and the kernel returns.  The
sessions whose tiles were not finished fail with LOC_ERR_TIMEOUT and stay failed; the others, and new
sessions on the same device, go on."""
import numpy as np
import pytest

import paper_1910_00572_gb300 as loc

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def hook_off_afterwards():
    yield
    loc.loc_debug_step_stall(0)


def session(H, W, K, seed=0, **kw):
    occ = (np.random.default_rng(seed).random((H, W)) < 0.1).astype(np.uint8)
    occ[0, 0] = 0
    return loc.loc_create(occ, loc.loc_params_default(H=H, W=W, K=K, cell_m=0.05, **kw))


def step(h):
    loc.loc_step(h, 0.03, 0.01, 0.02)


def beliefs_after(n, *shape, **kw):
    h = session(*shape, **kw)
    try:
        for _ in range(n):
            step(h)
        return loc.loc_belief(h)
    finally:
        loc.loc_destroy(h)


# one tile a CTA, and (565 x 576: 189 tiles of 28 x 64) more tiles than SMs; with and without the fused
# argmax; rows that TMA takes and rows that it does not
@pytest.mark.parametrize("H,W,K,tile,stall", [(28, 64, 8, 3, 1), (60, 128, 16, 16, 1), (565, 576, 9, 17, 2),
                                              (60, 61, 8, 0, 1), (565, 577, 9, 0, 2)], ids=str)
@pytest.mark.parametrize("storage", ["f32", "bf16"])
def test_a_withheld_tile_fails_the_handle_only(H, W, K, tile, stall, storage):
    kw = dict(tile=tile, storage=storage)
    want = beliefs_after(2, H, W, K, **kw)
    h = session(H, W, K, **kw)
    try:
        step(h)
        loc.loc_sync(h)
        loc.loc_debug_step_stall(stall)
        step(h)
        with pytest.raises(loc.LocError) as e:
            loc.loc_sync(h)
        assert e.value.status == loc.LOC_ERR_TIMEOUT
        loc.loc_debug_step_stall(0)
        with pytest.raises(loc.LocError) as e:
            step(h)
        assert e.value.status == loc.LOC_ERR_STATE
    finally:
        loc.loc_destroy(h)
    assert np.array_equal(beliefs_after(2, H, W, K, **kw), want)


@pytest.mark.parametrize("use_graph", [False, True])
def test_a_batch_that_gives_up_at_its_first_tile(use_graph):
    """Every CTA's first tile is withheld, before it has taken a second one: the sessions of the tiles
    in hand fail, nothing else is written, and a new batch matches the sessions stepped alone."""
    shapes = [(28, 64, 24), (56, 72, 16), (30, 200, 9)]
    want = [beliefs_after(2, *s, seed=n, tile=3) for n, s in enumerate(shapes)]
    for stall in (1, 0):
        hs = [session(*s, seed=n) for n, s in enumerate(shapes)]
        b = loc.loc_batch_create(hs, tile=3, use_graph=use_graph)
        try:
            loc.loc_batch_step(b, 0.03, 0.01, 0.02)
            loc.loc_batch_sync(b)
            loc.loc_debug_step_stall(stall)
            loc.loc_batch_step(b, 0.03, 0.01, 0.02)
            if stall:
                with pytest.raises(loc.LocError) as e:
                    loc.loc_batch_sync(b)
                loc.loc_debug_step_stall(0)
                assert e.value.status == loc.LOC_ERR_TIMEOUT
                for h in hs:                           # fewer tiles than CTAs: all of them were in hand
                    with pytest.raises(loc.LocError):
                        loc.loc_sync(h)
            else:
                loc.loc_batch_sync(b)
                for h, w in zip(hs, want):
                    assert np.array_equal(loc.loc_belief(h), w)
        finally:
            loc.loc_batch_destroy(b)
            for h in hs:
                loc.loc_destroy(h)


def test_a_batch_session_that_was_finished_stays_usable():
    """Every CTA's second tile is withheld.  The first session's tiles (the longest bins, so taken first, by
    eight CTAs) are first ones: they are recorded when a third tile is taken, and the session goes on.  The
    second session has six tiles a CTA and fails."""
    import torch
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    first, second = (28, 64 * 8, 12), (28 * 6, 64 * n_sm, 8)
    want = beliefs_after(2, *first, tile=3)
    hs = [session(*first), session(*second, seed=1)]
    b = loc.loc_batch_create(hs, tile=3)
    try:
        loc.loc_batch_step(b, 0.03, 0.01, 0.02)
        loc.loc_batch_sync(b)
        loc.loc_debug_step_stall(2)
        loc.loc_batch_step(b, 0.03, 0.01, 0.02)
        with pytest.raises(loc.LocError) as e:
            loc.loc_batch_sync(b)
        assert e.value.status == loc.LOC_ERR_TIMEOUT
        loc.loc_debug_step_stall(0)
        assert loc.loc_sync(hs[0]) >= 0
        assert np.array_equal(loc.loc_belief(hs[0]), want)
        with pytest.raises(loc.LocError):
            loc.loc_sync(hs[1])
    finally:
        loc.loc_batch_destroy(b)
        for h in hs:
            loc.loc_destroy(h)


def test_hook_arguments():
    for bad in (-1, 3):
        with pytest.raises(loc.LocError) as e:
            loc.loc_debug_step_stall(bad)
        assert e.value.status == loc.LOC_ERR_INVALID_ARG
