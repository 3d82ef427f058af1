"""Queued steps of small maps leave the GPU to other streams' kernels.  A step lets the next one of its
stream onto the SMs before it ends, and no more than the next one: eight streams of a 64 x 64 map hold
2 x 3 thread blocks each, so a ninth stream's step of three blocks finds idle SMs at once and takes about
what it takes on an idle GPU.  The bound, twice that, lies between 1.0 (one step ahead) and 3.6 (every
queued step ahead), both measured."""
import numpy as np
import pytest

import paper_1910_00572_gb300 as loc

pytestmark = pytest.mark.gpu


def test_a_step_beside_queued_steps_of_other_streams():
    import torch
    occ = np.zeros((64, 64), np.uint8)
    streams = [torch.cuda.Stream() for _ in range(9)]
    hs = [loc.loc_create(occ, loc.loc_params_default(H=64, W=64, K=128 if n < 8 else 16, cell_m=0.05,
                                                     stream=int(s.cuda_stream))) for n, s in enumerate(streams)]

    def step(h, n):
        loc.loc_step(h, 0.04 * (-1) ** n, 0.01 * (-1) ** n, 0.0)

    def latency(queued):
        out = []
        for rep in range(12):
            torch.cuda.synchronize()
            for n in range(queued):
                for h in hs[:8]:
                    step(h, n)
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(streams[8])
            step(hs[8], rep)
            b.record(streams[8])
            torch.cuda.synchronize()
            out.append(a.elapsed_time(b))
        return float(np.median(out[2:]))
    try:
        alone, beside = latency(0), latency(100)
        assert beside <= 2.0 * alone, (alone, beside)
    finally:
        for h in hs:
            loc.loc_destroy(h)
