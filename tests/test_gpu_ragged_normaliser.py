"""The normaliser of the streaming kernel on rows that TMA does not take is as precise as the generic
kernel's: two FP32 values are added before each compensated addition, so it is within 2^-24 relative of
the exact sum of the stored values (one rounding of each pair; the compensated sums add about 2^-47).

With taps of a single 1 (sigma 0, radii 2 and 3) and no motion the step only scales the belief, so every
fourth row holds s and the others s 2^-24.  The number of the former is just under a power of two, which
makes s = 1.004 x 2^n: s + s 2^-24 is then rounded by almost half a unit in the last place, and four rows
added up before a compensated addition would be off by 3 x 2^-24."""
import numpy as np
import pytest

import paper_1910_00572_gb300 as loc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", [loc.LOC_KERNEL_AUTO, loc.LOC_KERNEL_GENERIC], ids=["streaming", "generic"])
def test_pairs_of_values_are_summed_before_a_compensated_addition(kernel):
    import torch
    H, W, K = 40, 51, 8
    b = np.full((K, H, W), 2.0 ** -24, np.float32)
    b[:, ::4] = 1.0
    taken = []

    def alloc(n, stream):
        taken.append(torch.empty(n, dtype=torch.uint8, device="cuda"))
        return taken[-1].data_ptr()
    loc.loc_set_allocator(alloc, lambda p, stream: None)
    try:
        h = loc.loc_create(np.zeros((H, W), np.uint8), loc.loc_params_default(
            H=H, W=W, K=K, cell_m=0.05, sigma_xy_cells=0.0, sigma_theta_bins=0.0, r_xy=2, r_theta=3, kernel=kernel))
        loc.loc_set_belief(h, b)
        loc.loc_step(h, 0.0, 0.0, 0.0)
        z = loc.loc_stats(h)["last_Z"]
        stored = taken[1][:4 * K * H * W].view(torch.float32).cpu().numpy().reshape(K, H, W)
        loc.loc_destroy(h)
    finally:
        loc.loc_set_allocator(None, None)
    s = float(stored[0, 0, 0])
    assert (stored[:, ::4] == s).all() and (stored[:, 1] == s * 2.0 ** -24).all() and 1.0 < s * 4096 < 1.01
    exact = float(stored.astype(np.float64).sum())
    assert abs(z - exact) <= 2.0 ** -24 * exact + 1e-12 * exact, (z - exact) / exact * 2.0 ** 24
