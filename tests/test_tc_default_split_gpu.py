"""Default item split of the tensor-core sigma: items per SM by the number of
units, here its lower end (a few dozen units in all: 2 per SM), against the CPU
oracle and against the single-warp producer setting, bitwise. Tolerance as the
other FP16X2 sigma tests: 5e-6 of max|sigma| (operands and the intermediate in
22 bits, FP32 sums)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_small_plan_takes_two_items_per_sm():
    from oracle.nc import nc_terms
    from oracle.sigma import psi_layout, sigma_blocks, synthetic_ops
    from paper_2103_09976_gb300 import capi
    from synth import random_unit_vector
    left = [(1, -1, 70), (1, 1, 130), (2, 0, 96)]
    right = [(2, 0, 80), (3, -1, 129), (3, 1, 66)]
    ys = []
    for producers in (0, 1, 3):
        ctx = capi.dmrg_create(device=0, sigma_prec=capi.DMRG_FP16X2, tc_producers=producers)
        try:
            capi.dmrg_load_synthetic(ctx, 4, 8, 4, 0, left, right, 5)
            n = capi.dmrg_psi_layout(ctx)["size"]
            x, y = random_unit_vector(n, 6), np.full(n, np.nan)
            assert capi.dmrg_get_sigma_info(ctx)["tc_items_per_sm"] == 2   # what the plan will take
            capi.dmrg_sigma(ctx, -1, x, y)
            info = capi.dmrg_get_sigma_info(ctx)
        finally:
            capi.dmrg_destroy(ctx)
        assert info["tc_items_per_sm"] == 2 and info["tc_producers"] == (producers or 3)
        ys.append(y)
    bL, bR, oL, oR, _ = synthetic_ops(left, right, 4, 8, seed=5)
    lay, _ = psi_layout(bL, bR, (4, 0))
    ref = sigma_blocks(x, lay, nc_terms(4, 8), oL, oR)
    assert np.abs(ys[0] - ref).max() <= 5e-6 * np.abs(ref).max()
    assert np.array_equal(ys[0], ys[1]) and np.array_equal(ys[0], ys[2])
