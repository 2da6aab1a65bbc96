"""Small classes of the mixed-precision sigma (all blocks at most 32 wide) at
the edges of their 8 x 8 tiles, 16-row warps and 16-column contraction steps,
against the CPU oracle, in every mixed mode; operators used as stored and
transposed, identity factors included.

Tolerance: both products contract at most 32 terms and a tile sums a few
hundred products in FP32 groups of 8; operands carry at least 22 bits. Worst
case (32 + 32 + 8) 2^-24 + 3 * 2^-22 = 5e-6 of the largest product; rounding
errors of random sign stay below a tenth of that: bar 1e-6 of max|sigma|."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 1e-6
QS = [(0, 0), (1, -1), (1, 1), (2, -2), (2, 0), (2, 2), (3, -1), (3, 1), (4, 0)]  # right: (4 - N, -2Sz)


@pytest.mark.parametrize("prec", [1, 2, 3])
@pytest.mark.parametrize("left_dims,right_dims", [
    ((1, 2, 3, 4, 5, 6, 7, 8, 9), (9, 8, 7, 6, 5, 4, 3, 2, 1)),
    ((16, 15, 9, 8, 7, 1, 16, 13, 2), (1, 16, 8, 9, 16, 7, 3, 15, 16)),          # <= 16 class
    ((17, 16, 32, 31, 25, 24, 1, 8, 15), (32, 1, 17, 16, 24, 31, 32, 9, 8)),     # <= 32 class: one and two row tiles
    ((32, 32, 32, 32, 32, 32, 32, 32, 32), (32, 32, 32, 32, 32, 32, 32, 32, 32)),
])
def test_small_classes_match_oracle(prec, left_dims, right_dims):
    from oracle.nc import nc_terms
    from oracle.sigma import psi_layout, sigma_blocks, synthetic_ops
    from paper_2103_09976_gb300 import capi
    from synth import random_unit_vector
    left = [(n, s, d) for (n, s), d in zip(QS, left_dims)]
    right = sorted((4 - n, -s, d) for (n, s), d in zip(QS, right_dims))
    ctx = capi.dmrg_create(device=0, sigma_prec=prec)
    try:
        capi.dmrg_load_synthetic(ctx, 4, 8, 4, 0, left, right, 21)
        n = capi.dmrg_psi_layout(ctx)["size"]
        x = random_unit_vector(n, 22)
        y, y2 = np.full(n, np.nan), np.full(n, np.nan)
        capi.dmrg_sigma(ctx, -1, x, y)
        capi.dmrg_sigma(ctx, -1, x, y2)
    finally:
        capi.dmrg_destroy(ctx)
    bL, bR, oL, oR, _ = synthetic_ops(left, right, 4, 8, seed=21)
    lay, size = psi_layout(bL, bR, (4, 0))
    ref = sigma_blocks(x, lay, nc_terms(4, 8), oL, oR)
    assert np.abs(y - ref).max() <= TOL * np.abs(ref).max()
    assert np.array_equal(y, y2)
