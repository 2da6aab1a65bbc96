"""FP64 sigma on block shapes at the edges of the kernel's register tiles.

A warp owns 16 x 128 or 8 x 256 elements of an output tile, takes the
intermediate 32 columns at a time in groups of 8 (a last group of 2-4 columns
in natural order, others as even / odd columns) and contracts in steps of 4;
items share their tasks between 1, 2 or 4 warps. The dimensions below are the
edges of those splits and their neighbours.

Tolerance: every output is a sum of products of two contractions; a bound on
its rounding error is gamma_k with k the number of additions, at most about
300 + 300 per product and 200 products: 1e5 * 2^-53 = 1e-11 in the worst case,
and the square root of that, 1e-13, for rounding errors of random sign; bar
1e-12 of max|sigma| as in the other FP64 tests.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 1e-12

# target N = 4, 2Sz = 0: left (N, 2Sz) pairs with right (4 - N, -2Sz)
QS = [(0, 0), (1, -1), (1, 1), (2, -2), (2, 0), (2, 2), (3, -1), (3, 1), (4, 0)]


def _case(left_dims, right_dims):
    left = [(n, s, d) for (n, s), d in zip(QS, left_dims)]
    right = sorted((4 - n, -s, d) for (n, s), d in zip(QS, right_dims))
    return left, right


@pytest.mark.parametrize("left_dims,right_dims", [
    ((1, 2, 3, 4, 5, 6, 7, 8, 9), (9, 8, 7, 6, 5, 4, 3, 2, 1)),             # below one 8 x 8 group
    ((8, 15, 16, 17, 24, 25, 31, 32, 33), (33, 32, 31, 30, 29, 28, 27, 26, 25)),  # row slices, 32-column chunks
    ((1, 16, 40, 3, 12, 33, 7, 64, 1), (34, 66, 36, 120, 127, 128, 129, 130, 35)),  # 128 columns and past them
    ((5, 18, 2, 9, 33, 1, 4, 20, 6), (130, 7, 255, 1, 256, 12, 257, 3, 300)),  # 256 columns and past them
])
def test_sigma_f64_tile_edges_match_oracle(left_dims, right_dims):
    from oracle.nc import nc_terms
    from oracle.sigma import psi_layout, sigma_blocks, synthetic_ops
    from paper_2103_09976_gb300 import capi
    from synth import random_unit_vector
    left, right = _case(left_dims, right_dims)
    ctx = capi.dmrg_create(device=0)
    try:
        capi.dmrg_load_synthetic(ctx, 4, 8, 4, 0, left, right, 17)
        n = capi.dmrg_psi_layout(ctx)["size"]
        x = random_unit_vector(n, 18)
        y = np.full(n, np.nan)
        capi.dmrg_sigma(ctx, -1, x, y)
    finally:
        capi.dmrg_destroy(ctx)
    bL, bR, oL, oR, _ = synthetic_ops(left, right, 4, 8, seed=17)
    lay, size = psi_layout(bL, bR, (4, 0))
    assert size == n
    ref = sigma_blocks(x, lay, nc_terms(4, 8), oL, oR)
    assert np.abs(y - ref).max() <= TOL * np.abs(ref).max()


def test_transformation_of_wide_sectors_keeps_the_spectrum():
    """Right blocks built at full bond dimension (K=8: sectors up to 400 wide,
    several 16 x 128 pieces per tile) in random orthonormal bases represent H
    exactly: the lowest energy at the first bond is the stored FCI energy."""
    import json
    import os
    from paper_2103_09976_gb300 import capi
    from synth import random_integrals
    gold = json.load(open(os.path.join(os.path.dirname(__file__), "golden", "fci_energies.json")))["cfg1"]
    t, v = random_integrals(8, 0)
    ctx = capi.dmrg_create(device=0, seed=2)
    try:
        capi.dmrg_build_blocks(ctx, t, v, 8, 8, 0, 4096)
        q, d, _ = capi.dmrg_block_info(ctx, 1, 2)
        e, it, conv = capi.dmrg_davidson(ctx, 0, None, 1e-11)
    finally:
        capi.dmrg_destroy(ctx)
    assert d.max() > 256
    assert conv and abs(e - gold["energy"]) < 1e-9
