"""Branches of the device Davidson solver: register blocks of its vector
kernels (up to 8, 16 and 32 vectors), restarts, the projected eigenproblem with
and without a gap FP32 can see, and a direction that vanishes.

Energies are compared with numpy's eigvalsh of the dense H_eff, whose columns
are the library's FP64 sigma of unit vectors. A solve stops at |r|^2 < tol, and
an eigenvalue is off by at most |r|: bar |r| = 1e-7 plus 1e-12 |E| for FP64
rounding (an eigenvalue's error is of second order, so far less is met)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 1e-14


def _dense(capi, ctx, site, n):
    H = np.zeros((n, n))
    for j in range(n):
        e = np.zeros(n)
        e[j] = 1.0
        col = np.zeros(n)
        capi.dmrg_sigma(ctx, site, e, col)
        H[:, j] = col
    return H


@pytest.mark.parametrize("space", [3, 8, 9, 16, 17, 31, 32])
def test_subspace_sizes_and_restarts(space):
    from paper_2103_09976_gb300 import capi
    from synth import gaussian_sector_dims, mirrored_sectors, random_unit_vector
    left = gaussian_sector_dims(40, n_spatial=4, n_tot=6)
    right = mirrored_sectors(left, n_tot=6)
    ctx = capi.dmrg_create(device=0, dav_max_space=space, dav_max_iter=4000)
    try:
        capi.dmrg_load_synthetic(ctx, 8, 16, 6, 0, left, right, 9)
        n = capi.dmrg_psi_layout(ctx)["size"]
        H = _dense(capi, ctx, -1, n)
        x = random_unit_vector(n, 3)
        out = np.zeros(n)
        e, it, conv = capi.dmrg_davidson(ctx, -1, x, TOL, out)
    finally:
        capi.dmrg_destroy(ctx)
    assert n > 64 and conv
    w = np.linalg.eigvalsh(0.5 * (H + H.T))
    assert abs(e - w[0]) <= 1e-7 + 1e-12 * abs(w[0])
    assert abs(np.linalg.norm(out) - 1.0) < 1e-12
    assert np.linalg.norm(H @ out - e * out) < 2e-7


@pytest.mark.parametrize("levels", [(-1.0, -1.0, 0.5, 2.0, 2.0), (-1.0, -1.0 + 1e-9, 0.5, 0.75, 2.0),
                                    (0.0, 0.0, 0.0, 0.0, 0.0), (3.0, 4.0, 5.0, 6.0, 7.0)])
def test_degenerate_and_exhausted_spaces(levels):
    """One electron in five orbitals: five states. Equal or almost equal lowest
    levels leave the FP32 eigenvalues without a gap (the FP64 Jacobi decides);
    a space of five states is exhausted within five products, after which no
    direction is left."""
    from paper_2103_09976_gb300 import capi
    K = 5
    rng = np.random.default_rng(4)
    q, _ = np.linalg.qr(rng.standard_normal((K, K)))
    t = q @ np.diag(levels) @ q.T
    t = 0.5 * (t + t.T)
    ctx = capi.dmrg_create(device=0, seed=3, dav_max_iter=30)
    try:
        capi.dmrg_build_blocks(ctx, t, np.zeros((K, K, K, K)), K, 1, 1, 64)
        n = capi.dmrg_psi_layout(ctx, 0)["size"]
        e, it, conv = capi.dmrg_davidson(ctx, 0, None, 1e-18)
    finally:
        capi.dmrg_destroy(ctx)
    assert n == K
    assert conv and it <= K + 2
    assert abs(e - min(levels)) < 1e-9
