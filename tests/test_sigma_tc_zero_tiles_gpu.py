"""Output tiles without any product in the tensor-core sigma: their records
carry no unit, and a run of them follows the units of other tiles on the same
CTA. One sub-Hamiltonian whose only connected sectors are two of fourteen:
every other output block is exactly zero, the two connected ones match the
FP64 path (bar 5e-6 of max|sigma|: the mixed-precision bar of the other
tests)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [1, 2, 3])
@pytest.mark.parametrize("producers", [1, 3])
def test_tiles_without_products_are_zero(prec, producers):
    import torch
    from paper_2103_09976_gb300 import capi
    # sectors four electrons apart do not connect; (0, 0) and (2, 0) do, by the pair (0, 1) of rank 1
    left = [(0, 0, 40), (2, 0, 70)] + [(6 + 4 * k, 0, 300) for k in range(12)]
    N = 60
    right = sorted((N - n, -s, d + 3) for n, s, d in left)
    ctx = capi.dmrg_create(device=0, tc_producers=producers)
    try:
        capi.dmrg_load_synthetic_part(ctx, 4, 8, N, 0, left, right, 5, 1, 20)
        lay = capi.dmrg_psi_layout(ctx)
        n = lay["size"]
        x = torch.from_numpy(np.random.default_rng(2).standard_normal(n)).cuda()
        ref = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        capi.dmrg_sigma(ctx, -1, x, ref)
        capi.dmrg_sync(ctx)
        capi.dmrg_set_precision(ctx, prec)
        ys = []
        for _ in range(3):
            y = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            capi.dmrg_sigma(ctx, -1, x, y)
            capi.dmrg_sync(ctx)
            ys.append(y.cpu().numpy())
    finally:
        capi.dmrg_destroy(ctx)
    ref = ref.cpu().numpy()
    two = sum(int(a) * int(b) for a, b in zip(lay["m_l"][:2], lay["m_r"][:2]))
    assert not ref[two:].any() and ref[:two].any()
    for y in ys:
        assert not y[two:].any()
        assert np.abs(y[:two] - ref[:two]).max() <= 2e-5 * np.abs(ref).max() if prec == 1 else \
            np.abs(y[:two] - ref[:two]).max() <= 5e-6 * np.abs(ref).max()
        assert np.array_equal(y, ys[0])
