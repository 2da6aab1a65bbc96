"""Accuracy of the mixed sigma where all blocks are at most 32 wide (the small
classes alone), against the FP64 sigma of the same context.

Even psi: the error of FP32 arithmetic, in the 2-norm. The operands carry 24
(bf16 slices) or 22 bits (fp16): three roundings of at most 2^-25 or 2^-23
relative, uniform, are 3e-8 or 1.2e-7 / sqrt(3) each; the two products add some
four FP32 roundings of 2^-25. Bars 1.2e-7 and 1.8e-7; sums cut off instead of
rounded are at 3e-7.

Graded psi (a factor of 10 per electron off the middle, as Schmidt weights
fall): every block of sigma by itself. A block k electrons out gets most of
its value from psi two electrons further in, 10^-(k - 2) of the largest element.
FP16X2 holds psi to 2^-39 of its largest element: with k <= 8 that is 1.8e-6 of
those, about four times as much of their rms value; bar 1e-4 for cancellation
in blocks of a few elements. X = L psi on one scale for all blocks is ten
times further off than that."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BAR = {1: 1.2e-7, 2: 1.2e-7, 3: 1.8e-7}


def _errors(prec, nsp, ntot, M, grade, seed):
    from paper_2103_09976_gb300 import capi
    from synth import gaussian_sector_dims, mirrored_sectors
    two_sz = ntot % 2
    left = gaussian_sector_dims(M, n_spatial=nsp, n_tot=ntot, two_sz_tot=two_sz)
    right = mirrored_sectors(left, n_tot=ntot, two_sz_tot=two_sz)
    assert max(d for _, _, d in list(left) + list(right)) <= 32
    ctx = capi.dmrg_create(device=0)
    try:
        capi.dmrg_load_synthetic(ctx, 2 * nsp, 4 * nsp, ntot, two_sz, left, right, seed)
        lay = capi.dmrg_psi_layout(ctx)
        x = np.random.default_rng(seed).standard_normal(lay["size"])
        q = np.asarray(lay["q_l"]).reshape(-1, 2)
        parts = [slice(o, o + a * b) for o, a, b in zip(lay["offset"], lay["m_l"], lay["m_r"])]
        for s, (n, _) in zip(parts, q):
            x[s] *= grade ** abs(n - ntot / 2)
        x /= np.linalg.norm(x)
        ref, y = np.full_like(x, np.nan), np.full_like(x, np.nan)
        capi.dmrg_sigma(ctx, -1, x, ref)
        capi.dmrg_set_precision(ctx, prec)
        capi.dmrg_sigma(ctx, -1, x, y)
    finally:
        capi.dmrg_destroy(ctx)
    whole = np.linalg.norm(y - ref) / np.linalg.norm(ref)
    return whole, max(np.linalg.norm((y - ref)[s]) / np.linalg.norm(ref[s]) for s in parts)


@pytest.mark.parametrize("prec", [1, 2, 3])
@pytest.mark.parametrize("nsp,ntot,M", [(4, 8, 60), (12, 17, 200), (12, 17, 400), (18, 27, 500)])  # up to 4, 10, 21, 25 wide
def test_small_classes_have_the_error_of_fp32(prec, nsp, ntot, M):
    whole = np.mean([_errors(prec, nsp, ntot, M, 1.0, s)[0] for s in (1, 2, 3)])
    print(whole)
    assert whole < BAR[prec]


@pytest.mark.parametrize("prec", [1, 2, 3])
@pytest.mark.parametrize("nsp,ntot,M", [(8, 16, 150), (8, 16, 350)])
def test_blocks_of_a_graded_psi(prec, nsp, ntot, M):
    whole, worst = np.max([_errors(prec, nsp, ntot, M, 0.1, s) for s in (1, 2, 3)], axis=0)
    print(whole, worst)
    assert whole < BAR[prec] and worst < 1e-4
