"""Medium classes of the mixed-precision sigma (all blocks at most 64 wide, some
wider than 32) at the edges of their 8 x 8 tiles, 16-row warps (one to four per
term) and 16-column contraction steps; operators used as stored and
transposed, identity factors included.

The kernel of this class runs where it has 64 terms per SM or more. With 40
orbitals on each side the class has enough, which the host's plan check
asserts, and sigma is compared with the FP64 sigma of the same context; with 4
its terms are units of the tensor-core kernel, compared with the CPU oracle.

Tolerance: the arithmetic of the tensor-core sigma (operands and the
intermediate in 16 bits for BF16X2, 24 for BF16X3, 22 for FP16X2, FP32 sums),
so its bars: 2e-5 and 5e-6 of max|sigma|."""

import json
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = {1: 2e-5, 2: 5e-6, 3: 5e-6}
QS = [(0, 0), (1, -1), (1, 1), (2, -2), (2, 0), (2, 2), (3, -1), (3, 1), (4, 0)]  # right: (4 - N, -2Sz)


ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
DIMS = [
    ((33, 64, 1, 17, 48, 49, 63, 34, 2), (64, 3, 33, 40, 57, 1, 8, 48, 64)),
    ((64, 64, 64, 64, 64, 64, 64, 64, 64), (64, 64, 64, 64, 64, 64, 64, 64, 64)),
    ((5, 16, 31, 33, 47, 8, 65, 12, 40), (64, 40, 66, 33, 2, 50, 9, 61, 7)),     # some classes just above 64
]
# every number of 8-wide tiles: even and odd contractions on both sides, one to four row warps
EDGES = [
    ((33, 40, 41, 48, 49, 56, 57, 64, 8), (9, 15, 16, 17, 24, 25, 32, 64, 33)),
    ((1, 8, 9, 16, 17, 24, 25, 32, 64), (64, 57, 56, 49, 48, 41, 40, 34, 33)),
]


@pytest.fixture(scope="module")
def plan_check(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("plan") / "plan_check")
    csrc = os.path.join(ROOT, "paper_2103_09976_gb300", "csrc")
    subprocess.run(["g++", "-O2", "-std=c++17", "-pthread", "-I", csrc, os.path.join(ROOT, "tests", "host", "plan_check.cpp"),
                    os.path.join(csrc, "model.cpp"), "-o", out], check=True)
    return out


@pytest.mark.parametrize("left_dims,right_dims", DIMS + EDGES)
def test_medium_kernel_matches_fp64(plan_check, tmp_path, left_dims, right_dims):
    import torch
    from paper_2103_09976_gb300 import capi
    from synth import random_unit_vector
    left = [(n, s, d) for (n, s), d in zip(QS, left_dims)]
    right = sorted((4 - n, -s, d) for (n, s), d in zip(QS, right_dims))
    path = tmp_path / "sectors.txt"
    path.write_text(f"{len(left)} {len(right)}\n" + "".join("%d %d %d\n" % t for t in left + right))
    plan = json.loads(subprocess.run([plan_check, str(path), "40", "80", "4", "0", "nc", "medium"], check=True,
                                     capture_output=True, text=True).stdout)
    assert plan["errors"] == [] and plan["medium_items"] > 0
    # the check plans for 152 SMs; fewer need fewer terms
    assert torch.cuda.get_device_properties(0).multi_processor_count <= 152
    ctx = capi.dmrg_create(device=0)
    try:
        capi.dmrg_load_synthetic(ctx, 40, 80, 4, 0, left, right, 31)
        n = capi.dmrg_psi_layout(ctx)["size"]
        assert n == plan["psi_size"]
        x = random_unit_vector(n, 32)
        ref = np.full(n, np.nan)
        capi.dmrg_sigma(ctx, -1, x, ref)
        for prec in (1, 2, 3):
            capi.dmrg_set_precision(ctx, prec)
            y, y2 = np.full(n, np.nan), np.full(n, np.nan)
            capi.dmrg_sigma(ctx, -1, x, y)
            capi.dmrg_sigma(ctx, -1, x, y2)
            assert np.abs(y - ref).max() <= TOL[prec] * np.abs(ref).max(), prec
            assert np.array_equal(y, y2), prec
    finally:
        capi.dmrg_destroy(ctx)


@pytest.mark.parametrize("prec", [1, 2, 3])
@pytest.mark.parametrize("left_dims,right_dims", DIMS)
def test_medium_classes_match_oracle(prec, left_dims, right_dims):
    from oracle.nc import nc_terms
    from oracle.sigma import psi_layout, sigma_blocks, synthetic_ops
    from paper_2103_09976_gb300 import capi
    from synth import random_unit_vector
    left = [(n, s, d) for (n, s), d in zip(QS, left_dims)]
    right = sorted((4 - n, -s, d) for (n, s), d in zip(QS, right_dims))
    ctx = capi.dmrg_create(device=0, sigma_prec=prec)
    try:
        capi.dmrg_load_synthetic(ctx, 4, 8, 4, 0, left, right, 31)
        n = capi.dmrg_psi_layout(ctx)["size"]
        x = random_unit_vector(n, 32)
        y, y2 = np.full(n, np.nan), np.full(n, np.nan)
        capi.dmrg_sigma(ctx, -1, x, y)
        capi.dmrg_sigma(ctx, -1, x, y2)
    finally:
        capi.dmrg_destroy(ctx)
    bL, bR, oL, oR, _ = synthetic_ops(left, right, 4, 8, seed=31)
    lay, size = psi_layout(bL, bR, (4, 0))
    ref = sigma_blocks(x, lay, nc_terms(4, 8), oL, oR)
    assert np.abs(y - ref).max() <= TOL[prec] * np.abs(ref).max()
    assert np.array_equal(y, y2)
