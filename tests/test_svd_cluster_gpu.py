"""Decimation SVD (one-sided Jacobi): the cluster kernel at the edges of its
range (one column, odd and even counts, 32-element chunks, one or more pairs per
CTA, the shared-memory limit), blocks past it beside them on the grid-wide
kernel, both orientations, and graded, rank-deficient and zero spectra.

Tolerances: a rotation rounds each element at most three times (2^-53 of its
column), and d columns go through about 10 d rotations each, whose errors add as
a random walk: sqrt(3 * 10 * 256) * 1.1e-16 = 1e-14 at d = 256; bars at 4e-14 for
the largest of up to d^2 entries."""

import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SIZES = [(1, 1), (1, 40), (2, 5), (3, 1), (5, 5), (16, 16), (17, 33), (33, 17), (40, 7), (64, 64), (65, 31),
         (96, 160), (127, 128), (128, 129), (130, 130), (224, 223), (256, 90), (256, 256), (40, 257), (258, 60)]


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    from paper_2103_09976_gb300 import capi
    lib = os.path.dirname(os.path.abspath(capi.__file__))
    out = str(tmp_path_factory.mktemp("svd") / "svd_check")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(lib, "csrc"), "-I", os.path.join(cuda, "include"),
                    os.path.join(ROOT, "tests", "host", "svd_check.cpp"), "-o", out, os.path.join(lib, "libdmrg.so"),
                    "-L", os.path.join(cuda, "lib64"), "-lcudart", "-Wl,-rpath," + lib], check=True)
    return out


@pytest.mark.parametrize("left", [0, 1])
@pytest.mark.parametrize("spectrum", ["flat", "graded", "lowrank", "zero"])
def test_svd_kernels(checker, left, spectrum):
    args = [str(v) for dm in SIZES for v in dm]
    res = subprocess.run([checker, str(left), spectrum] + args, capture_output=True, text=True, timeout=300)
    assert res.returncode == 0, res.stderr
    rows = [line.split() for line in res.stdout.splitlines()]
    print(res.stdout)
    assert [(int(r[0]), int(r[1])) for r in rows] == SIZES
    assert [int(r[2]) for r in rows] == [0 if dm in ((40, 257), (258, 60)) else 1 for dm in SIZES]
    for r in rows:
        assert max(float(v) for v in r[3:]) < 4e-14, r
