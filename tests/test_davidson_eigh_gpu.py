"""Projected eigenproblem of the Davidson solver (its lowest pair, found in FP32
and refined in FP64): value, vector and time must not depend on a constant in
the Hamiltonian, and pairs that FP32 cannot tell apart are left to the FP64
Jacobi.

Bars: the refinement stops at a residual of 1e-15 |H|_F and evaluates it with
sums of 32 products, another 32 * 1.1e-16 of |H|_F at most: 5e-15; a value is off by
no more than its residual. A constant c enters the results through their own
rounding, 1.1e-16 |c|, and through the matrix, whose entries are the exact
ones here. Vectors of FP32 kept between calls: a rotation rounds by 6e-8, and a
call makes some 4 * 31 of them for each row: 7e-7 as a random walk, 1.4e-6 over the
four calls after which it is made good; bar 3e-6 for the largest of 1024 products."""

import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    from paper_2103_09976_gb300 import capi
    lib = os.path.dirname(os.path.abspath(capi.__file__))
    out = str(tmp_path_factory.mktemp("eigh") / "eigh_check")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(lib, "csrc"), "-I", os.path.join(cuda, "include"),
                    os.path.join(ROOT, "tests", "host", "eigh_check.cpp"), "-o", out, os.path.join(lib, "libdmrg.so"),
                    "-L", os.path.join(cuda, "lib64"), "-lcudart", "-Wl,-rpath," + lib], check=True)

    def call(constant, gap):
        res = subprocess.run([out, str(constant), str(gap)], capture_output=True, text=True, timeout=120)
        assert res.returncode == 0, res.stderr
        lines = [line.split() for line in res.stdout.splitlines()]
        print(res.stdout)
        return [[float(v) for v in r] for r in lines[:-1]], [float(v) for v in lines[-1][1:]]
    return call


@pytest.mark.parametrize("constant", [0.0, -88.0, -1e4])
@pytest.mark.parametrize("gap", [0.3, 1e-3, 1e-6, 1e-12, 0.0])
def test_lowest_pair(run, constant, gap):
    rows, _ = run(constant, gap)
    assert len(rows) == 32
    for k, value, resid, norm, orth in rows:
        const = 1.2e-16 * abs(constant)   # over |H - constant|_F >= 1 from k = 1 on
        assert value <= 5e-15 + const and resid <= 5e-15 + const, k
        assert norm <= 1e-14 and orth <= 3e-6, k


@pytest.mark.parametrize("gap", [0.3, 1e-3])
def test_time_does_not_depend_on_a_constant(run, gap):
    _, (plain, _) = run(0.0, gap)
    _, (shifted, _) = run(-1e4, gap)
    assert shifted <= 1.5 * plain, (plain, shifted)


def test_close_pairs_start_the_fp64_jacobi_from_the_fp32_vectors(run):
    _, (lowest, full) = run(0.0, 1e-12)
    assert lowest <= 0.7 * full, (lowest, full)
