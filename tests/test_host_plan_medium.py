"""Host logic of the tensor-core plan as the library builds it, with the class
of blocks of 33 - 64 in items of their own (one psi block each): the checks of
tests/host/plan_check.cpp hold, every product is in exactly one unit or
small-class item, and small problems keep that class in the units."""

import json
import os
import shutil
import subprocess

import pytest

from synth import gaussian_sector_dims, mirrored_sectors

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no C++ compiler")
    out = str(tmp_path_factory.mktemp("plan") / "plan_check")
    csrc = os.path.join(ROOT, "paper_2103_09976_gb300", "csrc")
    subprocess.run([gxx, "-O2", "-std=c++17", "-pthread", "-I", csrc, os.path.join(ROOT, "tests", "host", "plan_check.cpp"),
                    os.path.join(csrc, "model.cpp"), "-o", out], check=True)
    return out


@pytest.mark.parametrize("nsp,ntot,M,medium", [(54, 30, 2000, True), (27, 41, 1000, True), (8, 15, 600, False)])
def test_plan_with_medium_class(checker, tmp_path, nsp, ntot, M, medium):
    two_sz = ntot % 2
    left = gaussian_sector_dims(M, n_spatial=nsp, n_tot=ntot, two_sz_tot=two_sz)
    right = mirrored_sectors(left, n_tot=ntot, two_sz_tot=two_sz)
    path = tmp_path / "sectors.txt"
    with open(path, "w") as f:
        f.write(f"{len(left)} {len(right)}\n")
        for s in list(left) + list(right):
            f.write(" ".join(str(int(x)) for x in s) + "\n")
    args = [checker, str(path), str(2 * nsp), str(4 * nsp), str(ntot), str(two_sz), "nc"]
    got = json.loads(subprocess.run(args + ["medium"], check=True, capture_output=True, text=True).stdout)
    ref = json.loads(subprocess.run(args, check=True, capture_output=True, text=True).stdout)
    assert got["errors"] == [] and ref["errors"] == []
    assert got["plan_tasks"] == ref["plan_tasks"] and ref["medium_items"] == 0
    assert (got["medium_items"] > 0) == medium
    assert got["units"] < ref["units"] if medium else got["units"] == ref["units"]
