"""Task and plan construction where no thread can be started: the same lists,
built on the calling thread. The program runs with a thread stack (its stack
limit) larger than the address space it may use."""

import json
import os
import resource
import shutil
import subprocess

import pytest

from synth import gaussian_sector_dims, mirrored_sectors

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
GIB = 1 << 30


def _no_threads():
    resource.setrlimit(resource.RLIMIT_AS, (4 * GIB, 4 * GIB))
    resource.setrlimit(resource.RLIMIT_STACK, (64 * GIB, resource.getrlimit(resource.RLIMIT_STACK)[1]))


def test_lists_without_threads(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no C++ compiler")
    hard = resource.getrlimit(resource.RLIMIT_STACK)[1]
    if hard != resource.RLIM_INFINITY and hard < 64 * GIB:
        pytest.skip("the stack limit cannot be raised")
    out, csrc = str(tmp_path / "plan_check"), os.path.join(ROOT, "paper_2103_09976_gb300", "csrc")
    subprocess.run([gxx, "-O2", "-std=c++17", "-pthread", "-I", csrc, os.path.join(ROOT, "tests", "host", "plan_check.cpp"),
                    os.path.join(csrc, "model.cpp"), "-o", out], check=True)
    left = gaussian_sector_dims(250, n_spatial=12, n_tot=17, two_sz_tot=1)
    right = mirrored_sectors(left, n_tot=17, two_sz_tot=1)
    path = tmp_path / "sectors.txt"
    path.write_text(f"{len(left)} {len(right)}\n" + "".join("%d %d %d\n" % tuple(s) for s in list(left) + list(right)))
    args = [out, str(path), "24", "48", "17", "1", "nc", "medium"]
    ref = subprocess.run(args, check=True, capture_output=True, text=True).stdout
    got = subprocess.run(args, capture_output=True, text=True, preexec_fn=_no_threads)
    assert got.returncode == 0, got.stderr
    assert got.stdout == ref
    assert json.loads(ref)["errors"] == [] and json.loads(ref)["tasks"] > 2 * 6000
