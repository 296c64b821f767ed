"""The split of the CSR entries over warps (csrc/walk.cuh), compiled for the CPU with a warp of 32 fibers."""
from __future__ import annotations

import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def build_host(tmp, name):
    """Compiles tests/host/<name>.cpp against the library's headers; returns the program."""
    exe = os.path.join(str(tmp), name)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wno-unknown-pragmas", "-I",
                    os.path.join(ROOT, "paper_2504_17615_gb300", "csrc"), "-o", exe,
                    os.path.join(ROOT, "tests", "host", name + ".cpp")], check=True)
    return exe


@pytest.fixture(scope="module")
def walk_check(tmp_path_factory):
    return build_host(tmp_path_factory.mktemp("walk"), "walk_check")


# "any": offsets that decrease somewhere, which not every caller checks for; the walk has to end.  "even": no warp
# has far more to do than the others
@pytest.mark.parametrize("offsets", ["monotone", "any", "even"])
def test_walk(walk_check, offsets):
    r = subprocess.run([walk_check, offsets], capture_output=True, text=True, timeout=30)
    assert r.returncode == 0, r.stdout
