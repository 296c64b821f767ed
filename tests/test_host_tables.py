"""Sizes of the hash tables (csrc/tables.cuh), compiled for the CPU."""
from __future__ import annotations

import subprocess

from tests.test_host_walk import build_host


def test_sizes(tmp_path):
    r = subprocess.run([build_host(tmp_path, "tables_check")], capture_output=True, text=True, timeout=30)
    assert r.returncode == 0, r.stdout
