"""Shared-memory layout of the 3D plane convolution (csrc/plane_layout.cuh),
enumerated on the host: no half-warp access of 8-byte values meets a bank twice,
and every exchange reads a value where it was written, in a slot of its own."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_plane_layout_is_conflict_free(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("needs g++")
    exe = tmp_path / "plane_layout"
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1708_01663_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "plane_layout_host.cpp"), "-o", str(exe)], check=True)
    rows = [line.split() for line in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.splitlines()]
    assert len(rows) == 8
    for side, what, sharing, sound in rows:
        assert (sharing, sound) == ("1", "1"), (side, what)
