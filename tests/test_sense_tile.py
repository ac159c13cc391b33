"""The tiled storage of the sensing matrix (csrc/sense_tile.cuh), enumerated on the host: little padding, contiguous chunks,
no bank conflicts (tests/sense_tile_host.cpp)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_tiles(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("needs g++")
    exe = str(tmp_path / "sense_tile")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1708_01663_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "sense_tile_host.cpp"), "-o", exe], check=True)
    assert subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split() == ["0"]
