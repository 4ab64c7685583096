"""Indices of the bulk kernel, checked on the host."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def _run(tmp_path, name):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / name)
    subprocess.run([nvcc, "-O1", "-std=c++17", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2508_16387_gb300", "csrc"),
                    os.path.join(HERE, "native", name + ".cu"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout


def test_cells_outside_a_tile_read_written_slots(tmp_path):
    """Every slot of the shared plane that the states of cells outside the tile read (the material
    id there is an array index) is one that the plane's loads have written."""
    assert "unwritten slots read 0" in _run(tmp_path, "outside_check")


def test_mapped_positions_are_cells_of_the_grid(tmp_path):
    """A position anywhere in a tile or its halo, however short the axis, maps to a cell of it."""
    assert "positions outside 0 wrong 0" in _run(tmp_path, "map_check")


def test_requested_chunk_length_is_kept(tmp_path):
    """The z-length a caller asks for (m2c_set_tiling, a batch's tuning) is the one that runs; only
    the automatic one is evened out."""
    assert "wrong chunks 0" in _run(tmp_path, "chunk_check")
