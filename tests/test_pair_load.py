"""The two-cell FP64 sub-step's load of level n-1 (csrc/lap_int.cuh load_pair, sweep_flat.cuh flat_f64x2): the last cell of an odd row
stands beside the +x ghost, which a ghost thread of the same launch writes, so only the cell itself is read.  What the
cells become is compared with the oracle in test_fp64_pairs.py."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_last_cell_of_an_odd_row_is_read_alone(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "pair_load_check")
    subprocess.run([cxx, "-O0", "-std=c++17", "-o", exe, os.path.join(HERE, "native", "pair_load_check.cpp")], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True)
    assert out.stdout.split() == ["3", "5", "5", "5"]
