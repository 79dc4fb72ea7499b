"""Both integer forms of the FP64 Laplacian sum of one cell (csrc/lap_int.cuh) against the FP64 evaluation order, on the host: the
warp's vote (f64_update, csrc/cell.cuh) can send any accepted cell through lap6_rounded and any exact one through the sum."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.parametrize("seed", [1, 2])
def test_both_forms_of_every_accepted_cell(tmp_path, seed):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "lap_forms_check")
    subprocess.run([cxx, "-O2", "-ffp-contract=off", "-std=c++17", "-o", exe,
                    os.path.join(HERE, "native", "lap_forms_check.cpp")], check=True)
    out = subprocess.run([exe, "3000000", str(seed)], check=True, capture_output=True, text=True)
    cells, accepted, exact, mismatches = map(int, out.stdout.split())
    assert cells == 3000000 and accepted > cells // 2 and accepted // 4 < exact < accepted
    assert mismatches == 0
