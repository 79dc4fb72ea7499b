"""FP64 sub-steps with two cells per thread (csrc/lap_int.cuh lap6_units2, sweep_flat.cuh flat_f64x2): the pair's integer
forms give the bits of the FP64 evaluation order wherever they accept a stencil (host), and grids large enough for
pairs equal the oracle bit for bit for even, odd and single-cell rows under every boundary condition (GPU)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle as O
from paper_1602_05700_gb300 import inputs as I

torch = pytest.importorskip("torch")

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.parametrize("seed", [1, 2])
def test_pair_forms_equal_the_fp64_order(tmp_path, seed):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "lap_pair_check")
    subprocess.run([cxx, "-O2", "-ffp-contract=off", "-std=c++17", "-o", exe,
                    os.path.join(HERE, "native", "lap_pair_check.cpp")], check=True)
    out = subprocess.run([exe, "2000000", str(seed)], check=True, capture_output=True, text=True)
    cells, accepted, mismatches = map(int, out.stdout.split())
    assert cells == 4000000 and accepted > cells // 2
    assert mismatches == 0


def grids(shape, bc):
    import paper_1602_05700_gb300 as hg
    from tests.test_gpu_parity import BC_PAIRS, robin_cfl
    nx, ny, nz = shape
    h = 1.0 / 64
    dt = (robin_cfl(nx, ny, nz, h) if bc == "robin" else 0.5) * h / np.sqrt(3.0)
    origin = (-0.5 * nx * h, -0.5 * ny * h, -0.5 * nz * h)
    return (hg.Grid(nx, ny, nz, h, origin, 1.0, 1.0, dt, "f64", bc),
            O.Grid(nx, ny, nz, h, origin, 1.0, 1.0, dt, BC_PAIRS[bc]))


@pytest.mark.gpu
@pytest.mark.parametrize("bc", ["dirichlet", "robin", "periodic"])
@pytest.mark.parametrize("shape", [(100, 80, 75), (101, 77, 78), (1, 700, 858), (2, 601, 500), (3, 401, 499)])
def test_pairs_equal_the_oracle(shape, bc):
    assert shape[0] * shape[1] * shape[2] >= 600000
    g, og = grids(shape, bc)
    rho = I.noise(shape[::-1], 301, 0.0, 2.0) * (1.0 if bc == "robin" else 0.0)
    # noise within a factor of two, a steep slope through zero, and quiet cells: every form of the Laplacian sum
    phi0 = I.noise(shape[::-1], 302, -1.0, -0.5)
    phi0[:, : shape[1] // 3] *= np.linspace(-1.0, 1.0, shape[2])[:, None, None]
    phi0[:, -(shape[1] // 4):] = 0.0
    prev0 = phi0 * (1.0 + 1e-3 * I.noise(shape[::-1], 303, -1.0, 1.0))
    g.set_density(torch.from_numpy(rho).cuda())
    g.set_phi(torch.from_numpy(phi0).cuda(), torch.from_numpy(prev0).cuda())
    p, q = O.initial_state(og, rho, phi0=phi0, phi_prev0=prev0)
    g.step(5)
    O.run(og, p, q, rho, 5)
    assert np.array_equal(g.phi(torch.float64, "cpu"), p[1:-1, 1:-1, 1:-1])
    g.free()
