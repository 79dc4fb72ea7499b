"""The flat sub-step (one thread per group of cells, all ghosts in one launch): float grids against the z-marching sweep,
which a pinned block depth selects (the same arithmetic on the same values: every cell and ghost agrees bit for bit),
FP64 grids against the oracle bit for bit, for rows shorter than a group, ragged rows, single rows and planes, and
every boundary condition."""
import numpy as np
import pytest

import oracle as O
from paper_1602_05700_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1602_05700_gb300 as hg  # noqa: E402
from tests.test_gpu_parity import BC_PAIRS, robin_cfl  # noqa: E402


SHAPES = [(1, 1, 1), (3, 2, 1), (4, 1, 9), (5, 7, 3), (33, 17, 10), (129, 9, 6), (64, 64, 20)]


def case(shape, bc, prec):
    nx, ny, nz = shape
    h = 1.0 / 64
    dt = (robin_cfl(nx, ny, nz, h) if bc == "robin" else 0.5) * h / np.sqrt(3.0)
    origin = (-0.5 * nx * h, -0.5 * ny * h, -0.5 * nz * h)
    phi0 = I.noise(shape[::-1], 302, -1.0, -0.5)
    prev0 = phi0 + 1e-3 * I.noise(shape[::-1], 303, -1.0, 1.0)
    g = hg.Grid(nx, ny, nz, h, origin, 1.0, 1.0, dt, prec, bc)
    og = O.Grid(nx, ny, nz, h, origin, 1.0, 1.0, dt, BC_PAIRS[bc])
    return g, og, I.noise(shape[::-1], 301, 0.0, 2.0), phi0, prev0


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("bc", ["dirichlet", "robin", "periodic"])
def test_float_flat_equals_marching_sweep(bc, shape):
    out = []
    for depth in (0, 5):
        g, _, rho, phi0, prev0 = case(shape, bc, "f32k")
        g.set_block_depth(depth)
        g.set_density(torch.from_numpy(rho).cuda())
        g.set_phi(torch.from_numpy(phi0).cuda(), torch.from_numpy(prev0).cuda())
        g.step(11)
        out.append((g.phi_ghosted(), g.stats()["change_rel"]))
        g.free()
    assert np.array_equal(out[0][0], out[1][0])
    assert out[0][1] == out[1][1]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("bc", ["dirichlet", "robin", "periodic"])
def test_fp64_flat_equals_the_oracle(bc, shape):
    """Bit for bit; without a density where it would bring in a sum (the periodic mean, the Dirichlet monopole)."""
    g, og, rho, phi0, prev0 = case(shape, bc, "f64")
    if bc != "robin":
        rho = np.zeros_like(rho)
    g.set_density(torch.from_numpy(rho).cuda())
    g.set_phi(torch.from_numpy(phi0).cuda(), torch.from_numpy(prev0).cuda())
    p, q = O.initial_state(og, rho, phi0=phi0, phi_prev0=prev0)
    g.step(11)
    O.run(og, p, q, rho, 11)
    assert np.array_equal(g.phi(torch.float64, "cpu"), p[1:-1, 1:-1, 1:-1])
    g.free()


@pytest.mark.parametrize("prec", ["f32k", "f64"])
def test_small_slab_leaves_its_interface_ghosts_alone(prec):
    """A slab's interface ghost planes are supplied by the caller: the ghost threads skip those faces."""
    n, h = 12, 1.0 / 16
    out = []
    for depth in (0, 4):
        g = hg.Grid(n, n, n, h, (-0.5 * n * h,) * 3, 1.0, 1.0, 0.25 * h, prec, "robin", z_interfaces=3)
        g.set_block_depth(depth)
        g.set_phi(torch.from_numpy(I.noise((n, n, n), 311, -1.0, -0.5)).cuda())
        g.step(3)
        out.append(g.phi_ghosted())
        g.free()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("shape", [(1, 1, 1), (5, 7, 3), (130, 9, 6)])
@pytest.mark.parametrize("bc", ["dirichlet", "robin", "periodic"])
@pytest.mark.parametrize("prec", ["f32k", "f64"])
def test_small_adjoint_sum_is_linear_and_exact_for_one_step(prec, bc, shape):
    """The reverse sub-step adds level m to the running sum on the way.  One reverse step sums the injection alone:
    dL/drho = -(c dt)^2 4 pi G (lambda - mean if periodic); doubling the injection doubles a longer run's gradient
    exactly (a power of two commutes with every rounding)."""
    nx, ny, nz = shape
    h = 1.0 / 64
    dt = (robin_cfl(nx, ny, nz, h) if bc == "robin" else 0.5) * h / np.sqrt(3.0)
    g = hg.Grid(nx, ny, nz, h, (-0.5 * nx * h, -0.5 * ny * h, -0.5 * nz * h), 1.0, 1.0, dt, prec, bc)
    lam = I.noise(shape[::-1], 321, -1.0, 1.0).astype(np.float32).astype(np.float64)
    one = g.adjoint(torch.from_numpy(lam).cuda(), 1).cpu().numpy()
    want = -(dt * dt) * 4 * np.pi * (lam - (lam.mean() if bc == "periodic" else 0.0))
    assert np.abs(one - want).max() <= 4e-16 * dt * dt * 4 * np.pi
    a, b = (g.adjoint(torch.from_numpy(f * lam).cuda(), 7).cpu().numpy() for f in (1.0, 2.0))
    assert np.array_equal(2.0 * a, b)
    g.free()


@pytest.mark.parametrize("nx", [128, 136, 184, 248, 256, 132, 250])
@pytest.mark.parametrize("bc", ["dirichlet", "robin"])
def test_fused_tiles_that_share_columns(bc, nx):
    """The depth-2 kernel's last tile where nx is a multiple of 8 but not of 128 (it shares columns with its neighbour) and
    the general one elsewhere: exact mode bit for bit single sweeps, default mode within its roundings of them."""
    shape = (nx, 19, 37)
    out = {}
    for mode in ("single", "exact", "default"):
        g, _, rho, phi0, prev0 = case(shape, bc, "f32k")
        if mode != "single":
            g.set_temporal_depth(2)
            g.set_temporal_exact(mode == "exact")
        g.set_density(torch.from_numpy(rho).cuda())
        g.set_phi(torch.from_numpy(phi0).cuda(), torch.from_numpy(prev0).cuda())
        g.step(8)
        out[mode] = g.phi_ghosted()
        g.free()
    assert np.array_equal(out["single"], out["exact"])
    assert np.abs(out["single"] - out["default"]).max() <= 1e-6 * np.abs(out["single"]).max()
