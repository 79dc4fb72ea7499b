"""The fused depth-2 kernel where the last tile starts inside its neighbour (nx >= 128 a multiple of 8, not of 128): every column
has one tile that stores it.  In the default mode the two tiles round the columns next to a tile's edge by different forms
of the update, so with two writers a cell's float, its code and its increment could come from different blocks."""
import numpy as np
import pytest

from paper_1602_05700_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1602_05700_gb300 as hg  # noqa: E402
from tests.test_gpu_parity import robin_cfl  # noqa: E402

NY, NZ, H = 19, 37, 1.0 / 64


def grid(nx, bc, phi0, prev0, rho):
    dt = (robin_cfl(nx, NY, NZ, H) if bc == "robin" else 0.5) * H / np.sqrt(3.0)
    g = hg.Grid(nx, NY, NZ, H, (-0.5 * nx * H, -0.5 * NY * H, -0.5 * NZ * H), 1.0, 1.0, dt, "f32k", bc)
    g.set_temporal_depth(2)
    g.set_density(torch.from_numpy(rho).cuda())
    g.set_phi(torch.from_numpy(phi0).cuda(), torch.from_numpy(prev0).cuda())
    return g


def fields(nx):
    phi0 = I.noise((NZ, NY, nx), 421, -1.0, -0.5)
    return phi0, phi0 + 1e-3 * I.noise((NZ, NY, nx), 422, -1.0, 1.0), I.noise((NZ, NY, nx), 423, 0.0, 2.0)


@pytest.mark.parametrize("nx", [136, 184, 248, 392])
@pytest.mark.parametrize("bc", ["dirichlet", "robin"])
def test_runs_repeat_bit_for_bit(bc, nx):
    blobs = set()
    for _ in range(6):
        g = grid(nx, bc, *fields(nx))
        g.step(8)
        blobs.add(g.save_state())  # floats, codes, increments and ghosts
        g.free()
    assert len(blobs) == 1


@pytest.mark.parametrize("nx", [136, 184, 248])
def test_shared_columns_are_the_first_tiles(nx):
    """One fused pair: cells 0 .. 127 depend on cells 0 .. 129 alone, and the first tile of a longer row computes them alike."""
    wide = 264
    f = [v.copy() for v in fields(wide)]
    f[2][:] = 0.0
    out = []
    for n in (nx, wide):
        g = grid(n, "dirichlet", *(np.ascontiguousarray(v[:, :, :n]) for v in f))
        g.step(2)
        out.append(g.phi(torch.float64, "cpu")[:, :, :128])
        g.free()
    assert np.array_equal(out[0], out[1])
