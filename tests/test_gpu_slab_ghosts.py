"""A slab's interface ghost planes belong to the caller: no sweep writes them, while the other z face follows its boundary
condition.  Planes of known values are put on the interface faces of both time levels and read back two sub-steps later,
for every sweep a slab can take (flat, FP64 pairs, TMA-staged)."""
import ctypes

import numpy as np
import pytest

from paper_1602_05700_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1602_05700_gb300 as hg  # noqa: E402
from paper_1602_05700_gb300 import _lib  # noqa: E402
from tests.test_gpu_parity import robin_cfl  # noqa: E402


def put(g, side, plane):
    ny, nx = plane.shape
    raw = (plane.tobytes() if g.precision == _lib.HG_PREC_F64
           else plane.astype(np.float32).tobytes() + bytes(2 * nx * ny))  # floats, then codes of zero
    assert len(raw) == _lib.lib().hg_plane_bytes(g.handle)
    _lib.check(_lib.lib().hg_put_ghost_plane(g.handle, side, ctypes.create_string_buffer(raw, len(raw)), 0))


@pytest.mark.parametrize("interfaces", [1, 2, 3])
@pytest.mark.parametrize("prec,shape,depth", [("f32k", (12, 13, 14), 0), ("f32k", (140, 17, 14), 4), ("f64", (13, 12, 14), 0),
                                              ("f64", (101, 77, 78), 0)])
@pytest.mark.parametrize("bc", ["robin", "dirichlet"])
def test_sweeps_leave_interface_ghosts_alone(bc, prec, shape, depth, interfaces):
    nx, ny, nz = shape
    h = 1.0 / 64
    dt = (robin_cfl(nx, ny, nz, h) if bc == "robin" else 0.5) * h / np.sqrt(3.0)
    g = hg.Grid(nx, ny, nz, h, (-0.5 * nx * h, -0.5 * ny * h, -0.5 * nz * h), 1.0, 1.0, dt, prec, bc,
                z_interfaces=interfaces)
    if depth:
        g.set_block_depth(depth)
    g.set_phi(torch.from_numpy(I.noise(shape[::-1], 431, -1.0, -0.5)).cuda())
    free = g.phi_ghosted()  # the ghosts of the faces that are no interface, before any sub-step
    planes = {}
    for level in range(4):
        for side in (0, 1):
            if interfaces >> side & 1:
                want = I.noise((ny, nx), 440 + 2 * level + side, -1.0, -0.5).astype(np.float32).astype(np.float64)
                if level >= 2:  # the level of two sub-steps ago was put here then and must still be here
                    got = g.phi_ghosted()[0 if side == 0 else -1][1:-1, 1:-1]
                    assert np.array_equal(got, planes[side, level - 2])
                put(g, side, want)
                planes[side, level] = want
        g.step(1)
    after = g.phi_ghosted()
    for side in (0, 1):
        if not interfaces >> side & 1:
            a, b = (v[0 if side == 0 else -1][1:-1, 1:-1] for v in (free, after))
            assert np.array_equal(a, b) == (bc == "dirichlet")
    g.free()
