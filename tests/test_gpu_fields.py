"""Movement between dense arrays and the padded state, and -grad phi, over every access width of those kernels: rows of
whole 16-byte words or not, dense buffers on 16-byte boundaries or not, both dtypes and precisions.

Exact expectations: unpacking rounds hi + lo once; FP64 grids move values unchanged; a compensated-float grid holds
a seeded double to 2^-35 of its size (a float and an 11-bit remainder).  -grad phi: FP64 grids evaluate the same three
operations as numpy; float grids differ by the rounding of the 16-bit codes' sums, a few 2^-24 of max|phi| / 2h."""
import numpy as np
import pytest

from paper_1602_05700_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1602_05700_gb300 as hg  # noqa: E402

SHAPES = [(1, 1, 1), (2, 3, 4), (7, 5, 3), (64, 6, 5), (131, 9, 4), (260, 4, 3)]
DT = {"f32": torch.float32, "f64": torch.float64}


def dense(values, dtype, aligned):
    """A contiguous device tensor of the values, on a 16-byte boundary or one element past it."""
    t = torch.empty(values.size + 1, dtype=dtype, device="cuda")
    v = t[:-1] if aligned else t[1:]
    v.copy_(torch.from_numpy(values).reshape(-1))
    return v.view(values.shape)


def grid(shape, prec, bc="periodic"):
    nx, ny, nz = shape
    return hg.Grid(nx, ny, nz, 1.0 / 64, (-0.5, -0.5, -0.5), 1.0, 1.0, 0.25 / 64, prec, bc)


@pytest.mark.parametrize("aligned", [True, False])
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("prec", ["f32k", "f64"])
def test_seed_unpack_accel(prec, shape, aligned):
    nx, ny, nz = shape
    v = I.noise(shape[::-1], 501, -1.0, 1.0)
    special = [0.0, -0.0, 1e-30, -2.0 ** -70, 1.5 * 2.0 ** -71, 2.0 ** 100, 1.0 + 2.0 ** -24, 1.0 - 2.0 ** -25, 5e-324]
    v.reshape(-1)[: len(special)] = special[: v.size]
    for dt in ("f64", "f32"):
        g = grid(shape, prec)
        src = dense(v, DT[dt], aligned)
        g.set_phi(src)
        want = src.double().cpu().numpy()
        full = g.phi_ghosted()
        inner = full[1:-1, 1:-1, 1:-1]
        if prec == "f64" or dt == "f32":
            assert np.array_equal(inner, want)
        else:
            assert (np.abs(inner - want) <= 2.0 ** -35 * np.abs(want) + 1e-45).all()
        for odt in ("f64", "f32"):
            out = dense(np.zeros(shape[::-1]), DT[odt], aligned)
            hg._lib.check(hg._lib.lib().hg_get_phi(g.handle, out.data_ptr(), 1 if odt == "f64" else 0, 1))
            assert np.array_equal(out.cpu().numpy(), inner.astype(np.float64 if odt == "f64" else np.float32))
        acc = [dense(np.zeros(shape[::-1]), DT["f64" if prec == "f64" else "f32"], aligned) for _ in range(3)]
        g.accel(out=acc)
        c = slice(1, -1)
        inv = 1.0 / (2.0 * g.h)
        ref = [-(full[c, c, 2:] - full[c, c, :-2]) * inv, -(full[c, 2:, c] - full[c, :-2, c]) * inv,
               -(full[2:, c, c] - full[:-2, c, c]) * inv]
        for a, r in zip(acc, ref):
            a = a.cpu().numpy().astype(np.float64)
            if prec == "f64":
                assert np.array_equal(a, r)
            else:
                assert (np.abs(a - r) <= 4 * 2.0 ** -24 * (np.abs(r) + np.abs(full).max() * inv * 2.0 ** -20)).all()
        g.free()


@pytest.mark.parametrize("aligned", [True, False])
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("bc", ["periodic", "dirichlet"])
@pytest.mark.parametrize("prec", ["f32k", "f64"])
def test_density_source_and_mass(prec, bc, shape, aligned):
    """One sub-step from zero leaves phi = -s, s = (c dt)^2 4 pi (rho - mean): read back through the unpack kernel."""
    v = I.noise(shape[::-1], 502, 0.1, 2.0)
    for dt in ("f64", "f32"):
        g = grid(shape, prec, bc)
        src = dense(v, DT[dt], aligned)
        g.set_density(src)
        rho = src.double().cpu().numpy()
        mass = g.stats()["mass"]
        assert abs(mass - rho.sum() * g.h ** 3) <= 1e-14 * mass
        if bc == "periodic":
            g.step(1)
            s = (g.c * g.dt) ** 2 * 4 * np.pi * (rho - rho.mean())
            tol = 2e-15 if prec == "f64" else 3e-7  # float grids round the mean, the difference and the scale once each
            top = (g.c * g.dt) ** 2 * 4 * np.pi * rho.max()
            assert np.abs(g.phi(torch.float64, "cpu") + s).max() <= tol * top
        g.free()
